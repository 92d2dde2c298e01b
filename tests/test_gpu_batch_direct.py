"""Equi-joins of a batch without partitioning, against the CPU oracle: either
side built, tile edges (4096 rows), empty tables, keys with many rows on the
build side, joins whose pairs pass their room next to joins that fit theirs,
the empty-slot key 0, graphs on and off.  All values are integers: exact."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# (rows of R, rows of S, key domain)
JOINS = [(1, 1, 1), (4096, 4097, 3000), (9000, 100, 200), (0, 50, 10), (70, 0, 10), (20000, 30000, 1 << 20),
         (3000, 2900, 5), (5000, 40001, 6000), (12289, 12288, 40)]


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("pay", [False, True])
def test_batch_of_direct_joins(dt, graphs, pay):
    B.build()
    ctx = jn.Context(0)
    ctx.set_tuning(graphs=graphs)
    joins, exp = [], []
    for i, (nr, ns, dom) in enumerate(JOINS):
        r, s = (datagen.uniform_keys(n, -(dom // 2), dom - dom // 2, 90 + i, k, dtype=dt)
                for k, n in enumerate((nr, ns)))
        rp = datagen.uniform_int(nr, -(2 ** 31), 2 ** 31 - 1, 90 + i, 2) if pay else None
        sp = datagen.uniform_int(ns, -(2 ** 31), 2 ** 31 - 1, 90 + i, 3) if pay else None
        exp.append(O.sort_pairs(O.hash_join(*[x.numpy() if x is not None else None for x in (r, s, rp, sp)])))
        joins.append((jn.table(r.to(DEV), payload=rp.to(DEV) if pay else None),
                      jn.table(s.to(DEV), payload=sp.to(DEV) if pay else None), jn.JN_EQ, -1))
    pairs, first, cnt = jn.jn_batch(ctx, joins)
    assert cnt == [e.shape[0] for e in exp] == jn.jn_batch_count(ctx, joins)
    got = pairs.cpu().numpy()
    for i, e in enumerate(exp):
        assert np.array_equal(O.sort_pairs(got[first[i]:first[i] + cnt[i]]), e), i
    ctx.close()
