"""Partitioned int32 joins with the full table asked for (what the autotuner
picks for large uniform tables), whose items are counted and then written:
partitions of several chunks, repeated keys, the keys at the type's ends, both
paths and key types, the admission hook and outputs, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture()
def ctx():
    B.build()
    c = jn.Context(0)
    yield c
    c.close()


def columns(n, dom, stream, dt):
    k = datagen.uniform_keys(n, -(dom // 2), dom - dom // 2, 451, stream, dtype=dt)
    lim = torch.iinfo(dt)
    k[n // 2], k[n // 3], k[n // 4] = lim.min, lim.max, lim.min
    return k


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("path,bits", [(1, 1), (1, 7), (2, 2), (2, 6)])
@pytest.mark.parametrize("nr,ns,dom", [(40000, 50000, 30000), (9, 7, 5), (60001, 3000, 1 << 20)])
def test_items_counted_then_written(ctx, dt, path, bits, nr, ns, dom):
    r, s = columns(nr, dom, 0, dt), columns(ns, dom, 1, dt)
    exp = O.sort_pairs(O.hash_join(r.numpy(), s.numpy()))
    R, S = jn.table(r.to(DEV)), jn.table(s.to(DEV))
    ctx.set_tuning(hash_path=path, radix_bits=bits, table_rows=4096, heavy=0)
    host = torch.empty((exp.shape[0] + 1, 2), dtype=torch.int32)
    for out in (None, torch.empty((exp.shape[0], 2), dtype=torch.int32, device=DEV), host):
        got = jn.jn_hash(ctx, R, S, out=out)
        assert np.array_equal(O.sort_pairs(got.cpu().numpy()), exp)
    assert ctx.run_info()["hash_path"] in (1, 2)
    asked = []
    ctx.set_admission(lambda o, s: asked.append(o) or jn.JN_OK)
    assert np.array_equal(O.sort_pairs(jn.jn_hash(ctx, R, S).cpu().numpy()), exp)
    assert asked == [8 * exp.shape[0]]
    ctx.set_admission(None)
    if dt == torch.int32 and exp.shape[0]:
        ctx.set_profiling(True)
        ctx.reset_stats()
        jn.jn_hash(ctx, R, S)
        st = ctx.kernel_stats()
        assert st["hash_count"][0] == 1 and st["hash_emit"][0] == 1
