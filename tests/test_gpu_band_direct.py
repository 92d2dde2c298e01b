"""The direct band join (a sorted index of the smaller table, no
partitioning) against the CPU oracle: either side built (the condition on a
mirrored), tile edges (4096 rows), windows at the type's extremes, one key
value for all rows, clustered keys that pass the probe's limit (left to the
partitioned join), single joins and batches mixed with both kinds.  All
values are integers: comparisons are exact."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = jn.Context(0)
    yield c
    c.close()


def columns(n, span, seed, stream, dt, extremes):
    a = datagen.uniform_keys(n, -50, 50, seed, 2 * stream, dtype=dt)
    k = datagen.uniform_keys(n, -(span // 2), span - span // 2, seed, 2 * stream + 1, dtype=dt)
    if extremes and n > 8:
        lim = torch.iinfo(dt)
        k[1], k[2], a[1], a[2] = lim.min, lim.max, lim.min, lim.max
    return a, k


# (rows of R, rows of S, span of k, band, op, extremes)
CASES = [(1, 1, 1, 0, "EQ", False), (4097, 4095, 100000, 3, "LT", False), (300, 9000, 2000, 6, "GE", True),
         (9000, 300, 2000, 6, "GT", True), (8192, 40000, 1 << 20, 100, "NE", False), (5000, 12289, 1 << 30, 0, "ANY", True),
         (64, 5000, 1, 0, "LE", False), (20000, 3000, 9000, 1, "LE", True)]


def pairs_of(case, dt, seed):
    nr, ns, span, band, op, ext = case
    (ra, rk), (sa, sk) = columns(nr, span, seed, 0, dt, ext), columns(ns, span, seed, 1, dt, ext)
    exp = O.sort_pairs(O.band_join_sorted(ra.numpy(), rk.numpy(), sa.numpy(), sk.numpy(), getattr(O, op), band))
    return jn.table(ra.to(DEV), rk.to(DEV)), jn.table(sa.to(DEV), sk.to(DEV)), getattr(jn, "JN_" + op), band, exp


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
def test_direct_band_join(ctx, case, dt):
    R, S, op, band, exp = pairs_of(case, dt, 95)
    got = jn.jn_theta(ctx, R, S, op, band)
    assert np.array_equal(O.sort_pairs(got.cpu().numpy()), exp)
    pr = jn.pred(op, jn.JN_ANY, band)
    assert jn.jn_count(ctx, jn.JN_ALGO_THETA, R, S, pr) == exp.shape[0]
    assert jn.jn_aggregate(ctx, jn.JN_ALGO_THETA, R, S, pr) == (exp.shape[0], O.checksum_pairs(exp))


@pytest.mark.parametrize("graphs", [0, 1])
def test_direct_band_batch(graphs):
    B.build()
    c = jn.Context(0)
    c.set_tuning(graphs=graphs)
    cases = [pairs_of(x, torch.int32, 96 + i) for i, x in enumerate(CASES + [(0, 10, 5, 1, "EQ", False)])]
    joins = [x[:4] for x in cases]
    pairs, first, cnt = jn.jn_batch(c, joins)
    assert cnt == [x[4].shape[0] for x in cases] == jn.jn_batch_count(c, joins)
    got = pairs.cpu().numpy()
    for i, x in enumerate(cases):
        assert np.array_equal(O.sort_pairs(got[first[i]:first[i] + cnt[i]]), x[4]), i
    c.close()


def test_clustered_keys_stop_and_are_partitioned(ctx):
    # every other sampled row of the built table lies alone, the rows between
    # them on one value: the sample sees few candidates, the probe meets many
    n = 1 << 17
    k = torch.arange(n, dtype=torch.int32) * 1000
    k[torch.arange(n) % 32 != 0] = 7
    a = datagen.uniform_keys(n, 0, 100, 97, 0)
    sa, sk = datagen.uniform_keys(n, 0, 2, 97, 1), torch.full((n,), 7, dtype=torch.int32)
    sk[torch.arange(n) % 128 == 0] = 500
    R, S = jn.table(a.to(DEV), k.to(DEV)), jn.table(sa.to(DEV), sk.to(DEV))
    exp = O.band_join_sorted(a.numpy(), k.numpy(), sa.numpy(), sk.numpy(), O.LT, 2, count_only=True)
    assert jn.jn_count(ctx, jn.JN_ALGO_THETA, R, S, jn.pred(jn.JN_LT, jn.JN_ANY, 2)) == exp
