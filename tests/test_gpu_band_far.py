"""Band joins with a few keys far from the others, which put all other rows
into a few buckets of the direct join's index: against the CPU oracle, single
and in a batch, counted and written, and how long the direct join's kernels
take before such a join is left to the partitioned one."""
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


def columns(n, far, seed, stream, dt):
    a = datagen.uniform_keys(n, 0, 100, seed, 2 * stream, dtype=dt)
    k = datagen.uniform_keys(n, 0, 1 << 20, seed, 2 * stream + 1, dtype=dt)
    if far is not None:
        k[n // 3], k[n // 2] = far, -far
    return a, k


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("far", [30 << 20, 2 ** 31 - 1])
@pytest.mark.parametrize("nr,ns", [(1 << 14, 1 << 14), (40001, 1 << 16), (1 << 16, 9001)])
def test_far_keys_match_the_oracle(ctx, dt, far, nr, ns):
    (ra, rk), (sa, sk) = columns(nr, far, 401, 0, dt), columns(ns, far - 1, 401, 1, dt)
    exp = O.sort_pairs(O.band_join_sorted(ra.numpy(), rk.numpy(), sa.numpy(), sk.numpy(), O.LE, 1))
    R, S = jn.table(ra.to(DEV), rk.to(DEV)), jn.table(sa.to(DEV), sk.to(DEV))
    assert np.array_equal(O.sort_pairs(jn.jn_theta(ctx, R, S, jn.JN_LE, 1).cpu().numpy()), exp)
    pr = jn.pred(jn.JN_LE, jn.JN_ANY, 1)
    assert jn.jn_count(ctx, jn.JN_ALGO_THETA, R, S, pr) == exp.shape[0]
    assert jn.jn_aggregate(ctx, jn.JN_ALGO_THETA, R, S, pr) == (exp.shape[0], O.checksum_pairs(exp))
    # in a batch, between two joins that stay direct
    (qa, qk), (ta, tk) = columns(3000, None, 402, 0, dt), columns(5000, None, 402, 1, dt)
    Q, T = jn.table(qa.to(DEV), qk.to(DEV)), jn.table(ta.to(DEV), tk.to(DEV))
    near = O.sort_pairs(O.band_join_sorted(qa.numpy(), qk.numpy(), ta.numpy(), tk.numpy(), O.LE, 1))
    p, first, cnt = jn.jn_batch(ctx, [(Q, T, jn.JN_LE, 1), (R, S, jn.JN_LE, 1), (Q, T, jn.JN_LE, 1)])
    p = p.cpu().numpy()
    for i, e in enumerate((near, exp, near)):
        assert np.array_equal(O.sort_pairs(p[first[i]:first[i] + cnt[i]]), e)


def test_far_keys_are_noticed_before_the_probe(ctx):
    # 2^16 rows in the buckets of every window: the probe alone took 0.6 ms
    n = 1 << 16
    (ra, rk), (sa, sk) = columns(n, 2 ** 31 - 1, 403, 0, torch.int32), columns(n, None, 403, 1, torch.int32)
    R, S = jn.table(ra.to(DEV), rk.to(DEV)), jn.table(sa.to(DEV), sk.to(DEV))
    pr = jn.pred(jn.JN_LE, jn.JN_ANY, 0)
    jn.jn_count(ctx, jn.JN_ALGO_THETA, R, S, pr)
    ctx.set_profiling(True)
    ctx.reset_stats()
    jn.jn_count(ctx, jn.JN_ALGO_THETA, R, S, pr)
    ms = ctx.kernel_stats()
    ctx.set_profiling(False)
    assert ms["band_probe"][1] < 0.1 and ms["theta_count"][0] == 1
