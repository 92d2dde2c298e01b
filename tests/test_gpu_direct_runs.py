"""Long runs of the direct equi join (many build rows of a key, written apart
from the probe): lengths at the edges of the list's parts, probe rows of a
frequent key side by side, results past the room kept for pairs, single joins
and batches, against the CPU oracle, and that many pairs without a frequent
key stay with the direct join."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LENGTHS = (1, 4, 5, 127, 128, 129, 1023, 1024, 1025, 2049, 5000)  # rows of keys 1, 2, ..


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = jn.Context(0)
    yield c
    c.close()


def tables(dt, each):
    """A build side with keys of the given lengths and one row of key 0, and a
    probe side with `each` neighbouring rows of every key and others."""
    r = torch.cat([torch.full((n,), k + 1, dtype=dt) for k, n in enumerate(LENGTHS)] + [torch.zeros(1, dtype=dt)])
    r = r[torch.randperm(r.numel(), generator=torch.Generator().manual_seed(7))]
    s = torch.arange(-2, len(LENGTHS) + 3, dtype=dt).repeat_interleave(each)
    return r, torch.cat([s, datagen.uniform_keys(r.numel(), 100, 1 << 30, 411, 0, dtype=dt)])


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("each", [1, 3, 40])
def test_run_lengths(ctx, dt, swap, each):
    r, s = tables(dt, each)
    if swap:
        r, s = s, r
    exp = O.sort_pairs(O.hash_join(r.numpy(), s.numpy()))
    R, S = jn.table(r.to(DEV)), jn.table(s.to(DEV))
    assert np.array_equal(O.sort_pairs(jn.jn_hash(ctx, R, S).cpu().numpy()), exp)
    assert ctx.run_info()["hash_path"] == 3
    # a batch keeps 2.25 pairs a row at most: each = 1 fits beside other joins' room, 40 does not
    a = datagen.uniform_keys(3000, 0, 1000, 412, 0, dtype=dt)
    e2 = O.sort_pairs(O.hash_join(a.numpy(), a.numpy()))
    A = jn.table(a.to(DEV))
    p, first, cnt = jn.jn_batch(ctx, [(A, A, jn.JN_EQ, -1), (R, S, jn.JN_EQ, -1), (A, A, jn.JN_EQ, -1)])
    p = p.cpu().numpy()
    for i, e in enumerate((e2, exp, e2)):
        assert np.array_equal(O.sort_pairs(p[first[i]:first[i] + cnt[i]]), e)


def test_neighbouring_rows_of_a_frequent_key_share_the_device(ctx):
    # 2^20 pairs of 256 neighbouring probe rows: one block wrote them in 0.7 ms
    n = 1 << 14
    r, s = torch.arange(n, dtype=torch.int64) * 3, torch.arange(n, dtype=torch.int64) * 3 + 1
    r[100:4196], s[:256] = 1, 1
    R, S = jn.table(r.to(DEV)), jn.table(s.to(DEV))
    got = jn.jn_hash(ctx, R, S)
    ctx.set_profiling(True)
    ctx.reset_stats()
    got = jn.jn_hash(ctx, R, S).cpu().numpy()
    ms = ctx.kernel_stats()
    ctx.set_profiling(False)
    assert ms["direct_probe"][1] < 0.3
    assert np.array_equal(O.sort_pairs(got), O.sort_pairs(O.hash_join(r.numpy(), s.numpy())))


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
def test_many_pairs_without_a_frequent_key_stay_direct(ctx, dt):
    # 40 rows a key: 40 pairs a probe row, which were found, dropped and found again partitioned
    r = datagen.uniform_keys(16000, 0, 400, 413, 0, dtype=dt)
    s = datagen.uniform_keys(64000, 0, 400, 413, 1, dtype=dt)
    got = jn.jn_hash(ctx, jn.table(r.to(DEV)), jn.table(s.to(DEV)))
    assert ctx.run_info()["hash_path"] == 3
    assert np.array_equal(O.sort_pairs(got.cpu().numpy()), O.sort_pairs(O.hash_join(r.numpy(), s.numpy())))
