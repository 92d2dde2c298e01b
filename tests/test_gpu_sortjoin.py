"""The sort-merge join's kernels against the CPU oracle: chunks at the edges of
the sorting network's blocks, words of 32 and 64 bits, single keys that fill
chunks, chunks of distinct keys of one partition, results past the scratch
kept for them, both table sizes, both key types.  All values are integers:
comparisons are exact."""
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


def check(ctx, r, s, bits, rows):
    rp = datagen.uniform_int(len(r), -(2 ** 31), 2 ** 31 - 1, 95, 2)
    sp = datagen.uniform_int(len(s), -(2 ** 31), 2 ** 31 - 1, 95, 3)
    exp = O.sort_pairs(O.hash_join(r.numpy(), s.numpy(), rp.numpy(), sp.numpy()))
    R, S = jn.table(r.to(DEV), payload=rp.to(DEV)), jn.table(s.to(DEV), payload=sp.to(DEV))
    ctx.set_tuning(radix_bits=bits, table_rows=rows)
    try:
        assert np.array_equal(O.sort_pairs(jn.jn_sort_merge(ctx, R, S).cpu().numpy()), exp)
        assert jn.jn_count(ctx, jn.JN_ALGO_SORT, R, S) == exp.shape[0]
        assert jn.jn_aggregate(ctx, jn.JN_ALGO_SORT, R, S) == (exp.shape[0], O.checksum_pairs(exp))
        ctx.set_memory_limit(1 << 30)  # counted first, then written
        assert np.array_equal(O.sort_pairs(jn.jn_sort_merge(ctx, R, S).cpu().numpy()), exp)
    finally:
        ctx.set_memory_limit(0)
        ctx.set_tuning(radix_bits=0, table_rows=0)


@pytest.mark.parametrize("nr,ns,domain,bits", [(1, 1, 1, 0), (257, 255, 300, 1), (4097, 2049, 1 << 20, 1),
                                               (40000, 30000, 30000, 5), (9000, 100003, 900, 12),
                                               (70001, 5000, 40, 12), (70001, 5000, 70001, 11), (2500, 2600, 9, 0)])
@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("rows", [0, 1024])
def test_sort_join(ctx, nr, ns, domain, bits, dt, rows):
    r = datagen.uniform_keys(nr, -(domain // 2), domain - domain // 2, 95, 0, dtype=dt)
    s = datagen.uniform_keys(ns, -(domain // 2), domain - domain // 2, 95, 1, dtype=dt)
    lim = torch.iinfo(dt)
    if nr > 8 and ns > 8:
        r[3], s[5], r[7], s[2] = lim.min, lim.min, lim.max, lim.max
    check(ctx, r, s, bits, rows)


# Distinct keys that share the top 12 bits of the key hash (a product with
# 0x9E3779B1): every low bit pattern occurs, up to all ones.
@pytest.mark.parametrize("n", [255, 256, 257, 511, 513, 1025, 2047, 4095, 4096, 4097, 8192])
@pytest.mark.parametrize("bits", [0, 12])
def test_one_partition(ctx, n, bits):
    inv = pow(0x9E3779B1, -1, 1 << 32)
    x = (1 << 20) - 1 - np.arange(2 * n, dtype=np.int64) * ((1 << 20) // (2 * n))
    k = torch.from_numpy(((x.astype(np.uint64) * np.uint64(inv)) & np.uint64(0xFFFFFFFF)).astype(np.uint32).view(np.int32))
    check(ctx, k[0:n].flip(0).contiguous(), k[torch.arange(0, 2 * n, 3)], bits, 0)
