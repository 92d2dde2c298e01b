"""The partitioned hash join's shared-memory kernel against the CPU oracle:
partitions of many chunks and of almost no rows, keys with no, a few and many
further rows (runs, and runs a warp copies together), results past the scratch
kept for them, both partition paths, both table sizes, both key types.  All
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


# (rows of R, rows of S, key domain, partition bits; 0 = automatic)
CASES = [(1, 1, 1, 0), (4097, 2049, 1 << 20, 1), (40000, 30000, 1 << 17, 2), (40000, 30000, 30000, 5),
         (9000, 200003, 300, 3), (2500, 2600, 9, 0), (70001, 5000, 70001, 10), (8192, 512, 2, 1)]


@pytest.mark.parametrize("nr,ns,domain,bits", CASES)
@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("path,rows", [(2, 0), (2, 1024), (1, 0)])
def test_partition_join(ctx, nr, ns, domain, bits, dt, path, rows):
    r = datagen.uniform_keys(nr, -(domain // 2), domain - domain // 2, 91, 0, dtype=dt)
    s = datagen.uniform_keys(ns, -(domain // 2), domain - domain // 2, 91, 1, dtype=dt)
    lim = torch.iinfo(dt)
    if nr > 8 and ns > 8:
        r[3], s[5], r[7], s[2] = lim.min, lim.min, lim.max, lim.max
    rp = datagen.uniform_int(nr, -(2 ** 31), 2 ** 31 - 1, 91, 2)
    sp = datagen.uniform_int(ns, -(2 ** 31), 2 ** 31 - 1, 91, 3)
    exp = O.sort_pairs(O.hash_join(r.numpy(), s.numpy(), rp.numpy(), sp.numpy()))
    R, S = jn.table(r.to(DEV), payload=rp.to(DEV)), jn.table(s.to(DEV), payload=sp.to(DEV))
    ctx.set_tuning(hash_path=path, radix_bits=bits, table_rows=rows)
    try:
        got = jn.jn_hash(ctx, R, S)
        assert ctx.run_info()["hash_path"] == path
        assert np.array_equal(O.sort_pairs(got.cpu().numpy()), exp)
        assert jn.jn_count(ctx, jn.JN_ALGO_HASH, R, S) == exp.shape[0]
        assert jn.jn_aggregate(ctx, jn.JN_ALGO_HASH, R, S) == (exp.shape[0], O.checksum_pairs(exp))
        ctx.set_memory_limit(1 << 30)  # counted first, then written
        assert np.array_equal(O.sort_pairs(jn.jn_hash(ctx, R, S).cpu().numpy()), exp)
    finally:
        ctx.set_memory_limit(0)
        ctx.set_tuning(hash_path=0, radix_bits=0, table_rows=0)


# Eight segments of pairs in both passes: results past the scratch kept for
# them and under a memory limit (counted, then written at the segments'
# places), and, from 2^23 rows on, written in slices that are copied to a host
# buffer as they are finished, frequent keys' pairs behind them.
@pytest.mark.parametrize("algo", [jn.jn_hash, jn.jn_sort_merge])
@pytest.mark.parametrize("n,domain,host", [(300000, 60000, False), (300000, 60000, True), ((1 << 23) + 5, 1 << 24, True),
                                           ((1 << 23) + 5, 1 << 22, False)])
def test_segments(ctx, algo, n, domain, host):
    r = datagen.uniform_keys(n, 0, domain, 97, 0)
    s = datagen.uniform_keys(n, 0, domain, 97, 1)
    if n > 1 << 20:
        r[100:30100], s[7:207] = 12345, 12345
    exp = O.hash_join(r.numpy(), s.numpy(), np.arange(n, dtype=np.int32), np.arange(n, dtype=np.int32))
    R, S = jn.table(r.to(DEV)), jn.table(s.to(DEV))
    out = torch.empty((exp.shape[0] + 3, 2), dtype=torch.int32, pin_memory=True) if host else None
    ctx.set_tuning(radix_bits=10 if n < 1 << 20 else 13)
    try:
        for limit in (0, 8 << 30):
            ctx.set_memory_limit(limit)
            got = algo(ctx, R, S, out=out)
            got = got[: exp.shape[0]].cpu().numpy()
            word = lambda p: np.sort(np.ascontiguousarray(p).view(np.int64).ravel())
            assert np.array_equal(word(got), word(exp))
            if out is not None:
                out.zero_()
    finally:
        ctx.set_memory_limit(0)
        ctx.set_tuning(radix_bits=0)
