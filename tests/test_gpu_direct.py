"""The direct equi join (a hash table in global memory, no partitioning)
against the CPU oracle: tile edges, either side built, duplicate build keys
(runs), the empty-slot key 0 and the type's extremes, results larger than the
staging scratch, and the rule's far side.
All values are integers: comparisons are exact."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TILE = 256  # probe rows per block and round


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = jn.Context(0)
    yield c
    c.close()


def column(n, domain, seed, stream, dt):
    k = datagen.uniform_keys(n, -(domain // 2), domain - domain // 2, seed, stream, dtype=dt)
    lim = torch.iinfo(dt)
    for i, v in enumerate((0, lim.min, lim.max)):  # the empty marker and the extremes
        if n > 8:
            k[n // 2 + i] = v
    return k


# (rows of R, rows of S, key domain): one tile and its edges, S built (the
# smaller side), many rows per key (runs longer than a lane copies itself),
# keys shared by whole warps, more pairs than the staging scratch holds
CASES = [(1, 1, 1), (3, TILE - 1, 4), (300, TILE, 900), (300, TILE + 1, 20), (5 * TILE + 7, 129, 300),
         (70001, 70001, 1 << 20), (9000, 200003, 1000), (200003, 9000, 1000), (1000, 1001, 3), (40000, 64, 2)]


@pytest.mark.parametrize("nr,ns,domain", CASES)
@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("pay", [False, True])
def test_direct_join(ctx, nr, ns, domain, dt, pay):
    r, s = column(nr, domain, 71, 0, dt), column(ns, domain, 71, 1, dt)
    rp = datagen.uniform_int(nr, -(2 ** 31), 2 ** 31 - 1, 71, 2) if pay else None
    sp = datagen.uniform_int(ns, -(2 ** 31), 2 ** 31 - 1, 71, 3) if pay else None
    host = [x.numpy() if x is not None else None for x in (r, s, rp, sp)]
    R = jn.table(r.to(DEV), payload=rp.to(DEV) if pay else None)
    S = jn.table(s.to(DEV), payload=sp.to(DEV) if pay else None)
    exp = O.sort_pairs(O.hash_join(*host))
    got = jn.jn_hash(ctx, R, S)
    assert ctx.run_info()["hash_path"] == 3
    assert np.array_equal(O.sort_pairs(got.cpu().numpy()), exp)
    assert jn.jn_count(ctx, jn.JN_ALGO_HASH, R, S) == exp.shape[0]
    assert jn.jn_aggregate(ctx, jn.JN_ALGO_HASH, R, S) == (exp.shape[0], O.checksum_pairs(exp))


def test_direct_join_rule_and_outputs(ctx):
    # past the rule's size, and under any explicit partition knob, the
    # partitioned join runs; caller buffers (device off an 8-byte boundary,
    # host) and too small ones follow the output convention
    r, s = column(5000, 4000, 72, 0, torch.int32), column(9000, 4000, 72, 1, torch.int32)
    exp = O.sort_pairs(O.hash_join(r.numpy(), s.numpy()))
    m = exp.shape[0]
    R, S = jn.table(r.to(DEV)), jn.table(s.to(DEV))
    flat = torch.full((2 * m + 7,), -1, dtype=torch.int32, device=DEV)
    for out in (torch.full((m + 3, 2), -1, dtype=torch.int32, device=DEV), flat[1:2 * m + 7].view(-1, 2),
                torch.full((m + 3, 2), -1, dtype=torch.int32)):
        got = jn.jn_hash(ctx, R, S, out=out)
        assert ctx.run_info()["hash_path"] == 3
        assert np.array_equal(O.sort_pairs(got.cpu().numpy()), exp) and bool((out[m:] == -1).all())
    small = torch.zeros((m - 1, 2), dtype=torch.int32, device=DEV)
    with pytest.raises(jn.JoinError) as e:
        jn.jn_hash(ctx, R, S, out=small)
    assert e.value.status == jn.JN_ERR_CAPACITY and e.value.required == m and bool((small == 0).all())
    ctx.set_tuning(radix_bits=2)
    try:
        jn.jn_hash(ctx, R, S)
        assert ctx.run_info()["hash_path"] == 2
    finally:
        ctx.set_tuning(radix_bits=0)
    ctx.set_memory_limit(64 << 20)  # admitted by bytes: the scratch is held to the partitioned join's
    try:
        assert np.array_equal(O.sort_pairs(jn.jn_hash(ctx, R, S).cpu().numpy()), exp)
    finally:
        ctx.set_memory_limit(0)
