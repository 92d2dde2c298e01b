"""Large direct equi joins: several pairs a probe row, build sides with and
without repeated keys around the size where these are left to the partitioned
join, segmented results (2^23 probe rows and more) into new, device and host
outputs, the largest build side, star joins of as many rows, and that the
choice does not cost what it saves.  Keys are multiples of an odd number modulo
2^24, so the matching rows are known in closed form."""
import numpy as np
import pytest
import torch

from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
M = 1 << 20


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = jn.Context(0)
    yield c
    c.close()


def key(rank, dt):
    return ((rank * 0x9E3779B1) & ((1 << 24) - 1)).to(dt) - (1 << 23)


def ranks(n):
    return torch.arange(n, dtype=torch.int64, device=DEV)


def pair_words(p):
    return (p[:, 0].to(torch.int64) << 32 | p[:, 1].to(torch.int64)).sort()[0]


def check(got, d, ns, reps):
    """S row j has rank j % (2 d); R row i has rank i % d, `reps` times: the
    pairs of S row j (rank below d) are R rows rank, rank + d, .."""
    j = ranks(ns)
    rank = j % (2 * d)
    j, rank = j[rank < d], rank[rank < d]
    exp = torch.cat([(rank + k * d) << 32 | j for k in range(reps)]).sort()[0]
    assert torch.equal(pair_words(got.to(DEV)), exp)


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("d,reps,ns", [(1 << 22, 1, (1 << 23) + 5), ((1 << 21) + 3, 1, 3 * M + 1), (M + 7, 2, 4 * M + 1),
                                       (M + 7, 3, (1 << 23) + 9), (60001, 3, (1 << 23) + 3), (60001, 5, (1 << 23) + 3)])
def test_pairs(ctx, dt, d, reps, ns):
    nr = d * reps
    R, S = jn.table(key(ranks(nr) % d, dt)), jn.table(key(ranks(ns) % (2 * d), dt))
    check(jn.jn_hash(ctx, R, S), d, ns, reps)
    left = dt == torch.int32 and nr > 2 * M and reps > 1
    assert (ctx.run_info()["hash_path"] == 3) == (not left)
    total = reps * int(((ranks(ns) % (2 * d)) < d).sum())
    out = torch.empty((total + 1, 2), dtype=torch.int32, device=DEV)
    check(jn.jn_hash(ctx, R, S, out=out), d, ns, reps)
    host = torch.empty((total, 2), dtype=torch.int32, pin_memory=True)
    check(jn.jn_hash(ctx, R, S, out=host), d, ns, reps)
    with pytest.raises(jn.JoinError) as e:
        jn.jn_hash(ctx, R, S, out=out[: total - 1])
    assert e.value.status == jn.JN_ERR_CAPACITY and e.value.required == total


def test_past_the_largest_build_side(ctx):
    n = (1 << 22) + 1
    R, S = jn.table(key(ranks(n), torch.int32)), jn.table(key(ranks(n) % (2 * n), torch.int32))
    assert jn.jn_hash(ctx, R, S).shape[0] == n
    assert ctx.run_info()["hash_path"] != 3


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("reps", [1, 2])
def test_star_in_segments(ctx, dt, reps):
    # two rows a key of the first dimension: more triples than their room
    n, d1, d2 = (1 << 23) + 11, 50021, 70001
    i = ranks(n)
    r1, r2 = (i * 7919) % (d1 + 1000), (i * 104729) % (d2 + 1000)
    R = jn.table(key(r1, dt), key(r2, dt))
    S1, S2 = jn.table(key(ranks(d1 * reps) % d1, dt)), jn.table(key(ranks(d2), dt))
    both = (r1 < d1) & (r2 < d2)
    word = lambda r, s1, s2: ((r << 18 | s1) * (d2 + 1) + s2).sort()[0]
    exp = torch.cat([torch.stack([i[both], r1[both] + k * d1, r2[both]]) for k in range(reps)], 1)
    for out in (None, torch.empty((exp.shape[1], 3), dtype=torch.int32, device=DEV),
                torch.empty((exp.shape[1] + 2, 3), dtype=torch.int32, pin_memory=True)):
        t = jn.jn_star(ctx, R, S1, S2, out=out)
        torch.cuda.synchronize()
        t = t.to(DEV).to(torch.int64)
        assert t.shape[0] == exp.shape[1]
        assert torch.equal(word(t[:, 0], t[:, 1], t[:, 2]), word(*exp))
    assert ctx.run_info()["hash_path"] == 3


@pytest.mark.parametrize("nr,ns", [(2 * M, 32 * M), (4 * M, 16 * M)])
def test_two_rows_a_key_cost_no_more_than_partitioned(nr, ns):
    # found twice, they took 1.5 to 1.7 times as long
    B.build()
    c = jn.Context(0)
    r, s = (datagen.uniform_int(n, 0, nr // 2, 421, i, DEV, torch.int32) for i, n in enumerate((nr, ns)))
    R, S = jn.table(r), jn.table(s)
    ms = {}
    for path in (0, 2):
        c.set_tuning(hash_path=path)
        jn.jn_hash(c, R, S)
        c.set_profiling(True)
        best = 1e9
        for _ in range(5):
            c.reset_stats()
            jn.jn_hash(c, R, S)
            best = min(best, sum(v[1] for v in c.kernel_stats().values()))
        ms[path] = best
        c.set_profiling(False)
    c.close()
    assert ms[0] <= 1.15 * ms[2], ms
