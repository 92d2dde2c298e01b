"""Which equi-joins of a batch run without partitioning: batches of joins with
and without repeated build keys, alike and mixed with small and empty joins,
more of them than are looked at, graphs on and off; their pairs and counts
against closed forms, and that the choice does not cost what it saves."""
import pytest
import torch

from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def join(d, reps, ns, dt):
    """R row i has key i % d, S row j key j % (2 d): pairs (R row, S row)."""
    i, j = torch.arange(d * reps, device=DEV), torch.arange(ns, device=DEV)
    return (jn.table((i % max(d, 1)).to(dt)), jn.table((j % max(2 * d, 1)).to(dt)), jn.JN_EQ, -1)


def expected(d, reps, ns):
    j = torch.arange(ns, device=DEV)
    rank = j % max(2 * d, 1)
    j, rank = j[rank < d], rank[rank < d]
    return torch.cat([(rank + k * d) << 32 | j for k in range(reps)]).sort()[0] if reps else j


def words(p):
    return (p[:, 0].to(torch.int64) << 32 | p[:, 1].to(torch.int64)).sort()[0]


SMALL = [(0, 0, 50), (1, 1, 1), (700, 3, 900), (8192, 1, 8192)]
BATCHES = [[(50000, 1, 200001)] * 3 + SMALL, [(30000, 2, 100003)] * 20 + SMALL, [(1000, 100, 3000)] * 3,
           [(40000, 1, 300007), (20000, 3, 60001)] * 18 + SMALL, [(8193, 1, 8193)] * 40]


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("which", range(len(BATCHES)))
def test_pairs_of_either_choice(dt, graphs, which):
    B.build()
    c = jn.Context(0)
    c.set_tuning(graphs=graphs)
    joins = [join(*x, dt) for x in BATCHES[which]]
    pairs, first, cnt = jn.jn_batch(c, joins)
    # the joins' pairs follow one another in the batch's order
    assert first == [sum(cnt[:i]) for i in range(len(cnt))]
    for i, x in enumerate(BATCHES[which]):
        e = expected(*x) if x[0] else torch.empty(0, dtype=torch.int64, device=DEV)
        assert torch.equal(words(pairs[first[i]:first[i] + cnt[i]]), e), i
    assert jn.jn_batch_count(c, joins) == cnt
    c.close()


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("repeats", [False, True])
@pytest.mark.parametrize("n,f,k", [(1 << 14, 4, 128), (1 << 16, 1, 96), (1 << 18, 4, 12)])
def test_choice_costs_no_more_than_partitioned(dt, repeats, n, f, k):
    # left to themselves, batches with repeated int32 keys took twice as long
    B.build()
    c = jn.Context(0)
    joins = []
    for i in range(k):
        r = datagen.uniform_int(n, 0, n, 431, 2 * i, DEV, dt) if repeats else torch.arange(n, device=DEV).to(dt) * 7
        joins.append((jn.table(r), jn.table(datagen.uniform_int(n * f, 0, n * (1 if repeats else 7), 431, 2 * i + 1, DEV, dt)),
                      jn.JN_EQ, -1))
    ms = {}
    for rows in (0, 2048 if dt == torch.int32 else 1024):
        c.set_tuning(part_rows=rows)
        jn.jn_batch(c, joins)
        c.set_profiling(True)
        best = 1e9
        for _ in range(5):
            c.reset_stats()
            jn.jn_batch(c, joins)
            best = min(best, sum(v[1] for v in c.kernel_stats().values()))
        ms[rows] = best
        c.set_profiling(False)
    c.close()
    assert ms[0] <= 1.2 * max(v for rows, v in ms.items() if rows), ms
