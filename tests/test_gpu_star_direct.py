"""The one-pass star join (both dimensions' hash tables in global memory)
against the CPU oracle: one row, more than one block, duplicate keys on every
side, more triples than the staging scratch holds, the empty-slot key 0, and
a fact table smaller than a dimension (left to the two joins).  All values
are integers: comparisons are exact."""
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


def column(n, domain, seed, stream, dt):
    k = datagen.uniform_keys(n, -(domain // 2), domain - domain // 2, seed, stream, dtype=dt)
    lim = torch.iinfo(dt)
    for i, v in enumerate((0, lim.min, lim.max)):  # the empty marker and the extremes
        if n > 8:
            k[n // 2 + i] = v
    return k


@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("n,n1,n2,domain", [(1, 1, 1, 1), (1025, 40, 900, 60), (6000, 3000, 2000, 700),
                                            (3000, 700, 1100, 60), (2000, 9000, 10, 50)])
def test_one_pass_star_join(ctx, dt, n, n1, n2, domain):
    f1, f2 = column(n, domain, 73, 0, dt), column(n, domain, 73, 1, dt)
    d1, d2 = column(n1, domain, 73, 2, dt), column(n2, domain, 73, 3, dt)
    pays = [datagen.uniform_int(k, -(2 ** 31), 2 ** 31 - 1, 73, 4 + i) for i, k in enumerate((n, n1, n2))]
    exp = O.star_join(f1.numpy(), f2.numpy(), d1.numpy(), d2.numpy(), *[p.numpy() for p in pays])
    R = jn.table(f1.to(DEV), f2.to(DEV), pays[0].to(DEV))
    S1, S2 = jn.table(d1.to(DEV), payload=pays[1].to(DEV)), jn.table(d2.to(DEV), payload=pays[2].to(DEV))
    got = jn.jn_star(ctx, R, S1, S2).cpu().numpy()

    def canon(t):
        return t[np.lexsort((t[:, 2], t[:, 1], t[:, 0]))]

    assert np.array_equal(canon(got), canon(np.asarray(exp, dtype=np.int32).reshape(-1, 3)))
    assert jn.jn_star_count(ctx, R, S1, S2) == got.shape[0]
