"""One partition that holds every row of the largest probing table
(2^31 - 1 rows): the partitioned joins' kernels number a partition's S rows in
rounds, so the last round's numbers lie past 2^31.  The counts are known in
closed form."""
import pytest
import torch

from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
MOST = 2 ** 31 - 1


@pytest.fixture()
def tables():
    B.build()
    c = jn.Context(0)
    # no partition bits for so small an R, no set-aside of the frequent key
    c.set_tuning(heavy=0, prefilter=0, hash_path=1, part_rows=4096)
    r = torch.arange(1000, dtype=torch.int32)
    r[500] = 7
    R, S = jn.table(r.to(DEV)), jn.table(torch.full((MOST,), 7, dtype=torch.int32, device=DEV))
    yield c, R, S
    c.close()


@pytest.mark.parametrize("algo", [jn.JN_ALGO_HASH, jn.JN_ALGO_SORT])
def test_count_of_one_full_partition(tables, algo):
    c, R, S = tables
    assert jn.jn_count(c, algo, R, S) == 2 * MOST


def test_batch_count_of_one_full_partition(tables):
    c, R, S = tables
    assert jn.jn_batch_count(c, [(R, S, jn.JN_EQ, -1)]) == [2 * MOST]
