"""What holds when jn_star returns, whichever way the star join ran: its
triples are complete (a caller may read them on another stream), and the run's
information covers the scratch it held."""
import pytest
import torch

from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def tables(n, d):
    i = torch.arange(n, dtype=torch.int32, device=DEV)
    k = torch.arange(d, dtype=torch.int32, device=DEV)
    return jn.table(i % d, (i * 5) % d), jn.table(k), jn.table(k)


@pytest.mark.parametrize("caller_buffer", [False, True])
@pytest.mark.parametrize("path", [0, 2])
def test_triples_are_complete_on_return(caller_buffer, path):
    B.build()
    n, d = 1 << 26, 1 << 16
    args = tables(n, d)
    out = torch.empty((n, 3), dtype=torch.int32, device=DEV) if caller_buffer else None
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    c = jn.Context(0, stream)
    c.set_tuning(hash_path=path)
    jn.jn_star(c, *args, out=out)
    t = jn.jn_star(c, *args, out=out)
    assert stream.query()
    assert t.shape[0] == n and int(t[:, 0].to(torch.int64).sum()) == n * (n - 1) // 2
    c.close()


def test_run_info_covers_the_scratch_held():
    B.build()
    c = jn.Context(0)
    args = tables(100000, 5000)
    jn.jn_star(c, *args)
    info = c.run_info()
    # two hash tables of 8-byte slots and the kept triples at least
    assert info["hash_path"] == 3 and info["scratch_peak"] >= 2 * 5000 * 8 + 100000 * 12
    assert jn.jn_star_count(c, *args) == info["result"]
    assert 2 * 5000 * 8 <= c.run_info()["scratch_peak"] < info["scratch_peak"]
    c.close()
