"""A large result on its way to page-locked host memory, copied slice by slice
while later slices are written, when a later slice's launch fails (on the
host, jn_selftest_launches): once the call has returned its error nothing
writes the caller's buffer any more, and the context goes on."""
import pytest
import torch

from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_failed_slice_leaves_no_copy_behind():
    B.build()
    n = 1 << 25
    c = jn.Context(0)
    c.set_tuning(heavy=0, radix_bits=14)
    key = datagen.row_ids(n, DEV)
    R, S = jn.table(key), jn.table(key)
    out = torch.empty((n, 2), dtype=torch.int32, pin_memory=True)
    assert jn.jn_hash(c, R, S, out=out).shape[0] == n
    launches = c.run_info()["kernel_launches"]
    out.zero_()
    jn.jn_selftest_launches(c, launches)  # the last slice's
    with pytest.raises(jn.JoinError) as e:
        jn.jn_hash(c, R, S, out=out)
    # a few rows of each finished slice, read at once
    at_return = [out[q * n // 8: q * n // 8 + 64].clone() for q in (5, 4, 3, 2, 1, 0)]
    assert e.value.status == jn.JN_ERR_CUDA
    torch.cuda.synchronize()
    for q, rows in zip((5, 4, 3, 2, 1, 0), at_return):
        assert torch.equal(out[q * n // 8: q * n // 8 + 64], rows), q
    got = jn.jn_hash(c, R, S, out=out)
    assert torch.equal(got[:, 0], got[:, 1]) and torch.equal(got[:, 0].sort()[0], key.cpu())
    c.close()
