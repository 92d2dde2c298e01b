"""The screened one-pass nested loop against the CPU oracle: tile edges (4096
S rows, groups of 4 R rows), equality and band screens at the type's extremes,
bands too wide to screen, inputs whose rounds nearly all pass (the exact
rounds take over), and more pairs than its scratch holds (a second pass).
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


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = jn.Context(0)
    yield c
    c.close()


def columns(n, domain, seed, stream, dt):
    out = []
    for i in range(2):
        k = datagen.uniform_keys(n, -(domain // 2), domain - domain // 2, seed, 2 * stream + i, dtype=dt)
        lim = torch.iinfo(dt)
        if domain > 1 << 20 and n > 8:  # a wide domain reaches the extremes
            k[n // 3], k[n // 2] = lim.min, lim.max
        out.append(k)
    return out


# (rows of R, rows of S, domain, op on a, op on b, band)
CASES = [(1, 1, 1, "EQ", "ANY", -1), (5, 4097, 50, "EQ", "ANY", -1), (67, 4095, 4000, "LT", "EQ", -1),
         (1027, 8193, 1 << 24, "LT", "ANY", 200), (1027, 8193, 1 << 30, "GE", "ANY", 40000),
         (130, 5000, 1 << 24, "NE", "ANY", 0), (515, 4096, 1 << 16, "LE", "ANY", 9000),
         (300, 9000, 7, "EQ", "NE", -1), (900, 1200, 100, "GE", "LE", -1), (2000, 3000, 2, "ANY", "ANY", -1)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("dt", [torch.int32, torch.int64])
@pytest.mark.parametrize("second", [True, False])
def test_screened_nested_loop(ctx, case, dt, second):
    nr, ns, domain, oa, ok, band = case
    (ra, rb), (sa, sb) = columns(nr, domain, 81, 0, dt), columns(ns, domain, 81, 1, dt)
    op_a, op_k = getattr(O, oa), getattr(O, ok)
    if second:
        exp = O.nested_loop(ra.numpy(), sa.numpy(), rb.numpy(), sb.numpy(), op_a=op_a, op_k=op_k, band=band)
        R, S = jn.table(ra.to(DEV), rb.to(DEV)), jn.table(sa.to(DEV), sb.to(DEV))
    else:
        exp = O.nested_loop(ra.numpy(), sa.numpy(), op_a=op_a)
        R, S = jn.table(ra.to(DEV)), jn.table(sa.to(DEV))
    exp = O.sort_pairs(exp)
    pr = jn.pred(getattr(jn, "JN_" + oa), getattr(jn, "JN_" + ok), band)
    got = jn.jn_nested_loop(ctx, R, S, pr)
    assert np.array_equal(O.sort_pairs(got.cpu().numpy()), exp)
    assert jn.jn_count(ctx, jn.JN_ALGO_NLJ, R, S, pr) == exp.shape[0]
    assert jn.jn_aggregate(ctx, jn.JN_ALGO_NLJ, R, S, pr) == (exp.shape[0], O.checksum_pairs(exp))
