"""Joins on a device with little memory left: a join that keeps its pairs in
scratch still finishes where the exact output has no room beside them, down to
what the same join needs with nothing kept (its scratch under an admission
hook, which keeps no pairs, and the output).  Allocations are made to fail on
the host (jn_selftest_memory); no device memory is exhausted."""
import numpy as np
import pytest
import torch

from paper_1904_11201_gb300 import build as B
from paper_1904_11201_gb300 import datagen
from paper_1904_11201_gb300 import jn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def keys(n, dom, stream):
    return datagen.uniform_keys(n, 0, dom, 301, stream).to(DEV)


def hash_call(algo, nr, ns, **knobs):
    R, S = jn.table(keys(nr, nr, 0)), jn.table(keys(ns, nr, 1))

    def run(c, nothing_kept):
        # the partitioned join is what a run that keeps nothing falls back to
        c.set_tuning(**(knobs or ({"hash_path": 2} if nothing_kept else {"hash_path": 0})))
        return algo(c, R, S)
    return run


def band_call(nr, ns):
    ra, rk, sa, sk = keys(nr, 1000, 2), keys(nr, 4 * nr, 3), keys(ns, 1000, 4), keys(ns, 4 * nr, 5)
    R, S = jn.table(ra, rk), jn.table(sa, sk)
    return lambda c, _: jn.jn_theta(c, R, S, jn.JN_GE, 2)


def nested_call(nr, ns):
    R, S = jn.table(keys(nr, 3000, 6)), jn.table(keys(ns, 3000, 7))
    return lambda c, _: jn.jn_nested_loop(c, R, S)


def star_call(n, d1, d2):
    R, S1, S2 = jn.table(keys(n, d1, 8), keys(n, d2, 9)), jn.table(keys(d1, d1, 10)), jn.table(keys(d2, d2, 11))
    return lambda c, _: jn.jn_star(c, R, S1, S2)


def batch_call(band):
    joins = []
    for i in range(4):
        n = 20000 + 4097 * i
        joins.append((jn.table(keys(n, n, 20 + 8 * i)), jn.table(keys(3 * n, n, 21 + 8 * i)), jn.JN_EQ, -1))
        if band:
            joins.append((jn.table(keys(n, 1000, 22 + 8 * i), keys(n, 4 * n, 23 + 8 * i)),
                          jn.table(keys(3 * n, 1000, 24 + 8 * i), keys(3 * n, 4 * n, 25 + 8 * i)), jn.JN_LT, 2))
    return lambda c, _: jn.jn_batch(c, joins)[0]


CALLS = {
    "hash direct": lambda: hash_call(jn.jn_hash, 20000, 300000),
    "hash partitioned": lambda: hash_call(jn.jn_hash, 400000, 400001, radix_bits=9, heavy=0),
    "sort-merge": lambda: hash_call(jn.jn_sort_merge, 300000, 400001, radix_bits=8, heavy=0),
    "band direct": lambda: band_call(5000, 300000),
    "nested loop": lambda: nested_call(3000, 20000),
    "star": lambda: star_call(200000, 5000, 7000),
    "batch": lambda: batch_call(False),
    "batch with bands": lambda: batch_call(True),
}


@pytest.mark.parametrize("name", list(CALLS))
def test_little_memory_left(name):
    B.build()
    c = jn.Context(0)
    run = CALLS[name]()

    def rows(p):
        p = p.cpu().numpy()
        return p[np.lexsort(p.T)]

    c.set_admission(lambda out_bytes, scratch_bytes: jn.JN_OK)
    exp = run(c, True)
    least, out = c.run_info()["scratch_peak"], exp.numel() * 4
    exp = rows(exp)
    c.set_admission(None)
    assert np.array_equal(rows(run(c, False)), exp)
    most = c.run_info()["scratch_peak"]
    step = max(most - least, out) // 8
    for i in range(10):
        jn.jn_selftest_memory(c, least + out + 4096 + i * step)
        assert np.array_equal(rows(run(c, False)), exp), i
    # and with less than any way needs, the call says so and the context goes on
    jn.jn_selftest_memory(c, out // 2)
    with pytest.raises(jn.JoinError) as e:
        run(c, False)
    assert e.value.status == jn.JN_ERR_OOM
    jn.jn_selftest_memory(c, 0)
    assert np.array_equal(rows(run(c, False)), exp)
    c.close()
