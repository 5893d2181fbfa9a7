"""The stages of a search (orbg_tables.cpp) against every pattern of the order,
built for the host: no stage may end before a pattern it has not covered."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2202_13951_gb300", "csrc")


@pytest.fixture(scope="module")
def tables(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("tables") / "libtables_host.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                           "-I", "/usr/local/cuda/include",
                           os.path.join(HERE, "tables_host.cpp"),
                           os.path.join(CSRC, "orbg_tables.cpp"), "-o", out])
    return ctypes.CDLL(out)


def orders(kind, rng):
    """(n, cap, segment ends, J, beta) of one random order."""
    if kind == "by_weight":  # large intercepts: many pairs, few prefixes
        n = int(rng.integers(40, 256))
        return n, int(rng.integers(2000, 300_000)), [n], [int(rng.integers(50, 50_000))], \
            [int(rng.integers(1, 4))]
    n = int(rng.integers(2, 256))
    m = int(rng.integers(1, min(n, 5) + 1))
    ends = sorted(rng.choice(np.arange(1, n), m - 1, replace=False).tolist()) + [n]
    beta = rng.integers(1, 8, m)
    J = rng.integers(0, 80, m) - beta
    return n, int(rng.integers(1, 300_000)), ends, J.tolist(), beta.tolist()


@pytest.mark.parametrize("kind,seed", [("by_weight", 1), ("by_weight", 2), ("model", 3),
                                       ("model", 4), ("model", 5)])
def test_stages_cover_the_order(tables, kind, seed):
    rng = np.random.default_rng(seed)
    seen = 0
    for _ in range(60):
        n, cap, ends, J, beta = orders(kind, rng)
        m = len(J)
        what = ctypes.c_int()
        rc = tables.tables_check(n, ctypes.c_uint64(cap), m, (ctypes.c_int * (m + 1))(0, *ends),
                                 (ctypes.c_int64 * m)(*J), (ctypes.c_int64 * m)(*beta),
                                 int(rng.choice([8, 10, 13, 20])), ctypes.byref(what))
        assert rc <= 0, "check %d failed: n %d cap %d ends %s J %s beta %s" % (rc, n, cap, ends,
                                                                              J, beta)
        seen |= what.value if rc == 0 else 0
    assert seen & (1 if kind == "by_weight" else 6) == (1 if kind == "by_weight" else 6)
