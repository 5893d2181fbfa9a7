"""Orders close to one by Hamming weight (thousands of pairs, few prefixes):
phase 2 goes through the pairs, first alone, then with the prefixes in its
hash set.  Against the oracle, at any number of warps a block, with hits in
each part and none.  Whole numbers: equal or wrong."""
import numpy as np
import pytest

import oracle
from paper_2202_13951_gb300 import workloads
from test_gpu_parity import assert_same, gpu_batched, gpu_plain, orbg  # noqa: F401
from test_gpu_zpairs import repeated_columns

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = {
    # name: (H, blocks' Eb/N0, cap, order)
    # pairs alone up to the cap: no prefix of a position
    "no_prefix": (lambda: workloads.rlc(255, 231, 78).H, 4.5, 30000, ((), (40000,), (1,))),
    "pairs_then_triples": (lambda: workloads.rlc(255, 231, 79).H, 4.5, 100000,
                           ((), (40000,), (1,))),
    # 931 prefixes, up to two positions each
    "two_positions": (lambda: workloads.rlc(127, 106, 77).H, 2.5, 1_000_000, ((), (9000,), (1,))),
    # 6,441 pairs of which the first 670 or so alone
    "pairs_run_on": (lambda: workloads.rlc(127, 106, 77).H, 2.5, 100_000, ((), (50,), (1,))),
    "two_words": (lambda: workloads.rlc(181, 143, 71).H, 4.0, 60_000, ((), (20000,), (1,))),
    "four_words": (lambda: workloads.rlc(200, 100, 72).H, 4.5, 60_000, ((), (5000,), (1,))),
    "few_parity_bits": (lambda: workloads.rlc(96, 89, 73).H, 3.0, 100_000, ((), (3000,), (1,))),
    # many prefixes of one target, blocks that never decode
    "repeated_columns": (lambda: repeated_columns(96, 70, 74), 2.0, 60_000, ((), (3000,), (1,))),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_scan(orbg, name):  # noqa: F811
    make, ebn0, cap, model = CASES[name]
    H = make()
    n = H.shape[1]
    rng = np.random.default_rng(len(name))
    B = 60
    sigma = 10 ** (-ebn0 / 20.0) * 0.7
    llr = (2.0 * (-1.0 + sigma * rng.standard_normal((B, n))) / sigma ** 2).astype(np.float32)
    # a code word with two and with three unreliable bits wrong, at all depths
    for b in range(20, B):
        llr[b] = -rng.permutation(np.linspace(0.5, 8.0, n))
        llr[b, rng.choice(n, 2 + b % 2, replace=False)] *= -1
    llr = llr.astype(np.float32)
    want = oracle.decode_batch_mline(H, llr, cap, model)[:3]
    c = orbg.Code(H, max_query_cap=cap, model=model)
    assert_same(gpu_plain(orbg, c, llr, cap), want)
    cs = orbg.CodeSet([c])
    for warps in (8, 1, 7, 16):
        orbg.orbg_codeset_set_tuning(cs.handle, orbg.OrbgTuning(8, 0, 1, 1, warps))
        assert_same(gpu_batched(orbg, cs, llr, cap), want)
