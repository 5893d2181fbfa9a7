"""The fitted decoder's pair look-ups at their edges, against the oracle:
chunked pair sets, weights past the counted range and orders with fewer
patterns than the cap (both left to the tree search), wide syndromes, and
position 256 of n = 256.  Whole numbers: equal or wrong."""
import numpy as np
import pytest

import oracle
from paper_2202_13951_gb300 import workloads
from test_gpu_parity import assert_same, orbg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def noise(n, B, sigma, seed):
    rng = np.random.default_rng(seed)
    return (2.0 * (-1.0 + sigma * rng.standard_normal((B, n))) / sigma ** 2).astype(np.float32)


def nearly_flat(n, B, sigma, seed):
    """Reliabilities of a narrow range, errors anywhere: large intercepts, an
    order by Hamming weight first."""
    rng = np.random.default_rng(seed)
    mag = 1.0 + rng.permuted(np.tile(np.arange(1, n + 1) * 0.001, (B, 1)), axis=1)
    flip = rng.random((B, n)) < sigma
    return np.where(flip, mag, -mag).astype(np.float32)


CASES = {
    # name: (code, LLR maker, noise, cap, lines, divisible)
    "one_chunk": (lambda: workloads.rlc(100, 78, 81), noise, 0.55, 60000, 3, False),
    "several_chunks": (lambda: workloads.rlc(256, 232, 82), noise, 0.46, 400000, 3, False),
    "several_chunks_div": (lambda: workloads.rlc(255, 231, 83), noise, 0.46, 200000, 4, True),
    "past_the_count": (lambda: workloads.rlc(64, 40, 84), nearly_flat, 0.08, 50000, 1, False),
    "by_weight": (lambda: workloads.rlc(200, 180, 85), nearly_flat, 0.015, 30000, 2, False),
    "fewer_patterns": (lambda: workloads.rlc(13, 1, 86), noise, 4.0, 16000, 2, False),
    "two_words": (lambda: workloads.rlc(96, 56, 87), noise, 0.55, 100000, 2, False),
    "four_words": (lambda: workloads.rlc(160, 60, 88), noise, 0.5, 60000, 3, False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_fitted_pairs(orbg, name):  # noqa: F811
    make, inputs, sigma, cap, lines, div = CASES[name]
    code = make()
    llr = inputs(code.n, 48, sigma, 90 + len(name))
    want = oracle.decode_batch_fit(code.H, llr, cap, lines, div)
    c = orbg.Code(code.H, max_query_cap=1000)
    got = orbg.decode_fitted(c, torch.from_numpy(llr).cuda(), cap, lines, div)
    torch.cuda.synchronize()
    cw, q, ab = (x.cpu().numpy() for x in got[:3])
    assert_same((cw, q.astype(np.int64), ab), want[:3])


def test_position_256(orbg):  # noqa: F811
    """The most reliable of 256 positions flipped, alone and with others."""
    code = workloads.rlc(256, 236, 89)
    llr = nearly_flat(256, 12, 0.0, 91)
    order = np.argsort(np.abs(llr), axis=1, kind="stable")
    for b in range(12):
        llr[b, order[b, 255]] *= -1
        if b % 3:
            llr[b, order[b, b]] *= -1
    cap = 60000
    want = oracle.decode_batch_fit(code.H, llr, cap, 1, False)
    assert (want[1] == 257).any()
    c = orbg.Code(code.H, max_query_cap=1000)
    got = orbg.decode_fitted(c, torch.from_numpy(llr).cuda(), cap, 1, False)
    torch.cuda.synchronize()
    cw, q, ab = (x.cpu().numpy() for x in got[:3])
    assert_same((cw, q.astype(np.int64), ab), want[:3])
