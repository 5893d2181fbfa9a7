"""Phase 1's two bands, and its hand-over after each of them, against the
oracle.  A batch of at most two blocks a resident warp hands its blocks over
after the flat table and one of at most eight (forty with few parity bits)
after the first band, whatever the budget: here one warp an SM is resident and
the batches are larger.
Whole numbers: equal or wrong."""
import numpy as np
import pytest

import oracle
import oracle_pool
from paper_2202_13951_gb300 import workloads
from test_gpu_parity import assert_same, gpu_batched, orbg  # noqa: F401
from test_gpu_zpairs import CASES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TILE = 240  # different blocks of a batch
FLAT, BAND1, BAND2 = 256, 2375, 16857  # last queries of basic ORBGRAND's stages

#: besides the pair tables' cases: name -> (H, n, Eb/N0, cap, line)
LINES = {
    "line": (lambda: workloads.rlc(127, 109, 85).H, 127, 3.0, 40000, (5, 1)),
    "line_four_words": (lambda: workloads.rlc(150, 50, 86).H, 150, 4.5, 20000, (2, 3)),
    "two_words_past_128": (lambda: workloads.rlc(180, 140, 87).H, 180, 4.5, 30000, (0, 1)),
}

#: dB taken off a pair tables' case, so that more searches end in the bands
LOWER = {"four_words": 0.8, "unit_columns_first": 0.8, "cap_between_bands": 0.8,
         "repeated_columns": 0.5, "line_four_words": 0.8, "two_words_past_128": 0.5}


def noise(rng, B, n, ebn0):
    sigma = 10 ** (-ebn0 / 20.0) * 0.7
    llr = (2.0 * (-1.0 + sigma * rng.standard_normal((B, n))) / sigma ** 2).astype(np.float32)
    llr[0] = rng.permutation(np.linspace(-8, 8, n)).astype(np.float32)
    llr[1] = np.where(rng.random(n) < 0.3, 1.0, -1.0)  # every rank a tie
    return llr


@pytest.mark.parametrize("name", sorted(CASES) + sorted(LINES))
def test_bands(orbg, name):  # noqa: F811
    rng = np.random.default_rng(len(name) + 40)
    line = model = None
    if name in LINES:
        make, n, ebn0, cap, line = LINES[name]
    else:
        make, n, ebn0, cap, model = CASES[name]
    H = make()
    llr = noise(rng, TILE, n, ebn0 - LOWER.get(name, 0.0))
    if model is not None:
        want = oracle.decode_batch_mline(H, llr, cap, model)[:3]
    elif line is not None:
        want = oracle.decode_batch_mline(H, llr, cap, ((), line[:1], line[1:]))[:3]
    else:
        want = oracle.decode_batch(H, llr, cap)[:3]
    q = want[1].astype(np.int64)
    assert ((q > FLAT) & (q <= BAND1)).any()
    # a model's bands end elsewhere; with few parity bits no search lasts that long
    if model is None and cap > BAND2 and H.shape[0] > 10:
        assert ((q > BAND1) & (q <= BAND2)).any()
    cs = orbg.CodeSet([orbg.Code(H, max_query_cap=cap, line=line, model=model)])
    warps = torch.cuda.get_device_properties(0).multi_processor_count
    few = TILE * (2 * warps // TILE + 1)   # past two blocks a warp
    past = 40 if H.shape[0] <= 10 else 8
    many = TILE * (past * warps // TILE + 1)  # past that
    assert 2 * warps < few <= 8 * warps < many
    for B, budget in ((few, 1 << 25), (many, 1), (many, 1000), (many, 1 << 25)):
        orbg.orbg_codeset_set_tuning(cs.handle, orbg.OrbgTuning(1, 1, 4, budget, 8))
        assert_same(gpu_batched(orbg, cs, np.tile(llr, (B // TILE, 1)), cap),
                    [np.concatenate([w] * (B // TILE)) for w in want])


@pytest.fixture(scope="module")
def deep():
    """2,000 blocks of a code whose searches end in every stage, and past the
    last band's queries."""
    code = workloads.rlc(64, 44, 61)
    llr, _ = workloads.awgn_llr(code, 2000, 2.5, 63)
    cap = 30000
    want = oracle_pool.decode_batch(code.H, llr, cap)[:3]
    q = want[1].astype(np.int64)
    for lo, hi in ((1, FLAT), (FLAT, BAND1), (BAND1, BAND2), (BAND2, cap - 1)):
        assert ((q > lo) & (q <= hi)).sum() >= 10
    assert want[2].any()
    return code, llr, cap, want


@pytest.mark.parametrize("tuning", [(8, 1, 8, 1, 16), (1, 1, 1, 64, 4), (1, 1, 32, 4096, 1),
                                    (1, 1, 4, 16384, 8), (1, 1, 8, 10 ** 6, 16)],
                         ids=lambda t: "wpc%d_cps%d_grab%d_budget%d_hw%d" % t)
def test_budgets(orbg, deep, tuning):  # noqa: F811
    """Budgets below, between and past the bands' ends, and above the cap:
    blocks left open after the last band still reach phase 2."""
    code, llr, cap, want = deep
    cs = orbg.CodeSet([orbg.Code(code.H, max_query_cap=10 ** 5)])
    orbg.orbg_codeset_set_tuning(cs.handle, orbg.OrbgTuning(*tuning))
    assert_same(gpu_batched(orbg, cs, llr, cap), want)


def test_budgets_host_buffers(orbg, deep):  # noqa: F811
    """The same through the chunked path of host buffers: poisoned outputs,
    chunks of more than eight blocks a warp."""
    code, llr, cap, want = deep
    times = 70
    rows = np.tile(llr, (times, 1))
    B, n = rows.shape
    cs = orbg.CodeSet([orbg.Code(code.H, max_query_cap=10 ** 5)])
    orbg.orbg_codeset_set_tuning(cs.handle, orbg.OrbgTuning(1, 1, 4, 10 ** 6, 4))
    cw = np.full((B, n), 0xFF, np.uint8)
    q = np.full(B, 0xFFFFFFFF, np.uint32)
    ab = np.full(B, 0xFF, np.uint8)
    orbg.orbg_decode_batched(cs.handle, None, None, rows, B, cap, cw, None, q, ab)
    assert_same((cw, q.astype(np.int64), ab), [np.concatenate([w] * times) for w in want])
