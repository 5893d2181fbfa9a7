"""Codes of few parity bits: the flat table over the first band (up to ten of
them), the smaller chunks of pairs and the plain form's CTAs of four warps (up
to thirteen) and its handover, against the oracle.  Codes whose columns are mostly zero search on where dense
ones of so few rows end.  Whole numbers: equal or wrong."""
import numpy as np
import pytest

import oracle
from paper_2202_13951_gb300 import workloads
from test_gpu_parity import assert_same, gpu_batched, gpu_plain, orbg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def sparse(n, r, k, seed):
    """r rows, k nonzero columns among n, full rank."""
    rng = np.random.default_rng(seed)
    H = np.zeros((r, n), np.uint8)
    at = rng.choice(n, k, replace=False)
    H[:, at[:r]] = np.eye(r, dtype=np.uint8)
    H[:, at[r:]] = rng.integers(0, 2, (r, k - r))
    return H


CASES = {
    # name: (H, cap, order)
    "dense_64_10": (lambda: workloads.rlc(64, 54, 31).H, 100_000, None),
    "dense_256_9": (lambda: workloads.rlc(256, 247, 32).H, 100_000, None),
    "eleven_rows": (lambda: workloads.rlc(64, 53, 33).H, 100_000, None),
    "thirteen_rows_sparse": (lambda: sparse(90, 13, 16, 43), 300_000, None),
    "tiny": (lambda: workloads.rlc(12, 6, 34).H, 10_000, None),
    "cap_in_the_table": (lambda: sparse(100, 10, 12, 35), 700, None),
    "cap_at_its_end": (lambda: sparse(100, 10, 12, 36), 2375, None),
    "sparse_100": (lambda: sparse(100, 10, 12, 37), 1_000_000, None),
    "sparse_200": (lambda: sparse(200, 8, 10, 38), 300_000, None),
    "sparse_40": (lambda: sparse(40, 6, 8, 39), 200_000, None),
    "line": (lambda: sparse(127, 9, 12, 40), 100_000, ((), (5,), (1,))),
    "weightless": (lambda: sparse(60, 10, 14, 41), 30_000, ((20, 40), (-3, 10, 0), (3, 1, 2))),
    "segments": (lambda: sparse(127, 10, 14, 42), 300_000, ((7, 17), (3, 37, 58), (5, 2, 1))),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_few_rows(orbg, name):  # noqa: F811
    make, cap, model = CASES[name]
    H = make()
    r, n = H.shape
    rng = np.random.default_rng(len(name))
    B = 120
    llr = (2.0 * (-1.0 + 0.6 * rng.standard_normal((B, n)))).astype(np.float32)
    if name.startswith(("sparse", "thirteen", "cap", "line", "weight", "segm")):
        # a wrong bit at a given depth of the order, in a nonzero column
        for b in range(20, B):
            mag = np.linspace(0.5, 8.0, n)
            llr[b] = -rng.permutation(mag)
            cols = np.nonzero(H.any(axis=0))[0]
            llr[b, rng.choice(cols, 1 + b % 3, replace=False)] *= -1
    if model is None:
        want = oracle.decode_batch(H, llr, cap)[:3]
    else:
        want = oracle.decode_batch_mline(H, llr, cap, model)[:3]
    c = orbg.Code(H, max_query_cap=cap, model=model)
    assert_same(gpu_plain(orbg, c, llr, cap), want)
    cs = orbg.CodeSet([c])
    warps = torch.cuda.get_device_properties(0).multi_processor_count
    few, some, many = B, B * (8 * warps // B + 1), B * (40 * warps // B + 1)
    for blocks, budget in ((few, 1 << 25), (few, 1), (some, 1 << 25), (many, 1 << 25), (many, 300)):
        orbg.orbg_codeset_set_tuning(cs.handle, orbg.OrbgTuning(1, 1, 4, budget, 8))
        assert_same(gpu_batched(orbg, cs, np.tile(llr, (blocks // B, 1)), cap),
                    [np.concatenate([w] * (blocks // B)) for w in want])
