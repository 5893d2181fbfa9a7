"""Pair look-ups (prefix and pair of a pattern) at the edges of their tables,
against the oracle: orders of more pairs than one hash set holds, prefixes of
more positions than a record's first part, codes whose columns repeat or
whose first 32 rows say little, the two bands of phase 1 and its hand-over.
Whole numbers: equal or wrong."""
import numpy as np
import pytest

import oracle
from paper_2202_13951_gb300 import workloads
from test_gpu_parity import assert_same, gpu_batched, gpu_plain, orbg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def repeated_columns(n, k, seed):
    """A code with several equal parity-check columns."""
    code = workloads.rlc(n, k, seed)
    H = code.H.copy()
    H[:, 1] = H[:, 0]
    H[:, 5] = H[:, 4]
    H[:, 9] = H[:, 4]
    return H


CASES = {
    # name: (H, LLR blocks, cap, order)
    "cap_between_bands": (lambda: workloads.rlc(64, 44, 71).H, 64, 2.5, 3000, None),
    "past_the_bands": (lambda: workloads.rlc(128, 100, 72).H, 128, 2.0, 60000, None),
    "repeated_columns": (lambda: repeated_columns(48, 30, 73), 48, 2.0, 40000, None),
    "few_parity_bits": (lambda: workloads.rlc(90, 84, 74).H, 90, 3.0, 20000, None),
    "four_words": (lambda: workloads.rlc(160, 60, 75).H, 160, 4.5, 20000, None),
    "unit_columns_first": (lambda: workloads.rlc(100, 40, 76).H[:, ::-1].copy(), 100, 4.0, 20000,
                           None),
    # by Hamming weight first: 8,001 pairs, two hash sets
    "two_pair_chunks": (lambda: workloads.rlc(127, 106, 77).H, 127, 2.5, 60000,
                        ((), (9000,), (1,))),
    # 32,385 pairs of n = 255, eight sets
    "eight_pair_chunks": (lambda: workloads.rlc(255, 231, 78).H, 255, 4.5, 60000,
                          ((), (40000,), (1,))),
    # 6,441 pairs: the first 900, the first 2,047, then chunk by chunk
    "cuts_of_an_order": (lambda: workloads.rlc(127, 109, 81).H, 127, 2.5, 1_000_000,
                         ((7, 17), (3, 37, 58), (5, 2, 1))),
    # most look-ups of a band hit
    "many_hits_a_step": (lambda: workloads.rlc(256, 247, 82).H, 256, 5.0, 20000, None),
    "weightless_positions": (lambda: workloads.rlc(60, 40, 80).H, 60, 2.5, 30000,
                             ((20, 40), (-3, 10, 0), (3, 1, 2))),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_pair_tables(orbg, name):  # noqa: F811
    make, n, ebn0, cap, model = CASES[name]
    H = make()
    rng = np.random.default_rng(len(name))
    # pure noise around a code word: hits at all depths, some abandoned
    B = 60
    sigma = 10 ** (-ebn0 / 20.0) * 0.7
    llr = (2.0 * (-1.0 + sigma * rng.standard_normal((B, n))) / sigma ** 2).astype(np.float32)
    llr[0] = rng.permutation(np.linspace(-8, 8, n)).astype(np.float32)
    llr[1] = np.where(rng.random(n) < 0.3, 1.0, -1.0)
    if model is None:
        want = oracle.decode_batch(H, llr, cap)[:3]
    else:
        want = oracle.decode_batch_mline(H, llr, cap, model)[:3]
    c = orbg.Code(H, max_query_cap=cap, model=model)
    assert_same(gpu_plain(orbg, c, llr, cap), want)
    cs = orbg.CodeSet([c])
    for tuning in (None, (8, 0, 1, 1, 8), (8, 0, 1, 1000, 1), (8, 0, 1, 1 << 25, 16)):
        if tuning is not None:
            orbg.orbg_codeset_set_tuning(cs.handle, orbg.OrbgTuning(*tuning))
        assert_same(gpu_batched(orbg, cs, llr, cap), want)


def test_prefix_of_more_positions_than_a_record(orbg):  # noqa: F811
    """The sixteen lightest positions last in the order, patterns of seven
    of the eight others and a pair of light ones: prefixes of seven positions
    besides the light ones."""
    n, cap = 24, 2_600_000
    H = np.concatenate([np.eye(n - 1, dtype=np.uint8), np.ones((n - 1, 1), np.uint8)], axis=1)
    model = ((8,), (516, 500), (1, 1))
    llr = np.tile(-np.arange(1, n + 1, dtype=np.float32), (3, 1))
    for b, flips in enumerate(([0, 1, 2, 3, 4, 5, 6, 8, 9], [1, 2, 3, 4, 5, 6, 7, 10, 23],
                               [0, 2, 3, 4, 5, 6, 7, 22, 23])):
        llr[b, flips] *= -1
    want = oracle.decode_batch_mline(H, llr, cap, model)[:3]
    assert (want[1] > 1_800_000).any()
    c = orbg.Code(H, max_query_cap=cap, model=model)
    assert_same(gpu_plain(orbg, c, llr, cap), want)
    assert_same(gpu_batched(orbg, orbg.CodeSet([c]), llr, cap), want)


def test_per_code_launches(orbg):  # noqa: F811
    """A call large enough for one phase-1 launch per code, dense (one
    stride) with ids outside the set: each code's blocks as alone, the others
    flagged, their codewords untouched."""
    B, n, cap = 2 * 65536 + 5, 48, 20000
    codes = [workloads.rlc(n, 34, 81), workloads.rlc(n, 30, 82)]
    objs = [orbg.Code(c.H, max_query_cap=cap) for c in codes]
    rng = np.random.default_rng(83)
    cid = rng.integers(0, 2, B).astype(np.int32)
    bad = rng.choice(B, 50, replace=False)
    cid[bad] = rng.choice([-1, 2, 1 << 20], 50)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(84)
    llr = 4.0 * (-1.0 + 0.5 * torch.randn((B, n), generator=gen, device="cuda"))
    cs = orbg.CodeSet(objs)
    cw, q, ab = orbg.decode_batched(cs, llr, cap, code_id=torch.from_numpy(cid).cuda())
    torch.cuda.synchronize()
    for j, c in enumerate(objs):
        at = torch.from_numpy(np.nonzero(cid == j)[0]).cuda()
        alone = orbg.decode_batched(orbg.CodeSet([c]), llr[at].contiguous(), cap)
        for got, want in zip((cw[at], q[at], ab[at]), alone):
            assert torch.equal(got, want)
        pick = at[:40].cpu().numpy()
        want = oracle.decode_batch(codes[j].H, llr[at[:40]].cpu().numpy(), cap)[:3]
        assert_same((cw.cpu().numpy()[pick], q.cpu().numpy().astype(np.int64)[pick],
                     ab.cpu().numpy()[pick]), want)
    at = torch.from_numpy(bad).cuda()
    assert (q[at] == 0).all() and (ab[at] == 2).all() and (cw[at] == 255).all()
