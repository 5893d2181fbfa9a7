"""The fitted decoder at the batch sizes where it changes how long one warp
searches a block before a CTA takes it: the same outputs on both sides, and
as in a large batch, and the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2202_13951_gb300 import workloads
from test_gpu_parity import assert_same, orbg  # noqa: F401
from test_gpu_zfitpairs import noise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,sigma,sizes", [
    (128, 14, 0.55, (1, 303, 304, 305)),  # up to 38,912 positions
    (128, 15, 0.55, (32, 33)),            # past 14 parity bits, up to 32 blocks
    (72, 40, 0.55, (31, 32, 33, 540, 541)),
])
def test_batch_sizes(orbg, n, r, sigma, sizes):  # noqa: F811
    code = workloads.rlc(n, n - r, 95)
    cap, lines = 30000, 2
    llr = torch.from_numpy(noise(n, 700, sigma, 96)).cuda()
    c = orbg.Code(code.H, max_query_cap=1000)
    whole = orbg.decode_fitted(c, llr, cap, lines)
    want = oracle.decode_batch_fit(code.H, llr[:40].cpu().numpy(), cap, lines, False)
    # ends before, between and past the two lengths
    q = want[1].astype(np.int64)
    assert (q < 256).any() and ((q > 300) & (q < 1000)).any() and (q > 1200).any()
    assert_same([x[:40].cpu().numpy() for x in whole[:3]], want[:3])
    for B in sizes:
        part = orbg.decode_fitted(c, llr[:B].contiguous(), cap, lines)
        for got, w in zip(part, whole):
            assert torch.equal(got, w[:B])
