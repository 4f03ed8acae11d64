"""Rows up to the longest that is taken (8192 pixels): the winner-takes-all kernel
holds a row's right minima and left winners in shared memory beside its record
rings, and runs fewer warps where 16-bit records of 8 paths would not fit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cost", [sgm.SGM_COST_CENSUS, sgm.SGM_COST_SAD])
@pytest.mark.parametrize("D", [8, 128, 255])
def test_long_rows_match_the_oracle(D, cost):
    rng = np.random.default_rng(D)
    P1, P2 = (200, 800) if cost == sgm.SGM_COST_SAD else (8, 32)
    p = sgm.SgmParams(path_mask=sgm.SGM_PATHS_8, census_w=5, census_h=5, P1=P1, P2=P2, lr_tolerance=1, cost=cost)
    for W in (6800, 7000, 8192):
        left = rng.integers(0, 256, (2, W), dtype=np.uint8)
        right = np.roll(left, -min(D // 2, 40), axis=1)
        o = oracle.sgm(left, right, D, 5, 5, 0xFF, P1, P2, 1, p.median_k, stages=True, uv=False, cost=cost)
        with sgm.Handle(W, 2, D, p) as h:
            disp = torch.empty((2, W), dtype=torch.uint8, device="cuda")
            h.compute(torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda(), disp)
            assert np.array_equal(disp.cpu().numpy(), o["disp"]), (W, D)
