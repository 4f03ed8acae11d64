"""The 5x5 SAD cost kernel against the oracle: widths around its 15-pixel segments
and its CTAs' spans (60 to 480 pixels), odd heights, every number of slots, and
rectification maps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rect", [False, True])
@pytest.mark.parametrize("D", [1, 3, 9, 17, 32, 60, 64, 96, 128, 200, 255])
def test_sad_cost_volume_matches_the_oracle(D, rect):
    rng = np.random.default_rng(D)
    for W, H in ((1, 1), (14, 3), (15, 2), (16, 4), (59, 5), (61, 2), (121, 1), (241, 3), (481, 2)):
        left, right = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
        p = sgm.SgmParams(census_w=5, census_h=5, path_mask=sgm.SGM_PATHS_4, P1=200, P2=800, cost=sgm.SGM_COST_SAD)
        lo, ro = left, right
        with sgm.Handle(W, H, D, p) as h:
            if rect:
                maps = [rng.integers(0, n + 2, (H, W)).astype(np.uint16) for n in (W, H, W, H)]
                lo, ro = oracle.rectify(left, maps[0], maps[1]), oracle.rectify(right, maps[2], maps[3])
                sgm.sgm_set_rectification(h, *[torch.from_numpy(m.view(np.int16)).cuda() for m in maps])
            C = torch.full((H, W, D), -1, dtype=torch.int16, device="cuda")
            sgm.sgm_debug_cost(h, torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda(), C)
            got = C.cpu().numpy().view(np.uint16)
        assert np.array_equal(got, oracle.sad_cost_volume(lo, ro, D, 5, 5)), (W, H, D, rect)
