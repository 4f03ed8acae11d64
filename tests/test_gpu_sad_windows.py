"""The SAD cost kernel for any window against the oracle: widths around its 64-pixel
segments, heights around its 4 rows, every number of slots, and rectification maps;
and the 5x5 kernel with few slots, which only large images take."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rect", [False, True])
@pytest.mark.parametrize("D", [1, 8, 13, 16, 32, 50, 64, 96, 128, 150, 192, 200, 255])
def test_sad_cost_volume_matches_the_oracle(D, rect):
    rng = np.random.default_rng(D)
    for (W, H), (ww, wh) in zip(((1, 1), (63, 3), (64, 4), (65, 5), (130, 9)), ((3, 3), (1, 7), (7, 7), (11, 3), (9, 11))):
        left, right = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
        p = sgm.SgmParams(census_w=ww, census_h=wh, path_mask=1, P1=20, P2=80, cost=sgm.SGM_COST_SAD)
        lo, ro = left, right
        with sgm.Handle(W, H, D, p) as h:
            if rect:
                maps = [rng.integers(0, n + 2, (H, W)).astype(np.uint16) for n in (W, H, W, H)]
                lo, ro = oracle.rectify(left, maps[0], maps[1]), oracle.rectify(right, maps[2], maps[3])
                sgm.sgm_set_rectification(h, *[torch.from_numpy(m.view(np.int16)).cuda() for m in maps])
            C = torch.full((H, W, D), -1, dtype=torch.int16, device="cuda")
            sgm.sgm_debug_cost(h, torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda(), C)
            got = C.cpu().numpy().view(np.uint16)
        assert np.array_equal(got, oracle.sad_cost_volume(lo, ro, D, ww, wh)), (W, H, D, rect)


@pytest.mark.parametrize("W, H", [(481, 832), (61, 6558), (640, 625)])
@pytest.mark.parametrize("D", [3, 9, 32, 33, 64])
def test_large_images_of_few_slots_match_the_oracle(W, H, D):
    if D > 32:
        H = -(-90000 // W)  # the smallest that takes the 5x5 kernel
    rng = np.random.default_rng(W + D)
    left, right = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
    p = sgm.SgmParams(census_w=5, census_h=5, path_mask=1, P1=20, P2=80, cost=sgm.SGM_COST_SAD)
    with sgm.Handle(W, H, D, p) as h:
        C = torch.full((H, W, D), -1, dtype=torch.int16, device="cuda")
        sgm.sgm_debug_cost(h, torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda(), C)
        assert np.array_equal(C.cpu().numpy().view(np.uint16), oracle.sad_cost_volume(left, right, D, 5, 5))
