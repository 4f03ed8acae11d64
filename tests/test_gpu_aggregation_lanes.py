"""The aggregation kernel's lane widths and its wrapped diagonals against the oracle:
one size for each choice of pairs per lane, on either long axis, and square-ish
images in which every diagonal wraps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("turn", [False, True])
@pytest.mark.parametrize("W, H, D", [
    (120, 100, 32), (700, 60, 32), (1400, 40, 32),                 # 1/1, 1/4 and 2/4 pairs
    (150, 130, 64), (400, 100, 64), (430, 420, 64), (1500, 90, 64),  # 1/2, 1/4, 2/2, 2/4
    (110, 100, 128), (300, 60, 128), (130, 130, 90),               # 2/2, 2/4, 2/2
    (1240, 9, 96), (1230, 30, 65), (620, 9, 192), (440, 330, 192), (605, 40, 161),  # six pairs in the other directions
])
def test_lane_widths_match_the_oracle(W, H, D, turn):
    if turn:
        W, H = H, W
    rng = np.random.default_rng(W + D)
    left = rng.integers(0, 256, (H, W), dtype=np.uint8)
    right = np.roll(left, -min(D // 2, W - 1), axis=1)
    right[:, ::3] = rng.integers(0, 256, right[:, ::3].shape, dtype=np.uint8)
    P1, P2 = (193, 193) if D % 2 else (4, 96)
    p = sgm.SgmParams(census_w=9, census_h=7, path_mask=0xFF, P1=P1, P2=P2, lr_tolerance=1, median_k=3)
    o = oracle.sgm(left, right, D, 9, 7, 0xFF, P1, P2, 1, 3, stages=True, uv=False)
    with sgm.Handle(W, H, D, p) as h:
        L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
        S = torch.empty((H, W, D), dtype=torch.int16, device="cuda")
        disp = torch.empty((H, W), dtype=torch.uint8, device="cuda")
        sgm.sgm_debug_sum(h, L, R, S)
        h.compute(L, R, disp)
        assert np.array_equal(S.cpu().numpy().view(np.uint16), o["S"])
        assert np.array_equal(disp.cpu().numpy(), o["disp"])


@pytest.mark.parametrize("W, H", [(700, 560), (560, 700)])
def test_costs_beyond_l2_match_the_oracle(W, H):
    # 16-bit costs of 100 MB: the long axis is walked between the two sweeps
    rng = np.random.default_rng(W)
    left = rng.integers(0, 256, (H, W), dtype=np.uint8)
    right = np.roll(left, -40, axis=1)
    p = sgm.SgmParams(census_w=3, census_h=3, path_mask=0xFF, P1=200, P2=800, lr_tolerance=1, median_k=3,
                      cost=sgm.SGM_COST_SAD)
    o = oracle.sgm(left, right, 128, 3, 3, 0xFF, 200, 800, 1, 3, stages=True, uv=False, cost=sgm.SGM_COST_SAD)
    with sgm.Handle(W, H, 128, p) as h:
        disp = torch.empty((H, W), dtype=torch.uint8, device="cuda")
        S = torch.empty((H, W, 128), dtype=torch.int16, device="cuda")
        L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
        sgm.sgm_debug_sum(h, L, R, S)
        h.compute(L, R, disp)
        assert np.array_equal(S.cpu().numpy().view(np.uint16), o["S"])
        assert np.array_equal(disp.cpu().numpy(), o["disp"])
