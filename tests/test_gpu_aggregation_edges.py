"""The aggregation kernel at the edges of its cost ring, lane layouts and padding.

A warp's costs arrive through a ring of four stages of 8 or 16 steps, a lane
holds 4 to 32 disparities of a folded record, and padding slots hold a cost that
must neither win a minimum nor spoil a neighbour.  The sizes below put scanlines
just short of, at and past the stages; the penalties go up to the largest the
parameter check lets through, where a padding slot's path cost exceeds a byte.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (3, 8), (8, 7), (17, 9), (31, 33), (64, 32), (65, 15), (16, 129)]
DISPARITIES = [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 33, 48, 64, 65, 97, 127, 128, 129, 192, 255]


def check(W, H, D, cw, ch, mask, P1, P2, cost, cpl):
    rng = np.random.default_rng(1000 * D + 10 * W + H)
    left = rng.integers(0, 256, (H, W), dtype=np.uint8)
    right = np.roll(left, -min(D // 2, W - 1), axis=1)
    right[:, ::3] = rng.integers(0, 256, right[:, ::3].shape, dtype=np.uint8)
    o = oracle.sgm(left, right, D, cw, ch, mask, P1, P2, 1, 3, stages=True, uv=False, cost=cost)
    p = sgm.SgmParams(census_w=cw, census_h=ch, path_mask=mask, P1=P1, P2=P2, lr_tolerance=1, median_k=3, cost=cost)
    with sgm.Handle(W, H, D, p) as h:
        try:
            sgm.sgm_set_aggregation(h, 4, cpl)
        except sgm.SgmError as e:
            assert e.status == sgm.SGM_ERR_UNSUPPORTED
            return
        L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
        S = torch.empty((H, W, D), dtype=torch.int16, device="cuda")
        disp = torch.empty((H, W), dtype=torch.uint8, device="cuda")
        sgm.sgm_debug_sum(h, L, R, S)
        h.compute(L, R, disp)
        torch.cuda.synchronize()
        what = f"{W}x{H} D={D} cpl={cpl} P={P1}/{P2}"
        assert np.array_equal(S.cpu().numpy().view(np.uint16), o["S"]), what
        assert np.array_equal(disp.cpu().numpy(), o["disp"]), what


@pytest.mark.parametrize("cpl", [1, 2, sgm.SGM_AGG_CHUNKS_MIXED, 4])
@pytest.mark.parametrize("D", DISPARITIES)
def test_census_paths_match_the_oracle(D, cpl):
    for i, (W, H) in enumerate(SIZES):
        cw, ch = ((5, 5), (9, 7))[i % 2]
        most = 255 - (cw * ch - 1)  # the largest P2 that is taken
        P1, P2 = ((8, 32), (most, most), (0, most), (0, 0))[i % 4]
        check(W, H, D, cw, ch, (0xFF, 0x0F, 0x55, 0xA6)[i // 2 % 4], P1, P2, sgm.SGM_COST_CENSUS, cpl)


@pytest.mark.parametrize("D", DISPARITIES)
def test_sad_paths_match_the_oracle(D):
    for i, (W, H) in enumerate(SIZES):
        cw, ch, mask = ((5, 5, 0x0F), (3, 3, 0xFF), (11, 11, 0x02))[i % 3]
        top = cw * ch * 255
        most = min(32766, 65535 // bin(mask).count("1")) - top  # the largest P2 that is taken
        P1, P2 = ((20, 80), (most, most), (0, most))[i // 3 % 3]
        check(W, H, D, cw, ch, mask, P1, P2, sgm.SGM_COST_SAD, 1)
