"""Cost volume and planes end where their last record ends, for slot counts that
are no power of two as for the others: guard bytes behind them lie next to the
last byte a kernel may write."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

SLOTS = [(1, 8), (8, 8), (9, 16), (17, 32), (33, 64), (65, 96), (96, 96), (97, 128), (129, 160), (192, 192), (193, 224),
         (225, 256)]


@pytest.mark.parametrize("cost", [sgm.SGM_COST_CENSUS, sgm.SGM_COST_SAD])
@pytest.mark.parametrize("D, slots", SLOTS)
def test_a_handle_holds_the_slots_its_kernels_use(D, slots, cost):
    W, H, mask = 90, 31, 0x1F
    p = sgm.SgmParams(census_w=3, census_h=3, path_mask=mask, P1=20, P2=80, cost=cost)
    volume = W * H * slots * (2 if cost == sgm.SGM_COST_SAD else 1)
    codes = 0 if cost == sgm.SGM_COST_SAD else 2 * W * H * 4
    assert sgm.sgm_scratch_bytes(W, H, D, p)[0] == codes + 6 * volume + 4228 + W * H


@pytest.mark.parametrize("D, slots", SLOTS)
def test_the_static_array_is_laid_out_as_documented(D, slots):
    # a power of two of slots, by which shapes are taken or refused
    W, H, mask = 90, 31, 0x1F
    p = sgm.SgmParams(census_w=3, census_h=3, path_mask=mask, P1=20, P2=80)
    two = 8
    while two < D:
        two *= 2
    at = 0
    for part in (2 * W * H * 4, W * H * two, 5 * W * H * two, 4228):
        at = (at + part + 255) // 256 * 256
    assert sgm.sgm_scratch_bytes(W, H, D, p)[2] == at + W * H


@pytest.mark.gpu
@pytest.mark.parametrize("cost", [sgm.SGM_COST_CENSUS, sgm.SGM_COST_SAD])
@pytest.mark.parametrize("W, H, D", [(1240, 9, 96), (61, 47, 70), (97, 31, 160), (620, 9, 192), (45, 40, 200)])
def test_no_kernel_writes_past_the_last_record(W, H, D, cost):
    rng = np.random.default_rng(D)
    left = rng.integers(0, 256, (H, W), dtype=np.uint8)
    right = np.roll(left, -min(D // 2, W - 1), axis=1)
    P1, P2 = (200, 800) if cost == sgm.SGM_COST_SAD else (8, 64)
    p = sgm.SgmParams(census_w=5, census_h=5, path_mask=0xFF, P1=P1, P2=P2, lr_tolerance=1, median_k=3, cost=cost)
    o = oracle.sgm(left, right, D, 5, 5, 0xFF, P1, P2, 1, 3, uv=False, cost=cost)
    sgm.sgm_debug_canaries(True)
    try:
        h = sgm.Handle(W, H, D, p)
    finally:
        sgm.sgm_debug_canaries(False)
    with h:
        L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
        disp = torch.empty((H, W), dtype=torch.uint8, device="cuda")
        kernels = [sgm.SGM_COST_KERNEL_AUTO]
        if cost == sgm.SGM_COST_CENSUS and D <= 128:
            kernels.append(sgm.SGM_COST_KERNEL_TENSOR_CORES)
        for k in kernels:
            sgm.sgm_set_cost_kernel(h, k)
            h.compute(L, R, disp)
            assert np.array_equal(disp.cpu().numpy(), o["disp"]), k
        assert sgm.sgm_debug_check_canaries(h) == sgm.SGM_OK
