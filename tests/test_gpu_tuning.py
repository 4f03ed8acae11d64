"""The autotuner tries what a handle starts with, and only settings that differ."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


def inputs(W, H):
    rng = np.random.default_rng(W)
    left = rng.integers(0, 256, (H, W), dtype=np.uint8)
    L, R = torch.from_numpy(left).cuda(), torch.from_numpy(np.roll(left, -7, axis=1).copy()).cuda()
    return L, R, torch.empty((H, W), dtype=torch.uint8, device="cuda")


def best_time(h, L, R, disp, calls=20, runs=10):
    best = float("inf")
    for _ in range(runs):
        start, stop = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        start.record()
        for _ in range(calls):
            h.compute(L, R, disp)
        stop.record()
        torch.cuda.synchronize()
        best = min(best, start.elapsed_time(stop))
    return best


@pytest.mark.parametrize("tune_twice", [False, True])
def test_a_tuned_handle_is_no_slower_than_a_new_one(tune_twice):
    # 1000 x 600 starts with 5 blocks per SM; the next best, 4, takes 1.5 % longer
    # (289 and 294 us).  A second tuning starts from another setting.
    W, H, D = 1000, 600, 128
    p = sgm.SgmParams(census_w=9, census_h=7, path_mask=0xFF, P1=8, P2=95 - tune_twice, lr_tolerance=1, median_k=3)
    L, R, disp = inputs(W, H)
    with sgm.Handle(W, H, D, p) as h:
        start = sgm.sgm_get_aggregation(h)
        best_time(h, L, R, disp)
        sgm.sgm_autotune(h, L, R, disp)
        if tune_twice:
            sgm.sgm_set_aggregation(h, 2, 1)
            sgm.sgm_autotune(h, L, R, disp)
        tuned = sgm.sgm_get_aggregation(h)
        if tuned != start:
            best = {start: float("inf"), tuned: float("inf")}
            for _ in range(3):
                for setting in best:
                    sgm.sgm_set_aggregation(h, *setting)
                    best[setting] = min(best[setting], best_time(h, L, R, disp))
            assert best[tuned] <= 1.008 * best[start], (start, tuned)


@pytest.mark.parametrize("D", [66, 96, 130, 192, 224])
def test_settings_that_run_as_1_are_not_candidates(D):
    W, H = 260, 40
    p = sgm.SgmParams(census_w=9, census_h=7, path_mask=0xFF, P1=8, P2=92, lr_tolerance=1, median_k=3)
    L, R, disp = inputs(W, H)
    with sgm.Handle(W, H, D, p) as h:
        sgm.sgm_autotune(h, L, R, disp)
        assert sgm.sgm_get_aggregation(h)[1] == 1
