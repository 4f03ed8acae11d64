"""Planes of more than 2^32 units of 4 bytes: the columns of a tall image, whose
scanlines are few enough for the narrowest lanes.  A column's result depends on the
columns within D alone, so strips of the image are checked against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

pytestmark = pytest.mark.gpu


def test_tall_columns_of_16_bit_costs_match_the_oracle():
    W, H, D, mask = 2100, 65535, 40, 0x04
    if torch.cuda.mem_get_info()[0] < 50 << 30:
        pytest.skip("needs 50 GB of device memory")
    rng = np.random.default_rng(1)
    left = rng.integers(0, 256, (H, W), dtype=np.uint8)
    right = np.roll(left, -11, axis=1)
    p = sgm.SgmParams(census_w=1, census_h=1, path_mask=mask, P1=20, P2=80, lr_tolerance=-1, median_k=0,
                      cost=sgm.SGM_COST_SAD)
    disp = torch.full((H, W), 255, dtype=torch.uint8, device="cuda")
    with sgm.Handle(W, H, D, p) as h:
        h.compute(torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda(), disp)
        got = disp.cpu().numpy()
    for x0, skip in ((0, 0), (W - 56, D)):  # the second strip's first columns lack their right pixels
        o = oracle.sgm(left[:, x0:x0 + 56].copy(), right[:, x0:x0 + 56].copy(), D, 1, 1, mask, 20, 80, -1, 0, uv=False,
                       cost=sgm.SGM_COST_SAD)
        assert np.array_equal(got[:, x0 + skip:x0 + 56], o["disp"][:, skip:])
