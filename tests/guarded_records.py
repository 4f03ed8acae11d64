"""Runs the guarded build of the library (selected with SGM_LIBRARY) over the
records and work lists that tests/guarded_run.py does not reach: 96, 160, 192 and
224 slots, lanes of six pairs and their staged stores, the SAD kernels with and
without rectification maps, and costs of more than 100 MB, whose long axis is
walked second.  Checks each result against the CPU oracle and prints one JSON
line with the number of index-check hits.  Started by
tests/test_gpu_guarded_records.py in a process of its own."""
import json
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import torch  # noqa: E402

import oracle  # noqa: E402
from paper_1807_06271_gb300 import sgm  # noqa: E402

CENSUS, SAD = sgm.SGM_COST_CENSUS, sgm.SGM_COST_SAD
# W, H, D, cost, window, path mask, P1, P2, rectified
CASES = [
    (1240, 9, 96, CENSUS, (9, 7), 0xFF, 8, 96, False),   # six pairs per lane beside two
    (9, 1240, 70, CENSUS, (5, 5), 0xFF, 4, 24, False),
    (620, 9, 192, CENSUS, (9, 7), 0xFF, 8, 96, False),   # six pairs per lane beside four
    (9, 620, 161, CENSUS, (5, 5), 0xFF, 4, 24, False),
    (120, 41, 96, CENSUS, (7, 7), 0x0F, 8, 64, True),    # three quarters of a warp
    (77, 30, 130, CENSUS, (7, 5), 0xFF, 8, 64, False),   # 160 slots
    (50, 33, 200, CENSUS, (3, 3), 0x55, 8, 64, False),   # 224 slots
    (61, 20, 60, SAD, (5, 5), 0x55, 200, 800, False),
    (481, 188, 60, SAD, (5, 5), 0x55, 200, 800, False),
    (130, 11, 96, SAD, (5, 5), 0xFF, 200, 800, True),
    (67, 13, 3, SAD, (7, 7), 0x0F, 200, 800, False),
    (129, 9, 100, SAD, (3, 3), 0xFF, 200, 800, True),
    (700, 560, 128, SAD, (3, 3), 0xFF, 200, 800, False),  # 100 MB of costs
]


def main():
    sgm.sgm_debug_guard_hits(reset=True)
    bad = []
    for n, (W, H, D, cost, (cw, ch), mask, P1, P2, rect) in enumerate(CASES):
        rng = np.random.default_rng(n)
        left = rng.integers(0, 256, (H, W), dtype=np.uint8)
        right = np.roll(left, -min(D // 2, W - 1), axis=1)
        p = sgm.SgmParams(census_w=cw, census_h=ch, path_mask=mask, P1=P1, P2=P2, lr_tolerance=1, median_k=3, cost=cost)
        lo, ro = left, right
        with sgm.Handle(W, H, D, p) as h:
            if rect:
                maps = [rng.integers(0, m + 2, (H, W)).astype(np.uint16) for m in (W, H, W, H)]
                lo, ro = oracle.rectify(left, maps[0], maps[1]), oracle.rectify(right, maps[2], maps[3])
                on_device = [torch.from_numpy(m.view(np.int16)).cuda() for m in maps]
                sgm.sgm_set_rectification(h, *on_device)
            L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
            d = torch.empty((H, W), dtype=torch.uint8, device="cuda")
            h.compute(L, R, d)
            got = d.cpu().numpy()
        o = oracle.sgm(lo, ro, D, cw, ch, mask, P1, P2, 1, 3, uv=False, cost=cost)
        if not np.array_equal(got, o["disp"]):
            bad.append(f"{W}x{H}d{D} cost {cost}")
    torch.cuda.synchronize()
    print(json.dumps({"library": os.path.basename(sgm.library_path()), "hits": sgm.sgm_debug_guard_hits(),
                      "cases": len(CASES), "mismatches": bad}))


if __name__ == "__main__":
    main()
