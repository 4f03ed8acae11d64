"""The guarded build over folded records of 96 to 224 slots, the SAD kernels and
large cost volumes (tests/guarded_records.py), and that every unit that counts
index-check hits is read."""
import json
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_06271_gb300", "csrc")


def test_every_guarded_unit_is_summed():
    # a unit checks indices where it calls in_range, or reads pixels with rect_pixel
    with open(os.path.join(CSRC, "sgm_api.cu")) as f:
        api = f.read()
    summed = set(re.findall(r"(guard_hits_\w+)\(reset", api))
    for name in sorted(n for n in os.listdir(CSRC) if n.endswith(".cu")):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        if re.search(r"\b(in_range\(|rect_pixel<)", text):
            counters = set(re.findall(r"SGM_GUARD_COUNTER\((\w+)\)", text))
            assert counters and counters <= summed, f"{name} drops accesses out of range uncounted"


@pytest.mark.gpu
def test_guarded_records_stay_in_bounds_and_match_the_oracle():
    from paper_1807_06271_gb300 import build
    env = dict(os.environ, SGM_LIBRARY=build.build(guarded=True))
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "guarded_records.py")], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["library"] == "libsgm_guarded.so"
    assert out["mismatches"] == []
    assert out["hits"] == 0
