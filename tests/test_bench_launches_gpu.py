"""bench.py reports the launches that the library made, and the kernel that made them, at sizes on both
sides of the rule for two steps per launch."""
import json
import os
import subprocess
import sys

import pytest

from paper_1402_5487_gb300 import inputs as I
from paper_1402_5487_gb300 import plbm

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("prec,L", [("f32", 900), ("f32", 700), ("f32", 2047), ("bf16dev", 2076), ("f16dev", 1024), ("f64", 256)])
def test_launches_and_kernel_of_the_bench_line(prec, L):
    s = plbm.Solver(2, I.SET_013, 1.3, L, L, prec=prec)
    s.init(*I.kh_fields(L))
    s.step(8)
    n = s.step_launches
    s.close()
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--size", str(L), "--prec", prec, "--steps", "8", "--warmup", "4",
                          "--no-variants", "--no-cpu-baseline", "--no-e2e"], capture_output=True, text=True, check=True).stdout
    line = json.loads(out.strip().splitlines()[-1])
    assert line["gpu_launches"] == n and line["roofline"]["steps_per_launch"] == 8 / n
    assert ("two_steps" in line["roofline"]["kernel"]) == (n < 8)
    assert line["roofline"]["traffic"] is None   # no capture at this size
