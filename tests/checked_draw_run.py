"""Run by test_gpu_points_overflow.py in a child process with AF_CHECKED=1: the
point layer of the bounds-checked build with the draw's list as long as in
production (the road that ordinary frames take) and too short for the draw."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.path.insert(0, os.path.join(ROOT, "tests"))

from test_gpu_points_overflow import run_frames  # noqa: E402
from paper_2608_06412_gb300 import af  # noqa: E402

if __name__ == "__main__":
    assert os.environ.get("AF_CHECKED") == "1"
    assert b"checked" in af.load(build=False).af_version()
    for length in (None, 64):
        run_frames(length, dict(trig_sample=256), frames=2)
    print("CHECKED OK")
