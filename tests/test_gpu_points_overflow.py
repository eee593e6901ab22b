"""Draws of changed voxels that overflow the list of candidates: one CTA finds
the bound over all changed voxels, and the points queued are the oracle's --
with the list at its usual length, with room for some of the candidates, and
with room for one. The bounds-checked build takes the same roads as the usual
one (tests/checked_draw_run.py, in a child process)."""
import os
import subprocess
import sys

import pytest

from parity import to_dev
from paper_2608_06412_gb300 import af, synth, workload
from test_gpu_points import _compare, _pair

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_frames(length, over, frames=3):
    W = workload.single_frame()
    caps = dict(hash_capacity=1 << 15, pool_blocks=1 << 13, max_returns=1 << 13, max_points=1 << 10)
    if length is not None:
        os.environ["AF_DRAW_LIST"] = str(length)
    try:
        g, om, op = _pair(W, dict(dict(budget=700, capacity=1 << 14), **over), caps)
    finally:
        os.environ.pop("AF_DRAW_LIST", None)
    for f in range(frames):
        fr = synth.cone_frame(W.scene, 2500, 0.01, 300 + f, origin=(0.0, 0.03 * f, 0.01 * f))
        g.points_frame(to_dev(fr.pts), fr.pose)
        op.frame(fr.pts, fr.pose)
        _compare(g.points_export(), op.export(), f"frame {f}")
    assert g.sync_status() == 0


@pytest.mark.parametrize("length,sample", [(None, 256), (1, 256), (64, 256), (64, 40), (1000, 4096)])
def test_overflowed_draws(length, sample):
    run_frames(length, dict(trig_sample=sample))


def test_checked_build_takes_the_same_roads():
    af.load()  # builds both libraries if stale
    env = dict(os.environ, AF_CHECKED="1")
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "checked_draw_run.py")], env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "CHECKED OK" in r.stdout
