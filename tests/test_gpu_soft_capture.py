"""Soft calls and scans under stream capture: a capture records launches that
have not run yet, so it leaves the dense SDF view's state to eager calls, and a
replayed soft call brings the view up to the map as it then is -- compared bit
for bit with a map whose view is built whole."""
import numpy as np
import pytest

from paper_2608_06412_gb300 import af, synth, workload
from test_gpu_soft_views import CAPS, _pairs

pytestmark = pytest.mark.gpu


class Rig:
    """A map with a tool, scans to feed it, and pairs to ask it for."""

    def __init__(self):
        import torch
        self.W = workload.single_frame()
        self.scans = []
        for k in range(6):
            f = synth.cone_frame(self.W.scene, 1500, 0.01, 31 + k, origin=(0.0, 0.2 * k, 0.1 * k))
            self.scans.append((torch.from_numpy(f.pts).cuda(), f.pose))
        self.pairs = _pairs(self.W, 5000)
        self.c = torch.empty(5000, device="cuda")
        self.map = self.make(())

    def make(self, scans):
        m = af.Map(self.W.af_config(**CAPS))
        m.set_tool(self.W.af_tool(), self.W.dirs)
        m.soft_set_view(1)
        for k in scans:
            m.integrate_scan(*self.scans[k])
        return m

    def scan(self, k):
        self.map.integrate_scan(*self.scans[k])

    def soft(self):
        return self.map.soft_clearance_raw(*self.pairs, 1, out=self.c)

    def capture(self, call):
        import torch
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        # relaxed: the view's buffers may be allocated inside
        with torch.cuda.graph(g, capture_error_mode="relaxed"):
            call()
        return g

    def check(self, scans):
        """self.c is what a map of these scans gives with its view built whole."""
        import torch
        want = self.make(scans).soft_clearance_raw(*self.pairs, 1)
        assert torch.equal(self.c, want)
        assert (want < want.max() - 1e-3).any()   # some pairs see the surface


def test_first_build_under_capture():
    """The first soft call on a map is captured: an eager call made before the
    graph has run builds the view itself, and a replay builds it whole."""
    r = Rig()
    r.scan(0)
    g = r.capture(r.soft)
    r.soft()
    r.check([0])
    r.scan(1)
    g.replay()
    r.check([0, 1])
    r.scan(2)
    r.soft()
    r.check([0, 1, 2])


def test_captured_update_takes_the_scans_before_each_replay():
    r = Rig()
    r.scan(0)
    r.soft()
    r.scan(1)
    g = r.capture(r.soft)
    r.scan(2)
    r.soft()                # an eager call before the first replay
    r.check([0, 1, 2])
    r.scan(3)
    g.replay()
    r.check([0, 1, 2, 3])
    r.scan(4)
    r.scan(5)
    g.replay()
    r.check(range(6))


def test_two_soft_calls_and_a_scan_in_one_capture():
    import torch
    r = Rig()
    r.scan(0)
    r.soft()
    r.scan(1)
    torch.cuda.synchronize()
    first = torch.empty_like(r.c)

    def call():
        r.map.soft_clearance_raw(*r.pairs, 1, out=first)
        r.scan(2)
        r.soft()
        r.map.soft_clearance_raw(*r.pairs, 1, out=r.c)

    g = r.capture(call)
    g.replay()
    r.check([0, 1, 2])
    r.c.copy_(first)
    r.check([0, 1])


def test_scan_captured_early_and_replayed_late():
    """A captured scan keeps its scan number; replayed after later scans and a
    soft call, the next scan's update still takes its bricks."""
    r = Rig()
    r.scan(0)
    r.soft()
    g = r.capture(lambda: r.scan(1))
    for k in (2, 3):
        r.scan(k)
    r.soft()
    r.check([0, 2, 3])
    g.replay()
    # an empty scan: nothing of its own, but the view is out of date
    r.map.integrate_scan(r.scans[0][0][:0], r.scans[0][1])
    r.soft()
    r.check([0, 1, 2, 3])
