"""Refinement takes different kernels by the number of pairs and by where their
samples lie; what it gives does not depend on that. The same pairs in one call
(short way, then the general way for those it left) and in calls small enough
for the one kernel that does both: offsets, standoffs, C and the hard clearance
are the same bits."""
import pytest

from paper_2608_06412_gb300 import af, synth, workload
from test_gpu_soft_views import CAPS, _pairs

pytestmark = pytest.mark.gpu

N, PART = 20000, 4000


@pytest.mark.parametrize("view", [1, 2])
@pytest.mark.parametrize("tau_s", [0.005, 0.0005])   # weights against a bound, and against the minimum
@pytest.mark.parametrize("steps", [0, 1, 20])
def test_refinement_does_not_depend_on_the_calls_size(view, tau_s, steps):
    import torch
    W = workload.single_frame()
    m = af.Map(W.af_config(**CAPS))
    m.set_tool(W.af_tool(), W.dirs)
    m.soft_set_view(view)
    for k in range(2):
        f = synth.cone_frame(W.scene, 3000, 0.01, 51 + k, origin=(0.0, 0.2 * k, 0.0))
        m.integrate_scan(torch.from_numpy(f.pts).cuda(), f.pose)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert PART <= 64 * sm < N      # the sizes lie on both sides of the rule
    pts, u0, *par = _pairs(W, N)
    u0[::97] = float("nan")         # pairs without a start
    whole = [t.clone() for t in par]
    # large steps: some pairs leave the view, or come into it, on the way
    kw = dict(steps=steps, tau_s=tau_s, lr_dir=0.4, lr_h=0.05, h_max=0.4)
    whole += m.soft_refine(pts, u0, *whole, 1, **kw)
    parts = []
    for i in range(0, N, PART):
        j = slice(i, i + PART)
        p = [t[j].clone() for t in par]
        parts.append(p + list(m.soft_refine(pts[j], u0[j], *p, 1, **kw)))
    for w, p in zip(whole, map(torch.cat, zip(*parts))):
        assert torch.equal(torch.nan_to_num(w, nan=1e9), torch.nan_to_num(p, nan=1e9))
    assert steps < 20 or (whole[0] != par[0]).sum() > N // 50


@pytest.mark.parametrize("view", [1, 2])
def test_points_far_beyond_the_view_read_tau(view):
    """Cells up to 1e9 voxels from the box on either side: every sample reads
    tau, as for a pair that just leaves the box."""
    import torch
    W = workload.single_frame()
    m = af.Map(W.af_config(**CAPS))
    m.set_tool(W.af_tool(), W.dirs)
    m.soft_set_view(view)
    f = synth.cone_frame(W.scene, 3000, 0.01, 51)
    m.integrate_scan(torch.from_numpy(f.pts).cuda(), f.pose)
    far = [s * k * W.params["v"] for k in (9.9e8, 8.9e8, 7.0e8, 1e6, 2e3) for s in (1.0, -1.0)]
    pts = torch.tensor([[x if a == k else 1.0 for a in range(3)] for x in far for k in range(3)],
                       dtype=torch.float32, device="cuda")
    n = len(pts)
    u0 = torch.tensor([0.0, 0.0, 1.0], device="cuda").repeat(n, 1).contiguous()
    z = torch.zeros(n, device="cuda")
    cmin = torch.empty(n, device="cuda")
    c = m.soft_clearance_raw(pts, u0, z, z, z, 1, cmin=cmin)
    tool = W.af_tool()
    want = torch.tensor(W.params["tau"], dtype=torch.float32) - \
        torch.tensor(max(tool.radius, tool.corr_radius), dtype=torch.float32)
    assert (cmin == want.item()).all() and (c == c[0]).all()
