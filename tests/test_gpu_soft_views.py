"""The dense SDF view kept up to date scan by scan: after any run of scans
since the last soft call -- scan-centric, projective or batched, new bricks
and known ones, bricks on the faces of the map box -- the soft calls give
what they give on a map whose view is built whole."""
import numpy as np
import pytest

from paper_2608_06412_gb300 import af, synth, workload

pytestmark = pytest.mark.gpu

CAPS = dict(hash_capacity=1 << 14, pool_blocks=1 << 13, max_returns=4096, max_points=4096)


def _pairs(W, n=20000, seed=5):
    """Points over the box and one brick beyond it, with random directions."""
    import torch
    g = synth.rng(seed, 91)
    v = W.params["v"]
    lo = (np.array(W.dom_min) - 1) * 8 * v
    hi = (np.array(W.dom_min) + np.array(W.dom_bricks) + 1) * 8 * v
    u = g.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    return t(g.uniform(lo, hi, (n, 3))), t(u), t(g.normal(0, 0.1, n)), t(g.normal(0, 0.1, n)), \
        t(g.uniform(0, 0.05, n))


@pytest.mark.parametrize("how", ["scan", "projective", "batch"])
@pytest.mark.parametrize("tight", [False, True])
def test_updated_view_equals_whole(tight, how):
    import torch
    W = workload.single_frame()
    if tight:   # a box that cuts the scene on every axis
        lo, size = np.array(W.dom_min), np.array(W.dom_bricks)
        W.dom_min, W.dom_bricks = tuple(lo + size // 3), tuple(size - 2 * (size // 3))
    tool = W.af_tool()
    scans = []
    for k in range(5):
        f = synth.cone_frame(W.scene, 1500, 0.01, 11 + k, origin=(0.0, 0.2 * k, 0.1 * k))
        scans.append((torch.from_numpy(f.pts).cuda(), f.pose))

    def make():
        m = af.Map(W.af_config(**CAPS))
        m.set_tool(tool, W.dirs)
        m.soft_set_view(1)
        return m

    def integrate(m, batch, k):
        x, pose = scans[k]
        if how == "projective" and k % 2:
            m.integrate_scan_projective(x, pose, 64)
        elif how == "batch" and k % 2:
            e = torch.empty((0, 3), device="cuda")
            batch.tick([(x, pose, e, e, None, None)])
        else:
            m.integrate_scan(x, pose)

    pairs = _pairs(W)
    kept = make()
    kept_batch = af.Batch([kept])
    done = 0
    for upto in (1, 2, 2, 5):     # one scan, one more, none, three at once
        for k in range(done, upto):
            integrate(kept, kept_batch, k)
        done = upto
        whole = make()
        whole_batch = af.Batch([whole])
        for k in range(upto):
            integrate(whole, whole_batch, k)
        got = kept.soft_clearance_raw(*pairs[:2], *pairs[2:], 1)
        want = whole.soft_clearance_raw(*pairs[:2], *pairs[2:], 1)
        assert torch.equal(got, want)
        # refinement of pairs in and out of the view: C and the hard clearance at
        # the state it reports, whether a step takes the pair out or not
        for steps in (0, 3):
            a, b, h = (t.clone() for t in pairs[2:])
            c, cmin = kept.soft_refine(*pairs[:2], a, b, h, 1, steps=steps)
            hard = torch.empty_like(c)
            assert torch.equal(c, whole.soft_clearance_raw(*pairs[:2], a, b, h, 1, cmin=hard))
            assert torch.equal(cmin, hard)
            assert steps == 0 or not torch.equal(a, pairs[2])
        whole_batch.close()
        whole.close()
    far = got.max().item()
    assert (got < far - 1e-3).any()   # some pairs see the surface
