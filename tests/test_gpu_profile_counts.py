"""af_profile_read counts kernels: what each call launched, by the roads it
took."""
import pytest

from paper_2608_06412_gb300 import af, synth, workload
from test_gpu_soft_views import CAPS, _pairs

pytestmark = pytest.mark.gpu


def test_launch_counts():
    import torch
    W = workload.single_frame()
    m = af.Map(W.af_config(**CAPS))
    m.set_tool(W.af_tool(), W.dirs)
    m.soft_set_view(1)
    f = synth.cone_frame(W.scene, 3000, 0.01, 71)
    x = torch.from_numpy(f.pts).cuda()
    m.profile(True)
    m.profile_read(True)

    def counts(call):
        call()
        return {k: n for k, (n, _) in m.profile_read(True).items() if n}

    scan = dict(k_alloc=1, k_integrate=1, k_bitview=1)
    assert counts(lambda: m.integrate_scan(x, f.pose)) == scan
    assert counts(lambda: m.integrate_scan(x[:0], f.pose)) == dict(k_bitview=1)
    assert counts(lambda: m.integrate_scan_projective(x, f.pose, 64)) == dict(scan, k_integrate=2)
    pairs = _pairs(W, 30000)

    def refine(n):
        p = [t[:n].clone() for t in pairs]
        return lambda: m.soft_refine(*p, 1, steps=1)

    sm = torch.cuda.get_device_properties(0).multi_processor_count
    name = af.KERNELS[7]
    # the view's first build, then nothing to do; then the bricks of one scan
    assert counts(refine(500)) == {"k_views": 4, name: 1}
    assert counts(refine(500)) == {name: 1}
    m.integrate_scan(x, f.pose)
    m.profile_read(True)
    assert counts(refine(64 * sm)) == {"k_views": 2, name: 1}
    assert counts(refine(96 * sm)) == {name: 1}
    assert counts(refine(96 * sm + 1)) == {name: 2}
    for budget, n in ((-1, 1), (4, 3)):
        m.set_score_split(budget)
        assert counts(lambda: m.score(pairs[0], pairs[1])) == dict(k_score=n)
