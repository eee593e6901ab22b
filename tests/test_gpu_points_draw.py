"""The draw of changed voxels where its road changes: the largest draw that
goes through the candidate list and the smallest that does not, more drawn
than changed, a single one, the largest radius -- and the edges of the blocks
of 1,024 ids the selection works in, under budgets that end inside one."""
import pytest

from parity import to_dev
from paper_2608_06412_gb300 import synth, workload
from test_gpu_points import _compare, _pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [
    dict(trig_sample=4096), dict(trig_sample=4097), dict(trig_sample=1),
    dict(trig_sample=1 << 20), dict(trig_radius=7), dict(trig_radius=0),
    dict(budget=1023), dict(budget=1025), dict(budget=0),
], ids=lambda d: "-".join(f"{k}{v}" for k, v in d.items()))
def test_draw_and_selection_edges(over):
    W = workload.single_frame()
    caps = dict(hash_capacity=1 << 15, pool_blocks=1 << 13, max_returns=1 << 13, max_points=1 << 10)
    g, om, op = _pair(W, dict(dict(budget=700, capacity=1 << 14), **over), caps)
    for f in range(4):
        fr = synth.cone_frame(W.scene, 2500, 0.01, 300 + f, origin=(0.0, 0.03 * f, 0.01 * f))
        g.points_frame(to_dev(fr.pts), fr.pose)
        op.frame(fr.pts, fr.pose)
        _compare(g.points_export(), op.export(), f"frame {f}")
    for n in (1, 1024, 10 ** 6):
        g.points_drain(n)
        op.drain(n)
        _compare(g.points_export(), op.export(), f"drained {n}")
    assert g.sync_status() == 0
