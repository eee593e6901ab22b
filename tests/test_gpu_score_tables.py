"""Kernel tables of the scorer at their edges, labels and directions bit for
bit against the oracle: kernels of one row and of many, windows longer than a
word, empty kernels, axis-aligned and diagonal directions, both roads through
the search (all reads inside the box, and reads beyond its faces), points of
every parity, confidence gates at 0 and out of reach."""
import numpy as np
import pytest

import oracle
from parity import oracle_config, oracle_tool, to_dev
from paper_2608_06412_gb300 import af, synth, workload

pytestmark = pytest.mark.gpu

#: tool overrides: a needle of one row; no corridor; a corridor of three words
#: along an axis; an empty tool (self-exclusion beyond its length); strict
TOOLS = {
    "needle": dict(radius=0.005, length=0.3, self_excl=0.0, corr_radius=0.005, corr_length=0.7),
    "no_corridor": dict(corr_length=0.0, n_c=200),
    "long": dict(radius=0.05, length=0.9, corr_length=1.9, n_c=40),
    "empty_tool": dict(radius=0.01, length=0.02, self_excl=0.2),
    "strict": dict(strict=1, corr_length=0.3, n_c=3),
}


def _dirs():
    d = [[s * (k == a) for k in range(3)] for a in range(3) for s in (1.0, -1.0)]
    d += [[x, y, z] for x in (1, -1) for y in (1, -1) for z in (1, 0)]
    d = np.array(d, np.float64)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return np.concatenate([d.astype(np.float32), synth.fibonacci_dirs(23)])  # 37: a ragged group


@pytest.mark.parametrize("name", sorted(TOOLS))
@pytest.mark.parametrize("tight", [False, True])
@pytest.mark.parametrize("w_min", [0, 3, 1000])
def test_tables_at_their_edges(name, tight, w_min):
    import torch
    W = workload.single_frame()
    f = synth.cone_frame(W.scene, 3000, 0.01, 41)
    pts, nrm = synth.surface_points(f.world, f.normal, W.params["v"])
    pts, nrm = pts[::5], nrm[::5]
    if tight:    # a box that the kernels reach out of on every side
        W.dom_min, W.dom_bricks = (9, -4, -5), (8, 8, 10)
    W.params["w_min"] = w_min
    dirs = _dirs()
    g = af.Map(W.af_config(hash_capacity=1 << 14, pool_blocks=1 << 13, max_returns=4096,
                           max_points=4096))
    o = oracle.Map(oracle_config(W))
    for k in range(2):
        g.integrate_scan(to_dev(f.pts), f.pose)
        o.integrate(f.pts, f.pose)
    t = dict(W.tool(), **TOOLS[name])
    g.set_tool(af.ToolConfig(**t), dirs)
    inside = np.ones(len(pts), bool)
    if w_min == 0:   # points outside the box pass a gate of 0 as well
        idx = np.floor(pts.astype(np.float64) / np.float64(np.float32(W.params["v"]))).astype(int)
        lo = 8 * np.array(W.dom_min)
        inside = ((idx >= lo) & (idx < lo + 8 * np.array(W.dom_bricks))).all(1)
    pts, nrm = pts[inside], nrm[inside]
    lab, best = g.score(to_dev(pts), to_dev(nrm))
    torch.cuda.synchronize()
    ol, ob = o.score(oracle_tool(W, **TOOLS[name]), dirs, pts, nrm)
    assert g.sync_status() == 0
    np.testing.assert_array_equal(lab.cpu().numpy(), ol)
    np.testing.assert_array_equal(best.cpu().numpy(), ob)
    assert (ol == oracle.UNSCORED).all() == (w_min == 1000)
