"""Strict corridors (unknown voxels block) against the oracle, labels and
directions bit for bit: the nearest corridor entry is looked at with the arm
samples, so corridors of no entry, of one and of many, on maps whose space is
mostly unknown and mostly known, inside the box and beyond its faces, with the
search whole and shared out."""
import numpy as np
import pytest

import oracle
from parity import oracle_config, oracle_tool, to_dev
from paper_2608_06412_gb300 import af, synth, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("corr", [dict(corr_length=0.0), dict(corr_length=0.02, corr_radius=0.005),
                                  dict(corr_length=0.15), dict(corr_length=0.9)],
                         ids=["none", "one", "some", "many"])
@pytest.mark.parametrize("tight", [False, True])
@pytest.mark.parametrize("known", [False, True])
def test_strict_corridors(corr, tight, known):
    import torch
    W = workload.single_frame()
    if known:   # the band toward the sensor marks 60 cm of free space
        W.params.update(clear_samples=64, clear_hi=10.0)
    if tight:
        W.dom_min, W.dom_bricks = (9, -4, -5), (8, 8, 10)
    over = dict(strict=1, n_c=4, length=0.12, **corr)
    f = synth.cone_frame(W.scene, 6000, 0.01, 61)
    pts, nrm = synth.surface_points(f.world, f.normal, W.params["v"])
    pts, nrm = pts[::9], nrm[::9]
    g = af.Map(W.af_config(hash_capacity=1 << 15, pool_blocks=1 << 14, max_returns=1 << 13,
                           max_points=1 << 12))
    o = oracle.Map(oracle_config(W))
    for _ in range(3):
        g.integrate_scan(to_dev(f.pts), f.pose)
        o.integrate(f.pts, f.pose)
    dirs = synth.fibonacci_dirs(72)
    g.set_tool(af.ToolConfig(**dict(W.tool(), **over)), dirs)
    ol, ob = o.score(oracle_tool(W, **over), dirs, pts, nrm)
    for budget in (-1, 0, 3):
        g.set_score_split(budget)
        lab, best = g.score(to_dev(pts), to_dev(nrm))
        torch.cuda.synchronize()
        assert g.sync_status() == 0
        np.testing.assert_array_equal(lab.cpu().numpy(), ol)
        np.testing.assert_array_equal(best.cpu().numpy(), ob)
    assert (ol == 2).any()
