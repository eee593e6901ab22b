"""af_integrate_scan_noalloc (and the map path beside it) at the edges of their
tiles of returns and at several cube widths, against the oracle: one return, a
tile less one, one tile, one more, the scan sizes where the tile changes; cubes of 3, 9, 13 and 17 voxels (one and several offsets per thread);
dropped returns inside a tile; a box that cuts the cubes."""
import numpy as np
import pytest

import oracle
from parity import assert_maps_equal, gpu_voxels, oracle_config, oracle_voxels
from paper_2608_06412_gb300 import af, synth, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,radius", [(n, r) for n in (1, 3, 4, 5, 403, 3999, 4000, 4013)
                                      for r in (1, 4, 6, 8)] + [(39999, 2), (40003, 2)])
def test_box_tiles(radius, n):
    import torch
    W = workload.single_frame()
    over = dict(cube_radius=radius, w_cap=4)
    om = oracle.Map(oracle_config(W, **over))
    f = synth.cone_frame(W.scene, max(n, 450), 0.01, 23, origin=(0.0, 0.05, 0.0))
    pts = f.pts[:n].copy()
    if n > 5:
        pts[3] = np.nan          # dropped
        pts[5] = 1e-3            # too near
    box_min, box_dim = np.array([70, -22, -21]), np.array([63, 41, 37])
    count = int(np.prod(box_dim))
    vox = torch.zeros(count, dtype=torch.int64, device="cuda")
    flags = torch.zeros(count, dtype=torch.uint8, device="cuda")
    g = af.Map(W.af_config(**over, hash_capacity=1 << 14, pool_blocks=1 << 13, max_returns=1 << 16))
    for _ in range(2):
        g.integrate_scan(torch.from_numpy(pts).cuda(), f.pose)
        om.integrate(pts, f.pose)
        af.integrate_scan_noalloc(W.af_config(**over), torch.from_numpy(pts).cuda(), f.pose, box_min,
                                  box_dim, vox, flags)
    e = om.export()
    assert_maps_equal(gpu_voxels(g), oracle_voxels(om))
    rel = e["ijk"] - box_min
    ok = ((rel >= 0) & (rel < box_dim)).all(1)
    at = ((rel[:, 2] * box_dim[1] + rel[:, 1]) * box_dim[0] + rel[:, 0])[ok]
    want_v, want_f = np.zeros(count, np.int64), np.zeros(count, np.uint8)
    want_v[at] = (e["S"][ok].astype(np.int64) << 20) | e["w"][ok].astype(np.int64)
    want_f[at] = e["cleared"][ok] | (e["occ"][ok] << 1) | (e["known"][ok] << 2)
    assert n < 403 or (want_v != 0).sum() > 1000
    np.testing.assert_array_equal(vox.cpu().numpy(), want_v)
    np.testing.assert_array_equal(flags.cpu().numpy(), want_f)
