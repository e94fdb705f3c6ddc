"""Scan point Gaussians against the FP64 oracle where a normal's covariance can go
wrong: neighbourhoods from the smallest allowed to the largest, coincident
points, points on a line and on a plane, and a last warp with one point."""
import numpy as np
import pytest

from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kmin,k", [(3, 3), (3, 16), (5, 10), (16, 16)])
def test_scan_normals(oracle, kmin, k):
    from paper_2404_16370_gb300 import mp
    params = mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, 256)
    params.cov_min, params.cov_k = kmin, k
    rng = np.random.default_rng(kmin * 100 + k)
    r = params.r_cov
    blobs = [np.array([3.0 * b, 0, 0]) + 0.2 * r * rng.standard_normal((m, 3)) for b, m in enumerate(range(1, 19))]
    plane = np.array([0, 50.0, 0]) + np.c_[r * rng.random((60, 2)), np.zeros(60)]
    line = np.array([0, 80.0, 0]) + np.outer(0.1 * r * np.arange(12), [1.0, 0, 0])
    same = np.repeat([[0, 110.0, 1.0]], 20, 0)
    pts = np.concatenate(blobs + [plane, line, same]).astype(np.float32)
    pts = np.concatenate([pts, pts[:1] + 500.0])[: 8 * (len(pts) // 8) + 1]
    room = synth.box_room(1)
    c = mp.mp_init_map(room.map_points, params)
    try:
        mp.mp_init_particles(c, 256, poses=synth.box_room_particles(256, 3, room.half))
        mp.mp_set_scan(c, pts)
        mp.mp_run_stages(c, mp.MP_STAGE_SCAN)
        normals, valid = mp.mp_get_buffer(c, mp.MP_BUF_SCAN_NORMALS), mp.mp_get_buffer(c, mp.MP_BUF_SCAN_VALID)
    finally:
        mp.mp_destroy(c)
    ref, rvalid, _, covs = oracle.point_normals(pts, params.r_cov, k, kmin, want_covs=True)
    np.testing.assert_array_equal(valid, rvalid)
    lam = np.linalg.eigvalsh(covs.reshape(-1, 3, 3))
    gap = (lam[:, 1] - lam[:, 0]) / np.maximum(lam[:, 2], 1e-300)
    good = (rvalid > 0) & (gap > 1e-4)
    assert good.sum() > 60
    # both in FP64, rounded to float; the eigenvector moves by 2^-52 over the gap
    assert np.abs(normals[good] - ref[good]).max() < 2e-7
    assert np.all(np.isfinite(normals)) and np.all(normals[rvalid == 0] == 0)
