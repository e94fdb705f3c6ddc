"""The likelihood's two forms: point-major (a warp, or four, per particle; the
scan in parts of up to 1536 staged points, looked up 256 or 64 at a time and
queued in groups of 64) at the edges of those sizes, against the oracle; and
particle-major (many particles on a small map) against point-major, in every
precision. The scan that is read is the one prepared last, and the staged slots
beyond its points count for no pose."""
import numpy as np
import pytest

from gpu_util import check_sums
from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def room(oracle):
    w = synth.box_room_workload(n_particles=8192)
    scan = synth.scan(w.scene, w.gt[0], synth.spherical_dirs(3200), 0.02, 7)
    P = oracle.Params.box_room(4096)
    return dict(w=w, om=oracle.OracleMap(w.map_points, P), P=P, scan=scan)


def sums(room, poses, scan, precision=0):
    from paper_2404_16370_gb300 import mp
    n = len(poses)
    ctx = mp.mp_init_map(room["w"].map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, n))
    try:
        mp.mp_set_precision(ctx, precision)
        mp.mp_init_particles(ctx, n, poses=poses)
        mp.mp_set_scan(ctx, scan)
        mp.mp_run_stages(ctx, mp.MP_STAGE_SCAN | mp.MP_STAGE_LIKELIHOOD)
        return mp.mp_get_buffer(ctx, mp.MP_BUF_GN), mp.mp_get_buffer(ctx, mp.MP_BUF_SCAN_VALID)
    finally:
        mp.mp_destroy(ctx)


@pytest.mark.parametrize("n", [2, 1024, 1025])      # four warps a particle up to 1024, one beyond
@pytest.mark.parametrize("m", [64, 65, 255, 256, 257, 1536, 1537, 3200])
def test_point_major_sizes(room, oracle, n, m):
    # the densest part of the scan first, so that its points are valid and the
    # parts are full: m points are m staged points
    order = np.argsort(np.linalg.norm(room["scan"], axis=1), kind="stable")
    sc = np.ascontiguousarray(room["scan"][order][:m])
    gn, valid = sums(room, room["w"].particles[:n], sc)
    P = room["P"]
    sn, sv, _, _ = oracle.point_normals(sc, P.r_cov, P.cov_k, P.cov_min)
    assert np.array_equal(valid.astype(bool), sv.astype(bool))
    ref = oracle.likelihood(room["om"], room["w"].particles[:n], sc, sn, sv, P, amb_tol=1e-4)
    msg = check_sums(gn, ref)
    assert not msg, msg


def test_scan_order_changes_only_the_rounding(room):
    """The scan stage sorts the valid points: any input order of the same
    points gives the same sums up to FP32 rounding, and the same inliers."""
    poses = room["w"].particles[:1500]
    a, va = sums(room, poses, room["scan"][:1100])
    perm = np.random.default_rng(1).permutation(1100)
    b, vb = sums(room, poses, np.ascontiguousarray(room["scan"][:1100][perm]))
    assert np.array_equal(va[perm], vb)
    assert np.array_equal(a[:, 28], b[:, 28])
    assert np.all(np.abs(a - b) <= 2e-5 * (np.abs(a).max(axis=0, keepdims=True) + 1e-6))


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n,m", [(81920, 129), (82001, 700)])
def test_particle_major_equals_point_major(room, precision, n, m):
    """The same pairs with the same arithmetic, summed in another order: equal
    inliers, and sums within 1100 roundings of FP32 (6e-8 each) of their
    largest, 2e-5 with the cancellation between terms."""
    poses = np.tile(room["w"].particles, (n // 8192 + 1, 1))[:n]
    sc = np.ascontiguousarray(room["scan"][:m])
    pm, _ = sums(room, poses, sc, precision)
    pt, _ = sums(room, poses[:1500], sc, precision)
    assert np.array_equal(pm[:1500, 28], pt[:, 28])
    assert np.all(np.abs(pm[:1500] - pt) <= 2e-5 * (np.abs(pt).max(axis=0, keepdims=True) + 1e-6))
    assert np.array_equal(pm[:8192], pm[8192:16384])        # the same poses in other slots, to the last particle
    assert np.array_equal(pm[n - 1], pm[(n - 1) % 8192])


@pytest.mark.parametrize("n,precision", [(600, 0), (1500, 0), (1500, 1), (82001, 0), (82001, 1)])
def test_likelihood_reads_the_prepared_scan(room, n, precision):
    """A scan that is set but not prepared changes no sums: the likelihood
    reads the one the scan stage prepared last, all of it, though the new one
    is shorter."""
    from paper_2404_16370_gb300 import mp
    poses = np.tile(room["w"].particles, (11, 1))[:n]
    ctx = mp.mp_init_map(room["w"].map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, n))
    try:
        mp.mp_set_precision(ctx, precision)
        mp.mp_init_particles(ctx, n, poses=poses)
        mp.mp_set_scan(ctx, room["scan"])
        mp.mp_run_stages(ctx, mp.MP_STAGE_SCAN | mp.MP_STAGE_LIKELIHOOD)
        want = mp.mp_get_buffer(ctx, mp.MP_BUF_GN)
        mp.mp_set_scan(ctx, room["scan"][:20])
        mp.mp_run_stages(ctx, mp.MP_STAGE_LIKELIHOOD)
        np.testing.assert_array_equal(mp.mp_get_buffer(ctx, mp.MP_BUF_GN), want)
    finally:
        mp.mp_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("m", [9, 129])
def test_unused_slots_count_for_no_pose(room, precision, m):
    """The staged chunk's slots beyond the valid points stay outside the grid
    also for a stored quaternion that is not a unit one: (0.5, -0.5, 0, 0) maps
    (1, 1, 1) to 0, so the slot would land on the particle itself."""
    poses = np.zeros((82001, 7), np.float32)
    poses[:, :2] = 0.5, -0.5
    poses[:, 4:] = np.resize(room["w"].map_points, (82001, 3))
    order = np.argsort(np.linalg.norm(room["scan"], axis=1), kind="stable")
    sc = np.ascontiguousarray(room["scan"][order][:m])
    pm, valid = sums(room, poses, sc, precision)                # particle-major: the valid points alone
    for n in (600, 1500):
        pt, _ = sums(room, poses[:n], sc, precision)
        assert np.array_equal(pm[:n, 28], pt[:, 28]) and pt[:, 28].max() <= valid.sum()
        # the cost: 129 terms of one sign, each sum within 129 roundings of FP32 (6e-8)
        # (the other sums cancel under this rotation to their rounding)
        assert np.all(np.abs(pm[:n, 27] - pt[:, 27]) <= 2e-5 * np.abs(pt[:, 27]).max())


@pytest.fixture(scope="module")
def wide(room, oracle):
    """The room on a map of more than 512 voxels across (two far patches)."""
    y, z = np.meshgrid(0.1 * np.arange(5), 0.1 * np.arange(5))
    far = [np.c_[np.full(25, x), y.ravel(), z.ravel()] for x in (-30.0, 30.0)]
    pts = np.concatenate([room["w"].map_points, *far]).astype(np.float32)
    return dict(room, w=type("W", (), dict(map_points=pts, particles=room["w"].particles)),
                om=oracle.OracleMap(pts, room["P"]))


@pytest.mark.parametrize("n", [1, 127, 129, 1025])
@pytest.mark.parametrize("m", [40, 41, 127, 128, 129, 133, 700])
def test_wide_map_one_particle_a_thread(wide, oracle, n, m):
    # the densest part of the scan: m points are m staged points, in groups of four and chunks of 128
    order = np.argsort(np.linalg.norm(wide["scan"], axis=1), kind="stable")
    sc = np.ascontiguousarray(wide["scan"][order][:m])
    gn, valid = sums(wide, wide["w"].particles[:n], sc)
    P = wide["P"]
    sn, sv, _, _ = oracle.point_normals(sc, P.r_cov, P.cov_k, P.cov_min)
    assert np.array_equal(valid.astype(bool), sv.astype(bool))
    ref = oracle.likelihood(wide["om"], wide["w"].particles[:n], sc, sn, sv, P, amb_tol=1e-4)
    msg = check_sums(gn, ref)
    assert not msg, msg


def test_wide_map_sums_keep_their_bits(wide):
    """One particle a thread (up to 114688), pairs, and parts of the scan: the
    same sums, bit for bit."""
    poses = np.tile(wide["w"].particles, (16, 1))
    sc = np.ascontiguousarray(wide["scan"][:700])
    one, _ = sums(wide, poses[:8192], sc)
    for n in (114688, 114689, 131072):
        many, _ = sums(wide, poses[:n], sc)
        assert np.array_equal(many[:8192], one) and np.array_equal(many[n - 1], one[(n - 1) % 8192])
