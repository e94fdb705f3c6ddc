"""mp_gicp against the FP64 oracle at the sizes where its kernel can go wrong:
scans that end inside a tile of 64 target points, one scan much smaller than
the other, more source points than one round of the grid, every target point
twice (ties go to the smaller index), and a start too far for the last
iteration's correspondence to be the nearest point. A call whose buffers could
not be allocated leaves the context able to try again."""
import numpy as np
import pytest
from scipy.spatial.transform import Rotation

from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


def _T(rotvec, t):
    T = np.eye(4)
    T[:3, :3] = Rotation.from_rotvec(rotvec).as_matrix()
    T[:3, 3] = t
    return T


@pytest.mark.parametrize("n_src,n_tgt,twice,far", [(300, 2048, False, False), (2048, 321, False, False),
                                                   (450, 449, False, True), (512, 640, True, False),
                                                   (12000, 1500, False, False)])
def test_gicp_sizes(oracle, n_src, n_tgt, twice, far):
    from paper_2404_16370_gb300 import mp
    room = synth.box_room(1)
    params = mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, 1024)
    params.max_scan = 16384
    P = oracle.Params.box_room()
    motion = _T([0.02, -0.01, 0.04], [0.1, 0.06, -0.03])
    p0 = synth.box_room_gt_pose(room, 3)
    T1 = synth.pose_matrix(p0) @ motion
    s0 = synth.scan(room, p0, synth.spherical_dirs(n_tgt), 0.0, 1)
    s1 = synth.scan(room, synth.matrix_pose(T1), synth.spherical_dirs(n_src), 0.0, 2)
    if twice:
        s0 = np.concatenate([s0, s0])
    init = motion @ _T([0.0, 0.0, 0.1], [0.2, 0.0, 0.1]) if far else None
    c = mp.mp_init_map(room.map_points, params)
    try:
        g = mp.mp_gicp(c, s1, s0, init)
    finally:
        mp.mp_destroy(c)
    r = oracle.gicp(s1, s0, P, init)
    # a pair at the correspondence radius may fall on either side of it
    assert abs(g["n_corr"] - r["n_corr"]) <= 3 and r["n_corr"] > 50
    # FP32 sums of FP32 terms, each within a few 2^-24 of its value: the motion
    # and the Hessian follow to a few 1e-6 of their scale
    D = np.linalg.inv(g["T"]) @ r["T"]
    assert Rotation.from_matrix(D[:3, :3]).magnitude() < 1e-5 and np.linalg.norm(D[:3, 3]) < 1e-5
    assert np.abs(g["cov"] - r["cov"]).max() <= 1e-3 * np.abs(r["cov"]).max()


@pytest.mark.parametrize("which", [1, 2, 9, 13, 15])
def test_gicp_after_a_failed_allocation(which):
    """The knob makes one of the buffers' allocations fail: the call reports it,
    and the next one allocates all of them afresh and gives the same motion."""
    from paper_2404_16370_gb300 import mp
    room = synth.box_room(1)
    p0 = synth.box_room_gt_pose(room, 3)
    s0, s1 = (synth.scan(room, p0, synth.spherical_dirs(500), 0.02, k) for k in (1, 2))
    c, d = (mp.mp_init_map(room.map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, 64)) for _ in range(2))
    try:
        mp.mp_debug_set(c, mp.MP_DEBUG_FAIL_GICP_ALLOC, which)
        for _ in range(2):
            with pytest.raises(mp.MPError) as e:
                mp.mp_gicp(c, s1, s0)
            assert e.value.code == mp.MP_ENOMEM
        mp.mp_debug_set(c, mp.MP_DEBUG_FAIL_GICP_ALLOC, 0)
        a, b = mp.mp_gicp(c, s1, s0), mp.mp_gicp(d, s1, s0)
        assert np.array_equal(a["T"], b["T"]) and np.array_equal(a["cov"], b["cov"]) and a["n_corr"] == b["n_corr"]
    finally:
        mp.mp_destroy(c)
        mp.mp_destroy(d)
