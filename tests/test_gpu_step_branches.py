"""A step, whose scan kernels run beside the particles' on a second stream,
against the same stages run one by one: the same lists and scan Gaussians, and
the same log-likelihoods up to the order of their sums. Scans change from step
to step, so that one read too early or too late would show."""
import numpy as np
import pytest

from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 700, 20000])
def test_step_equals_its_stages(n):
    from paper_2404_16370_gb300 import mp
    room = synth.box_room(1)
    gt = synth.box_room_gt_pose(room, 3)
    poses = synth.box_room_particles(n, 3, room.half)
    scans = [synth.scan(room, gt, synth.spherical_dirs(m), 0.02, m) for m in (1500, 40, 3000, 700)]
    ctx = [mp.mp_init_map(room.map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, n)) for _ in range(2)]
    try:
        for scan in scans:
            for c in ctx:
                mp.mp_init_particles(c, n, poses=poses)
            mp.mp_step(ctx[0], scan)
            mp.mp_set_scan(ctx[1], scan)
            mp.mp_set_odometry(ctx[1], None, None)
            for bit in range(1, 9):
                mp.mp_run_stages(ctx[1], 1 << bit)
            for w in (mp.MP_BUF_SCAN_NORMALS, mp.MP_BUF_SCAN_VALID):
                np.testing.assert_array_equal(mp.mp_get_buffer(ctx[0], w), mp.mp_get_buffer(ctx[1], w))
            a, b = (mp.mp_get_buffer(c, mp.MP_BUF_LOGLIK).astype(np.float64) for c in ctx)
            # FP32 sums of 3000 terms of one sign, in any order
            assert np.abs(a - b).max() <= 1e-4 * np.abs(a).max()
            ids = [mp.mp_get_buffer(c, mp.MP_BUF_NBR_IDS) for c in ctx]
            np.testing.assert_array_equal(*ids)
    finally:
        for c in ctx:
            mp.mp_destroy(c)
