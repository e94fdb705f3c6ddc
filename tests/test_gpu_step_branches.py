"""A step, whose scan kernels run beside the particles' on a second stream,
against the same stages run one by one: the same lists and scan Gaussians, and
the same log-likelihoods up to the order of their sums. Scans change from step
to step, so that one read too early or too late would show. The second stream
has the priority of the caller's."""
import ctypes as C

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


@pytest.mark.parametrize("priority", [0, -1, -3])
def test_every_kernel_has_the_callers_priority(priority):
    """The stages captured into a graph (not run): each kernel node carries the
    priority of the stream that it was launched on."""
    import torch
    from paper_2404_16370_gb300 import mp
    stream = torch.cuda.Stream(priority=priority)
    cu, s = C.CDLL("libcuda.so.1"), C.c_void_p(stream.cuda_stream)
    room = synth.box_room(1)
    c = mp.mp_init_map(room.map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, 500), cuda_stream=stream.cuda_stream)
    graph = C.c_void_p()
    try:
        mp.mp_init_particles(c, 500, poses=synth.box_room_particles(500, 3, room.half))
        mp.mp_set_scan(c, synth.scan(room, synth.box_room_gt_pose(room, 3), synth.spherical_dirs(300), 0.02, 1))
        torch.cuda.synchronize()
        assert cu.cuStreamBeginCapture_v2(s, 2) == 0
        try:
            mp.mp_run_stages(c, mp.MP_STAGE_SCAN | mp.MP_STAGE_MERGE | mp.MP_STAGE_LIKELIHOOD)
        finally:
            assert cu.cuStreamEndCapture(s, C.byref(graph)) == 0
        count = C.c_size_t()
        assert cu.cuGraphGetNodes(graph, None, C.byref(count)) == 0
        nodes = (C.c_void_p * count.value)()
        assert cu.cuGraphGetNodes(graph, nodes, C.byref(count)) == 0
        got = []
        for node in nodes:
            kind, value = C.c_int(), (C.c_int * 16)()
            assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
            if kind.value == 0:   # a kernel; its attribute 8 is the priority
                assert cu.cuGraphKernelNodeGetAttribute(C.c_void_p(node), 8, value) == 0
                got.append(value[0])
    finally:
        mp.mp_destroy(c)
        if graph:
            cu.cuGraphDestroy(graph)
    assert len(got) == 5 and set(got) == {stream.priority}   # three of the scan, merge, likelihood
