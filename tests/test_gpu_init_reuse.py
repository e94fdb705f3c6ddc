"""Particles set again in a context that has stepped: as many (its buffers are
kept), more and fewer. The state is the one a fresh context starts from, and
poses go in and out of host and device memory alike; a device buffer that ends
beyond its allocation is refused; a refused call leaves the particles as they
were, and one that fails half-way leaves none."""
import ctypes as C

import numpy as np
import pytest

from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


def test_particles_set_again_start_afresh():
    import torch
    from paper_2404_16370_gb300 import mp
    room = synth.box_room(1)
    params = mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, 1000)
    scan = synth.scan(room, synth.box_room_gt_pose(room, 3), synth.spherical_dirs(300), 0.02, 1)
    which = [mp.MP_BUF_NBR_IDS, mp.MP_BUF_NBR_K, mp.MP_BUF_NBR_D, mp.MP_BUF_SORTED_IDS, mp.MP_BUF_VISIT_ORDER,
             mp.MP_BUF_LOGLIK, mp.MP_BUF_PSI, mp.MP_BUF_PHI, mp.MP_BUF_LOG_PRIOR, mp.MP_BUF_POSES]
    c = mp.mp_init_map(room.map_points, params)
    try:
        for n in (1000, 1000, 37, 2049, 2049):
            p = synth.box_room_particles(n, n, room.half).astype(np.float32)
            for poses in (p, torch.tensor(p, device="cuda")):
                mp.mp_init_particles(c, n, poses=poses)
                got = {w: mp.mp_get_buffer(c, w) for w in which}
                f = mp.mp_init_map(room.map_points, params)
                try:
                    mp.mp_init_particles(f, n, poses=p)
                    for w in which:
                        np.testing.assert_array_equal(got[w], mp.mp_get_buffer(f, w), err_msg=str(w))
                finally:
                    mp.mp_destroy(f)
                np.testing.assert_array_equal(got[mp.MP_BUF_POSES].reshape(n, 7), p)
                assert np.array_equal(got[mp.MP_BUF_SORTED_IDS], np.arange(n))
                ids = got[mp.MP_BUF_NBR_IDS].reshape(n, -1)
                assert np.array_equal(ids[:, 0], np.arange(n)) and np.all(ids[:, 1:] == -1)
                mp.mp_step(c, scan)
                on_device = torch.empty((n, 7), device="cuda")
                on_host = np.empty((n, 7), np.float32)
                mp.mp_get_posterior(c, poses_out=on_device)
                best, prob = mp.mp_get_posterior(c, poses_out=on_host)
                assert np.array_equal(on_device.cpu().numpy(), on_host) and not np.array_equal(on_host, p)
                assert np.any(np.all(on_host == best, 1)) and 0 < prob <= 1
    finally:
        mp.mp_destroy(c)


def test_device_buffers_beyond_their_allocation_are_refused():
    """Poses, probabilities and sums go straight to device memory by a kernel:
    where the caller's allocation is too short for them the call is refused, as
    the copy of the same size is, and the context goes on."""
    import torch
    from paper_2404_16370_gb300 import mp
    torch.zeros(1, device="cuda")
    cu, L = C.CDLL("libcuda.so.1"), mp.lib()
    room = synth.box_room(1)
    n = 300
    p = synth.box_room_particles(n, 3, room.half).astype(np.float32)
    c = mp.mp_init_map(room.map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, n))

    def alloc(count):
        d = C.c_uint64()
        assert cu.cuMemAlloc_v2(C.byref(d), C.c_size_t(count)) == 0
        return d

    short, whole = alloc(1024), alloc(29 * 4 * n)
    try:
        mp.mp_init_particles(c, n, poses=p)
        calls = {"posterior": lambda d: L.mp_get_posterior(c, C.c_void_p(d), None, None, None),
                 "probabilities": lambda d: L.mp_get_posterior(c, None, C.c_void_p(d), None, None),
                 "poses": lambda d: L.mp_get_buffer(c, mp.MP_BUF_POSES, C.c_void_p(d), C.c_int64(7 * n)),
                 "sums": lambda d: L.mp_get_buffer(c, mp.MP_BUF_GN, C.c_void_p(d), C.c_int64(29 * n)),
                 "set": lambda d: L.mp_set_buffer(c, mp.MP_BUF_POSES, C.c_void_p(d), C.c_int64(7 * n))}
        for name, call in calls.items():
            assert call(short.value) == mp.MP_ECUDA, name
            assert "beyond its device allocation" in mp.mp_last_error(c), name
            assert call(whole.value + 29 * 4 * n - 1024) == mp.MP_ECUDA, name     # in the middle of one
        for name in ("sums", "probabilities", "posterior", "poses", "set"):      # the last: what "poses" wrote
            assert calls[name](whole.value) == mp.MP_OK, name
        end = whole.value + (29 - 7) * 4 * n                                     # up to the allocation's last byte
        assert calls["poses"](end) == mp.MP_OK and calls["set"](end) == mp.MP_OK
        np.testing.assert_array_equal(mp.mp_get_buffer(c, mp.MP_BUF_POSES).reshape(n, 7), p)
    finally:
        mp.mp_destroy(c)
        for d in (short, whole):
            cu.cuMemFree_v2(C.c_uint64(d.value))


def test_refused_and_failed_initialisation():
    import torch
    from paper_2404_16370_gb300 import mp
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    room = synth.box_room(1)
    n = 300
    p = synth.box_room_particles(n, 3, room.half).astype(np.float32)
    scan = synth.scan(room, synth.box_room_gt_pose(room, 3), synth.spherical_dirs(300), 0.02, 1)
    c = mp.mp_init_map(room.map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, n))
    short = C.c_uint64()
    assert cu.cuMemAlloc_v2(C.byref(short), C.c_size_t(1024)) == 0
    try:
        mp.mp_init_particles(c, n, poses=p)
        with pytest.raises(mp.MPError) as e:
            mp.mp_init_particles(c, 2 * n, lo=np.ones(6, np.float32), hi=np.zeros(6, np.float32))
        assert e.value.code == mp.MP_EINVAL
        np.testing.assert_array_equal(mp.mp_get_buffer(c, mp.MP_BUF_POSES).reshape(-1, 7), p)
        mp.mp_step(c, scan)
        mp.mp_get_posterior(c)
        assert mp.lib().mp_init_particles(c, 2 * n, None, None, C.c_void_p(short.value), None) == mp.MP_ECUDA
        with pytest.raises(mp.MPError) as e:
            mp.mp_step(c, scan)
        assert e.value.code == mp.MP_ENOTINIT
        mp.mp_init_particles(c, n, poses=p)
        mp.mp_step(c, scan)
        best, prob = mp.mp_get_posterior(c)
        assert np.isfinite(best).all() and 0 < prob <= 1
    finally:
        mp.mp_destroy(c)
        cu.cuMemFree_v2(short)
