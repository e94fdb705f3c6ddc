"""Particles set again in a context that has stepped: as many (its buffers are
kept), more and fewer. The state is the one a fresh context starts from, and
poses go in and out of host and device memory alike."""
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
