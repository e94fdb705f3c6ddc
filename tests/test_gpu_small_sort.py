"""The sorts of an instance (one CTA, one cooperative launch of a CTA per 1024
particles, radix passes as launches) against their definition: the stable bucket
order, ranks and segments, and the visiting order, at the edges of their ranges
and tiles and with one, two and four radix passes."""
import numpy as np
import pytest

from gpu_util import visit_order
from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 3584, 3585, 5120, 16385, 100001, 155648, 155649, 400001, 1245185])
@pytest.mark.parametrize("bits", [1, 8, 13, 26])
def test_small_sort(n, bits):
    from paper_2404_16370_gb300 import mp
    room = synth.box_room(1)
    poses = synth.box_room_particles(n, 3)
    p = mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, n, n_buckets_log2=bits)
    ctx = mp.mp_init_map(room.map_points, p)
    try:
        mp.mp_init_particles(ctx, n, poses=poses)
        mp.mp_set_step_index(ctx, 5)
        mp.mp_run_stages(ctx, mp.MP_STAGE_LSH | mp.MP_STAGE_SORT)
        b = mp.mp_get_buffer(ctx, mp.MP_BUF_BUCKETS)
        ids = mp.mp_get_buffer(ctx, mp.MP_BUF_SORTED_IDS)
        seg = mp.mp_get_buffer(ctx, mp.MP_BUF_SEGMENTS)
        visit = mp.mp_get_buffer(ctx, mp.MP_BUF_VISIT_ORDER)
        info = mp.mp_map_info(ctx)
    finally:
        mp.mp_destroy(ctx)
    assert np.array_equal(ids, np.argsort(b, kind="stable"))
    sb = b[ids]
    assert np.array_equal(seg[:, 0], np.searchsorted(sb, b, "left"))
    assert np.array_equal(seg[:, 1], np.searchsorted(sb, b, "right"))
    assert np.array_equal(visit, visit_order(ids, poses[:, 4:7], info))
