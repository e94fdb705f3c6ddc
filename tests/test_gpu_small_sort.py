"""The one-CTA sort of instances of at most 16384 particles against the general
one's definition: the stable bucket order, ranks and segments, and the visiting
order, at the edges of its rows of 1024 and with one, two and four radix passes."""
import numpy as np
import pytest

from gpu_util import visit_order
from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 4096, 15360, 16383, 16384, 16385])
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
