"""The posterior stage's forms against the oracle's Eq. 11: one CTA (no grid
barrier), one cluster (129 to 1024 particles), blocks of 128 and of 256
particles with lists of at most 16 and 32 entries held in registers, and lists
read by every sweep when the particle blocks outnumber the resident CTAs."""
import numpy as np
import pytest

from paper_2404_16370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,iters", [(1, 4, 3), (128, 16, 10), (129, 32, 3), (256, 16, 10), (257, 5, 0), (700, 16, 9), (1024, 32, 10), (1025, 16, 2), (3001, 17, 9), (38000, 32, 2),
                                       (40001, 32, 3), (79001, 16, 3), (300, 16, 10), (19456, 32, 3), (19457, 16, 3)])
def test_posterior_forms(oracle, n, K, iters):
    from paper_2404_16370_gb300 import mp
    rng = np.random.default_rng(n + K)
    ids = rng.integers(0, n, (n, K)).astype(np.int32)
    ids[rng.random((n, K)) < 0.3] = -1
    ids[:, 0] = np.arange(n)
    kk = rng.uniform(0.05, 1.0, (n, K)).astype(np.float32)
    kk[n // 3] = 0                                   # no weight at all: the particle keeps its value
    loglik = (-rng.uniform(0, 80, n)).astype(np.float32)
    logprior = -rng.uniform(0, 5, n)
    room = synth.box_room(1)
    poses = synth.box_room_particles(n, 3)
    ctx = mp.mp_init_map(room.map_points, mp.mp_default_params(mp.MP_PRESET_BOX_ROOM, n, K=K, post_iters=iters))
    try:
        mp.mp_init_particles(ctx, n, poses=poses)
        mp.mp_set_buffer(ctx, mp.MP_BUF_NBR_IDS, ids)
        mp.mp_set_buffer(ctx, mp.MP_BUF_NBR_K, kk)
        mp.mp_set_buffer(ctx, mp.MP_BUF_LOGLIK, loglik)
        mp.mp_set_buffer(ctx, mp.MP_BUF_LOG_PRIOR, logprior)
        mp.mp_run_stages(ctx, mp.MP_STAGE_POSTERIOR)
        post = mp.mp_get_buffer(ctx, mp.MP_BUF_POST)
        best, best_p = mp.mp_get_posterior(ctx)
    finally:
        mp.mp_destroy(ctx)
    _, p_ref, b_ref = oracle.posterior(logprior, loglik.astype(np.float64), ids, kk.astype(np.float64), iters,
                                       oracle.Params().post_floor)
    # FP64 sums of at most n terms
    assert np.allclose(post, p_ref, rtol=1e-10, atol=1e-300)
    assert np.array_equal(best, poses[b_ref]) and abs(best_p - p_ref[b_ref]) < 1e-12
