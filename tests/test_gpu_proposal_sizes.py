"""The proposal network's outputs, loss and gradient against the FP64 oracle at
batches that end inside the tiles of the head's products (16 rows, 128 of K)
and of the pooled rows (64), and at scans of one point, one tile and more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,P", [(1, 1), (1, 128), (2, 384), (3, 2), (5, 1024), (17, 1), (64, 1), (129, 1), (133, 2)])
def test_network_sizes(B, P):
    import torch
    from oracle import proposal as PN
    from paper_2404_16370_gb300 import mp, proposal as PR
    rng = np.random.default_rng(100 * B + P)
    p = PN.init_params(5)
    k = 0
    for s in PN.SHAPES:
        m = int(np.prod(s))
        if len(s) == 1:
            p[k:k + m] = rng.normal(0, 0.1, m)
        k += m
    scans = rng.normal(0, 3.0, (B, P, 3)).astype(np.float32)
    y = np.concatenate([rng.normal(0, 1, (B, 3)), rng.uniform(-np.pi, np.pi, (B, 1)), rng.normal(0, 0.5, (B, 2))],
                       1).astype(np.float32)
    net = mp.mp_pn_create(P, B, PR.IN_SCALE, PR.SCALE, PR.OFFSET, seed=3)
    try:
        n = mp.mp_pn_num_params(net)
        mp.mp_pn_set_params(net, torch.tensor(p, dtype=torch.float32, device="cuda"))
        p32, o = torch.empty(n, device="cuda"), torch.empty((B, mp.MP_PN_OUT), device="cuda")
        mp.mp_pn_get_params(net, p32)
        xs, ys = torch.tensor(scans, device="cuda"), torch.tensor(y, device="cuda")
        loss, grad = torch.zeros(1, device="cuda"), torch.empty(n, device="cuda")
        mp.mp_pn_forward(net, xs, o)
        mp.mp_pn_loss_grad(net, xs, ys, loss, grad)
        mp.mp_pn_status(net)
        o, grad, p64 = o.cpu().numpy(), grad.cpu().numpy(), p32.cpu().numpy().astype(np.float64)
    finally:
        mp.mp_pn_destroy(net)
    form = P % 128 == 0   # the tensor-core form's roundings, else plain FP32
    ref = PN.forward(p64, scans.astype(np.float64), PR.IN_SCALE, bf16_form=form)
    L_ref, g_ref = PN.loss_grad(p64, scans.astype(np.float64), y.astype(np.float64), PR.IN_SCALE, bf16_form=form)
    # FP32 sums of at most 416 terms, and of the pooled rows for the gradients:
    # sqrt(416 * 256 * 133) 2^-24 of the terms' scale at the most
    assert np.abs(o - ref["o"]).max() <= 1e-5 * max(1.0, np.abs(ref["o"]).max())
    assert abs(float(loss.item()) - L_ref) <= 1e-5 * max(1.0, abs(L_ref))
    k = 0
    for s in PN.SHAPES:
        m = int(np.prod(s))
        gb, rb = grad[k:k + m], g_ref[k:k + m]
        assert np.linalg.norm(gb - rb) <= 1e-4 * (np.linalg.norm(rb) + 1e-12), s
        k += m
