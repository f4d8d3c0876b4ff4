"""The network's inference at every layout of its features: 16, 32, 48, 64 and 80 operand columns (2 L + 1
features), the U feature first, in the middle and last of its group of eight, many tiles per CTA at 14
sites and 32 sites (the U feature behind all 64 bits)."""
import numpy as np
import pytest

import ed_inputs
from oracle import basis as obasis
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nu,nd", [(4, 2, 2), (7, 3, 3), (8, 4, 3), (11, 2, 4), (14, 5, 6), (15, 2, 4), (16, 3, 3),
                                     (19, 2, 3), (23, 2, 2), (24, 2, 3), (31, 2, 2), (32, 2, 2), (32, 31, 2)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_inference_against_oracle(L, nu, nd, dtype):
    """The oracle's forward pass rounds weights, U / 8 and h1 to bfloat16 as the kernel does. What is left:
    tanh's approximation (2^-10 relative with a factor 2), the bfloat16 rounding of an h1 off by that (one
    unit, 2^-8 relative), and FP32 sums (1e-5 of their terms)."""
    import torch
    import paper_1511_00863_gb300 as ed
    U = 2.5
    up, dn = obasis.species_states(L, nu), obasis.species_states(L, nd)
    b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
    net = ed.ed_mlp_create(L, 13)
    try:
        dim = ed.ed_basis_dims(b)[2]
        P = omlp.param_count(L)
        params = (np.random.default_rng(6).normal(size=P) * 0.2).astype(np.float32)

        class V:
            __cuda_array_interface__ = {"shape": (P,), "typestr": "<f4", "data": (ed.ed_mlp_params(net)[0], False), "version": 3}
        torch.as_tensor(V(), device="cuda").copy_(torch.tensor(params))
        out = torch.full((dim,), float("nan"), dtype=torch.float32 if dtype == "f32" else torch.float64, device="cuda")
        ed.ed_mlp_infer(net, b, U, out)
        got = out.double().cpu().numpy()
    finally:
        ed.ed_mlp_destroy(net)
        ed.ed_basis_destroy(b)
    assert np.all(np.isfinite(got))
    pick = np.unique(np.concatenate([np.random.default_rng(1).integers(0, dim, 20000), np.arange(min(dim, 300)),
                                     np.arange(max(0, dim - 300), dim)]))
    x = omlp.features(up[pick // len(dn)], dn[pick % len(dn)], L, U)
    a, z, (_, h1, h2) = omlp.forward(params, x, L)
    W1, b1, W2, b2, W3, b3 = (omlp.bf16_round(w) for w in omlp.unpack(params, L))
    f32, tanh, bf = 1e-5, 2.0**-10, 2.0**-8
    dh1 = f32 * (np.abs(x) @ np.abs(W1) + np.abs(b1)) + tanh * np.abs(h1)
    dh1 = dh1 + bf * np.abs(h1)
    dh2 = dh1 @ np.abs(W2) + f32 * (np.abs(h1) @ np.abs(W2) + np.abs(b2)) + tanh * np.abs(h2)
    d = dh2 @ np.abs(W3) + f32 * (np.abs(h2) @ np.abs(W3) + np.abs(b3))
    err = np.abs(np.log(np.abs(got[pick])) - a)
    assert np.all(err <= d[:, 0]), float(np.max(err / d[:, 0]))
    sure = np.abs(z) > d[:, 1]
    assert sure.mean() > 0.3 and np.all(np.sign(got[pick][sure]) == np.where(z[sure] >= 0, 1.0, -1.0))
