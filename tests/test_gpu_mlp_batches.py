"""The network's gradient over batches of more tiles than resident CTAs (a CTA adds up several
tiles), at the smallest and largest numbers of sites, and its accumulation error."""
import numpy as np
import pytest

import ed_inputs
from oracle import basis as obasis
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


def _view(ptr, n):
    import torch

    class V:
        __cuda_array_interface__ = {"shape": (n,), "typestr": "<f4", "data": (ptr, False), "version": 3}
    return torch.as_tensor(V(), device="cuda")


class _Net:
    def __init__(self, L, nu, nd, seed):
        import torch
        import paper_1511_00863_gb300 as ed
        self.ed, self.L = ed, L
        self.b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
        self.up, self.dn = obasis.species_states(L, nu), obasis.species_states(L, nd)
        self.dim = ed.ed_basis_dims(self.b)[2]
        self.net = ed.ed_mlp_create(L, 7)
        self.P = omlp.param_count(L)
        self.params = (np.random.default_rng(seed).normal(size=self.P) * 0.2).astype(np.float32)
        _view(ed.ed_mlp_params(self.net)[0], self.P).copy_(torch.tensor(self.params))
        torch.cuda.synchronize()

    def grad(self, U, idx, target, scale):
        import torch
        loss, g = self.ed.ed_mlp_loss_grad(self.net, self.b, U, torch.as_tensor(idx, device="cuda"),
                                           torch.as_tensor(target, device="cuda"), scale)
        return loss, _view(g, self.P).double().cpu().numpy()

    def __enter__(self):
        return self

    def __exit__(self, *_):
        self.ed.ed_mlp_destroy(self.net)
        self.ed.ed_basis_destroy(self.b)


# 32 sites: 65 features, the U feature in a row of W1 and a column of the tile of its own
@pytest.mark.parametrize("L,nu,nd", [(6, 3, 2), (13, 2, 3), (32, 2, 1)])
@pytest.mark.parametrize("n", [63, 64, 65, 40001])
def test_gradient_of_many_tiles_vs_oracle(L, nu, nd, n):
    U = 3.0
    rng = np.random.default_rng(n)
    with _Net(L, nu, nd, 4) as N:
        idx = rng.integers(0, N.dim, size=n)
        target = rng.normal(size=n) * 0.05
        target[n // 2] = 0.0
        loss, g = N.grad(U, idx, target, 100.0)
        x = omlp.features(N.up[idx // len(N.dn)], N.dn[idx % len(N.dn)], L, U)
        L_ref, g_ref = omlp.loss_and_grad(N.params.astype(np.float64), x, target, 100.0, L)
        assert abs(loss - L_ref) <= 1e-5 * abs(L_ref)
        assert np.max(np.abs(g - g_ref)) <= 1e-4 * np.max(np.abs(g_ref)), np.max(np.abs(g - g_ref))


@pytest.mark.parametrize("L", [6, 32])
def test_accumulation_error_does_not_grow_with_the_samples(L):
    """2^22 equal samples: their mean gradient is that of one sample (1/n is a power of two), up to the
    rounding of the sums: 64 samples of a tile, the tiles of a CTA (65,536 over two CTAs per SM), the
    CTAs' sums in eight parts, 2^-24 each at most."""
    import torch
    n, U, scale = 1 << 22, 3.0, 50.0
    with _Net(L, 2, 1, 4) as N:
        one = N.grad(U, np.array([3]), np.array([0.04]), scale)[1]
        many = N.grad(U, np.full(n, 3), np.full(n, 0.04), scale)[1]
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    chain = 64 + -(-(n // 64) // ctas) + -(-ctas // 8) + 8
    assert np.count_nonzero(one) > 64 * 64
    assert np.all(np.abs(many - one) <= chain * 2.0**-24 * np.abs(one)), np.max(np.abs(many - one)[one != 0] / np.abs(one[one != 0]))
