"""The row-ordered H.v's tables, sorted on the device: the longest rows (24,310 and 27,132 columns, not
multiples of 32), 16 amplitude classes (the most) and 17 (none of these tables), equal counts everywhere
(a complete graph: the order is the ranks') and hardly any hops, against the oracle."""
import itertools

import numpy as np
import pytest

import ed_inputs
from oracle import complex_hopping as ch
from oracle import hamiltonian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nu,nd", [(17, 2, 8), (19, 2, 6)])
def test_longest_rows(L, nu, nd):
    import torch
    import paper_1511_00863_gb300 as ed
    bonds, t, U = ed_inputs.ring_bonds(L), 0.7, 1.9
    b = ed.ed_build_basis(L, bonds, nu, nd)
    try:
        dim = ed.ed_basis_dims(b)[2]
        x = torch.tensor(ed_inputs.uniform_pm1(3, dim), dtype=torch.float32, device="cuda")
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, t, U, x, y)
        got, xr = y.cpu().numpy(), x.cpu().numpy().astype(np.float64)
    finally:
        ed.ed_basis_destroy(b)
    assert np.all(np.isfinite(got))
    pick = np.random.default_rng(2).integers(0, dim, 100000)
    want = hamiltonian.hv_rows(L, bonds, nu, nd, t, U, xr, pick)
    scale = hamiltonian.hv_abs_rows(L, bonds, nu, nd, t, U, xr, pick)
    assert np.all(np.abs(got[pick] - want) <= 4 * (2 * L + 2) * 2.0**-24 * scale + 1e-300)


@pytest.mark.parametrize("classes", [1, 5, 16, 17])
@pytest.mark.parametrize("nu,nd", [(2, 3), (3, 2)])
def test_amplitude_classes(classes, nu, nd):
    import torch
    import paper_1511_00863_gb300 as ed
    L, t, U = 16, 0.7, 1.9
    bonds = np.array(list(itertools.combinations(range(L), 2)), dtype=np.int32)
    amp = 1.0 + 0.1 * np.arange(classes)  # real: an amplitude and its conjugate are one class
    tb = amp[np.random.default_rng(classes).permutation(len(bonds)) % classes] * np.where(np.arange(len(bonds)) % 3, 1, -1)
    b = ed.ed_build_basis(L, bonds, nu, nd, t_bond=tb)
    try:
        dim = ed.ed_basis_dims(b)[2]
        raw = ed_inputs.uniform_pm1(5, 2 * dim)
        x = torch.tensor(raw[0::2] + 1j * raw[1::2], device="cuda")
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, t, U, x, y)
        got, xr = y.cpu().numpy(), x.cpu().numpy()
    finally:
        ed.ed_basis_destroy(b)
    H = ch.hamiltonian_csr_complex(L, bonds, tb, nu, nd, t, U)
    bound = 4 * (2 * len(bonds) + 2) * 2.0**-53 * (abs(H) @ np.abs(xr)) + 1e-300
    assert np.all(np.abs(got - H @ xr) <= bound)


@pytest.mark.parametrize("bonds", [[], [(0, 1)], [(0, 15), (3, 4), (4, 3)]])
def test_few_hops(bonds):
    import torch
    import paper_1511_00863_gb300 as ed
    L, nu, nd, t, U = 16, 2, 3, 0.7, 1.9
    bonds = np.array(bonds, dtype=np.int32).reshape(-1, 2)
    b = ed.ed_build_basis(L, bonds, nu, nd)
    try:
        dim = ed.ed_basis_dims(b)[2]
        x = torch.tensor(ed_inputs.uniform_pm1(6, dim), device="cuda")
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, t, U, x, y)
        got, xr = y.cpu().numpy(), x.cpu().numpy()
    finally:
        ed.ed_basis_destroy(b)
    pick = np.arange(dim)
    want = hamiltonian.hv_rows(L, bonds, nu, nd, t, U, xr, pick)
    scale = hamiltonian.hv_abs_rows(L, bonds, nu, nd, t, U, xr, pick)
    assert np.all(np.abs(got - want) <= 4 * (2 * len(bonds) + 2) * 2.0**-53 * scale + 1e-300)
