"""The row-ordered H.v (rows that fit in shared memory twice, at least 64 of them and 96 columns)
against the oracle: odd and even row lengths (wide and single loads), up lists longer than a
warp, amplitude classes (few: summed by class; all different: the plain kernels), sign flips
between equal amplitudes, and the Lanczos-fused form."""
import numpy as np
import pytest

import ed_inputs
from oracle import complex_hopping as ch
from oracle import hamiltonian
from oracle import lanczos as olz

pytestmark = pytest.mark.gpu

# sites, up, down -> rows x columns: 105 x 105, 91 x 1001, 165 x 462, 66 x 495, 286 x 78 (short
# rows: not this kernel), 120 x 210
SIZES = [(15, 2, 2), (14, 2, 4), (11, 3, 5), (12, 2, 4), (13, 3, 2), (10, 3, 4)]
EPS = {"f64": 2.0**-53, "f32": 2.0**-24, "c64": 2.0**-53, "c32": 2.0**-24}


def _bonds(L, n, seed):
    r = np.random.default_rng(seed)
    return np.array([r.permutation(L)[:2] for _ in range(n)], dtype=np.int32)


def _amplitudes(kind, n):
    r = np.random.default_rng(3)
    if kind == "few":
        v = np.exp(0.7j)
        return np.array([1.0, -1.0, 1.0j, v, -v, np.conj(v), 0.3])[r.integers(0, 7, n)]
    return r.uniform(0.5, 1.5, n) * np.exp(1j * r.uniform(-3, 3, n)) if kind == "many" else None


@pytest.mark.parametrize("L,nu,nd", SIZES)
@pytest.mark.parametrize("dtype,kind", [("f64", None), ("f32", None), ("c64", None), ("c64", "few"), ("c32", "few"),
                                        ("c64", "many"), ("c32", "many")])
def test_hv_against_oracle(L, nu, nd, dtype, kind):
    import torch
    import paper_1511_00863_gb300 as ed
    bonds = _bonds(L, 60, L)
    tb = _amplitudes(kind, len(bonds))
    b = ed.ed_build_basis(L, bonds, nu, nd, t_bond=tb)
    try:
        dim = ed.ed_basis_dims(b)[2]
        cx = dtype[0] == "c"
        raw = ed_inputs.uniform_pm1(17, 2 * dim)
        x = torch.tensor(raw[0::2] + 1j * raw[1::2] if cx else raw[:dim],
                         dtype={"f64": torch.float64, "f32": torch.float32, "c64": torch.complex128,
                                "c32": torch.complex64}[dtype], device="cuda")
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, 0.7, 1.9, x, y)
        got, xr = y.cpu().numpy(), x.cpu().numpy().astype(np.complex128 if cx else np.float64)
    finally:
        ed.ed_basis_destroy(b)
    H = ch.hamiltonian_csr_complex(L, bonds, np.ones(len(bonds)) if tb is None else tb, nu, nd, 0.7, 1.9) if cx \
        else hamiltonian.hamiltonian_csr(L, bonds, nu, nd, 0.7, 1.9)
    bound = 4 * (2 * len(bonds) + 2) * EPS[dtype] * (abs(H) @ np.abs(xr)) + 1e-300
    assert np.all(np.abs(got - H @ xr) <= bound)


@pytest.mark.parametrize("dtype,kind", [("c64", "few"), ("c64", "many"), ("f64n", None)])
def test_lanczos_against_oracle(dtype, kind):
    import paper_1511_00863_gb300 as ed
    L, nu, nd = 14, 2, 4
    bonds = _bonds(L, 60, 5)
    tb = _amplitudes(kind, len(bonds))
    b = ed.ed_build_basis(L, bonds, nu, nd, t_bond=tb)
    try:
        dim = ed.ed_basis_dims(b)[2]
        r = ed.ed_lanczos_solve(b, 0.7, 1.9, ed.make_opts(max_steps=12, tol=0.0, seed=9, dtype=dtype))
    finally:
        ed.ed_basis_destroy(b)
    if tb is None:
        H = hamiltonian.hamiltonian_csr(L, bonds, nu, nd, 0.7, 1.9)
        mv, n = (lambda v: H @ v), dim
    else:
        mv, n = ch.real_view_matvec(ch.hamiltonian_csr_complex(L, bonds, tb, nu, nd, 0.7, 1.9)), 2 * dim
    ref = olz.lanczos(mv, olz.normalized_start(ed_inputs.start_vector_raw(9, n)), max_steps=12, reorth=False,
                      fixed_steps=True)
    assert np.allclose(r["alpha"], ref.alpha, rtol=1e-11, atol=1e-11)
    assert np.allclose(r["beta"][:11], np.asarray(ref.beta)[:11], rtol=1e-11, atol=1e-11)
