"""Which kernel ed_hv takes for a basis (row-ordered or row-staged) by row length and row count:
both sides of every line against the oracle, on bases large enough that a CTA takes several row
groups, with odd row counts (the last pair of rows half empty) and row lengths that are and are not
multiples of 16 bytes; and short rows of a large basis are not left to the kernel that serves long
ones."""
import numpy as np
import pytest

import ed_inputs
from oracle import complex_hopping as ch
from oracle import hamiltonian

pytestmark = pytest.mark.gpu

EPS = {"f64": 2.0**-53, "f32": 2.0**-24, "c64": 2.0**-53, "c32": 2.0**-24}


def _torch_dtype(dtype):
    import torch
    return {"f64": torch.float64, "f32": torch.float32, "c64": torch.complex128, "c32": torch.complex64}[dtype]


# rows x columns, row-ordered: 1,287 x 1,287 and 3,003 x 2,002 (pairs of rows, one left over; odd and
# 2 mod 4 columns), 1,820 x 560, 1,287 x 286, 462 x 330; row-staged: 1,716 x 715, 12,870 x 120, 3,003 x 105
@pytest.mark.parametrize("dtype,L,nu,nd", [("f32", 13, 5, 5), ("f32", 14, 6, 5), ("f32", 16, 4, 3), ("f32", 11, 5, 4),
                                           ("f32", 13, 6, 4), ("f32", 16, 8, 2), ("f32", 15, 5, 2), ("f64", 13, 5, 3),
                                           ("f64", 13, 6, 4), ("f64", 15, 5, 2)])
def test_real_rows_against_oracle(dtype, L, nu, nd):
    import torch
    import paper_1511_00863_gb300 as ed
    bonds, t, U = ed_inputs.ring_bonds(L), 0.7, 1.9
    b = ed.ed_build_basis(L, bonds, nu, nd)
    try:
        up, dn, dim = ed.ed_basis_dims(b)
        x = torch.tensor(ed_inputs.uniform_pm1(23, dim), dtype=_torch_dtype(dtype), device="cuda")
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, t, U, x, y)
        got, xr = y.cpu().numpy(), x.cpu().numpy().astype(np.float64)
    finally:
        ed.ed_basis_destroy(b)
    assert np.all(np.isfinite(got))
    # 20,000 elements of random rows, and the first and last four rows whole
    pick = np.unique(np.concatenate([np.random.default_rng(1).integers(0, dim, 20000), np.arange(4 * dn),
                                     np.arange(dim - 4 * dn, dim)]))
    want = hamiltonian.hv_rows(L, bonds, nu, nd, t, U, xr, pick)
    scale = hamiltonian.hv_abs_rows(L, bonds, nu, nd, t, U, xr, pick)
    assert np.all(np.abs(got[pick] - want) <= 4 * (2 * len(bonds) + 2) * EPS[dtype] * scale + 1e-300)


# row-ordered: 1,287 x 286 (several row groups per CTA), 91 x 364 (c32); row-staged: 1,365 x 455 (c32),
# 3,003 x 105 without classes
@pytest.mark.parametrize("dtype,L,nu,nd,classes", [("c64", 13, 5, 3, True), ("c32", 13, 5, 3, True), ("c64", 13, 5, 3, False),
                                                   ("c32", 13, 5, 3, False), ("c32", 14, 2, 3, True),
                                                   ("c32", 15, 4, 3, False), ("c64", 15, 5, 2, False),
                                                   ("c64", 15, 5, 2, True)])
def test_complex_rows_against_oracle(dtype, L, nu, nd, classes):
    import torch
    import paper_1511_00863_gb300 as ed
    bonds, t, U = ed_inputs.ring_bonds(L), 0.7, 1.9
    v = np.exp(0.7j)
    tb = np.array([1.0, -v, np.conj(v), v])[np.arange(len(bonds)) % 4] if classes else None
    b = ed.ed_build_basis(L, bonds, nu, nd, t_bond=tb)
    try:
        dim = ed.ed_basis_dims(b)[2]
        raw = ed_inputs.uniform_pm1(29, 2 * dim)
        x = torch.tensor(raw[0::2] + 1j * raw[1::2], dtype=_torch_dtype(dtype), device="cuda")
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, t, U, x, y)
        got, xr = y.cpu().numpy(), x.cpu().numpy().astype(np.complex128)
    finally:
        ed.ed_basis_destroy(b)
    H = ch.hamiltonian_csr_complex(L, bonds, np.ones(len(bonds)) if tb is None else tb, nu, nd, t, U)
    bound = 4 * (2 * len(bonds) + 2) * EPS[dtype] * (abs(H) @ np.abs(xr)) + 1e-300
    assert np.all(np.abs(got - H @ xr) <= bound)


@pytest.mark.parametrize("dtype", ["f32", "c32"])
def test_short_rows_are_not_left_to_the_long_row_kernel(dtype):
    """12,870 rows of 120 columns: the row-staged ed_hv takes 0.4 (FP32) and 0.6 (complex FP32) of the
    time of the fused Lanczos H.v of the same basis, which reads and writes one vector more; the
    row-ordered kernel 0.84 and 1.2."""
    import torch
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(16, ed_inputs.ring_bonds(16), 8, 2)
    try:
        dim = ed.ed_basis_dims(b)[2]
        x = torch.ones(dim, dtype=_torch_dtype(dtype), device="cuda")
        y = torch.empty_like(x)
        st = ed.ed_lanczos_init(b, ed.make_opts(max_steps=200, tol=0.0, dtype=dtype))
        hv, fused = [], []
        try:
            for _ in range(6):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                ed.ed_hv(b, 1.0, 4.0, x, y)
                e[0].record()
                for _ in range(40):
                    ed.ed_hv(b, 1.0, 4.0, x, y)
                e[1].record()
                torch.cuda.synchronize()
                hv.append(e[0].elapsed_time(e[1]) / 40)
                fused.append(ed.ed_lanczos_run(st, 1.0, 4.0, 20, time_hv=True) / 20)
        finally:
            ed.ed_lanczos_destroy(st)
        assert min(hv) <= 0.75 * min(fused), (min(hv), min(fused))
    finally:
        ed.ed_basis_destroy(b)
