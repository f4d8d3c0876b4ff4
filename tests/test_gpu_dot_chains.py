"""a_j of the FP32 runs: a thread adds the products of all its rows as a compensated FP32 pair, whose error
grows with their number and not with its square."""
import math

import numpy as np
import pytest

import ed_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "c32"])
def test_equal_products_sum_exactly(dtype):
    """t = 0, a constant f_1 and one down particle: w = U f_1 on the states whose down site is doubly
    occupied (half of them) and 0 elsewhere, so a_1 is a sum of equal products, known from one of them.
    705,432 rows of 22 columns: up to 600 row groups per CTA, 4 products of a thread in each. Bound: an
    addition of a renormalised pair rounds twice, by 2^-25 of a low part of 2^-24 of the sum (and the
    product's error), so 2400 2^-48; the FP64 sums 100 2^-53."""
    import torch
    import paper_1511_00863_gb300 as ed
    L, f = 22, np.float32
    b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), L // 2, 1)
    try:
        dim = ed.ed_basis_dims(b)[2]
        f1 = torch.full((dim,), 0.731, dtype=torch.float32 if dtype == "f32" else torch.complex64, device="cuda")
        count = math.comb(L - 1, L // 2 - 1) * L
        worst = 0.0
        for U in (1.1, 1.7, 2.3, 3.1, 4.7, 5.9, 6.7, 7.3):
            st = ed.ed_lanczos_init(b, ed.make_opts(max_steps=4, tol=0.0, dtype=dtype), f1=f1)
            try:
                sc = f(ed.ed_lanczos_buffers(st)["scale_next"])  # the kernel's factor of f_1
                alpha = ed.ed_lanczos_step(st, 0.0, U)[1]
            finally:
                ed.ed_lanczos_destroy(st)
            x = f(0.731)
            want = float(f(sc * f(f(U) * x))) * float(f(sc * x)) * count
            worst = max(worst, abs(alpha - want) / want)
        assert worst <= 2400 * 2.0**-48 + 100 * 2.0**-53, worst
    finally:
        ed.ed_basis_destroy(b)
