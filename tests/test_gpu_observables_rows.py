"""Double occupancy of few long rows, whose runs are cut by their number: one row, an empty and a full up
species, run lengths at and beside every limit, against the oracle on the same vector; and one row is
not left to a few warps."""
import time

import numpy as np
import pytest

import ed_inputs
from oracle import observables

pytestmark = pytest.mark.gpu


# rows x columns: 1 x 12,376, 1 x 24,310, 1 x 17, 1 x 184,756 (empty up species), 17 x 24,310, 136 x 680,
# 91 x 3,432, 560 x 560 and 715 x 715 (either side of four warps per SM on 152 SMs), 3,432 x 91
@pytest.mark.parametrize("L,nu,nd", [(17, 17, 11), (17, 0, 8), (17, 17, 1), (20, 0, 10), (17, 1, 8), (17, 2, 3),
                                     (14, 12, 7), (16, 3, 13), (13, 4, 9), (14, 7, 2)])
def test_against_oracle(L, nu, nd):
    import torch
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
    try:
        dim = ed.ed_basis_dims(b)[2]
        psi = torch.tensor(ed_inputs.uniform_pm1(11, dim), device="cuda")
        D, site = ed.ed_double_occupancy(b, psi)
    finally:
        ed.ed_basis_destroy(b)
    Dr, site_r = observables.double_occupancy(L, nu, nd, psi.cpu().numpy())
    assert abs(D - Dr) <= 1e-13 * max(1.0, Dr)
    assert np.allclose(site, site_r, rtol=1e-13, atol=1e-15)


def test_one_row_is_spread_over_the_chip():
    """12,376 states in one row against 48,400 in 220 rows: with six warps on the one row its call took
    three times as long as the other."""
    import torch
    import paper_1511_00863_gb300 as ed
    t = []
    for L, nu, nd in [(17, 17, 11), (12, 3, 3)]:
        b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
        try:
            psi = torch.tensor(ed_inputs.uniform_pm1(11, ed.ed_basis_dims(b)[2]), device="cuda")
            ts = []
            for _ in range(25):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                ed.ed_double_occupancy(b, psi)
                ts.append(time.perf_counter() - t0)
        finally:
            ed.ed_basis_destroy(b)
        t.append(sorted(ts)[12])
    assert t[0] <= 2 * t[1], t
