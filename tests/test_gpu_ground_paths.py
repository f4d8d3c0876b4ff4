"""ed_lanczos_ground_state keeps the Lanczos vectors and sums them in one pass when the device
has room for them, and regenerates them step by step when it has not: the same psi either way,
bit for bit (both sum the same integers). ed_double_occupancy by runs of down states."""
import numpy as np
import pytest

import ed_inputs

pytestmark = pytest.mark.gpu


def test_kept_and_regenerated_vectors_give_the_same_psi():
    import torch
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(14, ed_inputs.ring_bonds(14), 7, 6)
    try:
        dim = ed.ed_basis_dims(b)[2]
        psi = [torch.empty(dim, dtype=torch.float64, device="cuda") for _ in range(2)]
        opts = ed.make_opts(max_steps=200, tol=1e-12, seed=4)
        res = [ed.ed_lanczos_ground_state(b, 1.0, 4.0, opts, psi[0])]
        # about 75 vectors of 83 MB: with 1 GB free (and the memory kept from the first call)
        # half of it does not hold them
        torch.cuda.synchronize()
        hog = torch.empty(max(0, torch.cuda.mem_get_info()[0] - (1 << 30)), dtype=torch.uint8, device="cuda")
        try:
            res.append(ed.ed_lanczos_ground_state(b, 1.0, 4.0, opts, psi[1]))
        finally:
            del hog
            torch.cuda.empty_cache()
        assert res[0] == res[1] and res[0]["steps"] > 45
        assert torch.equal(psi[0], psi[1])
    finally:
        ed.ed_basis_destroy(b)


@pytest.mark.parametrize("L,nu,nd", [(6, 3, 3), (12, 0, 5), (12, 5, 0), (12, 10, 2), (13, 2, 6), (14, 12, 7)])
@pytest.mark.parametrize("reorth", [0, 1])
def test_small_ground_states_and_double_occupancy(L, nu, nd, reorth):
    """Odd row lengths, one species, more than 8 particles (two passes over a run), a run limit
    inside a row (C(14, 7) = 3432 down states, runs of 2048)."""
    import torch
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
    try:
        up, dn, dim = ed.ed_basis_dims(b)
        psi = torch.empty(dim, dtype=torch.float64, device="cuda")
        r = ed.ed_lanczos_ground_state(b, 1.0, 3.0, ed.make_opts(max_steps=150, tol=1e-13, seed=6, reorth=reorth),
                                       psi, raise_not_converged=False)
        y = torch.empty_like(psi)
        ed.ed_hv(b, 1.0, 3.0, psi, y)
        assert abs(float(psi.norm()) - 1.0) <= 1e-12
        assert float((y - r["E0"] * psi).norm()) <= 1e-4 and abs(float(psi @ y) - r["E0"]) <= 1e-8
        # any vector: against plain sums, n sites x dim terms of relative rounding eps
        v = torch.randn(dim, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        D, site = ed.ed_double_occupancy(b, v)
        p2 = (v.cpu().numpy() ** 2).reshape(up, dn)
        bits = lambda n: np.array([s for s in range(1 << L) if bin(s).count("1") == n])  # noqa: E731
        ub, db = bits(nu), bits(nd)
        want = np.array([p2[np.ix_((ub >> i) & 1 == 1, (db >> i) & 1 == 1)].sum() for i in range(L)]) / p2.sum()
        assert np.all(np.abs(site - want) <= 1e-12 * np.maximum(want, 1e-3))
        assert abs(D - want.sum()) <= 1e-12 * max(want.sum(), 1e-3)
    finally:
        ed.ed_basis_destroy(b)
