"""The convergence test of ed_lanczos_solve runs beside the steps, several steps per check on
small bases: the run must end at the first step that passes the stated rule, with E0(j) of every
step, at every check stride (8, 4, 2 and 1 steps by the vector's length) and step limit."""
import numpy as np
import pytest

import ed_inputs

pytestmark = pytest.mark.gpu


def _lowest(a, b):
    return np.linalg.eigvalsh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))[0]


@pytest.mark.parametrize("L,nu,nd", [(12, 3, 3), (12, 6, 4), (13, 6, 6), (14, 7, 6)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_stops_at_the_first_step_that_passes(L, nu, nd, dtype):
    import paper_1511_00863_gb300 as ed
    tol = 1e-9 if dtype == "f64" else 1e-6
    b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
    try:
        for limit in (1, 2, 7, 200):
            r = ed.ed_lanczos_solve(b, 1.0, 4.0, ed.make_opts(max_steps=limit, tol=tol, seed=3, dtype=dtype),
                                    raise_not_converged=False)
            n, E, a, bt = r["steps"], r["E0_hist"], r["alpha"], r["beta"]
            assert len(E) == len(a) == len(bt) == n and E[-1] == r["E0"]
            passed = [j for j in range(2, n + 1)
                      if abs(E[j - 1] - E[j - 2]) <= tol * max(abs(E[j - 1]), 1.0)]
            assert passed == ([n] if r["status"] == 0 else [])
            assert (r["status"] == 0) == (limit == 200) and (n == limit or limit == 200)
            for j in range(1, n + 1):
                T = np.abs(a[:j]).max() + 2 * np.abs(bt[:j]).max()
                assert abs(E[j - 1] - _lowest(a[:j], bt[:j])) <= 8 * 2.0**-52 * T
    finally:
        ed.ed_basis_destroy(b)


def test_breakdown_ends_a_checked_run():
    """Two sites, one particle each, U = 0: the Krylov space has at most 3 states, so a run
    longer than that ends by breakdown, not by the convergence test of a later step."""
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(2, ed_inputs.ring_bonds(2), 1, 1)
    try:
        r = ed.ed_lanczos_solve(b, 1.0, 0.0, ed.make_opts(max_steps=200, tol=1e-14, seed=2))
        assert r["status"] == ed.ED_BREAKDOWN and r["steps"] <= 3
        assert abs(r["E0"] + 4.0) <= 1e-12
    finally:
        ed.ed_basis_destroy(b)
