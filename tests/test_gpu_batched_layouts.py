"""Batched solves over both layouts of an instance (row-ordered H.v with rows padded to 4 elements;
dense rows element by element): row lengths that are and are not multiples of 4, rows shorter than
the row-ordered kernel takes, few rows, and groups of one and of many CTAs in one batch."""
import numpy as np
import pytest

import ed_inputs

pytestmark = pytest.mark.gpu

# rows x columns: 66 x 924, 462 x 330, 165 x 462, 126 x 126, 78 x 286 and 286 x 286, 252 x 252 (row
# ordered); 924 x 66, 70 x 70, 12 x 495, 55 x 330 (dense)
SYSTEMS = [(12, 2, 6), (11, 5, 4), (11, 3, 5), (9, 4, 4), (13, 2, 3), (13, 3, 3), (10, 5, 5), (12, 6, 2), (8, 4, 4),
           (12, 1, 4), (11, 2, 4)]


@pytest.mark.parametrize("schedule", [0, 3, 5, 6])
@pytest.mark.parametrize("form,tol", [("f32", 1e-6), ("f64n", 1e-10), ("mixed", 1e-10)])
def test_layouts_agree_with_single_solves(form, tol, schedule):
    import paper_1511_00863_gb300 as ed
    bases = [ed.ed_build_basis(L, ed_inputs.ring_bonds(L), u, d) for L, u, d in SYSTEMS]
    Us = [2.0 + 0.5 * i for i in range(len(bases))]
    try:
        ref = np.array([ed.ed_lanczos_solve(b, 1.0, U, ed.make_opts(max_steps=300, tol=1e-13, seed=2))["E0"]
                        for b, U in zip(bases, Us)])
        ts = [1.0] * len(bases)
        if form == "mixed":
            r = ed.ed_lanczos_solve_batched_mixed(bases, ts, Us, ed.make_opts(max_steps=200, tol=1e-8, seed=2, dtype="f32",
                                                                              schedule=schedule),
                                                  refine_steps=200, refine_tol=1e-13)
        else:
            r = ed.ed_lanczos_solve_batched(bases, ts, Us, ed.make_opts(
                max_steps=200, tol=1e-8 if form == "f32" else 1e-13, seed=2, dtype=form, schedule=schedule))
        assert np.all(np.abs(r["E0"] - ref) <= tol * np.abs(ref))
        assert np.all(r["inst_status"] == 2)
    finally:
        for b in bases:
            ed.ed_basis_destroy(b)
