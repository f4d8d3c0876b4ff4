"""Lanczos steps on long vectors of few rows, where every row group of the fused H.v has a CTA of its own
and the update sums the H.v's records: a_j and b_{j+1} against those of the native FP64 run, whose H.v is
another kernel, and of longer vectors of more rows, where the H.v's last CTA finishes a_j."""
import numpy as np
import pytest

import ed_inputs

pytestmark = pytest.mark.gpu

STEPS = 6
# the vectors' own rounding, over the hops of a row and the steps so far
TOL = {"f64": 1e-12, "f32": 2e-6, "c32": 2e-6}


# 120 x 12,870, 136 x 24,310 (int64: two slices), 153 x 18,564 and 190 x 15,504 (complex: one CTA to an
# SM and some rows more than SMs), 560 x 12,870; 1,820 x 1,820 and 1,716 x 1,287 (tickets)
@pytest.mark.parametrize("L,nu,nd", [(16, 2, 8), (17, 2, 8), (18, 2, 6), (20, 2, 5), (16, 3, 8), (16, 4, 4), (13, 6, 5)])
@pytest.mark.parametrize("dtype", ["f64", "f32", "c32"])
def test_against_native(L, nu, nd, dtype):
    import torch
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
    try:
        dim = ed.ed_basis_dims(b)[2]
        f1 = torch.empty(dim, dtype=torch.float64, device="cuda")
        ed.ed_start_vector(dim, 9, f1)
        run = {}
        for dt, x in [("native", f1), (dtype, f1.to({"f64": torch.float64, "f32": torch.float32,
                                                      "c32": torch.complex64}[dtype]))]:
            code = ed.ED_F64_NATIVE if dt == "native" else dt
            run[dt] = ed.ed_lanczos_solve(b, 1.0, 4.0, ed.make_opts(max_steps=STEPS, tol=0.0, dtype=code), f1=x)
    finally:
        ed.ed_basis_destroy(b)
    got, want = run[dtype], run["native"]
    scale = np.abs(want["alpha"]).max() + 2 * want["beta"].max()
    assert got["steps"] == want["steps"] == STEPS
    for k in ("alpha", "beta"):
        assert np.all(np.abs(got[k] - want[k]) <= TOL[dtype] * scale), (k, got[k] - want[k])
