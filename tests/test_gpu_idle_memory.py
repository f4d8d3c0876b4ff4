"""Memory that the library's pools hold idle (vectors of earlier ground-state calls, stores of batched
solves) counts as free: later calls get it, nothing fails or is cut short for it, and a large
ground-state call leaves no work vectors behind."""
import pytest

import ed_inputs

pytestmark = pytest.mark.gpu

GB = 1 << 30


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _hog(leave):
    import torch
    return torch.empty(max(0, _free() - leave), dtype=torch.uint8, device="cuda")


@pytest.fixture()
def idle():
    """A basis alive and at least 7 GB idle in the pool: the vectors of a 14-site ground state."""
    import torch
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(14, ed_inputs.ring_bonds(14), 7, 7)
    psi = torch.empty(ed.ed_basis_dims(b)[2], dtype=torch.float64, device="cuda")
    r = ed.ed_lanczos_ground_state(b, 1.0, 4.0, ed.make_opts(max_steps=200, tol=1e-12, seed=3), psi)
    assert r["steps"] * psi.numel() * 8 > 6 * GB
    del psi
    torch.cuda.empty_cache()
    yield ed
    ed.ed_basis_destroy(b)
    torch.cuda.empty_cache()


def test_work_vectors_get_idle_memory(idle):
    ed = idle
    b = ed.ed_build_basis(16, ed_inputs.ring_bonds(16), 8, 8)
    hog = _hog(GB)
    try:
        st = ed.ed_lanczos_init(b, ed.make_opts(max_steps=5, tol=0.0, dtype="f64"))  # 2 x 1.3 GB
        ed.ed_lanczos_run(st, 1.0, 4.0, 2)
        assert ed.ed_lanczos_energy(st)[1] == 2
        ed.ed_lanczos_destroy(st)
    finally:
        del hog
        ed.ed_basis_destroy(b)


def test_mixed_solve_counts_idle_memory(idle):
    ed = idle
    b = ed.ed_build_basis(14, ed_inputs.ring_bonds(14), 7, 6)  # 41 MB a vector: 1 GB free is 11 of them
    opts = ed.make_opts(max_steps=60, tol=1e-8, dtype="f32", seed=5)
    try:
        hog = _hog(GB)
        try:
            tight = ed.ed_lanczos_solve_mixed(b, 1.0, 4.0, opts, refine_steps=64, refine_tol=1e-12)
        finally:
            del hog
    finally:
        ed.ed_basis_destroy(b)
    b = ed.ed_build_basis(14, ed_inputs.ring_bonds(14), 7, 6)
    try:
        roomy = ed.ed_lanczos_solve_mixed(b, 1.0, 4.0, opts, refine_steps=64, refine_tol=1e-12)
    finally:
        ed.ed_basis_destroy(b)
    assert roomy["steps32"] > 20 and tight["steps32"] == roomy["steps32"] and tight["E0"] == roomy["E0"]


def test_batched_solve_gets_idle_memory(idle):
    ed = idle
    b = ed.ed_build_basis(12, ed_inputs.ring_bonds(12), 6, 6)  # 850,000 states: 0.68 GB of FP32 vectors at 200 steps
    hog = _hog(GB)
    try:
        r = ed.ed_lanczos_solve_batched_mixed([b] * 4, [1.0] * 4, [1.0, 2.0, 3.0, 4.0],
                                              ed.make_opts(max_steps=200, tol=1e-6, seed=1, dtype="f32", schedule=5),
                                              raise_not_converged=False)
        assert r["E0"].shape == (4,)
    finally:
        del hog
        ed.ed_basis_destroy(b)


def test_large_ground_state_leaves_no_work_vectors():
    import torch
    import paper_1511_00863_gb300 as ed
    b = ed.ed_build_basis(16, ed_inputs.ring_bonds(16), 8, 7)  # two vectors of 1.2 GB
    try:
        psi = torch.empty(ed.ed_basis_dims(b)[2], dtype=torch.float64, device="cuda")
        hog = _hog(int(2.5 * psi.numel() * 8) + (256 << 20))  # no room for kept vectors: none idle afterwards
        try:
            before = _free()
            ed.ed_lanczos_ground_state(b, 1.0, 4.0, ed.make_opts(max_steps=4, tol=0.0, seed=4), psi)
            assert before - _free() <= 256 << 20
        finally:
            del hog
    finally:
        ed.ed_basis_destroy(b)
        torch.cuda.empty_cache()
