"""The row-ordered H.v's tables with complex amplitudes: the two directions of a bond are two classes, so
a chunk of 32 columns can need more table rows than the lattice has bonds. A complete bipartite lattice
with one complex amplitude, behind a few bonds of other amplitudes by which the columns are sorted
first, against the oracle."""
import itertools
import random

import numpy as np
import pytest

import ed_inputs
from oracle import complex_hopping as ch


def _lattice(extra):
    """13 sites: `extra` bonds inside the halves, each with an amplitude of its own, then all 42 between them."""
    L, h = 13, 6
    inner = [(a, b) for a in range(L) for b in range(a + 1, L) if (a < h) == (b < h)]
    inner = random.Random(0).sample(inner, extra)
    bonds = inner + [(a, b) for a in range(h) for b in range(h, L)]
    tb = np.array([1.0 + 0.125 * k for k in range(extra)] + [np.exp(0.7j)] * (h * (L - h)))
    return L, np.array(bonds, dtype=np.int32), tb


def _chunk_rows(L, bonds, tb, n):
    """Table rows of the chunks: columns by hop counts, class by class, the most hops of each class in 32."""
    s = np.array(sorted(sum(1 << i for i in c) for c in itertools.combinations(range(L), n)))
    amps = []
    cnt = np.zeros((2 * len(bonds), len(s)), dtype=np.int64)  # by class
    for (i, j), v in zip(bonds, tb):
        for a, hop in ((v, ~(s >> i) & (s >> j) & 1), (np.conj(v), (s >> i) & ~(s >> j) & 1)):
            c = next((k for k, w in enumerate(amps) if a in (w, -w)), None)
            if c is None:
                c = len(amps)
                amps.append(a)
            cnt[c] += hop
    cnt = cnt[:len(amps), np.lexsort(-cnt[:len(amps)][::-1])]
    return np.array([cnt[:, k:k + 32].max(axis=1).sum() for k in range(0, len(s), 32)])


@pytest.mark.parametrize("extra", [6, 8])
def test_lattices_need_more_rows_than_bonds(extra):
    L, bonds, tb = _lattice(extra)
    assert _chunk_rows(L, bonds, tb, 6).mean() > len(bonds)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["c64", "c32"])
@pytest.mark.parametrize("extra", [6, 8])
def test_against_oracle(extra, dtype):
    import torch
    import paper_1511_00863_gb300 as ed
    (L, bonds, tb), nu, nd, t, U = _lattice(extra), 2, 6, 0.7, 1.9
    b = ed.ed_build_basis(L, bonds, nu, nd, t_bond=tb)
    try:
        dim = ed.ed_basis_dims(b)[2]
        raw = ed_inputs.uniform_pm1(5, 2 * dim)
        x = torch.tensor(raw[0::2] + 1j * raw[1::2], device="cuda")
        x = x.to({"c64": torch.complex128, "c32": torch.complex64}[dtype])
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, t, U, x, y)
        got, xr = y.cpu().numpy(), x.cpu().numpy().astype(np.complex128)
    finally:
        ed.ed_basis_destroy(b)
    H = ch.hamiltonian_csr_complex(L, bonds, tb, nu, nd, t, U)
    eps = {"c64": 2.0**-53, "c32": 2.0**-24}[dtype]
    bound = 4 * (2 * len(bonds) + 2) * eps * (abs(H) @ np.abs(xr)) + 1e-300
    assert np.all(np.abs(got - H @ xr) <= bound)
