"""Rounding of ed_hv is the same whichever kernel a basis takes: the hops of each species are added in table
order with their signs alone, each sum is multiplied by -t, the diagonal comes last. With t = 1, U = 4 and
at most two doubly occupied sites every product is exact, so numpy gives the same bits."""
import numpy as np
import pytest

import ed_inputs

pytestmark = pytest.mark.gpu


def _hop_sums(tab, x, axis):
    """Sum over the hops of a species in table order (tab: [maxhops][n] entries target | sign << 31)."""
    n = x.shape[axis]
    acc = np.zeros_like(x)
    for row in tab:
        tgt, ok = row & 0x3FFFFFFF, (row & 0x3FFFFFFF) < n
        v = np.take(x, np.where(ok, tgt, 0), axis=axis)
        s = np.where(ok, np.where(row >> 31, -1, 1), 0).astype(x.real.dtype)
        acc = acc + v * (s[:, None] if axis == 0 else s[None, :])
    return acc


# row-staged: 3,003 x 105, 12,870 x 120, 1,287 x 78; row-ordered: 455 x 560 (f32, f64), 816 x 153 (few rows)
@pytest.mark.parametrize("L,nu,nd", [(15, 5, 2), (16, 8, 2), (13, 5, 2), (18, 3, 2)])
@pytest.mark.parametrize("dtype", ["f64", "f32", "c64", "c32"])
def test_bits(L, nu, nd, dtype):
    import torch
    import paper_1511_00863_gb300 as ed

    def table(ptr, rows, cols):
        class V:
            __cuda_array_interface__ = {"shape": (rows, cols), "typestr": "<i4", "data": (ptr, False), "version": 3}
        return torch.as_tensor(V(), device="cuda").cpu().numpy().view(np.uint32)

    b = ed.ed_build_basis(L, ed_inputs.ring_bonds(L), nu, nd)
    try:
        up, dn, dim = ed.ed_basis_dims(b)
        tb = ed.ed_basis_tables(b)
        hu, hd = table(tb["hop_up"], tb["maxhops_up"], up), table(tb["hop_dn"], tb["maxhops_dn"], dn)
        bits = [table(p, 1, n)[0] for p, n in ((tb["up_bits"], up), (tb["dn_bits"], dn))]
        raw = ed_inputs.uniform_pm1(31, 2 * dim)
        x = torch.tensor(raw[0::2] + 1j * raw[1::2] if dtype[0] == "c" else raw[:dim])
        x = x.to({"f64": torch.float64, "f32": torch.float32, "c64": torch.complex128, "c32": torch.complex64}[dtype])
        x = x.cuda()
        y = torch.full_like(x, float("nan"))
        ed.ed_hv(b, 1.0, 4.0, x, y)
        got, xr = y.cpu().numpy().reshape(up, dn), x.cpu().numpy().reshape(up, dn)
    finally:
        ed.ed_basis_destroy(b)
    both = bits[0][:, None] & bits[1][None, :]
    n = sum(((both >> np.uint32(i)) & np.uint32(1)).astype(np.int64) for i in range(L))
    hops = -(_hop_sums(hd, xr, 1) + _hop_sums(hu, xr, 0))
    want = hops + (4 * n).astype(xr.real.dtype) * xr
    assert np.array_equal(got, want), np.abs(got - want).max()
