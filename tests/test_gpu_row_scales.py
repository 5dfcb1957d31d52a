"""Rows of H and S of different size. The fixed-point Krylov kernel holds all coefficients of a matrix in
one scale, so it is used only where the row sums lie within 2^5 of one another. An atom's basis functions
are scaled by s: columns whose cluster does not hold the atom stay the same, to the bit where the FP64
kernel takes them, while the fixed-point one rounds with the matrix's largest entries."""
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


def _poles(s_atom, r_cluster=4.3):
    import paper_1210_1531_gb300 as eg
    pos, box = wl.diamond((4, 4, 4), sigma=0.05, seed=3)
    s = eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, 20, 0.1, 4.0 * len(pos))
    H, S = s.hs()
    rp, ci = s.pattern()
    rows = torch.repeat_interleave(torch.arange(len(pos), device="cuda"), (rp[1:] - rp[:-1]).long())
    d = torch.ones(len(pos), dtype=torch.float64, device="cuda")
    d[0] = s_atom
    f = (d[rows] * d[ci.long()])[:, None, None]
    s.set_hs(H * f, S * f)
    spread = 0.0
    for X in (H * f, S * f):
        sums = torch.zeros(len(pos), 4, dtype=torch.float64, device="cuda").index_add_(0, rows, X.abs().sum(2))
        spread = max(spread, float(sums.max() / sums.min()))
    s.green_columns()
    p = torch.tensor(pos, device="cuda")
    step = p - p[0]
    b = torch.tensor(box, device="cuda")
    step = step - b * torch.round(step / b)
    far = ((step ** 2).sum(1) > (r_cluster + 1e-9) ** 2).repeat_interleave(4)
    return s.spectra()["eps"][far], spread


@pytest.mark.parametrize("s_atom", [2.0, 8.0, 16.0, 0.125])
def test_which_kernel_takes_them(s_atom):
    want, spread = _poles(64.0)
    assert spread > 256.0                       # the FP64 kernel's
    got, spread = _poles(s_atom)
    assert torch.equal(got, want) == (spread > 32.0)
    assert float((got - want).abs().max()) <= 1e-10
