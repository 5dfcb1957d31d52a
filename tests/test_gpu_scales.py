"""H and S in other units: multiplied by a power of two, which is exact, they give the poles of the
original in those units. Bound: the two agree as two runs of the recursion in different arithmetic do
(1e-12 of the largest pole, for a space far from exhausted)."""
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


def _poles(h_exp, s_exp, reorth):
    import paper_1210_1531_gb300 as eg
    pos, box = wl.diamond((2, 2, 2), sigma=0.05, seed=3)
    s = eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), 0.0, 12, 0.1, 4.0 * len(pos), reorth=reorth)
    H, S = s.hs()
    s.set_hs(H * 2.0 ** h_exp, S * 2.0 ** s_exp)
    assert s.green_columns() == 0
    return s.spectra()["eps"] * 2.0 ** (s_exp - h_exp)


@pytest.mark.parametrize("s_exp", [-64, -40, 40, 64, 130, 200, 300])
@pytest.mark.parametrize("reorth", [0, 1])
def test_scaled_overlap(s_exp, reorth):
    want = _poles(0, 0, reorth)
    assert float((_poles(0, s_exp, reorth) - want).abs().max()) <= 1e-12 * float(want.abs().max())


@pytest.mark.parametrize("h_exp", [-300, -140, -70, 90, 126, 140, 300])
@pytest.mark.parametrize("reorth", [0, 1])
def test_scaled_hamiltonian(h_exp, reorth):
    want = _poles(0, 0, reorth)
    assert float((_poles(h_exp, 0, reorth) - want).abs().max()) <= 1e-12 * float(want.abs().max())
