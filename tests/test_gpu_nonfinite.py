"""What is not a number is reported and not dropped. Slater-Koster systems without finite H and S (two atoms in one place, a model with a NaN or an
infinity) are refused, as the integers of the fixed-point kernel cannot carry what is not a number."""
import dataclasses

import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu
NAN, INF = float("nan"), float("inf")


@pytest.mark.parametrize("change, code", [
    (dict(Es=NAN), -3), (dict(Es=INF), -3), (dict(Ep=NAN), -3), (dict(Ep=-INF), -3), (dict(V0=0), -3), (dict(V0=3), -3),
    (dict(pair=0.0), -2), (dict(pair=1e-200), -2)])
@pytest.mark.parametrize("cells, r_cluster", [((2, 2, 2), 0.0), ((6, 6, 6), 5.0)])   # one column a CTA, four
def test_refused(change, code, cells, r_cluster):
    import paper_1210_1531_gb300 as eg
    pos, box = wl.diamond(cells, sigma=0.05, seed=3)
    sk = wl.sk_params()
    if "pair" in change:
        pos[5] = pos[4] + change["pair"]
    elif "V0" in change:
        sk = dataclasses.replace(sk, V0=tuple(NAN if k == change["V0"] else v for k, v in enumerate(sk.V0)))
    else:
        sk = dataclasses.replace(sk, **change)
    s = eg.System(torch.tensor(np.ascontiguousarray(pos), device="cuda"), box, sk, r_cluster, 12, 0.1, 4.0 * len(pos))
    with pytest.raises(eg.ElsesError) as err:
        s.green_columns()
    assert err.value.code == code


@pytest.mark.parametrize("t, code", [(1e150, 0), (1.2e154, -5)])
def test_qr_sweep_that_overflows(t, code):
    """Two atoms coupled by t: the projected matrix ((0, t), (t, 0)) is finite and so is t^2, but not the
    2 t^2 of the first rotation."""
    import paper_1210_1531_gb300 as eg
    pos = np.array([[0.0, 0.0, 0.0], [0.3, 0.2, 0.1]])
    s = eg.System(torch.tensor(pos, device="cuda"), np.array([60.0] * 3), wl.sk_params(), 0.0, 2, 0.1, 8.0)
    rp = torch.tensor([0, 2, 4], dtype=torch.int32, device="cuda")
    ci = torch.tensor([0, 1, 0, 1], dtype=torch.int32, device="cuda")
    blocks = lambda on, off: torch.eye(4, dtype=torch.float64, device="cuda") * \
        torch.tensor([on, off, off, on], dtype=torch.float64, device="cuda")[:, None, None]   # noqa: E731
    s.set_hs(blocks(0.0, t), blocks(1.0, 0.0), rp, ci)
    if code == 0:
        assert s.green_columns() == 0
        want = torch.tensor([-t, t], dtype=torch.float64, device="cuda")
        assert float((s.spectra()["eps"] / want - 1.0).abs().max()) <= 1e-15
        return
    with pytest.raises(eg.ElsesError) as err:
        s.green_columns()
    assert err.value.code == code
