"""Slater-Koster systems without finite H and S (two atoms in one place, a model with a NaN or an
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
