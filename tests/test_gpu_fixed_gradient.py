"""The bases that the fixed-point Krylov kernel keeps for the exact gradient (its store form), at the sizes
where its work is split: dOmega/dH and dOmega/dS against those over the FP64 kernel's bases, which takes
over where an atom on its own has its functions scaled (that atom's block aside). Spaces far from
exhausted, where the gradient moves by some 100 times the rounding of the bases: 1e-11 of its largest."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, nu, r_cluster, reorth", [
    (63, 5, 0.0, 0), (64, 2, 0.0, 1), (65, 12, 0.0, 0), (64, 33, 0.0, 1),      # one column a CTA
    (330, 18, 0.0, 1), (512, 24, 4.4, 0), (512, 30, 6.0, 1), (500, 30, 5.1, 0),   # four
])
def test_gradient(n, nu, r_cluster, reorth):
    import paper_1210_1531_gb300 as eg
    side = max(2, int(np.ceil(((n - 1) / 8) ** (1 / 3))))
    pos, box = wl.diamond((side, side, side), sigma=0.08, seed=3)
    box = np.array(box, dtype=np.float64)
    pos = np.concatenate([pos[:n - 1], [[0.0, 0.0, box[2] + 10.0]]])
    box[2] += 20.0
    make = lambda: eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, nu, 0.1,  # noqa: E731
                             4.0 * n, exact_forces=True, reorth=reorth)
    sk, caller, fp64 = make(), make(), make()
    H, S = sk.hs()
    caller.set_hs(H, S)
    d = torch.ones_like(H)
    d[-1] = 1024.0
    fp64.set_hs(H * d, S * d)
    for s in (sk, caller, fp64):
        s.green_columns()
    mu, _ = fp64.find_mu()
    want = fp64.omega_gradient(mu)
    for s in (sk, caller):
        for g, w in zip(s.omega_gradient(mu), want):
            assert float((g - w)[:-1].abs().max()) <= 1e-11 * float(w[:-1].abs().max())
