"""mu of the bisection in one launch against its form of one launch per step, where N(mu) is steep (kT = 1
eV smears the gap), at pole counts around the edges of its grid. Both sum up to 1e6 terms in different
orders, N to within 1e-10, and stop at a bracket of 1e-13: mu agrees to 2e-13 + 1e-10 / N'(mu)."""
import numpy as np
import pytest
import torch

import workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, nu", [(2, 4), (32, 4), (33, 4), (64, 30), (512, 21), (4096, 10), (10400, 30)])
def test_same_mu(n, nu):
    import paper_1210_1531_gb300 as eg
    side = max(2, int(np.ceil((n / 8) ** (1 / 3))))
    pos, box = wl.diamond((side, side, side), sigma=0.05, seed=5)
    pos = np.ascontiguousarray(pos[:n])
    s = eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), 0.0 if n <= 64 else 4.0, nu, 1.0, 4.0 * n)
    s.green_columns()
    sp = s.spectra()
    mu, _ = s.find_mu()
    mu1, _, _ = eg.find_mu_static(sp["eps"], sp["c"], sp["d"], sp["nu_eff"], 1.0, 4.0 * n)
    slope = (s.energies(mu + 1e-4)["N"] - s.energies(mu - 1e-4)["N"]) / 2e-4
    assert slope > 0.1      # mu is determined to 1e-9 at least
    assert abs(mu - mu1) <= gu.mu_tolerance(s, mu)
