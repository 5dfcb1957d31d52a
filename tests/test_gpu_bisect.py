"""The bisection in one launch (elses_find_mu) against its form of one launch per step
(elses_find_mu_static), at pole counts around the edges of its grid: one block, part of a block's
poles, one block per SM, two per SM.

Both take the same decisions from sums of up to 5e6 terms in different orders, which differ by less than
1e-13 of N; mu moves by that divided by dN/dmu, and both stop at the same tolerance."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eg():
    import paper_1210_1531_gb300
    return paper_1210_1531_gb300


@pytest.mark.parametrize("n, nu", [(1, 3), (32, 4), (33, 4), (64, 30), (512, 21), (4096, 10), (10400, 30)])
def test_one_launch_matches_one_per_step(eg, n, nu):
    side = max(2, int(np.ceil((n / 8) ** (1 / 3))))
    pos, box = wl.diamond((side, side, side), sigma=0.05, seed=5)
    pos = np.ascontiguousarray(pos[:n])
    s = eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), 0.0 if n <= 64 else 4.0, nu, 0.1, 4.0 * n)
    s.green_columns()
    sp = s.spectra()
    mu, n_at = s.find_mu()
    mu1, n1, _ = eg.find_mu_static(sp["eps"], sp["c"], sp["d"], sp["nu_eff"], 0.1, 4.0 * n)
    assert abs(n_at - n1) <= 1e-11 * n
    # where the density of states vanishes mu is not determined to better than the sums: compare N there
    assert abs(mu - mu1) <= 1e-10 * (1.0 + abs(mu1)) or abs(n_at - 4.0 * n) <= 1e-11 * n
