"""The QR chase on tridiagonals that split: block systems whose Krylov spaces decouple, equal and
vanishing diagonals, nu 1 to 3. Poles against NumPy's on the same dense pencil; both are backward
stable, so they agree to a few nu eps of the largest eigenvalue."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, nu", [(1, 1), (2, 2), (2, 3), (4, 16), (9, 36), (16, 64)])
@pytest.mark.parametrize("kind", ["dense", "zero diagonal", "small entries"])
def test_poles_of_the_whole_space(n, nu, kind):
    import paper_1210_1531_gb300 as eg
    rng = np.random.default_rng(n)
    pos = np.arange(n)[:, None] * np.array([[0.3, 0.2, 0.1]])
    s = eg.System(torch.tensor(pos, device="cuda"), np.array([60.0] * 3), wl.sk_params(), 0.0, nu, 0.1, 4.0 * n)
    m = 4 * n
    H = rng.standard_normal((m, m))
    H = H + H.T
    if kind == "zero diagonal":
        np.fill_diagonal(H, 0.0)
    if kind == "small entries":      # graded: entries down to 1e-12 of the largest
        g = 10.0 ** (-12.0 * np.arange(m) / max(1, m - 1))
        H = H * np.minimum.outer(g, g)
    blocks = lambda X: torch.tensor(X.reshape(n, 4, n, 4).transpose(0, 2, 1, 3).reshape(n * n, 4, 4).copy(),  # noqa: E731
                                    device="cuda")
    rp = torch.arange(0, n * n + 1, n, dtype=torch.int32, device="cuda")
    ci = torch.arange(n, dtype=torch.int32, device="cuda").repeat(n)
    s.set_hs(blocks(H), blocks(np.eye(m)), rp, ci)
    s.green_columns()
    sp = s.spectra()
    eps, c, ne = (sp[k].cpu().numpy() for k in ("eps", "c", "nu_eff"))
    scale = np.abs(np.linalg.eigvalsh(H)).max()
    for j in range(m):
        e, w = eps[j, :ne[j]], c[j, :ne[j]] ** 2
        assert np.all(np.diff(e) >= 0.0)
        # moments of column j, which its space of nu steps reproduces: e_j^T H^k e_j = sum w e^k
        v = np.zeros(m)
        v[j] = 1.0
        for k in range(min(2 * int(ne[j]), 6)):
            assert abs((w * (e / scale) ** k).sum() - v[j]) <= 64 * nu * 2.0 ** -52
            v = H @ v / scale
