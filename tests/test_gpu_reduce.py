"""The reduction's first-order form (S' = I to 2^-32) at the sizes where its lanes split: nu below, at and
past a warp, and the rows of the three vectors past it. The Krylov space spans the whole space, so
the density matrix is the dense one: rho = sum 2 f(e) y y^T over the pencil's eigenvectors, with both
sides' rounding of a few eps times nu and the condition of S below 10."""
import numpy as np
import pytest
import scipy.linalg
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, nu", [(1, 4), (2, 8), (7, 28), (8, 32), (9, 36), (16, 64)])
def test_density_matrix_of_the_whole_space(n, nu):
    import paper_1210_1531_gb300 as eg
    rng = np.random.default_rng(n)
    pos = np.arange(n)[:, None] * np.array([[0.3, 0.2, 0.1]])
    s = eg.System(torch.tensor(pos, device="cuda"), np.array([60.0] * 3), wl.sk_params(), 0.0, nu, 0.1, 4.0 * n)
    m = 4 * n
    H, S = rng.standard_normal((2, m, m))
    H, S = H + H.T, np.eye(m) + 0.1 * (S + S.T) / np.sqrt(m)
    blocks = lambda X: torch.tensor(X.reshape(n, 4, n, 4).transpose(0, 2, 1, 3).reshape(n * n, 4, 4).copy(),  # noqa: E731
                                    device="cuda")
    rp = torch.arange(0, n * n + 1, n, dtype=torch.int32, device="cuda")
    ci = torch.arange(n, dtype=torch.int32, device="cuda").repeat(n)
    s.set_hs(blocks(H), blocks(S), rp, ci)
    s.green_columns()
    assert int(s.spectra()["nu_eff"].min()) == nu
    rho, rho_e = s.density_matrix(0.0)
    e, Y = scipy.linalg.eigh(H, S)
    f2 = 2.0 / (np.exp(e / 0.1) + 1.0)
    for got, w in ((rho, f2), (rho_e, f2 * e)):
        want = (Y * w) @ Y.T
        got = got.cpu().numpy().reshape(n, n, 4, 4).transpose(0, 2, 1, 3).reshape(m, m)
        # f changes by de / (4 kT): eigenvalue errors of nu eps |H| count ten times over
        assert np.abs(got - want).max() <= 64 * nu * 2.0 ** -52 * np.abs(e).max() / 0.1
