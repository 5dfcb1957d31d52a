"""How far rho and rho_E of spaces that span the whole system are from the dense pencil's, whose eigenvectors
are corrected to first order in long double (an error of 1e-19 or so): the root mean square over the
pattern, as the geometric mean over 150 small systems (singular numbers differ by rounding luck; the mean
does not). Bounds: the figures of rotations that form T's entries from four products each and the
general reduction, 5.0e-16 (two classical passes) and 4.6e-16 (second pass from S'), rho_E 5.9e-15 and
5.3e-15 eV."""
import numpy as np
import pytest
import scipy.linalg as sl
import torch

import workloads as wl

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _dense(X, rp, ci, n):
    D = np.zeros((n, 4, n, 4))
    D[np.repeat(np.arange(n), np.diff(rp)), :, ci, :] = X
    return D.reshape(4 * n, 4 * n)


def _reference(H, S, kT):
    e, Y = sl.eigh(H, S)
    Hl, Sl, Yl = (x.astype(LD) for x in (H, S, Y))
    A, B = Yl.T @ Hl @ Yl, Yl.T @ Sl @ Yl
    el = np.diag(A) / np.diag(B)
    D = el[None, :] - el[:, None]
    D[np.abs(D) < 1e-7] = LD(1e30)          # equal levels: any basis of theirs gives the same rho
    C = (A - B * el[None, :]) / D
    np.fill_diagonal(C, (1 - np.diag(B)) / 2)
    Y = Yl + Yl @ C
    f = 2 / (np.exp(np.clip(el / LD(kT), -700, 700)) + 1)
    return [((Y * w) @ Y.T).astype(np.float64) for w in (f, f * el)]


@pytest.mark.parametrize("reorth, bound, bound_e", [(0, 5.0e-16, 5.9e-15), (1, 4.6e-16, 5.3e-15)])
def test_geometric_mean(reorth, bound, bound_e):
    import paper_1210_1531_gb300 as eg
    logs = []
    for n in (8, 10, 12, 14, 16):
        for seed in range(3, 33):
            pos, box = wl.diamond((2, 2, 2), sigma=0.05, seed=seed)
            s = eg.System(torch.tensor(np.ascontiguousarray(pos[:n]), device="cuda"), box, wl.sk_params(), 0.0, 4 * n,
                          0.1, 4.0 * n, reorth=reorth)
            try:
                s.green_columns()
            except eg.ElsesError as err:     # S is not positive definite
                assert err.code == -2
                continue
            H, S = (x.cpu().numpy() for x in s.hs())
            rp, ci = (x.cpu().numpy() for x in s.pattern())
            on = _dense(np.ones_like(H), rp, ci, n)
            want = _reference(_dense(H, rp, ci, n), _dense(S, rp, ci, n), 0.1)
            got = (_dense(x.cpu().numpy(), rp, ci, n) for x in s.density_matrix(0.0))
            logs.append([0.5 * np.log((((g - w) * on) ** 2).sum() / on.sum()) for g, w in zip(got, want)])
    assert len(logs) >= 100
    rho, rho_e = np.exp(np.mean(logs, axis=0))
    assert rho <= bound and rho_e <= bound_e, (rho, rho_e)
