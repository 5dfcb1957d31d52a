"""The exact gradient of a system that keeps no bases (elses_omega_gradient without exact_forces): it builds
the columns once more with the kernel that the energy pass used, so that it is the gradient over kept
bases, bit for bit. Also where the space is nearly or wholly exhausted, and other arithmetic gives other
bases: two atoms to a cluster, nu at and past the cluster's orbitals."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [
    (3, 12, 0.0), (9, 36, 0.0), (10, 64, 0.0),        # exhausted spaces, one column a CTA
    (64, 30, 0.0), (512, 24, 4.4), (512, 40, 2.7),    # whole system; ragged clusters; a few atoms each
    (350, 6, 0.0),                                    # clusters the fixed-point kernel leaves to the FP64 one
    (4096, 8, 4.0),                                   # built and taken in several parts
]


def _system(n, nu, r_cluster, caller, **kw):
    import paper_1210_1531_gb300 as eg
    side = max(2, int(np.ceil((n / 8) ** (1 / 3))))
    pos, box = wl.diamond((side, side, side), sigma=0.05, seed=3)
    pos = np.ascontiguousarray(pos[:n])
    s = eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, nu, 0.1, 4.0 * n, **kw)
    if caller:
        H, S = s.hs()
        if caller == "uneven":    # an atom's functions scaled: rows too unlike for the fixed-point form
            d = torch.ones(n, dtype=torch.float64, device="cuda")
            d[0] = 1024.0
            rp, ci = s.pattern()
            rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
            f = (d[rows] * d[ci.long()])[:, None, None]
            H, S = H * f, S * f
        s.set_hs(H, S)
    s.green_columns()
    return s


def _outcome(call):
    """The call's result, or the code it is refused with (an exhausted space that is too far gone)."""
    import paper_1210_1531_gb300 as eg
    try:
        return call()
    except eg.ElsesError as refused:
        return refused.code


@pytest.mark.parametrize("n, nu, r_cluster", SHAPES)
@pytest.mark.parametrize("reorth", [0, 1])
@pytest.mark.parametrize("caller", ["", "own", "uneven"])
def test_same_with_and_without_kept_bases(n, nu, r_cluster, reorth, caller):
    kept = _outcome(lambda: _system(n, nu, r_cluster, caller, exact_forces=True, reorth=reorth))
    built = _outcome(lambda: _system(n, nu, r_cluster, caller, reorth=reorth, k3_lanes=32))
    if isinstance(kept, int):
        assert kept == built and caller == "uneven"
        return
    mu, _ = kept.find_mu()
    want, got = (_outcome(lambda: s.omega_gradient(mu)) for s in (kept, built))
    if isinstance(want, int):
        assert want == got and caller == "uneven"
        return
    for w, g in zip(want, got):
        assert torch.equal(g, w)
    # and of a range of atoms: integer sums, rounded once each
    cut = n // 3
    low, high = built.omega_gradient(mu, 0, cut), built.omega_gradient(mu, cut, n)
    for w, a, b in zip(want, low, high):
        assert float((a + b - w).abs().max()) <= 4.0 * 2.0 ** -53 * float(torch.maximum(a.abs(), b.abs()).max())


@pytest.mark.parametrize("n, nu, r_cluster", [(64, 30, 0.0), (211, 20, 0.0), (512, 24, 4.4), (4096, 8, 4.0)])
@pytest.mark.parametrize("caller", ["", "own"])
def test_two_pass(n, nu, r_cluster, caller):
    """V formed by another kernel: the same to rounding, for spaces far from exhausted."""
    kept = _system(n, nu, r_cluster, caller, exact_forces=True, reorth=1)
    two = _system(n, nu, r_cluster, caller, exact_forces=True, reorth=1, two_pass=True)
    mu, _ = kept.find_mu()
    for w, g in zip(kept.omega_gradient(mu), two.omega_gradient(mu)):
        assert float((g - w).abs().max()) <= 1e-11 * float(w.abs().max())
