"""Poles, density matrix and G(z) of the fixed-point Krylov kernel against the FP64 one, on the systems that
are hardest for vectors of one scale: graphite around diamond grains, whose layers hang together by
bonds near the cutoff, so that parts of a cluster are reached late and with amplitudes of 2^-20 to 2^-70;
dense disordered carbon with close pairs; strongly displaced diamond. The FP64 kernel takes over where one atom's
basis functions are scaled by 32; columns whose cluster does not hold that atom are the same.

Bounds. The poles of both kernels are within 3e-10 eV of an 80-bit recursion's in the worst columns of such
systems (weights of 1e-7 to 1e-4), so the two within 6e-10. rho: 1e-12 of the largest entry, the gate between
the FP64 forms. G(z) at 0.2 eV off the axis: a pole of weight w that is off by e moves G by w e / 0.04, and
w e is below 5e-12: 2.5e-10 at most, and 1e-12 of G in the root mean square."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu

CLASSES = ((100, 20), (140, 30), (1 << 30, 40))


def _structure(kind):
    if kind == "composite":
        pos, box, _ = wl.composite(32768)
        return pos, box, 6.0, CLASSES
    if kind == "amorphous":
        return (*wl.amorphous((8, 8, 8), seed=7), 5.0, ())
    return (*wl.diamond((8, 8, 8), sigma=0.1, seed=1210), 6.0, ())


@pytest.mark.parametrize("kind, reorth, z", [("composite", 1, False), ("composite", 0, False), ("amorphous", 1, True),
                                             ("amorphous", 0, False), ("diamond", 1, True), ("diamond", 0, False)])
def test_against_the_fp64_kernel(kind, reorth, z):
    import paper_1210_1531_gb300 as eg
    pos, box, r_cluster, classes = _structure(kind)
    n = len(pos)
    make = lambda: eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, 30, 0.1, 4.0 * n,  # noqa: E731
                             nu_classes=classes, schedule=1, reorth=reorth)
    fixed, fp64 = make(), make()
    H, S = fixed.hs()
    rp, ci = fixed.pattern()
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    d = torch.ones(n, dtype=torch.float64, device="cuda")
    d[0] = 32.0
    f = (d[rows] * d[ci.long()])[:, None, None]
    fp64.set_hs(H * f, S * f)
    del H, S, f
    for s in (fixed, fp64):
        assert s.green_columns() == 0
    step = pos - pos[0]
    step -= box * np.rint(step / box)
    same = torch.tensor((step ** 2).sum(1) > (r_cluster + 1e-9) ** 2, device="cuda")    # by atom
    a, b = fixed.spectra(), fp64.spectra()
    columns = same.repeat_interleave(4)
    assert torch.equal(a["nu_eff"], b["nu_eff"]) and int(columns.sum()) > 0.95 * 4 * n
    inside = torch.arange(a["eps"].shape[1], device="cuda")[None, :] < a["nu_eff"][:, None]
    assert float(((a["eps"] - b["eps"]).abs() * (inside & columns[:, None])).max()) <= 6e-10
    blocks = same[ci.long()]                            # block (I, J) holds columns of J
    mu, _ = fixed.find_mu()
    for x, y in zip(fixed.density_matrix(mu), fp64.density_matrix(mu)):
        assert float((x - y)[blocks].abs().max()) <= 1e-12 * float(x[blocks].abs().max())
    if z:
        for zz in (-12 + 0.2j, -2 + 0.2j, 4 + 0.2j, 30 + 0.2j):
            x, y = (s.green_columns(z=[zz])[blocks] for s in (fixed, fp64))
            assert float((x - y).abs().max()) <= 2.5e-10
            assert float((x - y).norm()) <= 1e-12 * float(x.norm())
