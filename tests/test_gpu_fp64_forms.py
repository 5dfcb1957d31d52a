"""The FP64 Krylov kernels in their two-centre forms, half-warp and whole-warp columns: on Slater-Koster
systems that the fixed-point kernel leaves to them. Either clusters past its largest (360 atoms, 23 slots of
16), or rows of very different size (on-site energies of 0.01 eV and an atom on its own in a vacuum)."""
import dataclasses

import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


def _large(nu=8, **kw):
    import paper_1210_1531_gb300 as eg
    pos, box = wl.diamond((4, 4, 3), sigma=0.05, seed=3)
    return eg.System(torch.tensor(np.ascontiguousarray(pos[:360]), device="cuda"), box, wl.sk_params(), 0.0, nu, 0.1,
                     1440.0, **kw)


def _uneven(r_cluster, nu=16, **kw):
    import paper_1210_1531_gb300 as eg
    pos, box = wl.diamond((4, 4, 4), sigma=0.08, seed=3)
    box = np.array(box, dtype=np.float64)
    pos = np.concatenate([pos, [[0.0, 0.0, box[2] + 10.0]]])
    box[2] += 20.0
    sk = dataclasses.replace(wl.sk_params(), Es=-0.01, Ep=0.01)
    return eg.System(torch.tensor(pos, device="cuda"), box, sk, r_cluster, nu, 0.1, 4.0 * len(pos), **kw)


def test_both_forms_are_timed():
    """More launches than with the half-warp form switched off."""
    launches = {lanes: _large(autotune=True, k3_lanes=lanes).stats()["launches"] for lanes in (0, 32)}
    assert launches[0] > launches[32]


@pytest.mark.parametrize("r_cluster", [3.9, 4.4, 5.1, 6.0])
@pytest.mark.parametrize("reorth", [0, 1])
def test_half_warp_columns_match_whole_warp_ones(r_cluster, reorth):
    """Both sum in FP64 in other orders: rho within the FP64 forms' gate of 1e-12 of its largest entry."""
    half, whole = (_uneven(r_cluster, reorth=reorth, schedule=1, k3_lanes=lanes) for lanes in (0, 32))
    for s in (half, whole):
        assert s.green_columns() >= 0
    assert any(cap % 32 == 16 for cap in half.autotune_shapes())
    assert not any(cap % 32 == 16 for cap in whole.autotune_shapes())
    assert torch.equal(half.spectra()["nu_eff"], whole.spectra()["nu_eff"])
    mu, _ = whole.find_mu()
    for x, y in zip(half.density_matrix(mu), whole.density_matrix(mu)):
        assert float((x - y).abs().max()) <= 1e-12 * float(y.abs().max())
        assert not torch.equal(x, y)        # (two FP64 forms; the fixed-point kernel's would be one)


@pytest.mark.parametrize("system", [lambda **kw: _large(nu=20, **kw), lambda **kw: _uneven(4.4, **kw)])
def test_kept_bases_in_fp64(system):
    """Exact forces over kept bases against those over bases built again: the same to the bit."""
    kept, two = system(exact_forces=True), system()
    for s in (kept, two):
        s.green_columns()
    mu, _ = kept.find_mu()
    want = kept.omega_gradient(mu)
    built = system(k3_lanes=32)
    built.green_columns()
    for w, g in zip(want, built.omega_gradient(mu)):
        assert torch.equal(g, w)
    for w, g in zip(want, two.omega_gradient(mu)):      # V of half-warp columns
        assert float((g - w).abs().max()) <= 1e-11 * float(w.abs().max())
