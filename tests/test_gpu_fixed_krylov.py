"""The fixed-point Krylov kernel (Slater-Koster systems) against the FP64 one, which the same H and S
take when the caller sets them (elses_set_hs), at the sizes where the former's work is split: the
units of a thread (128 and 384 threads), vectors in tensor memory, shared memory and scratch, the
first steps in FP64, clusters it leaves to the FP64 kernel, both Gram-Schmidt forms, kept bases.

Both round at the level of 2^-53 of H's and S's rows; rho moves by that times the column's
conditioning, for which the two FP64 forms are gated at 1e-12 of the largest entry."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu

RHO_TOL = 1e-12


@pytest.fixture(scope="module")
def eg():
    import paper_1210_1531_gb300
    return paper_1210_1531_gb300


def _system(n, seed=3):
    """n atoms of a displaced diamond in its periodic box (whole cells kept, the rest vacancies)."""
    side = max(2, int(np.ceil((n / 8) ** (1 / 3))))
    pos, box = wl.diamond((side, side, side), sigma=0.08, seed=seed)
    return np.ascontiguousarray(pos[:n]), box


def _pair(eg, pos, box, r_cluster, nu, **kw):
    make = lambda: eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, nu, 0.1,  # noqa: E731
                             4.0 * len(pos), **kw)
    a, b = make(), make()
    b.set_hs(*a.hs())
    return a, b


@pytest.mark.parametrize("n, nu, r_cluster, reorth", [
    (1, 3, 0.0, 0), (2, 8, 0.0, 1),                                  # a single atom, a pair
    (63, 1, 0.0, 0), (64, 2, 0.0, 1), (65, 3, 0.0, 0),               # one column per CTA: 126, 128, 130 units
    (64, 4, 0.0, 0), (65, 5, 0.0, 1), (64, 33, 0.0, 0),              # around the FP64 steps; past a warp of vectors
    (72, 64, 0.0, 1),                                                # the largest nu
    (330, 18, 0.0, 1), (340, 12, 0.0, 0),                            # the largest cluster, and one past it
    (512, 21, 4.3, 0), (512, 30, 6.0, 1), (500, 30, 5.1, 0),         # four columns per CTA, ragged clusters
])
def test_matches_the_fp64_kernel(eg, n, nu, r_cluster, reorth):
    pos, box = _system(n)
    a, b = _pair(eg, pos, box, r_cluster, nu, reorth=reorth)
    a.green_columns()
    b.green_columns()
    mu, _ = a.find_mu()
    sa, sb = a.spectra(), b.spectra()
    assert torch.equal(sa["nu_eff"], sb["nu_eff"])
    for x, y in zip(a.density_matrix(mu), b.density_matrix(mu)):
        assert float((x - y).abs().max()) <= RHO_TOL * float(y.abs().max())
    ea, eb = a.energies(mu), b.energies(mu)
    assert abs(ea["E_band"] - eb["E_band"]) <= 1e-12 * abs(eb["E_band"])


def test_results_do_not_depend_on_batches_or_schedule(eg):
    pos, box = _system(512)
    args = (torch.tensor(pos, device="cuda"), box, wl.sk_params(), 5.5, 24, 0.1, 2048.0)
    ref = eg.System(*args).energy_force()
    for kw in (dict(schedule=1), dict(schedule=1, batch_atoms=100, keep_factors=1000), dict(two_pass=True)):
        got = eg.System(*args, **kw).energy_force()
        assert got[0] == ref[0] and got[1] == ref[1] and torch.equal(got[3], ref[3]), kw


def test_overlap_that_is_not_positive_definite_is_reported(eg):
    sk = wl.sk_params()
    bad = type(sk)(**{**sk.__dict__, "S0": tuple(6.0 * s for s in sk.S0)})
    pos, box = _system(64)
    s = eg.System(torch.tensor(pos, device="cuda"), box, bad, 0.0, 12, 0.1, 256.0)
    with pytest.raises(eg.ElsesError) as err:
        s.green_columns()
    assert err.value.code == -2
