"""The fixed-point Krylov kernel, of Slater-Koster systems and of a caller's matrices (elses_set_hs),
against the FP64 one, which takes over where the rows of H or S differ too much in size: the basis
functions of an atom on its own are scaled by 32, which is exact and changes nothing but that atom's
block of rho. At the sizes where the work is split: the
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


def _forms(eg, n, r_cluster, nu, **kw):
    """The system of n atoms (the last on its own in a vacuum), the same as caller matrices, the same
    with the last atom's functions scaled, and that scale by block of H, S and rho."""
    pos, box = _system(n - 1)
    box = np.array(box, dtype=np.float64)
    pos = np.concatenate([pos, [[0.0, 0.0, box[2] + 10.0]]])
    box[2] += 20.0
    make = lambda: eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, nu, 0.1,  # noqa: E731
                             4.0 * n, **kw)
    sk, caller, fp64 = make(), make(), make()
    H, S = sk.hs()
    caller.set_hs(H, S)
    d = torch.ones_like(H)
    d[-1] = 1024.0
    assert int(sk.pattern()[0][-2]) == len(H) - 1
    fp64.set_hs(H * d, S * d)
    return sk, caller, fp64, d


@pytest.mark.parametrize("n, nu, r_cluster, reorth", [
    (2, 3, 0.0, 0), (3, 8, 0.0, 1),                                  # single atoms, a pair
    (63, 1, 0.0, 0), (64, 2, 0.0, 1), (65, 3, 0.0, 0),               # one column per CTA: 126, 128, 130 units
    (64, 4, 0.0, 0), (65, 5, 0.0, 1), (64, 33, 0.0, 0),              # around the FP64 steps; past a warp of vectors
    (72, 64, 0.0, 1),                                                # the largest nu
    (330, 18, 0.0, 1), (340, 12, 0.0, 0),                            # the largest cluster, and one past it
    (512, 21, 4.3, 0), (512, 30, 6.0, 1), (500, 30, 5.1, 0),         # four columns per CTA, ragged clusters
])
def test_matches_the_fp64_kernel(eg, n, nu, r_cluster, reorth):
    sk, caller, fp64, d = _forms(eg, n, r_cluster, nu, reorth=reorth)
    for s in (sk, caller, fp64):
        s.green_columns()
    mu, _ = fp64.find_mu()
    ref = [x * d for x in fp64.density_matrix(mu)]
    e_ref, sp_ref = fp64.energies(mu)["E_band"], fp64.spectra()
    for s in (sk, caller):
        assert torch.equal(s.spectra()["nu_eff"], sp_ref["nu_eff"])
        for x, y in zip(s.density_matrix(mu), ref):
            assert float((x - y).abs().max()) <= RHO_TOL * float(y.abs().max())
        assert abs(s.energies(mu)["E_band"] - e_ref) <= 1e-12 * abs(e_ref)


def test_caller_matrices_under_capture_and_after_other_matrices(eg):
    """The choice of kernel is made on the device with every set_hs, also in a captured one."""
    sk, caller, fp64, d = _forms(eg, 64, 0.0, 12)
    H, S = sk.hs()
    caller.green_columns()
    fp64.green_columns()
    want, want64 = caller.spectra()["eps"].clone(), fp64.spectra()["eps"].clone()
    Hin, Sin = H.clone(), S.clone()
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=st):
            caller.set_hs(Hin, Sin, stream=st)
    for f, w in ((1.0, want), (d, want64), (1.0, want)):
        Hin.copy_(H * f)
        Sin.copy_(S * f)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        caller.set_hs(Hin, Sin)
        caller.green_columns()
        assert torch.equal(caller.spectra()["eps"], w)


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
