"""The projected reduction around 2^-40, where its first-order form (S' = I + E) hands over to Cholesky. An
antisymmetric part d A of the caller's S goes into S' as E of that size, as Gram-Schmidt, which takes its
products the other way round, does not see it. rho then moves by d D; D is taken at d = 2^-30 (Cholesky; what
is quadratic in d is below 1e-16 there), and every d from 2^-46 to 2^-34 has to give rho(0) + d D.
Bound 2e-13: ten times what the forms of the FP64 kernels differ by on such a system; leaving E out would
be off by d |D|, 1e-12 and more at 2^-40."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [12, 33])
def test_rho_is_linear_in_the_antisymmetric_part(nu):
    import paper_1210_1531_gb300 as eg
    pos, box = wl.diamond((2, 2, 2), sigma=0.05, seed=3)
    n = len(pos)
    s = eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), 0.0, nu, 0.1, 4.0 * n)
    H, S = s.hs()
    rp, ci = (x.cpu().numpy() for x in s.pattern())
    rows = np.repeat(np.arange(n), np.diff(rp))
    A = np.random.default_rng(5).standard_normal((n, n, 4, 4))
    A = A - A.transpose(1, 0, 3, 2)
    A = torch.tensor(A[rows, ci], device="cuda")

    def rho(d):
        s.set_hs(H, S + d * A)
        s.green_columns()
        return s.density_matrix(3.0)[0].clone()

    zero = rho(0.0)
    D = (rho(2.0 ** -30) - zero) * 2.0 ** 30
    assert float(D.abs().max()) > 1.0
    for k in range(34, 47):
        assert float((rho(2.0 ** -k) - zero - 2.0 ** -k * D).abs().max()) <= 2e-13, k
