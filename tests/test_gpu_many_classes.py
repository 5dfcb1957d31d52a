"""More cluster size classes than sixteen, the one with the most atoms last: each class launch has a work
queue of its own, as the classes run at the same time. The work-queue form against the static order, bit
for bit."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


def _islands():
    """Pieces of displaced diamond of 24 to 296 atoms, and many of 8, each on its own, 38 A apart."""
    pos, _ = wl.diamond((6, 6, 6), sigma=0.05, seed=3)
    centre = pos.mean(axis=0)
    order = np.argsort(np.linalg.norm(pos - centre, axis=1))
    sizes = [16 * k + 8 for k in range(1, 19)] + [8] * 100
    sites = np.stack(np.meshgrid(*[np.arange(5)] * 3, indexing="ij"), -1).reshape(-1, 3) * 38.0 + 19.0
    return np.concatenate([pos[order[:s]] - centre + sites[i] for i, s in enumerate(sizes)]), np.full(3, 190.0)


@pytest.mark.parametrize("lanes", [0, 32])
def test_queues_of_their_own(lanes):
    import paper_1210_1531_gb300 as eg
    pos, box = _islands()
    make = lambda schedule: eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), 12.0, 8, 0.1,  # noqa: E731
                                      4.0 * len(pos), schedule=schedule, k3_lanes=lanes)
    static, queued = make(0), make(1)
    static.green_columns()
    want = static.spectra()
    sizes = np.diff(static.clusters()[0].cpu().numpy())
    slots = -(-sizes // (32 if lanes else 16))
    if lanes == 0:
        assert len(np.unique(slots)) > 16 and np.bincount(slots).argmax() == 1
    for _ in range(8):
        queued.green_columns()
        got = queued.spectra()
        assert torch.equal(got["nu_eff"], want["nu_eff"]) and torch.equal(got["eps"], want["eps"])
        assert torch.equal(got["c"], want["c"])
