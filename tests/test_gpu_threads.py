"""Systems of different cluster sizes driven from several threads at once, a stream each: a kernel's
shared-memory limit is one for all of them, and every thread gets the results it gets alone."""
import threading

import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [((4, 4, 4), 6.0, 30, 1), ((2, 2, 2), 0.0, 8, 0), ((4, 4, 4), 4.3, 20, 0), ((3, 3, 3), 0.0, 40, 1)]


def _pass(shape, stream):
    import paper_1210_1531_gb300 as eg
    cells, r_cluster, nu, reorth = shape
    pos, box = wl.diamond(cells, sigma=0.05, seed=3)
    with torch.cuda.stream(stream):
        s = eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, nu, 0.1, 4.0 * len(pos),
                      reorth=reorth, schedule=1)
        out = s.energy_force()
        stream.synchronize()
        return out[1], out[3].clone()


def test_threads_get_what_they_get_alone():
    want = [_pass(s, torch.cuda.Stream()) for s in SHAPES]
    got = [[] for _ in SHAPES]

    def work(k):
        stream = torch.cuda.Stream()
        for _ in range(6):
            got[k].append(_pass(SHAPES[k], stream))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(SHAPES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w, g in zip(want, got):
        assert len(g) == 6 and all(e == w[0] and torch.equal(f, w[1]) for e, f in g)
