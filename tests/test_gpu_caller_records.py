"""elses_set_hs and the fixed-point kernel's records of the caller's blocks: whichever way H and S came
to be written (a call, or a replay of a captured one, before or after other calls), the columns are
those of the matrices written last; and the call allocates nothing, so that another stream may be
captured around it."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eg():
    import paper_1210_1531_gb300
    return paper_1210_1531_gb300


def _system(eg, cells=(2, 2, 2), r_cluster=0.0, nu=12, **kw):
    pos, box = wl.diamond(cells, sigma=0.05, seed=3)
    return eg.System(torch.tensor(pos, device="cuda"), box, wl.sk_params(), r_cluster, nu, 0.1, 4.0 * len(pos), **kw)


def _poles(s):
    s.green_columns()
    return s.spectra()["eps"].clone()


def test_columns_are_of_the_matrices_written_last(eg):
    s, own = _system(eg), _system(eg)
    H, S = own.hs()
    want = {}
    for f in (1.0, 1.25, 0.5):
        own.set_hs(H * f, S)
        want[f] = _poles(own)
    Hin, Sin = H.clone(), S.clone()
    st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(st), torch.cuda.graph(g, stream=st):
        s.set_hs(Hin, Sin, stream=st)            # the first set_hs of the system is a captured one

    def replay(f):
        Hin.copy_(H * f)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()

    replay(1.0)
    assert torch.equal(_poles(s), want[1.0])
    s.set_hs(H * 1.25, S)
    assert torch.equal(_poles(s), want[1.25])
    replay(0.5)
    assert torch.equal(_poles(s), want[0.5])
    replay(1.0)
    assert torch.equal(_poles(s), want[1.0])


def test_a_replay_leaves_the_records_of_a_rebuilt_system_alone(eg):
    """After a rebuild the two-centre form is in use; what a replay then writes is not its input."""
    s = _system(eg)
    want, (H, S) = _poles(s), s.hs()
    st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(st), torch.cuda.graph(g, stream=st):
        s.set_hs(H, S, stream=st)
    s.rebuild(s._pos)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(_poles(s), want)


def test_set_hs_while_another_stream_is_captured(eg):
    s, own = _system(eg), _system(eg)
    H, S = own.hs()
    own.set_hs(H, S)
    x = torch.zeros(4, device="cuda")
    st, other, g = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        g.capture_begin()
        x += 1
        s.set_hs(H, S, stream=other)
        g.capture_end()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 1.0 and torch.equal(_poles(s), _poles(own))


def test_set_hs_allocates_nothing(eg):
    s = _system(eg, cells=(16, 16, 16), r_cluster=4.0, nu=6)
    H, S = s.hs()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s.set_hs(H, S)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    assert np.isfinite(float(_poles(s).sum()))
