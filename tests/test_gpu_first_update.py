"""The first update collides the state in the buffer, whoever put it there."""
import ctypes as C

import numpy as np
import pytest

from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (40, 48)


def _sim(seed, stream=None):
    r, u = I.random_flow(SHAPE, 2, seed=seed, rho_amp=0.005, u_amp=0.02)
    s = X.Simulation(9, (48, 40), 1.5, "bgk", "f32", stream=stream)
    s.init(r.astype(np.float32), u.astype(np.float32))
    return s, r.astype(np.float32), u.astype(np.float32)


def test_populations_written_after_init():
    """The pointer of xlb_populations stays valid until the next xlb_step, over
    an xlb_init too."""
    a, r, u = _sim(101)
    b, _, _ = _sim(102)
    pa, plane = X.xlb_populations(a.ctx)
    a.init(r, u)
    pb, _ = X.xlb_populations(b.ctx)
    a.synchronize()
    b.synchronize()
    assert C.CDLL("libcuda.so.1").cuMemcpyDtoD_v2(C.c_uint64(pa), C.c_uint64(pb), C.c_size_t(9 * plane * 4)) == 0
    for n in (1, 3):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0], b.populations()[0])
    a.step(1)  # and a later xlb_init starts from its fields again
    a.init(r, u)
    c, _, _ = _sim(101)
    a.step(4)
    c.step(4)
    assert np.array_equal(a.populations()[0], c.populations()[0])
    for s in (a, b, c):
        s.close()


@pytest.mark.parametrize("n", [1, 3])
def test_replayed_first_update_takes_the_restored_state(n):
    """A capture of the first updates after xlb_init, replayed on a state
    restored since."""
    st = torch.cuda.Stream()
    a, _, _ = _sim(103, st.cuda_stream)
    b, _, _ = _sim(104)
    start = b.state_get().copy()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.step(n)
    a.state_set(start)
    with torch.cuda.stream(st):
        g.replay()
    st.synchronize()
    b.step(n)
    assert np.array_equal(a.populations()[0], b.populations()[0])
    a.close()
    b.close()
