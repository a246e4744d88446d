"""The first update collides the state in the buffer, whoever put it there."""
import ctypes as C

import numpy as np
import pytest

from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu



# FP32 D3Q19 forms f_0 again from the initial fields where it may
def _sim(shape, seed, stream=None):
    r, u = I.random_flow(shape, len(shape), seed=seed, rho_amp=0.005, u_amp=0.02)
    s = X.Simulation(9 if len(shape) == 2 else 19, tuple(reversed(shape)), 1.5, "bgk", "f32", stream=stream)
    s.init(r.astype(np.float32), u.astype(np.float32))
    return s, r.astype(np.float32), u.astype(np.float32)


@pytest.mark.parametrize("shape", [(40, 48), (10, 12, 20)])
def test_populations_written_after_init(shape):
    """The pointer of xlb_populations stays valid until the next xlb_step, over
    an xlb_init too."""
    a, r, u = _sim(shape, 101)
    b, _, _ = _sim(shape, 102)
    pa, plane = X.xlb_populations(a.ctx)
    a.init(r, u)
    pb, _ = X.xlb_populations(b.ctx)
    a.synchronize()
    b.synchronize()
    assert C.CDLL("libcuda.so.1").cuMemcpyDtoD_v2(C.c_uint64(pa), C.c_uint64(pb), C.c_size_t(a.Q * plane * 4)) == 0
    for n in (1, 3):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0], b.populations()[0])
    a.step(1)  # and a later xlb_init starts from its fields again
    a.init(r, u)
    c, _, _ = _sim(shape, 101)
    a.step(4)
    c.step(4)
    assert np.array_equal(a.populations()[0], c.populations()[0])
    for s in (a, b, c):
        s.close()


@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("shape", [(40, 48), (10, 12, 20)])
def test_replayed_first_update_takes_the_restored_state(shape, n):
    """A capture of the first updates after xlb_init, replayed on a state
    restored since."""
    st = torch.cuda.Stream()
    a, _, _ = _sim(shape, 103, st.cuda_stream)
    b, _, _ = _sim(shape, 104)
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


@pytest.mark.parametrize("storage,solid", [("bf16", 0.0), ("f32", 0.05)])
def test_first_update_is_no_slower_than_a_local_collision(storage, solid):
    """After a restored state the first update collides what is stored."""
    shape = (128, 256, 256)
    st = torch.cuda.Stream()
    s = X.Simulation(19, tuple(reversed(shape)), 1.5, "bgk", storage, stream=st.cuda_stream)
    if solid:
        s.set_mask(I.random_obstacle_mask(shape, solid, seed=105))
    r, u = torch.ones(shape, device="cuda"), torch.full((3,) + shape, 0.01, device="cuda")
    torch.cuda.synchronize()
    s.init(r, u)
    start = s.state_get().copy()
    us = []
    for restored in (False, True):
        best = []
        for _ in range(10):
            s.state_set(start) if restored else s.init(r, u)
            s.synchronize()
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record(st)
            s.step(1)
            e[1].record(st)
            s.synchronize()
            best.append(e[0].elapsed_time(e[1]))
        us.append(min(best))
    s.close()
    assert us[0] < 1.1 * us[1]
