"""The first update collides the state in the buffer, whoever put it there."""
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
