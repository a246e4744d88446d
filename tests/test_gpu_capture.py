"""Updates captured in a caller's CUDA graph: an even number of them ends in the
buffer it began in, so replays go on from each other, whichever kernel takes
them (resident, tiled, overlapping launches, boundary passes)."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from parity_util import Case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(shape):
    d = len(shape)
    r, u = I.random_flow(shape, d, seed=71, rho_amp=0.005, u_amp=0.02)
    m = np.where(I.random_obstacle_mask(shape, 0.04, seed=72) > 0, O.WALL, O.FLUID).astype(np.uint8)
    if d == 3:
        m = I.lid_driven_cavity_mask(shape[2], shape[1], shape[0])
    return Case(9 if d == 2 else 19, shape, 1.5, "bgk", mask=m, lid=(1.0, (0.03, 0.0, 0.0)) if d == 3 else None,
                rho0=r, u0=u)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("shape,n", [((60, 70), 6), ((500, 610), 2), ((500, 610), 10), ((500, 610), 64),
                                     ((13, 21, 35), 4), ((12, 20, 32), 4)])
def test_replayed_capture_continues(shape, n, storage):
    c = _case(shape)
    sims = []
    for replay in (True, False):
        s = torch.cuda.Stream()
        sim = X.Simulation(c.q, tuple(reversed(shape)), 1.5, "bgk", storage, stream=s.cuda_stream)
        sim.set_mask(c.mask)
        sim.set_bc(X.XLB_CELL_LID, 1.0, (0.03, 0.0, 0.0))
        sim.init(c.rho0.astype(np.float32), c.u0.astype(np.float32))
        sim.step(n)
        if replay:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                sim.step(n)
            with torch.cuda.stream(s):
                for _ in range(3):
                    g.replay()
            s.synchronize()
        else:
            sim.step(3 * n)
        sims.append(sim)
    fl = O.fluid_like(c.mask)
    assert np.array_equal(sims[0].populations()[0][:, fl], sims[1].populations()[0][:, fl])
    for x, y in zip(sims[0].macroscopic(), sims[1].macroscopic()):
        assert np.array_equal(x, y)
    for sim in sims:
        sim.close()
