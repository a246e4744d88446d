"""The serialized state of a run is a function of the run: also the slots of
solid cells, whatever the buffers held before."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from parity_util import Case

pytestmark = pytest.mark.gpu


# (whole multiples of 256 bytes a plane: no padding; an obstacle that is not a
# face plane, which single updates rewrite)
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", [(64, 66), (250, 512)])  # one launch a call; tiles
def test_equal_runs_give_equal_bytes(shape, storage):
    r, u = I.random_flow(shape, 2, seed=96, rho_amp=0.005, u_amp=0.02)
    m = np.where(I.random_obstacle_mask(shape, 0.05, seed=97) > 0, O.WALL, O.FLUID).astype(np.uint8)
    s = Case(9, shape, 1.5, "bgk", mask=m, rho0=r, u0=u).gpu_sim(storage)
    states = []
    for n in (4, 10, 13):
        for _ in range(2):
            s.init(r.astype(np.float32), u.astype(np.float32))
            s.step(n)
            states.append(s.state_get().copy())
            # another run between, launch by launch, leaves both buffers changed
            s.init(None, -u.astype(np.float32))
            for _ in range(n):
                s.step(1)
        assert np.array_equal(states[-1], states[-2])
    s.close()
