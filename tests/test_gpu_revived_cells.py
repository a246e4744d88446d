"""Solid cells that a new mask turns into fluid in mid-run start from what the run
has left in their slots, not from what a buffer happened to hold or from the
kernel that took the updates."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from parity_util import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape,bc", [((64, 66), False), ((250, 512), False), ((250, 512), True)])
def test_equal_runs_revive_equal_cells(shape, bc, storage):
    """Obstacles of several cells; another run between leaves both buffers changed."""
    r, u = I.random_flow(shape, 2, seed=161, rho_amp=0.005, u_amp=0.02)
    m = np.zeros(shape, np.uint8)
    m[20:30, 20:33] = O.WALL
    m[40:43, 10:50] = O.WALL
    s = Case(9, shape, 1.5, "bgk", mask=m, rho0=r, u0=u).gpu_sim(storage)
    out = []
    for k in range(2):
        s.set_mask(m)
        s.init(r.astype(np.float32), u.astype(np.float32))
        s.step(30)
        if bc:  # (a change that turns the state into its post-stream form first)
            s.set_bc(O.LID, 1.0, (0.0, 0.0, 0.0))
        s.set_mask(np.zeros(shape, np.uint8))
        s.step(3)
        out.append(s.populations()[0].copy())
        s.set_mask(m)
        s.init(None, -3 * u.astype(np.float32))
        for _ in range(30 + k):
            s.step(1)
    assert np.array_equal(out[0], out[1])
    s.close()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("left,right", [(O.WALL, O.WALL), (O.WALL, O.EQ), (O.LID, O.WALL)])
def test_x_faces_served_in_the_pull_or_by_links(left, right, storage):
    """One wall distance of 1/2, the halfway rule, makes links serve the x-faces."""
    sh = (8, 10, 37)
    m = np.zeros(sh, np.uint8)
    m[:, :, 0] = left
    m[:, :, -1] = right
    r, u = I.random_flow(sh, 3, seed=162, rho_amp=0.005, u_amp=0.02)
    c = Case(19, sh, 1.5, "bgk", mask=m, lid=(1.0, (0.0, 0.02, 0.01)), eq=(1.0, (0.01, 0.0, 0.0)), rho0=r, u0=u)
    a, b = c.gpu_sim(storage), c.gpu_sim(storage)
    lat = np.asarray(O.Lattice(19).c)
    x, cx = (1, -1) if left == O.WALL else (35, 1)
    i = [k for k in range(1, 19) if tuple(lat[k]) == (cx, 0, 0)][0]
    b.set_wall_distances([x + 37 * (4 + 10 * 3)], [i], [0.5])
    free = np.zeros(sh, np.uint8)
    for s in (a, b):
        s.step(5)
    assert np.array_equal(a.populations()[0][:, m == 0], b.populations()[0][:, m == 0])
    for s in (a, b):
        s.set_mask(free)
    assert np.array_equal(a.populations()[0], b.populations()[0])
    a.close()
    b.close()
