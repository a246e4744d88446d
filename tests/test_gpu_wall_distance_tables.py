"""The wall distances by cell that the tiled D2Q9 kernel reads: only where it can
run, whatever the order of the list, and the last entry of a link counts."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from parity_util import Case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_no_table_where_tiles_never_run():
    """4096^2 cells: launched one by one, so the call leaves no table of that
    size behind."""
    n = 4096
    m = np.zeros((n, n), np.uint8)
    m[2000:2003, 2000:2003] = O.WALL
    s = X.Simulation(9, (n, n), 1.5, "bgk", "f32")
    s.set_mask(m)
    s.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s.set_wall_distances([1999 + n * 2001], [1], [0.3])
    s.synchronize()
    assert before - torch.cuda.mem_get_info()[0] < 16 << 20
    s.close()


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_shuffled_and_repeated_links(storage):
    ny, nx = 200, 320
    m = I.channel_2d_mask(nx, ny)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    m[(x - 90.2) ** 2 + (y - 99.6) ** 2 <= 12.7 ** 2] = O.WALL
    cells, dirs, q = I.ball_links(m, (90.2, 99.6), 12.7, O.Lattice(9).c)
    rng = np.random.default_rng(121)
    k = rng.permutation(len(cells))
    r, u = I.random_flow((ny, nx), 2, seed=122, rho_amp=0.005, u_amp=0.02)
    case = Case(9, (ny, nx), 1.6, "bgk", mask=m, rho0=r, u0=u)
    a, b = case.gpu_sim(storage), case.gpu_sim(storage)
    a.set_wall_distances(np.concatenate([cells[::3], cells[k]]), np.concatenate([dirs[::3], dirs[k]]),
                         np.concatenate([1.0 - q[::3], q[k]]))
    b.set_wall_distances(cells, dirs, q)
    X.xlb_profile_enable(b.ctx, True)  # every update by itself
    fl = O.fluid_like(m)
    for n in (2, 25):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl]), n
        assert np.array_equal(a.wall_force(), b.wall_force())
    a.close()
    b.close()
