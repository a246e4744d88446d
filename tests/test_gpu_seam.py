"""Curved walls across the periodic seams: D2Q9 calls of several updates (on the
tiled kernel) against single updates, bit for bit, the stochastic rounding of
BF16 ghost values included (it is keyed by the slot they are written to)."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from parity_util import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("center", [(100.4, 0.3), (0.2, 90.7), (0.4, 199.6)], ids=["y", "x", "corner"])
def test_bouzidi_body_across_a_seam(center, storage):
    ny, nx = 200, 320
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    dx, dy = (x - center[0] + nx / 2) % nx - nx / 2, (y - center[1] + ny / 2) % ny - ny / 2
    m = np.where(dx ** 2 + dy ** 2 <= 8.3 ** 2, O.WALL, O.FLUID).astype(np.uint8)
    c = np.asarray(O.Lattice(9).c)
    rng = np.random.default_rng(98)
    links = [(xx + nx * yy, i) for yy, xx in np.argwhere(m == O.FLUID) for i in range(1, 9)
             if m[(yy + c[i, 1]) % ny, (xx + c[i, 0]) % nx] == O.WALL]
    cells, dirs = (np.array(a) for a in zip(*links))
    q = rng.uniform(0.05, 0.95, len(cells))
    r, u = I.random_flow((ny, nx), 2, seed=99, rho_amp=0.005, u_amp=0.02)
    case = Case(9, (ny, nx), 1.6, "bgk", mask=m, rho0=r, u0=u)
    a, b = case.gpu_sim(storage), case.gpu_sim(storage)
    for s in (a, b):
        s.set_wall_distances(cells, dirs, q)
    X.xlb_profile_enable(b.ctx, True)
    fl = O.fluid_like(m)
    for n in (3, 24):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl]), n
        assert np.array_equal(a.wall_force(), b.wall_force())
    a.close()
    b.close()
