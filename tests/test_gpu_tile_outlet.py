"""Bodies that reach the column before the OUTLET plane: D2Q9 calls of several
updates (which may run on the tiled kernel) against single updates, bit for bit.
Profiling a context makes it launch every update by itself."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X

pytestmark = pytest.mark.gpu

STORAGES = ["f32", "f16", "bf16"]


def _channel(body):
    """Channel of 420 x 150 cells, INLET and OUTLET planes, and a body: where
    `body` (x, y grids -> bool) holds, off the planes and the walls."""
    ny, nx = 150, 420
    m = I.channel_2d_mask(nx, ny)
    m[1:-1, 0] = O.INLET
    m[1:-1, -1] = O.OUTLET
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    b = body(x, y)
    b[[0, -1], :] = False
    b[:, [0, 1, -1]] = False
    m[b] = O.WALL
    return m


def _links(m, owner):
    """Links (cell, direction toward a body cell, q) of the cells of type owner."""
    c = np.asarray(O.Lattice(9).c)
    rng = np.random.default_rng(91)
    out = []
    for y, x in np.argwhere(m == owner):
        for i in range(1, 9):
            xw, yw = x + c[i, 0], y + c[i, 1]
            if 0 <= xw < m.shape[1] and 0 < yw < m.shape[0] - 1 and m[yw, xw] == O.WALL:
                out.append((x + m.shape[1] * y, i, rng.uniform(0.05, 0.95)))
    return out


def _sims(m, storage, links=()):
    u = np.zeros((2,) + m.shape, np.float32)
    u[0] = 0.04 * O.fluid_like(m)
    sims = []
    for _ in range(2):
        s = X.Simulation(9, (m.shape[1], m.shape[0]), 1.5, "bgk", storage)
        s.set_mask(m)
        s.set_bc(X.XLB_CELL_INLET, 1.0, (0.04, 0.0, 0.0))
        if links:
            s.set_wall_distances(*(np.array(a) for a in zip(*links)))
        s.init(np.ones(m.shape, np.float32), u)
        sims.append(s)
    X.xlb_profile_enable(sims[1].ctx, True)
    return sims


def _compare(a, b, m):
    fl = O.fluid_like(m)
    for n in (2, 5, 30):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl]), n
        assert np.array_equal(a.wall_force(), b.wall_force())
    assert np.all(np.isfinite(a.macroscopic()[1]))
    a.close()
    b.close()


@pytest.mark.parametrize("storage", STORAGES)
def test_wall_distances_of_outlet_cells(storage):
    """A curved body beside the outlet: its links to OUTLET cells take wall
    distances too."""
    m = _channel(lambda x, y: (x - 416.0) ** 2 + (y - 70.3) ** 2 <= 6.2 ** 2)
    links = _links(m, O.FLUID) + _links(m, O.OUTLET)
    assert _links(m, O.OUTLET)
    a, b = _sims(m, storage, links)
    _compare(a, b, m)


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("body", [lambda x, y: (x >= 410) & (abs(y - 75) <= 3),  # a plate that ends at the outlet
                                  lambda x, y: (y <= 1) | (y >= 148),           # walls two cells thick
                                  lambda x, y: (x == 418) & (y == 40)],         # one cell
                         ids=["plate", "thick", "cell"])
def test_wall_before_the_outlet(body, storage):
    """An OUTLET cell whose neighbour at x - 1 is a WALL cell."""
    m = _channel(body)
    a, b = _sims(m, storage)
    _compare(a, b, m)


@pytest.mark.parametrize("storage", STORAGES)
def test_body_one_cell_off_the_outlet(storage):
    """The nearest body that leaves the OUTLET plane's neighbours FLUID."""
    m = _channel(lambda x, y: (x >= 410) & (x <= 417) & (abs(y - 75) <= 3))
    links = _links(m, O.FLUID)
    a, b = _sims(m, storage, links)
    _compare(a, b, m)
