"""Wall distances on the links of WALL x-face planes, which 16-bit storage keeps
in the link table: every kernel applies them, in whatever calls the updates are
taken."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from parity_util import Case

pytestmark = pytest.mark.gpu


def _x_links(m):
    """Links of the cells beside the WALL planes x = 0 and x = nx - 1, away from
    the other planes' cells, with seeded distances."""
    d = m.ndim
    c = np.asarray(O.Lattice(9 if d == 2 else 19).c)
    rng = np.random.default_rng(92)
    nx = m.shape[-1]
    cells, dirs = [], []
    for side, x in ((-1, 1), (1, nx - 2)):
        for i in range(1, c.shape[0]):
            if c[i, 0] != side:
                continue
            at = np.argwhere(m[..., x] == O.FLUID)
            at = at[np.all((at >= 2) & (at < np.array(m.shape[:-1]) - 2), axis=1)]
            cells.append(np.ravel_multi_index(tuple(at.T) + (np.full(len(at), x),), m.shape))
            dirs.append(np.full(len(at), i))
    cells, dirs = np.concatenate(cells), np.concatenate(dirs)
    return cells, dirs, rng.uniform(0.05, 0.95, len(cells)).astype(np.float32)


def _case(shape):
    m = np.zeros(shape, np.uint8)
    m[..., 0] = m[..., -1] = O.WALL
    r, u = I.random_flow(shape, len(shape), seed=93, rho_amp=0.005, u_amp=0.02)
    return Case(9 if len(shape) == 2 else 19, shape, 1.5, "bgk", mask=m, rho0=r, u0=u)


def _sim(c, storage, variant, links):
    s = c.gpu_sim(storage, variant)
    if links is not None:
        s.set_wall_distances(*links)
    return s


@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_distances_in_one_cell_and_vector_kernels(storage):
    c = _case((10, 12, 36))
    links = _x_links(c.mask)
    a, b, h = _sim(c, storage, "direct", links), _sim(c, storage, "vec2", links), _sim(c, storage, "direct", None)
    fl = O.fluid_like(c.mask)
    for n in (1, 6):
        for s in (a, b, h):
            s.step(n)
        assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl])
        assert np.array_equal(a.wall_force(), b.wall_force())
    assert not np.array_equal(a.populations()[0][:, fl], h.populations()[0][:, fl])  # the distances act
    for s in (a, b):  # and halfway walls come back without them
        s.set_wall_distances([], [], [])
        s.step(5)
    assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl])
    for s in (a, b, h):
        s.close()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_distances_in_calls_of_one_and_of_several_updates(storage):
    c = _case((203, 301))
    links = _x_links(c.mask)
    a, b = _sim(c, storage, "auto", links), _sim(c, storage, "auto", links)
    fl = O.fluid_like(c.mask)
    a.step(9)
    for _ in range(9):
        b.step(1)
    assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl])
    assert np.array_equal(a.wall_force(), b.wall_force())
    a.close()
    b.close()
