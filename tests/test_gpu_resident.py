"""The resident D2Q9 kernel (a domain in the shared memory of one cluster, many
updates in one launch) and the tiled one (larger lattices, several updates per
launch) against the update-by-update kernels, bit for bit:
profiling a context makes it launch every update by itself.  Sizes at the
edges of its shapes: fewer rows than blocks, one and two cells per thread and
more, rows that do not divide among the blocks, odd and even update counts,
domains that only fit packed, and the limit beyond which calls are launched as
before."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from parity_util import Case

pytestmark = pytest.mark.gpu


def _case(nx, ny, collision="bgk", walls=True):
    r, u = I.random_flow((ny, nx), 2, seed=61, rho_amp=0.005, u_amp=0.02)
    m = None
    if walls:
        m = I.channel_2d_mask(nx, ny)
        m[I.random_obstacle_mask((ny, nx), 0.07, seed=62) > 0] = O.WALL
    return Case(9, (ny, nx), 1.6, collision, mask=m, force=(2e-5, -1e-5, 0.0) if walls else None, rho0=r, u0=u)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny,collision,walls", [
    (1, 1, "bgk", False), (7, 3, "bgk", False), (33, 16, "bgk", True), (45, 47, "kbc", True),
    (128, 128, "bgk", False), (129, 127, "bgk", True), (131, 200, "kbc", False), (256, 250, "bgk", True),
    (1000, 17, "bgk", True), (400, 300, "bgk", False)])
def test_resident_equals_update_by_update(nx, ny, collision, walls, storage):
    c = _case(nx, ny, collision, walls)
    a, b = c.gpu_sim(storage), c.gpu_sim(storage)
    X.xlb_profile_enable(b.ctx, True)
    fl = O.fluid_like(c.mask)
    for n in (1, 2, 5, 8):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl]), n
    for x, y in zip(a.macroscopic(), b.macroscopic()):  # the ghost values of the last state
        assert np.array_equal(x, y)
    if walls:
        assert np.array_equal(a.wall_force(), b.wall_force())
    a.close()
    b.close()


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_batch_shapes_equal_per_domain_launches(storage):
    sizes = [(1, 1), (5, 2), (200, 14), (90, 90), (256, 40), (256, 128), (250, 127), (300, 160), (310, 300)]
    doms = []
    for nx, ny in sizes:  # the last does not fit a cluster: it takes the queue
        c = _case(nx, ny)
        m = c.mask if ny > 2 else np.zeros((ny, nx), np.uint8)
        doms.append(dict(nx=nx, ny=ny, mask=m.astype(np.uint8), force=(1e-5, 0.0)))
    a, b = X.Batch(doms, 1.4, storage), X.Batch(doms, 1.4, storage)
    for x in (a, b):
        x.set_masks()
        x.init()
    for n in (9, 12):
        a.step(n)
        b.step_per_domain(n)
        for (ra, ua), (rb, ub) in zip(a.macroscopic(), b.macroscopic()):
            assert np.array_equal(ra, rb) and np.array_equal(ua, ub), n
    a.close()
    b.close()


def test_resident_segments_of_a_tape():
    """An open tape records its checkpoints between the launches."""
    c = _case(60, 40, walls=False)
    g = []
    for k in (4, 50):
        s = c.gpu_sim()
        X.xlb_tape_begin(s.ctx, 23, k)
        s.step(23)
        seed = np.ones((40, 60), np.float32)
        X.xlb_adjoint_seed_macro(s.ctx, seed, None)
        X.xlb_adjoint_step(s.ctx, 23)
        out = np.empty((40, 60), np.float32)
        X.xlb_adjoint_init_grad(s.ctx, out, None)
        g.append(out)
        s.close()
    assert np.array_equal(g[0], g[1])


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny,collision,walls", [
    (160, 150, "bgk", False), (301, 203, "bgk", True), (257, 499, "kbc", True), (1200, 40, "bgk", True)])
def test_tiles_equal_update_by_update(nx, ny, collision, walls, storage):
    c = _case(nx, ny, collision, walls)
    a, b = c.gpu_sim(storage), c.gpu_sim(storage)
    X.xlb_profile_enable(b.ctx, True)
    fl = O.fluid_like(c.mask)
    for n in (1, 2, 17):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl]), n
    if walls:
        assert np.array_equal(a.wall_force(), b.wall_force())
    a.close()
    b.close()


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("graph", [0, 9])
@pytest.mark.parametrize("n_d,inlet,bouzidi", [(10, "zou_he", True), (20, "regularized", True), (14, "zou_he", False)])
def test_tiles_with_inflow_outflow_and_curved_walls(n_d, inlet, bouzidi, graph, storage):
    from test_gpu_cylinder import Cyl
    c = Cyl(n_d=n_d, u_mean=0.04, inlet=inlet, bouzidi=bouzidi)
    a, b = c.gpu(storage), c.gpu(storage)
    a.set_step_graph(graph)
    X.xlb_profile_enable(b.ctx, True)
    fl = O.fluid_like(c.mask)
    for n in (2, 3, 40):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations()[0][:, fl], b.populations()[0][:, fl]), n
        assert np.array_equal(a.wall_force(), b.wall_force())
    a.close()
    b.close()


@pytest.mark.parametrize("T,k,chunks", [(1, 1, (1,)), (2, 2, (2,)), (12, 4, (12,)), (13, 4, (5, 6, 2)), (9, 20, (4, 5)),
                                        (11, 5, (10, 1)), (8, 1, (8,))])
def test_last_tape_segment_needs_no_recomputation(T, k, chunks):
    """The forward pass keeps the last segment's states in the tape slots: the
    gradient equals the one of a forward pass that profiles (and so launches
    every update by itself and keeps nothing), in any chunks, and the state
    between the chunks is the live one."""
    sh = (6, 7, 10)
    r, u = I.random_flow(sh, 3, seed=81, rho_amp=0.01, u_amp=0.02)
    m = I.lid_driven_cavity_mask(10, 7, 6)
    c = Case(19, sh, 1.4, "bgk", mask=m, lid=(1.0, (0.03, 0.0, 0.0)), rho0=r, u0=u)
    out = []
    for mode in ("keep", "profile", "mixed"):
        s = c.gpu_sim()
        X.xlb_tape_begin(s.ctx, T, k)
        for i, n in enumerate(chunks):
            X.xlb_profile_enable(s.ctx, mode == "profile" or (mode == "mixed" and i % 2 == 1))
            s.step(n)
            mid = s.macroscopic()
        X.xlb_adjoint_seed_macro(s.ctx, np.ones(sh, np.float32), None)
        X.xlb_adjoint_step(s.ctx, T)
        g = np.empty(sh, np.float32)
        X.xlb_adjoint_init_grad(s.ctx, g, None)
        out.append((g,) + mid)
        s.close()
    for other in out[1:]:
        for x, y in zip(out[0], other):
            assert np.array_equal(x, y)
