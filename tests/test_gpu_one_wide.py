"""Lattices one cell wide in x: against the FP64 oracle, and no slower than the
same number of cells in one row (rows of one cell would leave 127 of 128 lanes
idle)."""
import time

import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from parity_util import Case, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("q,shape", [(9, (1, 1)), (9, (129, 1)), (9, (700, 1)), (19, (1, 130, 1)), (19, (9, 31, 1)),
                                     (27, (6, 50, 1))])
def test_one_wide_lattices_match_oracle(q, shape, storage):
    r, u = I.random_flow(shape, len(shape), seed=141, rho_amp=0.005, u_amp=0.02)
    m = np.zeros(shape, np.uint8)
    if shape[-2] > 30:
        m[..., 0, :] = O.WALL
        m[..., 7, :] = O.WALL
    c = Case(q, shape, 1.4, "bgk", mask=m, rho0=r, u0=u)
    (_, uo), _ = c.oracle(12)
    _, ug = c.gpu(12, storage)
    fl = O.fluid_like(c.mask)
    assert rel_l2(ug[:, fl], uo[:, fl]) <= (1e-4 if storage == "f32" else 5e-3)


def test_one_wide_costs_what_one_row_costs():
    us = {}
    for dims in ((1, 1000000), (1000000, 1)):
        s = X.Simulation(9, dims, 1.4, "bgk", "f32")
        rho = torch.ones(dims[1], dims[0], device="cuda")
        u = torch.zeros(2, dims[1], dims[0], device="cuda")
        torch.cuda.synchronize()
        s.init(rho, u)
        best = []
        for call in (lambda: s.step(1), lambda: s.macroscopic(rho, u)):
            t = []
            for _ in range(8):
                s.synchronize()
                t0 = time.perf_counter()
                call()
                s.synchronize()
                t.append(time.perf_counter() - t0)
            best.append(min(t))
        us[dims] = best
        s.close()
    for one, row in zip(us[(1, 1000000)], us[(1000000, 1)]):
        assert one < 4 * row
