"""xlb_reduce sums the fluid-like cells alone, whatever the EQ cells prescribe."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from parity_util import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,shape", [(9, (60, 70)), (19, (12, 14, 33)), (27, (9, 10, 17))])
def test_mass_and_momentum_beside_eq_cells(q, shape):
    d = len(shape)
    m = I.random_obstacle_mask(shape, 0.2, seed=131, code=O.EQ)
    m[I.random_obstacle_mask(shape, 0.1, seed=132) > 0] = O.WALL
    r, u = I.random_flow(shape, d, seed=133, rho_amp=0.005, u_amp=0.02)
    s = Case(q, shape, 1.5, "bgk", mask=m, eq=(1.01, (0.1, 0.05, 0.02)), rho0=r, u0=u).gpu_sim()
    fl = O.fluid_like(m)
    for n in (0, 1, 4):
        s.step(n)
        rho, vel = s.macroscopic()
        rho, vel = rho.astype(np.float64), vel.astype(np.float64)
        mass, mom = s.reduce()
        # (FP32 observables: a few roundings of 6e-8 each)
        assert abs(mass - rho[fl].sum()) <= 1e-6 * rho[fl].sum()
        for a in range(d):
            want = (rho * vel[a])[fl]
            assert abs(mom[a] - want.sum()) <= 1e-6 * rho[fl].sum()
    s.close()
