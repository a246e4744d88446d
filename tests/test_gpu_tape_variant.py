"""A change of the bulk variant while a tape is open: the adjoint replays the
segments from the checkpoints with the variant of the moment."""
import numpy as np
import pytest

from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from parity_util import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,k", [(12, 4), (7, 3), (5, 1)])
@pytest.mark.parametrize("taken,replayed", [("direct", "vec2"), ("direct", "vec"), ("vec2", "direct")])
def test_variant_changed_before_the_adjoint(taken, replayed, T, k):
    sh = (8, 12, 36)
    r, u = I.random_flow(sh, 3, seed=94, rho_amp=0.005, u_amp=0.02)
    c = Case(19, sh, 1.5, "bgk", mask=I.lid_driven_cavity_mask(36, 12, 8), lid=(1.0, (0.03, 0.0, 0.0)), rho0=r, u0=u)
    out = []
    for later in (taken, replayed):
        s = c.gpu_sim("f16", taken)
        X.xlb_tape_begin(s.ctx, T, k)
        s.step(T)
        s.set_kernel(later)
        X.xlb_adjoint_seed_macro(s.ctx, np.random.default_rng(95).standard_normal(sh).astype(np.float32), None)
        X.xlb_adjoint_step(s.ctx, T)
        g, gu = np.empty(sh, np.float32), np.empty((3,) + sh, np.float32)
        X.xlb_adjoint_init_grad(s.ctx, g, gu)
        out.append((g, gu))
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
