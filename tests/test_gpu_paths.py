"""Which D2Q9 calls take several updates in a launch, by the kernels they queue:
the other tests compare such calls with single updates and would hold as well
if both went the same way."""
import numpy as np
import pytest

from oracle import lbm as O
from paper_2311_16080_gb300 import inputs as I
from paper_2311_16080_gb300 import xlb as X
from graph_util import kernels_of
from parity_util import Case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 40


def _kernels(shape, storage, variant="auto", prepare=None, mask=None, steps=N):
    st = torch.cuda.Stream()
    r, u = I.random_flow(shape, 2, seed=111, rho_amp=0.005, u_amp=0.02)
    if mask is None:
        mask = np.where(I.random_obstacle_mask(shape, 0.05, seed=112) > 0, O.WALL, O.FLUID).astype(np.uint8)
    s = X.Simulation(9, (shape[1], shape[0]), 1.5, "bgk", storage, stream=st.cuda_stream)
    s.set_kernel(variant)
    s.set_mask(mask)
    if prepare:
        prepare(s)
    s.init(r.astype(np.float32), u.astype(np.float32))
    s.step(1)
    n = kernels_of(st.cuda_stream, lambda: s.step(steps))
    s.close()
    return n


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_small_lattices_take_one_launch(storage):
    assert _kernels((64, 66), storage) <= 3  # and the ghost values of the last state


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", [(150, 420), (203, 301), (200, 320), (250, 512)])
def test_larger_lattices_take_several_updates_a_launch(shape, storage):
    assert _kernels(shape, storage) < N // 2


def test_profiled_updates_are_launched_one_by_one():
    assert _kernels((64, 66), "f32", prepare=lambda s: X.xlb_profile_enable(s.ctx, True)) >= N


@pytest.mark.parametrize("storage,variant", [("f32", "direct"), ("f16", "vec"), ("bf16", "vec2")])
@pytest.mark.parametrize("shape", [(64, 68), (200, 320)])
def test_a_chosen_variant_launches_every_update(shape, storage, variant):
    assert _kernels(shape, storage, variant) >= N


# (us launched one by one / together: 4.6 / 9.2, 8.3 / 12.8, 28.3 / 42.9, 84.8 / 128.6)
@pytest.mark.parametrize("shape,storage,n", [((128, 128), "f32", 2), ((599, 601), "f16", 2), ((1000, 1200), "f16", 4),
                                             ((1000, 1200), "f16", 12), ((800, 900), "bf16", 24)])
def test_calls_that_gain_nothing_launch_every_update(shape, storage, n):
    assert _kernels(shape, storage, mask=np.zeros(shape, np.uint8), steps=n) == n
