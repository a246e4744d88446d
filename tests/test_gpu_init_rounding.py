"""f_0 in BF16 storage is the FP32 f_0 rounded by the published rule: 16 random bits
per value from a hash of the cell and of the FP32 bits of its values."""
import numpy as np
import pytest

from paper_2311_16080_gb300 import inputs as I
from parity_util import Case

pytestmark = pytest.mark.gpu

M = 0xFFFFFFFF


def _fmix32(h):
    h = h ^ (h >> 16)
    h = h * 0x85EBCA6B & M
    h = h ^ (h >> 13)
    h = h * 0xC2B2AE35 & M
    return h ^ (h >> 16)


def _rounded(f32):
    """BF16 bits of the deviations f32 [Q, cells]."""
    b = f32.view(np.uint32).astype(np.uint64)
    s0 = _fmix32((np.arange(b.shape[1], dtype=np.uint64) * 0x9E3779B9 & M) ^ np.bitwise_xor.reduce(b, axis=0))
    out, m, a = [], 747796405, 2891336453
    for row in b:
        out.append(((row + ((s0 * m & M) + a & M) // 65536 & M) // 65536).astype(np.uint16))
        m, a = m * 747796405 & M, (a * 747796405 + 2891336453) & M
    return np.stack(out)


@pytest.mark.parametrize("q,shape", [(9, (60, 70)), (9, (33, 128)), (19, (12, 14, 20)), (27, (9, 10, 17))])
def test_bf16_initial_state_is_the_rounded_fp32_one(q, shape):
    r, u = I.random_flow(shape, len(shape), seed=171, rho_amp=0.01, u_amp=0.03)
    c = Case(q, shape, 1.4, rho0=r, u0=u)
    a, b = c.gpu_sim("f32"), c.gpu_sim("bf16")
    f32, bf16 = a.populations()[0].reshape(q, -1).copy(), b.populations()[0].reshape(q, -1)
    assert np.array_equal(_rounded(f32), bf16)
    a.close()
    b.close()
