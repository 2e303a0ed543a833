"""lbm_init at the ends of the range: float pairs (FP32 and 16-bit storage) hold neither the squares of huge gradients nor
all bits of tiny values, and such nodes are formed in FP64.  Each FP32 lattice against an FP64 one with the same
inputs, whose populations rounded to FP32 it holds."""
import numpy as np
import pytest
import torch

from paper_1704_07559_gb300 import lbm
from test_gpu_parity import f64, rates

pytestmark = pytest.mark.gpu


def states(q, dims, drho, u, g, **kw):
    """The FP32 lattice's populations, and the FP64 one's rounded to FP32."""
    out = []
    for precision in ("fp32", "fp64"):
        lat = lbm.Lattice(q, *dims, rates=rates(q, 0.6), precision=precision, **kw)
        out.append(lat.init(drho, u, g).get_state().float().cpu().numpy())
    return out


# an ulp of FP32 beside the rounding itself
def close(a, b):
    return np.all(np.abs(a.astype(np.float64) - b) <= 2.0 ** -23 * np.abs(b) + 2.0 ** -149)


@pytest.mark.parametrize("q,dims", [(19, (33, 4, 3)), (15, (20, 3, 3)), (9, (40, 5, 1))])
@pytest.mark.parametrize("n", [0.7, 1.3])
@pytest.mark.parametrize("size", [3e18, 2e19, 1e25, 1e30])
def test_power_law_with_huge_gradients(q, dims, n, size):
    d = 2 if q == 9 else 3
    shape = dims[::-1]
    g = np.zeros((d * d,) + shape)
    g[1, :, 1, 3::5] = size
    g[0, :, 2, 1::7] = -size
    a, b = states(q, dims, np.zeros(shape), np.zeros((d,) + shape), g, closure="powerlaw", pl_n=n, pl_k=0.02)
    assert np.all(np.isfinite(b)) and close(a, b)


@pytest.mark.parametrize("q,dims", [(19, (33, 4, 3)), (15, (20, 3, 3)), (9, (40, 5, 1))])
@pytest.mark.parametrize("n,K", [(0.95, 0.116), (1.05, 1.0), (0.98, 0.3)])
def test_power_law_with_tiny_gradients(q, dims, n, K):
    d = 2 if q == 9 else 3
    shape = dims[::-1]
    rng = np.random.default_rng(2)
    g = rng.standard_normal((d * d,) + shape) * 10.0 ** rng.uniform(-26, -12, size=shape)
    a, b = states(q, dims, np.zeros(shape), np.zeros((d,) + shape), g, closure="powerlaw", pl_n=n, pl_k=K)
    assert close(a, b)


@pytest.mark.parametrize("q,dims", [(19, (33, 14, 13)), (9, (140, 45, 1))])
@pytest.mark.parametrize("closure", ["newton", "smag"])
@pytest.mark.parametrize("gradient", [False, True])
def test_values_below_the_pairs_range_are_rounded_once(q, dims, closure, gradient):
    """Nodes whose values all lie below 2^-103, where a pair's low part is subnormal: bit for bit the FP64 result."""
    d = 2 if q == 9 else 3
    shape = dims[::-1]
    rng = np.random.default_rng(4)
    size = 10.0 ** rng.uniform(-36, -33, size=shape)
    drho, u = rng.standard_normal(shape) * size, rng.standard_normal((d,) + shape) * size
    g = rng.standard_normal((d * d,) + shape) * size if gradient else None
    a, b = states(q, dims, drho, u, g, closure=closure, smag_cs=0.17)
    assert np.array_equal(a.view(np.int32), b.view(np.int32)), int((a != b).sum())
