"""lbm_init in float pairs (FP32 and 16-bit storage) and in FP64, over lattices, closures, walls and
forces, against the oracle, and its infinities and NaN against the FP64 lattice's.

Bounds.  FP64: 1e-13 of max|f|.  FP32: one rounding to nearest, 2^-24 |f|, of a value that is within
2^-40 of max|f| (a float pair holds 2^-46 of each of some 30 terms).  16-bit storage rounds that once
more: 2^-11 (FP16; its subnormal spacing 2^-25) or 2^-8 (BF16)."""
import numpy as np
import pytest
import torch

from test_gpu_parity import Case, f64

pytestmark = pytest.mark.gpu

EPS = {"fp64": (0.0, 0.0), "fp32": (2.0 ** -24, 0.0), "fp16s": (2.0 ** -24 + 2.0 ** -11, 2.0 ** -25),
       "bf16s": (2.0 ** -24 + 2.0 ** -8, 0.0)}
WALLS = dict(bc=["periodic"] * 2 + ["wall", "lid"] + ["periodic"] * 2, lid={3: (0.05, 0.0, 0.01)})
CASES = [
    (19, (33, 7, 5), "fp32", "smag", dict(force=[1e-4, -2e-4, 3e-5])),
    (19, (64, 5, 4), "fp32", "newton", WALLS),
    (19, (1, 9, 3), "fp16s", "smag", dict(force_field=True)),
    (19, (40, 6, 5), "bf16s", "newton", {}),
    (19, (17, 4, 3), "fp64", "smag", dict(force=[1e-4, 0, 0], **WALLS)),
    (15, (35, 6, 4), "fp32", "smag_dev", dict(force_field=True)),
    (15, (18, 6, 4), "fp16s", "smag", WALLS),
    (9, (130, 9, 1), "fp32", "powerlaw", dict(pl=(0.7, 0.02), bc=["wall"] * 3 + ["lid"], lid={3: (0.1, 0, 0)})),
    (9, (31, 8, 1), "fp64", "smag", dict(force=[1e-5, 2e-5])),
]


@pytest.mark.parametrize("gradient", [False, True])
@pytest.mark.parametrize("q,dims,precision,closure,extra", CASES)
def test_init_is_the_rounded_oracle(q, dims, precision, closure, extra, gradient):
    c = Case(q, dims, precision=precision, closure=closure, tau=0.6, **extra)
    g = c.g if gradient else None
    c.lat.init(c.drho, c.u, g)
    fg = f64(c.lat.get_state())
    F = c.oforce
    if c.ffield is not None and precision != "fp64":
        F = F.astype(np.float32).astype(np.float64)  # the lattice holds the field in its compute type
    fo = c.G.init(c.drho, c.u, g, force=F)
    rel, sub = EPS[precision]
    scale = np.abs(fo).max()
    tol = rel * np.abs(fo) + sub + (1e-13 if precision == "fp64" else 2.0 ** -40) * scale
    assert np.all(np.abs(fg - fo) <= tol), float((np.abs(fg - fo) / tol).max())


def test_zero_tiny_huge_and_non_finite_inputs_as_in_fp64():
    """Zeros, values whose squares leave the FP32 range and non-finite inputs: FP32 storage holds the
    FP64 lattice's populations, rounded (infinite where those are beyond the FP32 range)."""
    a = Case(19, (40, 3, 3), precision="fp32", closure="smag", force=[1e-5, 0, 0])
    b = Case(19, (40, 3, 3), precision="fp64", closure="smag", force=[1e-5, 0, 0])
    drho, u, g = a.drho.copy(), a.u.copy(), a.g.copy()
    drho[:, :, 0:4], u[:, :, :, 0:4], g[:, :, :, 0:4] = 0.0, 0.0, 0.0
    drho[1, 1, 8], drho[1, 1, 10] = np.inf, np.nan
    u[0, 1, 1, 12], u[1, 1, 1, 14], u[2, 1, 1, 16] = 1e25, -1e19, np.nan
    g[3, 1, 1, 18], g[0, 1, 1, 20] = 1e30, np.inf
    u[:, 1, 1, 22] = 1e-40
    drho[1, 1, 24] = 1e300
    for c in (a, b):
        c.lat.init(drho, u, g)
    fa, fb = f64(a.lat.get_state()), f64(b.lat.get_state())
    with np.errstate(over="ignore"):
        fr = fb.astype(np.float32).astype(np.float64)
    assert np.array_equal(np.isnan(fa), np.isnan(fr))
    assert np.array_equal(np.isinf(fa), np.isinf(fr))
    ok = np.isfinite(fr)
    ordinary = np.abs(fr) < 1.0
    tol = 2.0 ** -23 * np.abs(fb[ok]) + np.where(ordinary[ok], 2.0 ** -40, 0.0)
    assert np.all(np.abs(fa[ok] - fb[ok]) <= tol)
