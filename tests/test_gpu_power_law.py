"""The power-law closure's iteration from a guess against the oracle's plain sweeps: tau and
S at every node of states that reach the clamps, stay between them, are at rest, or are dominated by the
dilatation that the guess leaves out; and the parameters that keep plain sweeps.

Bars: the repository's for S and tau (FP64 1e-12, FP32 1e-5 of the largest), the stopping rule being
1e-13 and 1e-6 and the map's slope at most 1/2."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1704_07559_gb300 import lbm
from test_gpu_parity import TOL, f64, rates, relerr

pytestmark = pytest.mark.gpu


def states(q, shape, kind, seed=3):
    rng = np.random.default_rng(seed)
    w = O.tables(q)[1].reshape((q,) + (1,) * len(shape))
    f = w * rng.normal(scale=1e-3, size=shape)
    amp = 10.0 ** rng.uniform(-9, -2, size=shape)  # strain over seven decades, node by node
    noise = rng.normal(size=(q,) + shape)
    if kind == "dilated":  # the energy moment only, over a shear a thousandth of it
        T = O.tables(q)[2]
        noise = 1e-3 * noise + T[1].reshape((q,) + (1,) * len(shape)) * rng.normal(size=shape)
    f = f + w * amp * noise
    if kind == "rest":
        f[:] = 0.0
    return f


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["mixed", "dilated", "rest"])
@pytest.mark.parametrize("n,extra", [(0.5, {}), (0.8, {}), (1.5, {}), (1.0, {}), (0.5, dict(pl_max_iter=47)),
                                     (1.2, dict(pl_tau_min=0.6, pl_tau_max=0.9)), (0.45, {}), (0.7, dict(pl_k=0.0))])
@pytest.mark.parametrize("q,dims", [(9, (67, 9, 1)), (19, (35, 5, 3))])
def test_tau_and_strain_match_plain_sweeps(q, dims, n, extra, kind, precision):
    shape = dims[::-1]
    kw = dict(pl_k=2e-3 * 100.0 ** (n - 0.5), pl_tau_min=0.505, pl_tau_max=5.0, pl_max_iter=64)
    kw.update(extra)
    f = states(q, shape, kind)
    lat = lbm.Lattice(q, *dims, rates=rates(q, 0.8), precision=precision, closure="powerlaw", formula="chai", pl_n=n,
                      **kw)
    lat.set_state(torch.from_numpy(f).to(device="cuda", dtype=lat.storage_dtype))
    fin = f64(lat.get_state())
    p = O.make_params(q, rates(q, 0.8), closure=O.POWERLAW, formula=O.CHAI, pl_n=n,
                      pl_tol=1e-14 if precision == "fp64" else 1e-7, **kw)
    out = O.Grid(p, *dims).readout(fin)
    for formula in ("chai", "yu"):
        S, tau = lat.strain_rate(formula, with_tau=True)
        assert relerr(f64(tau), out["tau"]) <= TOL[precision]["S"]
        assert relerr(f64(S), out["S"]) <= TOL[precision]["S"]
