"""lbm_adjoint by its ways of launching and of keeping states: the same steps on the same states, so the functional, the
gradient and the final state are equal bit for bit."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1704_07559_gb300 import inputs as I
from paper_1704_07559_gb300 import lbm
from test_gpu_parity import rates

pytestmark = pytest.mark.gpu


def lattice(dims, precision="fp32", closure="smag", formula="yu", **kw):
    nx, ny, nz = dims
    drho, u = I.random_fourier(nx, ny, nz, kmax=2, rms=0.02, seed=6)
    g = I.gaussian_force(3, (nz, ny, nx), std=1e-5, seed=5)
    lat = lbm.Lattice(19, nx, ny, nz, rates=rates(19, 0.55), precision=precision, closure=closure, formula=formula,
                      smag_cs=0.17, force_field=torch.from_numpy(g), **kw)
    lat.init(drho, u)
    return lat, lat.get_state().clone()


def run(lat, f0, T, seg=None, schedule="auto"):
    lat.set_schedule(schedule)
    lat.set_state(f0)
    L, grad = lat.adjoint(T, seg)
    lat.status()
    return L, grad, lat.get_state().clone()


def same(a, b):
    return np.isfinite(a[0]) and a[0] == b[0] and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])


@pytest.mark.parametrize("closure", ["newton", "smag"])
@pytest.mark.parametrize("formula", ["yu", "chai"])
@pytest.mark.parametrize("dims", [(96, 12, 6), (33, 9, 5)])
def test_schedules_agree(dims, closure, formula):
    lat, f0 = lattice(dims, closure=closure, formula=formula)
    ref = run(lat, f0, 13, 4, "per_step")
    for schedule in ("stream", "auto"):
        assert same(run(lat, f0, 13, 4, schedule), ref)
        assert same(run(lat, f0, 13, None, schedule), ref)


def test_every_state_of_a_long_run_kept():
    """More steps than one multi-step launch takes (4096), through the C ABI with a workspace that holds every state."""
    T, seg = 4200, 64
    lat, f0 = lattice((16, 4, 3))
    ref = run(lat, f0, T, seg, "per_step")
    need = ctypes.c_int64()
    lat._check(lbm.lib().lbm_adjoint_workspace(lat.ctx, T, seg, ctypes.byref(need)))
    state = -(-19 * lat.stride * 4 // 256) * 256
    nbytes = need.value + T * state
    work = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    grad, loss = torch.empty_like(ref[1]), ctypes.c_double()
    for schedule in ("stream", "per_step"):
        lat.set_schedule(schedule)
        lat.set_state(f0)
        lat._check(lbm.lib().lbm_adjoint(lat.ctx, T, seg, ctypes.c_void_p(work.data_ptr() + (-work.data_ptr()) % 256), nbytes,
                                         ctypes.c_void_p(grad.data_ptr()), ctypes.byref(loss)))
        lat.status()
        assert same((loss.value, grad, lat.get_state()), ref)
