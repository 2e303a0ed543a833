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


def kept(lat, f0, T, seg, schedule):
    """The call with a workspace that holds every state, through the C ABI."""
    need = ctypes.c_int64()
    lat._check(lbm.lib().lbm_adjoint_workspace(lat.ctx, T, seg, ctypes.byref(need)))
    size = lat.storage_dtype.itemsize
    nbytes = need.value + T * (-(-19 * lat.stride * size // 256) * 256)
    work = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    grad = torch.empty((3,) + lat.shape, dtype=torch.float64, device="cuda")
    loss = ctypes.c_double()
    lat.set_schedule(schedule)
    lat.set_state(f0)
    lat._check(lbm.lib().lbm_adjoint(lat.ctx, T, seg, ctypes.c_void_p(work.data_ptr() + (-work.data_ptr()) % 256), nbytes,
                                     ctypes.c_void_p(grad.data_ptr()), ctypes.byref(loss)))
    lat.status()
    return loss.value, grad, lat.get_state().clone()


def test_every_state_of_a_long_run_kept():
    """More steps than one multi-step launch takes (4096)."""
    lat, f0 = lattice((16, 4, 3))
    ref = run(lat, f0, 4200, 64, "per_step")
    for schedule in ("stream", "per_step"):
        assert same(kept(lat, f0, 4200, 64, schedule), ref)


@pytest.mark.parametrize("precision,closure,schedule", [("fp32", "smag", "stream"), ("fp32", "newton", "per_step"),
                                                        ("fp32", "newton", "stream"), ("fp64", "smag", "auto")])
@pytest.mark.parametrize("T,seg", [(13, 2), (13, 4), (13, 5), (16, 4), (9, 2)])
def test_recomputed_segments_equal_kept_states(precision, closure, schedule, T, seg):
    """Pairs whose workspace is smaller than that of every state, so that a given seg does recompute: segments that
    divide T, leave a remainder and leave one step."""
    lat, f0 = lattice((96, 12, 6), precision=precision, closure=closure)
    need, every = ctypes.c_int64(), ctypes.c_int64()
    lat._check(lbm.lib().lbm_adjoint_workspace(lat.ctx, T, seg, ctypes.byref(need)))
    lat._check(lbm.lib().lbm_adjoint_workspace(lat.ctx, T, T, ctypes.byref(every)))
    assert need.value < every.value
    assert same(run(lat, f0, T, seg, schedule), kept(lat, f0, T, seg, schedule))


@pytest.mark.parametrize("total,free,kept", [(64, 0, True), (63, 4, True), (63, 3, False), (8, 4, True), (8, 3, False),
                                             (7, 100, False)])
def test_default_leaves_memory_free(monkeypatch, total, free, kept):
    """Every state is kept where they take a 64th of the device's memory at most, or an eighth of it and a quarter of what
    is free (both given here in multiples of what they take); the checkpoints are used otherwise."""
    lat, f0 = lattice((16, 8, 8))
    every = ctypes.c_int64()
    lat._check(lbm.lib().lbm_adjoint_workspace(lat.ctx, 9, 9, ctypes.byref(every)))

    class Device:
        total_memory = total * every.value

    sizes, empty = [], torch.empty
    monkeypatch.setattr(torch, "empty", lambda *shape, **kw: sizes.append(shape[0]) or empty(*shape, **kw))
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: Device)
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda d: (free * every.value, Device.total_memory))
    lat.adjoint(9)
    assert (sizes[0] >= every.value) == kept
