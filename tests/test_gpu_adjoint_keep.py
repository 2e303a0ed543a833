"""lbm_adjoint with room for every state (the binding's default where memory allows) against checkpoints with
recomputation: the same steps on the same states, so the functional, the gradient and the final state
are equal bit for bit, for segments that divide T, leave a remainder, and hold one step."""
import numpy as np
import pytest
import torch

from paper_1704_07559_gb300 import inputs as I
from paper_1704_07559_gb300 import lbm
from test_gpu_parity import rates

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,closure,schedule", [("fp32", "smag", "stream"), ("fp32", "newton", "per_step"),
                                                        ("fp32", "smag", "auto"), ("fp64", "smag", "auto")])
@pytest.mark.parametrize("T", [1, 2, 3, 13, 16])
def test_keeping_every_state_equals_recomputation(precision, closure, schedule, T):
    nx, ny, nz = 300, 12, 6
    drho, u = I.random_fourier(nx, ny, nz, kmax=2, rms=0.02, seed=6)
    g = I.gaussian_force(3, (nz, ny, nx), std=1e-5, seed=5)
    lat = lbm.Lattice(19, nx, ny, nz, rates=rates(19, 0.55), precision=precision, closure=closure, smag_cs=0.17,
                      force_field=torch.from_numpy(g))
    lat.set_schedule(schedule)
    lat.init(drho, u)
    f0 = lat.get_state().clone()
    seg = max(1, round(T ** 0.5))
    out = []
    for s in (None, seg):
        lat.set_state(f0)
        L, grad = lat.adjoint(T, s)
        lat.status()
        out.append((L, grad, lat.get_state().clone()))
    assert out[0][0] == out[1][0] and np.isfinite(out[0][0])
    assert torch.equal(out[0][1], out[1][1])
    assert torch.equal(out[0][2], out[1][2])


def test_without_room_the_checkpoints_are_used(monkeypatch):
    lat = lbm.Lattice(19, 16, 8, 8, rates=rates(19, 0.55), closure="smag", smag_cs=0.17,
                      force_field=torch.zeros(3, 8, 8, 16))
    lat.init(np.zeros((8, 8, 16)), 0.01 * np.ones((3, 8, 8, 16)))
    f0 = lat.get_state().clone()
    a = lat.adjoint(9)
    sizes, empty = [], torch.empty

    def scarce(*shape, **kw):  # the first allocation, room for every state, fails
        sizes.append(shape[0])
        if len(sizes) == 1:
            raise torch.cuda.OutOfMemoryError("out of memory")
        return empty(*shape, **kw)

    lat.set_state(f0)
    monkeypatch.setattr(torch, "empty", scarce)
    b = lat.adjoint(9)
    assert sizes[1] < sizes[0]
    assert a[0] == b[0] and torch.equal(a[1], b[1])
