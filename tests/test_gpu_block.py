"""Several steps of a small FP32 D2Q9 lattice per launch (shared-memory tiles) against one launch per step: every
node's arithmetic is the same, so the states are equal bit for bit.  Sizes on and beside the tiles' edges
(32 x 16, 32 x 20), down to one node; periodic, walled and moving faces; each closure; uniform and field forces;
step counts that leave a remainder."""
import numpy as np
import pytest
import torch

from test_gpu_parity import Case

pytestmark = pytest.mark.gpu

CAVITY = dict(bc=["wall"] * 3 + ["lid"], lid={3: (0.1, 0.02, 0)})
CASES = [
    ((64, 32, 1), "newton", "yu", {}),
    ((65, 33, 1), "newton", "chai", dict(force=[1e-5, -2e-5])),
    ((31, 47, 1), "smag", "chai", CAVITY),
    ((97, 16, 1), "smag", "yu", dict(bc=["periodic"] * 2 + ["wall", "lid"], lid={3: (0.05, 0, 0)}, force=[1e-5, 0])),
    ((40, 70, 1), "powerlaw", "chai", dict(pl=(0.6, 0.01), **CAVITY)),
    ((33, 17, 1), "smag_dev", "yu", dict(force_field=True)),
    ((5, 3, 1), "smag", "yu", dict(force=[1e-5, 0])),
    ((2, 1, 1), "newton", "yu", {}),
    ((3, 40, 1), "powerlaw", "yu", dict(pl=(1.3, 0.05), bc=["wall", "lid", "periodic", "periodic"], lid={1: (0, 0.1, 0)})),
    ((1, 1, 1), "newton", "yu", dict(bc=["wall"] * 4)),
    ((256, 256, 1), "newton", "yu", CAVITY),
    ((1283, 83, 1), "smag", "chai", dict(force=[1e-5, 0], **CAVITY)),  # enough tiles for the higher form (32 x 20)
    ((320, 330, 1), "newton", "yu", {}),
    ((640, 160, 1), "powerlaw", "chai", dict(pl=(0.6, 0.01), **CAVITY)),
]


@pytest.mark.parametrize("nsteps", [4, 11])
@pytest.mark.parametrize("dims,closure,formula,extra", CASES)
def test_blocked_steps_equal_per_step(dims, closure, formula, extra, nsteps):
    c = Case(9, dims, precision="fp32", closure=closure, formula=formula, tau=0.6, **extra)
    c.lat.init(c.drho, c.u, c.g)
    f0 = c.lat.get_state().clone()
    c.lat.set_schedule("per_step").step(nsteps)
    ref = c.lat.get_state().clone()
    c.lat.set_state(f0)
    before = np.array(c.lat.stats())
    c.lat.set_schedule("auto").step(nsteps)
    assert tuple(np.array(c.lat.stats()) - before) == (nsteps, nsteps // 4 + nsteps % 4)
    got = c.lat.get_state()
    assert torch.equal(got.view(torch.int32), ref.view(torch.int32)), int((got != ref).sum())


def test_lagged_closure_and_large_power_law_lattices_step_one_by_one():
    for dims, closure in (((64, 32, 1), "smag_lagged"), ((1024, 513, 1), "powerlaw")):
        c = Case(9, dims, precision="fp32", closure=closure, tau=0.6, pl=(0.7, 0.01))
        c.lat.init(c.drho, c.u, c.g).step(8)
        assert c.lat.stats() == (8, 8)


WALLED = dict(bc=["wall"] * 4)
ROUTES = [  # dims, closure, what else, whether tiles are taken: they are where they step faster (step_block.cuh)
    ((256, 256), "newton", {}, True),
    ((600, 600), "newton", {}, True),
    ((700, 700), "newton", {}, False),
    ((1000, 1000), "newton", {}, False),
    ((1000, 1000), "newton", WALLED, True),
    ((1000, 1000), "smag", WALLED, True),
    ((1000, 1000), "smag", dict(force=[1e-6, 0], **WALLED), False),
    ((1000, 1000), "smag_dev", dict(force=[1e-6, 0], **WALLED), True),
    ((1500, 1400), "newton", dict(force=[1e-6, 0]), True),
    ((1500, 1400), "smag", {}, False),
    ((1500, 1400), "smag_dev", {}, True),
    ((1, 20000), "newton", {}, False),
    ((20000, 1), "newton", {}, False),
    ((20000, 5), "smag", WALLED, False),
    ((28, 20000), "newton", WALLED, True),
    ((3, 6000), "newton", {}, True),
    ((512, 512), "powerlaw", dict(pl=(0.6, 0.01)), True),
    ((600, 600), "powerlaw", dict(pl=(0.6, 0.01)), False),
    ((700, 700), "powerlaw", dict(pl=(0.6, 0.01), **WALLED), True),
    ((1000, 1000), "powerlaw", dict(pl=(1.0, 0.01), **WALLED), True),
    ((1500, 1400), "powerlaw", dict(pl=(1.0, 0.01), force=[1e-6, 0], **WALLED), True),
    ((1500, 1400), "powerlaw", dict(pl=(1.0, 0.01)), False),
]


@pytest.mark.parametrize("dims,closure,extra,tiles", ROUTES)
def test_tiles_are_taken_where_they_step_faster(dims, closure, extra, tiles):
    c = Case(9, dims + (1,), precision="fp32", closure=closure, tau=0.6, **extra)
    c.lat.init(c.drho, c.u).step(8)
    assert c.lat.stats() == (8, 2 if tiles else 8)
