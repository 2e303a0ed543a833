"""Rows that nearly fill whole blocks of threads, and rows that do not: each map from threads to nodes (the plain grid
with idle threads at the row ends, node order, and the multi-step launch's walk with and without padded rows)
against the oracle, one step at a time, and the multi-step schedule against one launch per step bit for bit.

Blocks hold 128 threads (64 in FP64), one node each or two in 16-bit storage with nx even; a 16th of a row may stay idle."""
import pytest
import torch

from test_gpu_parity import Case

pytestmark = pytest.mark.gpu

WALL_X = ["wall"] * 2 + ["periodic"] * 4
WALL_Y = ["periodic"] * 2 + ["wall"] * 2 + ["periodic"] * 2
CASES = [(19, "fp16s", 242), (19, "bf16s", 250), (15, "bf16s", 254), (15, "fp16s", 240), (19, "fp16s", 486),
         (19, "fp32", 121), (15, "fp32", 127), (19, "fp32", 120), (19, "fp64", 61), (15, "fp64", 63), (19, "fp64", 60)]


@pytest.mark.parametrize("bc", [None, WALL_X, WALL_Y])
@pytest.mark.parametrize("q,precision,nx", CASES)
def test_every_node_is_stepped_once(q, precision, nx, bc):
    c = Case(q, (nx, 11, 5), precision=precision, closure="smag", formula="yu", tau=0.55, bc=bc, force=[1e-5, 0, 0])
    c.check_init()
    c.check_step()
    if precision == "fp64":
        return
    f0 = c.lat.get_state().clone()
    ref = c.lat.set_schedule("per_step").step(7).get_state().clone()
    c.lat.set_state(f0)
    got = c.lat.set_schedule("stream").step(7).status().get_state()
    bits = torch.int16 if got.element_size() == 2 else torch.int32
    assert torch.equal(got.view(bits), ref.view(bits))


@pytest.mark.parametrize("nx", [66, 128, 131])
@pytest.mark.parametrize("bc", [None, ["wall"] * 4])
def test_every_node_of_a_2d_fp64_lattice_is_stepped_once(nx, bc):
    c = Case(9, (nx, 260, 1), precision="fp64", closure="smag", formula="chai", tau=0.55, bc=bc, force=[1e-5, 0])
    c.check_init()
    c.check_step()
