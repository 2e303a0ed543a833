"""States of 16-bit Smagorinsky lattices stepped by Chai's route, bit for bit as recorded
(tests/golden/chai_16bit_states.json: SHA-256 of the populations).  Their FP32 arithmetic is rounded to the storage each
step, and a different last place grows to a storage rounding everywhere within some 20 steps, so its order is part of
the result.  Even and odd rows (two nodes and one node to a thread), walls, uniform and per-node forces."""
import hashlib
import json
import os

import numpy as np
import pytest
import torch

from paper_1704_07559_gb300 import lbm

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "chai_16bit_states.json")
SHEAR = {19: (9, 11, 13, 14, 15), 15: (9, 10, 11, 12, 13)}
WALLS = ["periodic"] * 2 + ["wall"] * 2 + ["periodic"] * 2


def rates(q, s):
    r = [0, 1.19, 1.4, 0, 1.2, 0, 1.2, 0, 1.2] + ([s, 1.4, s, 1.4, s, s, s, 1.98, 1.98, 1.98] if q == 19 else [s] * 5 + [1.98])
    return [float(x) for x in r]


def weights(q):
    return np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12 if q == 19 else [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8)


def final_state(q, precision, nx, flow, schedule):
    """Raw bits of the populations after 20 steps from fixed ones (built on the host)."""
    ny, nz = 10, 6
    rng = np.random.default_rng(17)
    f = weights(q)[:, None, None, None] * (1.0 + 0.05 * rng.standard_normal((q, nz, ny, nx))) - weights(q)[:, None, None, None]
    kw = {}
    if flow == "channel":
        kw.update(bc=WALLS, force=[1e-5, 0.0, 0.0])
    elif flow == "field":
        kw.update(force_field=torch.from_numpy(1e-5 * rng.standard_normal((3, nz, ny, nx))))
    lat = lbm.Lattice(q, nx, ny, nz, rates=rates(q, 1 / 0.53), precision=precision, closure="smag", formula="chai",
                      smag_cs=0.17, **kw)
    lat.set_state(torch.from_numpy(f).float().to(lat.storage_dtype).cuda())
    lat.set_schedule(schedule).step(20).status()
    return lat.get_state().view(torch.int16).cpu().numpy()


def digest(bits):
    return hashlib.sha256(np.ascontiguousarray(bits).astype("<i2").tobytes()).hexdigest()


CASES = [(q, p, nx, flow) for q in (19, 15) for p in ("fp16s", "bf16s") for nx in (34, 33) for flow in ("box", "channel", "field")]


@pytest.mark.gpu
@pytest.mark.parametrize("schedule", ["per_step", "stream"])
@pytest.mark.parametrize("q,precision,nx,flow", CASES)
def test_state_is_the_recorded_one(q, precision, nx, flow, schedule):
    with open(GOLDEN) as fh:
        want = json.load(fh)
    got = digest(final_state(q, precision, nx, flow, schedule))
    assert got == want["%d %s %d %s" % (q, precision, nx, flow)]


@pytest.mark.gpu
@pytest.mark.parametrize("q", [19, 15])
@pytest.mark.parametrize("nx", [34, 33])
def test_each_viscous_moment_relaxes_at_its_own_rate(q, nx):
    """Fixed rates that differ from one viscous moment to the next (accepted on Chai's route), against FP64 storage:
    one step apart by a rounding to FP16 (2^-11) of the largest population."""
    r = rates(q, 1.0)
    for k, s in zip(SHEAR[q], (0.6, 0.9, 1.2, 1.5, 1.8)):
        r[k] = s
    rng = np.random.default_rng(3)
    f = weights(q)[:, None, None, None] * 0.05 * rng.standard_normal((q, 4, 5, nx))
    f = torch.from_numpy(f).half()
    out = []
    for precision in ("fp16s", "fp64"):
        lat = lbm.Lattice(q, nx, 5, 4, rates=r, precision=precision, closure="newton", formula="chai")
        lat.set_state(f.to(lat.storage_dtype).cuda())
        out.append(lat.step(1).get_state().double())
    assert float((out[0] - out[1]).abs().max()) <= 2.0 ** -11 * float(out[1].abs().max())
