"""What a user of this library has it do, as cases that can be timed and checked one by one.

Each case goes through the public binding (paper_1704_07559_gb300.lbm): a `Lattice` that the
program keeps, and one call or one short sequence of calls on it.  Four kinds:

  advance   n time steps and then what the program reads: a checkpoint of the populations, the
            macroscopic fields, or S by both formulas
  diagnose  the read-outs of a running simulation: S with tau, the macroscopic fields, the sums
  setup     the initial state from given fields and velocity gradients, as a checkpoint
  adjoint   one gradient of the dissipation functional with respect to the force field

The inputs are synthetic flows made from the seed: a few dozen divergence-free Fourier modes (and
the laminar profile in a channel), as populations in equilibrium plus the first-order viscous
part, which is what a checkpoint of a running simulation holds.  `exact` steps the same
populations in 64 bits with plain torch operations and dense matrices, from the formulas alone.
"""
import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_1704_07559_gb300 import lbm

DEVICE = "cuda"

# float operations of one node update by the shorter (Yu) route: two transforms, the equilibrium,
# the closure and the relaxation (additions and multiplications counted one by one)
FLOPS = {9: 170, 15: 330, 19: 420}
BYTES = {"fp64": 8, "fp32": 4, "fp16s": 2, "bf16s": 2}


# ---------------------------------------------------------------------------------- the cases


def _advance(lattice, precision, closure, formula, flow, nx, ny, nz, steps, out, tau0=0.51, n_index=1.0):
    return {"kind": "advance", "lattice": lattice, "precision": precision, "closure": closure, "formula": formula,
            "flow": flow, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "out": out, "tau0": tau0, "n_index": n_index}


def listed():
    chan = ("channel", 256, 128, 128, 20, "state")
    cases = {
        # the smallest call: a 32^3 FP64 Taylor-Green-like box advanced one step at a time with S
        # read by both formulas after each, the paper's correctness run; launches and latency count
        "box32_fp64_both_s": _advance(19, "fp64", "newton", "yu", "box", 32, 32, 32, 1, "both_s", tau0=0.6),
        # a small 2D lid-driven cavity, as a validation study runs it: many steps of little work
        "cavity256_d2q9_fp32": _advance(9, "fp32", "newton", "yu", "cavity", 256, 256, 1, 50, "macro"),
        # a 64^3 periodic box: a state that stays in cache, read out every 20 steps
        "box64_fp32_yu": _advance(19, "fp32", "smag", "yu", "box", 64, 64, 64, 20, "macro"),
        # large-eddy channel with walls and a body force, the library's ordinary work: FP32 by both
        # routes, and the reduced-precision forms (D3Q19 FP16, D3Q15 BF16) at the same size
        "channel_fp32_yu": _advance(19, "fp32", "smag", "yu", *chan),
        "channel_fp32_chai": _advance(19, "fp32", "smag", "chai", *chan),
        "channel_fp16_yu": _advance(19, "fp16s", "smag", "yu", *chan),
        "channel_d3q15_bf16_chai": _advance(15, "bf16s", "smag", "chai", *chan),
        # a large shear-thinning cavity (power law n = 0.5, tau by per-node fixed point), Chai's route
        "cavity4096_powerlaw_chai": _advance(9, "fp32", "powerlaw", "chai", "cavity", 4096, 4096, 1, 8, "state",
                                             n_index=0.5),
        # the largest: a 512^3 box of decaying turbulence in FP16 storage
        "box512_fp16_yu": _advance(19, "fp16s", "smag", "yu", "box", 512, 512, 512, 10, "state"),
        # one gradient of flow control: forward steps, checkpoints, recomputation, reverse sweep
        "adjoint128": {"kind": "adjoint", "nx": 128, "ny": 128, "nz": 128, "T": 64, "closure": "smag"},
        # the read-outs of a running channel with ragged sizes: S and tau, fields, conserved sums
        "diagnose_fp32_chai": {"kind": "diagnose", "lattice": 19, "precision": "fp32", "closure": "smag",
                               "formula": "chai", "flow": "channel", "nx": 200, "ny": 150, "nz": 97, "tau0": 0.51,
                               "n_index": 1.0},
        # the start of a run from given fields, with the first-order non-equilibrium part
        "setup192_fp32": {"kind": "setup", "precision": "fp32", "closure": "smag", "nx": 192, "ny": 192, "nz": 192},
    }
    return [dict(c, name=k) for k, c in cases.items()]


def _size(rng, lo, hi):
    """A size between lo and hi, spread over the logarithm; a third are made odd."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n | 1 if rng.random() < 1 / 3 else n


def draw(rng):
    kind = rng.choice(["box", "box", "channel", "channel", "channel", "cavity", "cavity", "adjoint", "diagnose", "setup"])
    formula = rng.choice(["yu", "chai"])
    if kind == "adjoint":
        return {"kind": "adjoint", "nx": _size(rng, 16, 128), "ny": _size(rng, 16, 128), "nz": _size(rng, 16, 128),
                "T": rng.randint(2, 48), "closure": rng.choice(["newton", "smag"])}
    if kind == "setup":
        return {"kind": "setup", "precision": rng.choice(["fp64", "fp32", "fp16s"]),
                "closure": rng.choice(["newton", "smag"]), "nx": _size(rng, 16, 192), "ny": _size(rng, 16, 192),
                "nz": _size(rng, 16, 192)}
    if kind == "diagnose":
        return {"kind": "diagnose", "lattice": rng.choice([15, 19]), "precision": rng.choice(["fp64", "fp32"]),
                "closure": "smag", "formula": formula, "flow": rng.choice(["box", "channel"]),
                "nx": _size(rng, 24, 256), "ny": _size(rng, 24, 192), "nz": _size(rng, 24, 128), "tau0": 0.51,
                "n_index": 1.0}
    if kind == "cavity":
        closure = rng.choice(["newton", "powerlaw"])
        return _advance(9, rng.choice(["fp32", "fp32", "fp64"]), closure, formula, "cavity", _size(rng, 64, 2048),
                        _size(rng, 64, 2048), 1, rng.randint(1, 20), "state",
                        n_index=round(rng.uniform(0.5, 1.5), 2) if closure == "powerlaw" else 1.0)
    lattice = rng.choice([15, 19, 19])
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16s", "bf16s"])
    closure = rng.choice(["smag", "smag", "newton", "smag_dev", "smag_lagged"] if precision in ("fp64", "fp32")
                         else ["smag", "newton"])
    if precision == "fp64":
        dims = [_size(rng, 16, 128) for _ in range(3)]
    elif kind == "box":
        dims = [_size(rng, 24, 384) for _ in range(3)]
    else:
        dims = [_size(rng, 48, 384), _size(rng, 32, 192), _size(rng, 32, 192)]
    return _advance(lattice, precision, closure, formula, kind, *dims, rng.randint(1, 24), "state")


# ---------------------------------------------------------------------------------- the model


def _velocities(q):
    """The library's velocity order (rows of three integers)."""
    if q == 9:
        return [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
    c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    if q == 15:
        return c + [(x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)]
    return (c + [(x, y, 0) for y in (1, -1) for x in (1, -1)] + [(x, 0, z) for z in (1, -1) for x in (1, -1)] +
            [(0, y, z) for z in (1, -1) for y in (1, -1)])


def _weights(q):
    by = {9: {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}, 15: {0: 2 / 9, 1: 1 / 9, 3: 1 / 72}, 19: {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}}[q]
    return [by[x * x + y * y + z * z] for x, y, z in _velocities(q)]


def _moment_row(q, x, y, z):
    s = x * x + y * y + z * z
    if q == 9:
        return [1, -4 + 3 * s, 4 - 21 * s / 2 + 9 * s * s / 2, x, (3 * s - 5) * x, y, (3 * s - 5) * y, x * x - y * y, x * y]
    if q == 15:
        return [1, s - 2, (15 * s * s - 55 * s + 32) / 2, x, (5 * s - 13) * x / 2, y, (5 * s - 13) * y / 2, z,
                (5 * s - 13) * z / 2, 3 * x * x - s, y * y - z * z, x * y, y * z, x * z, x * y * z]
    p, w = 3 * x * x - s, y * y - z * z
    return [1, 19 * s - 30, (21 * s * s - 53 * s + 24) / 2, x, (5 * s - 9) * x, y, (5 * s - 9) * y, z, (5 * s - 9) * z, p,
            (3 * s - 5) * p, w, (3 * s - 5) * w, x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
            (x * x - y * y) * z]


VISCOUS = {9: (7, 8), 15: (9, 10, 11, 12, 13), 19: (9, 11, 13, 14, 15)}


def _rates(q, tau0):
    s = 1 / tau0
    if q == 9:
        return [0, 1.19, 1.4, 0, 1.2, 0, 1.2, s, s]
    if q == 15:
        return [0, 1.19, 1.4, 0, 1.2, 0, 1.2, 0, 1.2, s, s, s, s, s, 1.98]
    return [0, 1.19, 1.4, 0, 1.2, 0, 1.2, 0, 1.2, s, 1.4, s, 1.4, s, s, s, 1.98, 1.98, 1.98]


LID = 0.05  # lid speed of the cavities


def _model(case):
    """What the case's lattice is, as the keywords of lbm.Lattice and as numbers for `exact`."""
    kind = case["kind"]
    q = case.get("lattice", 19)
    flow = case.get("flow", "box")
    closure = case["closure"]
    tau0 = case.get("tau0", 0.51)
    kw = {"precision": case.get("precision", "fp32"), "closure": closure, "formula": case.get("formula", "yu"),
          "smag_cs": 0.17}
    bc, lid, force = ["periodic"] * 6, {}, [0.0, 0.0, 0.0]
    if flow == "channel":
        bc[2] = bc[3] = "wall"
        force = [1e-6, 0.0, 0.0]
    elif flow == "cavity":
        bc = ["wall", "wall", "wall", "lid", "periodic", "periodic"]
        lid = {3: (LID, 0.0, 0.0)}
        # Reynolds number 1000: nu = U L / 1000, and for the power law K = U^(2-n) L^n / 1000
        n = case["n_index"]
        K = LID ** (2 - n) * case["nx"] ** n / 1000
        if closure == "powerlaw":
            kw.update(pl_n=n, pl_k=K, pl_tau_min=0.505, pl_tau_max=5.0)
        tau0 = min(max(0.5 + 3 * LID * case["nx"] / 1000, 0.51), 1.5)
    if any(force):
        kw["force"] = force
    kw.update(bc=bc, lid_u=lid, rates=_rates(q, tau0))
    return q, kw, force, tau0, kind


# ---------------------------------------------------------------------------------- the inputs


def _flow(case, seed, dtype=torch.float32):
    """(drho, u, grad) of the synthetic flow: fields (nz, ny, nx), (3, ...), (9, ...) or None."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    flat = nz == 1
    g = torch.Generator().manual_seed(1000 + int(seed))
    xs = [torch.arange(n, dtype=torch.float64) for n in (nx, ny, nz)]
    u = torch.zeros((3, nz, ny, nx), dtype=dtype, device=DEVICE)
    want_grad = case["kind"] == "setup"
    grad = torch.zeros((9, nz, ny, nx), dtype=dtype, device=DEVICE) if want_grad else None
    drho = torch.zeros((nz, ny, nx), dtype=dtype, device=DEVICE)
    rms = {"box": 0.03, "channel": 0.01, "cavity": 0.01}[case.get("flow", "box")]
    kmax, modes = 8, 16
    for _ in range(modes):
        while True:
            k = torch.randint(-kmax, kmax + 1, (3,), generator=g).double()
            if flat:
                k[2] = 0
            if 0 < float((k * k).sum()) <= kmax * kmax:
                break
        kk = k * 2 * math.pi / torch.tensor([nx, ny, nz], dtype=torch.float64)  # per lattice unit
        a = torch.randn(3, generator=g, dtype=torch.float64)
        if flat:
            a[2] = 0
        a = a - kk * (a @ kk) / (kk @ kk)
        a = a * (rms * math.sqrt(2 / modes) / max(float(a.norm()), 1e-3)) * (0.5 + float(torch.rand(1, generator=g)))
        phase = 2 * math.pi * float(torch.rand(1, generator=g))
        ph = [(kk[d] * xs[d]).to(dtype).to(DEVICE) for d in range(3)]
        arg = ph[0][None, None, :] + ph[1][None, :, None] + (ph[2] + phase)[:, None, None]
        c = torch.cos(arg)
        s = torch.sin(arg) if want_grad else None
        for d in range(3):
            if float(a[d]):
                u[d].add_(c, alpha=float(a[d]))
            if want_grad:
                for e in range(3):
                    grad[3 * d + e].add_(s, alpha=-float(a[d] * kk[e]))
        drho.add_(c, alpha=2e-3 * (float(torch.rand(1, generator=g)) - 0.5))
        del arg, c, s
    if case.get("flow") == "channel":
        y = (torch.arange(ny, dtype=torch.float64) + 0.5) / ny
        u[0].add_((0.4 * y * (1 - y)).to(dtype).to(DEVICE)[None, :, None])
    return drho, u, grad


def _populations(case, seed, q, tau0, dtype):
    """Equilibrium plus the first-order viscous part of the flow, as q populations of `dtype`."""
    drho, u, _ = _flow(case, seed)
    c, w = _velocities(q), _weights(q)
    d = 2 if q == 9 else 3
    uu = (u * u).sum(0)
    grads = {}  # du_a/dx_b + du_b/dx_a by central differences (one cell inside, whatever the faces)
    for a in range(d):
        for b in range(a, d):
            x = lambda v, ax: (torch.roll(v, -1, 2 - ax) - torch.roll(v, 1, 2 - ax)) * 0.5  # noqa: E731
            grads[a, b] = (x(u[a], b) + x(u[b], a)) * 0.5
    div = sum(grads[a, a] for a in range(d))
    f = torch.empty((q,) + tuple(drho.shape), dtype=dtype, device=DEVICE)
    for i in range(q):
        cu = sum(c[i][a] * u[a] for a in range(d))
        if isinstance(cu, (int, float)):
            cu = torch.zeros_like(drho)
        neq = -div / 3
        for a in range(d):
            for b in range(a, d):
                if c[i][a] * c[i][b]:
                    neq = neq + (1 if a == b else 2) * c[i][a] * c[i][b] * grads[a, b]
        f[i] = w[i] * (drho + 3 * cu + 4.5 * cu * cu - 1.5 * uu) - (3 * w[i] * tau0) * neq
    return f


STORAGE = {"fp64": torch.float64, "fp32": torch.float32, "fp16s": torch.float16, "bf16s": torch.bfloat16}


def _force_field(case, seed):
    g = torch.Generator(device=DEVICE).manual_seed(2000 + int(seed))
    return torch.randn((3, case["nz"], case["ny"], case["nx"]), generator=g, device=DEVICE) * 1e-5


def _given(case, seed):
    """What the program has in hand: the model and its input tensors."""
    q, kw, force, tau0, kind = _model(case)
    if kind == "setup":
        return q, kw, force, tau0, tuple(t.double() for t in _flow(case, seed, torch.float64))
    return q, kw, force, tau0, _populations(case, seed, q, tau0, STORAGE[kw["precision"]])


def prepare(case, seed):
    q, kw, _, tau0, given = _given(case, seed)
    if case["kind"] == "adjoint":
        g = _force_field(case, seed).requires_grad_()
        lat = lbm.Lattice(q, case["nx"], case["ny"], case["nz"], force_field=g.detach(), **kw)
        return {"case": case, "lat": lat, "f0": given, "g": g}
    lat = lbm.Lattice(q, case["nx"], case["ny"], case["nz"], **kw)
    if case["kind"] == "setup":
        return {"case": case, "lat": lat, "fields": given,
                "out": torch.empty((q,) + lat.shape, dtype=lat.storage_dtype, device=DEVICE)}
    lat.set_state(given)
    if lat.tau is not None:
        lat.tau.fill_(tau0)
    state = {"case": case, "lat": lat}
    if case.get("out") == "state":
        state["out"] = torch.empty((q,) + lat.shape, dtype=lat.storage_dtype, device=DEVICE)
    return state


# ---------------------------------------------------------------------------------- one pass


def run(state):
    case, lat = state["case"], state["lat"]
    kind = case["kind"]
    if kind == "adjoint":
        g = state["g"]
        g.grad = None
        loss = lbm.DissipationLoss.apply(g, lat, state["f0"], case["T"])
        loss.backward()
        return {"loss": loss.detach().to(g.dtype), "grad": g.grad}
    if kind == "setup":
        lat.init(*state["fields"])
        return lat.get_state(out=state["out"])
    if kind == "diagnose":
        S, tau = lat.strain_rate(with_tau=True)
        drho, u = lat.macroscopic()
        return {"S": S, "tau": tau, "drho": drho, "u": u, "sums": lat.sums()}
    lat.step(case["steps"])
    if case["out"] == "both_s":
        return {"yu": lat.strain_rate("yu"), "chai": lat.strain_rate("chai")}
    if case["out"] == "macro":
        drho, u = lat.macroscopic()
        return {"drho": drho, "u": u}
    f = lat.get_state(out=state["out"])
    return f if lat.tau is None else {"f": f, "tau": lat.tau}  # the lagged closure's tau is state too


# ---------------------------------------------------------------------------------- what it costs


def work(case):
    """Bytes: the state once in and once out per pass, and what the pass returns besides; a pass of
    several steps cannot do without reading the first state and writing the last (its steps in
    between are counted as operations only).  Flops: one node update per node and step."""
    kind, q = case["kind"], case.get("lattice", 19)
    N = case["nx"] * case["ny"] * case["nz"]
    precision = case.get("precision", "fp32")
    b, d = BYTES[precision], 2 if q == 9 else 3
    cb = 8 if precision == "fp64" else 4
    ns = 3 if d == 2 else 6
    if kind == "adjoint":
        # f0, the force field in and the gradient out; a reverse step is two node updates and a half
        return {"bytes": N * (q * 4 + 3 * 4 + 3 * 4), "flops": N * FLOPS[q] * case["T"] * 3.5}
    if kind == "setup":
        return {"bytes": N * (13 * 8 + 2 * q * b + q * b), "flops": N * FLOPS[q]}
    if kind == "diagnose":
        return {"bytes": N * (q * b + (ns + 2 + d) * cb), "flops": N * FLOPS[q] * 0.6}
    outs = {"state": 2 * q * b, "macro": (1 + d) * cb, "both_s": 2 * ns * cb}[case["out"]]
    return {"bytes": N * (2 * q * b + outs), "flops": N * FLOPS[q] * (case["steps"] + (1 if case["out"] == "both_s" else 0))}


# ---------------------------------------------------------------------------------- in 64 bits


class _Exact:
    """The model in 64 bits with dense matrices: pull, moments, S, closure, relaxation."""

    def __init__(self, case):
        self.q, kw, self.force, self.tau0, _ = _model(case)
        q = self.q
        self.kw, self.d = kw, 2 if q == 9 else 3
        self.c, self.w = _velocities(q), _weights(q)
        M = torch.tensor([_moment_row(q, *c) for c in self.c], dtype=torch.float64, device=DEVICE).T.contiguous()
        self.T, self.Ti = M, torch.linalg.inv(M)
        s = torch.tensor(kw["rates"], dtype=torch.float64, device=DEVICE)
        visc = torch.zeros(q, dtype=torch.bool, device=DEVICE)
        visc[list(VISCOUS[q])] = True
        self.fixed = torch.where(visc, torch.zeros_like(s), s)
        self.visc = visc.double()
        self.ab = [(a, a) for a in range(self.d)] + ([(0, 1)] if self.d == 2 else [(0, 1), (1, 2), (0, 2)])
        cc = torch.tensor([[c[a] * c[b] for c in self.c] for a, b in self.ab], dtype=torch.float64, device=DEVICE)
        self.A = -1.5 * (cc @ self.Ti) * self.fixed  # S = A mn + (1/tau) B mn, rho0 = 1
        self.B = -1.5 * (cc @ self.Ti) * self.visc
        self.twice = torch.tensor([1.0 if a == b else 2.0 for a, b in self.ab], dtype=torch.float64, device=DEVICE)
        self.lagged = None  # the lagged closure's stored tau

    def pull(self, f):
        g = torch.empty_like(f)
        walls = [a for a in range(self.d) if self.kw["bc"][2 * a] != "periodic"]
        for i, c in enumerate(self.c):
            g[i] = torch.roll(f[i], c[::-1], (0, 1, 2))
            back = self.c.index((-c[0], -c[1], -c[2]))
            hit = [a for a in walls if c[a]]
            plane = {a: (slice(None),) * (2 - a) + ((0 if c[a] > 0 else -1),) for a in hit}
            for a in hit:
                face = 2 * a + (0 if c[a] > 0 else 1)
                lid = self.kw["lid_u"].get(face, (0.0, 0.0, 0.0))
                g[i][plane[a]] = f[back][plane[a]] + 6 * self.w[i] * sum(x * y for x, y in zip(c, lid))
            for n, a in enumerate(hit):
                for b in hit[n + 1:]:
                    at = [slice(None)] * 3
                    at[2 - a], at[2 - b] = 0 if c[a] > 0 else -1, 0 if c[b] > 0 else -1
                    g[i][tuple(at)] = f[back][tuple(at)]
        return g

    def node(self, p, F=None, tau=None):
        """(drho, u, mn, Fbar, S, tau) of pulled populations p (q, ...)."""
        F = self.force if F is None else F
        drho = p.sum(0)
        j = [sum(c[a] * p[i] for i, c in enumerate(self.c) if c[a]) + 0.5 * F[a] for a in range(self.d)]
        jj, jF = sum(x * x for x in j), sum(x * y for x, y in zip(j, F))
        eff, Fbar = [], []
        for c, w, x in zip(self.c, self.w, p):
            cj, cF = sum(c[a] * j[a] for a in range(self.d)), sum(c[a] * F[a] for a in range(self.d))
            fb = w * (3 * cF - 3 * jF + 9 * cj * cF)
            eff.append(x - w * (drho + 3 * cj + 4.5 * cj * cj - 1.5 * jj) + 0.5 * fb)
            Fbar.append(fb + torch.zeros_like(drho))
        mn = torch.einsum("kq,q...->k...", self.T, torch.stack(eff))
        del eff
        A = torch.einsum("ck,k...->c...", self.A, mn)
        B = torch.einsum("ck,k...->c...", self.B, mn)
        norm = lambda S: torch.sqrt(2 * torch.einsum("c,c...->...", self.twice, S * S))  # noqa: E731
        closure, c3 = self.kw["closure"], 3 * self.kw["smag_cs"] ** 2
        t = torch.full_like(drho, self.tau0)
        if closure == "smag":
            for _ in range(6):
                t = self.tau0 + c3 * norm(A + B / t)
        elif closure == "smag_dev":
            for _ in range(40):
                t = self.tau0 + c3 * norm(B / t)
        elif closure == "smag_lagged":
            t = tau if tau is not None else t
        elif closure == "powerlaw":
            for _ in range(60):
                t = 0.5 + 3 * self.kw["pl_k"] * norm(A + B / t) ** (self.kw["pl_n"] - 1)
                t = t.clamp(self.kw["pl_tau_min"], self.kw["pl_tau_max"])
        S = A + B / t
        if closure == "smag_lagged":
            self.lagged = self.tau0 + c3 * norm(S)
        return drho, torch.stack(j), mn, Fbar, S, t

    def collide(self, p, F=None, tau=None):
        _, _, mn, Fbar, _, t = self.node(p, F, tau)
        relax = mn * self.fixed.view((-1,) + (1,) * (mn.dim() - 1))
        relax = relax + mn * self.visc.view((-1,) + (1,) * (mn.dim() - 1)) / t
        return p - torch.einsum("qk,k...->q...", self.Ti, relax) + torch.stack(Fbar)

    def step(self, f, F=None):
        p = self.pull(f)
        out = torch.empty_like(p)
        lag = torch.empty_like(p[0]) if self.kw["closure"] == "smag_lagged" else None
        rows = max(1, (1 << 23) // (p.shape[2] * p.shape[3]))  # z planes, or y rows, at a time
        ax = 1 if p.shape[1] > 1 else 2
        rows = rows if ax == 1 else max(1, (1 << 23) // p.shape[3])
        tau = self.lagged
        for k in range(0, p.shape[ax], rows):
            m = min(rows, p.shape[ax] - k)
            part = self.collide(p.narrow(ax, k, m), F, None if tau is None else tau.narrow(ax - 1, k, m))
            out.narrow(ax, k, m).copy_(part)
            if lag is not None:
                lag.narrow(ax - 1, k, m).copy_(self.lagged)
        if lag is not None:
            self.lagged = lag
        return out


def _exact_adjoint(case, seed, f0):
    x = _Exact(case)
    g = _force_field(case, seed).double().requires_grad_()
    one = lambda f, g: x.collide(x.pull(f), [g[0], g[1], g[2]])  # noqa: E731
    f = f0.double()
    for _ in range(case["T"]):
        f = checkpoint(one, f, g, use_reentrant=False)

    def total(f, g):
        _, _, _, _, S, t = x.node(x.pull(f), [g[0], g[1], g[2]])
        return ((t - 0.5) / 3 * torch.einsum("c,c...->...", x.twice, S * S)).sum()

    loss = checkpoint(total, f, g, use_reentrant=False)
    loss.backward()
    return {"loss": loss.detach(), "grad": g.grad}


def exact(case, seed):
    q, _, _, _, given = _given(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed, given)
    x = _Exact(case)
    if case["kind"] == "setup":
        return _exact_setup(x, *given)
    f = given.double()
    del given
    if case["kind"] == "diagnose":
        drho, u, _, _, S, t = x.node(x.pull(f))
        sums = torch.stack([drho.sum()] + [v.sum() for v in u])
        return {"S": S, "tau": t, "drho": drho, "u": u, "sums": sums}
    for _ in range(case["steps"]):
        f = x.step(f)
    if case["out"] == "state":
        return f if x.lagged is None else {"f": f, "tau": x.lagged}
    drho, u, _, _, S, _ = x.node(x.pull(f), tau=x.lagged)
    return {"yu": S, "chai": S} if case["out"] == "both_s" else {"drho": drho, "u": u}


def _exact_setup(x, drho, u, grad):
    """f_eq plus the first-order moments of eq. (YuLuobasis) on D3Q19, un-streamed (periodic box)."""
    G = grad.view((3, 3) + tuple(drho.shape))
    div = G[0, 0] + G[1, 1] + G[2, 2]
    E = (G + G.transpose(0, 1)) / 2
    t = torch.full_like(drho, x.tau0)
    if x.kw["closure"] == "smag":
        t = x.tau0 + 3 * x.kw["smag_cs"] ** 2 * torch.sqrt(2 * (E * E).sum((0, 1)))
    mn = torch.zeros((x.q,) + tuple(drho.shape), dtype=torch.float64, device=DEVICE)
    mn[1] = -38 / (3 * x.kw["rates"][1]) * div
    mn[9] = -2 * t / 3 * (3 * G[0, 0] - div)
    mn[11] = -2 * t / 3 * (G[1, 1] - G[2, 2])
    for k, (a, b) in ((13, (0, 1)), (14, (1, 2)), (15, (0, 2))):
        mn[k] = -2 * t / 3 * E[a, b]
    f = torch.einsum("qk,k...->q...", x.Ti, mn)
    uu = (u * u).sum(0)
    for i, c in enumerate(x.c):
        cu = sum(c[a] * u[a] for a in range(3))
        f[i] += x.w[i] * (drho + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
        f[i] = torch.roll(f[i].clone(), tuple(-v for v in c[::-1]), (0, 1, 2))
    return f
