"""Performance cases of the LBMTau1 step: what users have this library do.

Every case drives the public entry points of
``paper_1912_09327_gb300.binding`` (``Domain``, ``Batch``) and returns the whole
resulting state.  The sizes are those of the library's own configurations,
tests and benchmark (channel 64 x 32, cavity 256^2 .. 8192^2, periodic boxes
and porous samples up to 4096^2, the batched mix of sides 64 .. 1024, the
multiphase drop) or ragged ones of the same range.

``advance`` cases step a domain by ``steps`` in one call and read the residual,
as a solver does that tests for convergence at intervals (Section 3 of
arXiv:1912.09327 tests the cavity every 1000 steps), and take a device copy of
the state.  ``monitor`` cases test after every step (the channel's criterion of
the same section).  ``restart`` cases load a state from the host, step and
read it back.  ``batch`` cases advance many domains together by one chunk and
read all residuals, as the serving loop does.  Every pass goes on from the
state the previous one left, as a time loop does.
"""
import math

import numpy as np
import torch

from paper_1912_09327_gb300 import binding, serving, workloads

ES = {"f32": 4, "f16": 2, "bf16": 2}
DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
# the storage formats' exact scales of rho - 1 and j (include/lbmtau1.h)
SCALE = {"f32": (1.0, 1.0), "f16": (1024.0, 64.0), "bf16": (1.0, 1.0)}
# floating-point operations per lattice update of the moments-only closed
# form: about 20 to turn a node into its six quantities, 50 for the nine-point
# sums of three moments; the pseudo-potential force adds about 25
FLOPS, FLOPS_SC = 70.0, 25.0

_STREAM = []


def stream():
    """The program's stream (one for all domains; not the default stream)."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def listed():
    return [
        # the Poiseuille channel of Section 3 at its test size: pure latency
        dict(name="channel_64x32", kind="advance", geom="channel", nx=64,
             ny=32, steps=1000, storage="f32"),
        # smallest point of the single-domain sweep, a small cavity solve
        dict(name="cavity_256", kind="advance", geom="cavity", nx=256, ny=256,
             steps=500, storage="f32"),
        # the lid-driven cavity configuration, one convergence interval
        dict(name="cavity_1024", kind="advance", geom="cavity", nx=1024,
             ny=1024, steps=1000, storage="f32"),
        # a porous sample of ragged size: walls in every tile
        dict(name="porous_2040x1531", kind="advance", geom="porous", nx=2040,
             ny=1531, steps=200, storage="f32"),
        # all-fluid periodic box of the bandwidth sweep, larger than L2
        dict(name="box_4096", kind="advance", geom="box", nx=4096, ny=4096,
             steps=100, storage="f32"),
        # a large cavity: a long time loop over memory
        dict(name="cavity_8192", kind="advance", geom="cavity", nx=8192,
             ny=8192, steps=100, storage="f32"),
        # a channel whose residual is tested after every step
        dict(name="monitor_4001x2047", kind="monitor", geom="channel", nx=4001,
             ny=2047, steps=10, storage="f32"),
        # 16-bit storage, stochastic rounding (its default)
        dict(name="cavity_f16_4096x2500", kind="advance", geom="cavity",
             nx=4096, ny=2500, steps=100, storage="f16"),
        dict(name="channel_bf16_1101x900", kind="advance", geom="channel",
             nx=1101, ny=900, steps=200, storage="bf16"),
        # the multiphase drop of Section 4
        dict(name="drop_2048", kind="advance", geom="drop", nx=2048, ny=2048,
             steps=100, storage="f32"),
        # one chunk of the batched mix / the serving loop: 48 domains
        dict(name="batch_48", kind="batch", count=48, lo=64, hi=1024, mix=0,
             steps=200, storage="f32"),
        # resume from a host checkpoint, step, write the next checkpoint
        dict(name="restart_2000x1500", kind="restart", geom="cavity", nx=2000,
             ny=1500, steps=50, storage="f32"),
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance"] * 7 + ["monitor", "batch", "restart"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(12, 56), lo=64, hi=1024,
                    mix=rng.randrange(1 << 16), steps=rng.choice([100, 200]),
                    storage="f32")
    if kind == "monitor":
        return dict(kind=kind, geom=rng.choice(["channel", "cavity", "box"]),
                    nx=_side(rng, 256, 4400), ny=_side(rng, 256, 4400),
                    steps=rng.randint(4, 12), storage="f32")
    if kind == "restart":
        return dict(kind=kind, geom=rng.choice(["channel", "cavity"]),
                    nx=_side(rng, 256, 2400), ny=_side(rng, 256, 2400),
                    steps=rng.randint(20, 80), storage="f32")
    geom = rng.choice(["channel", "cavity", "cavity", "box", "porous", "drop"])
    storage = "f32" if geom == "drop" else rng.choice(["f32", "f32", "f16",
                                                       "bf16"])
    hi = {"porous": 2200, "drop": 2200}.get(geom, 6000)
    nx, ny = _side(rng, 48, hi), _side(rng, 32, hi)
    # between 60 and 1000 steps (16-bit: 200), fewer on large domains
    steps = int(min(1000 if storage == "f32" else 200,
                    max(60, 1.0e9 / (nx * ny))))
    return dict(kind=kind, geom=geom, nx=nx, ny=ny,
                steps=steps - rng.randint(0, 9), storage=storage)


# ---- inputs ----

def _noise(shape, seed, amp):
    """amp * N(0, 1) fields for rho - 1, u_x, u_y, drawn on one block of at
    most 512 x 512 and repeated."""
    rng = np.random.default_rng(seed)
    t = tuple(min(512, s) for s in shape)
    reps = tuple(-(-s // b) for s, b in zip(shape, t))
    return [np.tile(amp * rng.standard_normal(t), reps)[:shape[0], :shape[1]]
            for _ in range(3)]


def _problem(geom, nx, ny, seed, amp=1e-3):
    """A workload of the library with a small random perturbation on its fluid
    nodes (the seed's part of the input, with a porous sample's discs)."""
    if geom == "channel":
        p = workloads.channel(nx, max(ny, 5))
    elif geom == "cavity":
        p = workloads.cavity(nx, 0.1, ny=max(ny, 4))
    elif geom == "porous":
        p = workloads.mixed_domain("porous", nx, ny, seed) \
            if min(nx, ny) < 512 else workloads.porous(nx, seed=seed, ny=ny)
    elif geom == "drop":
        p = workloads.drop(nx, ny=ny)
    else:
        p = workloads.Problem("box", np.zeros((ny, nx), np.uint8),
                              (True, True), (0.0, 0.0), np.ones((ny, nx)),
                              np.zeros((ny, nx)), np.zeros((ny, nx)))
    d, u, v = _noise(p.mask.shape, seed + 1, amp)
    fluid = p.mask == 0
    d *= fluid
    p.rho = p.rho * (1.0 + d)
    p.jx = p.jx + p.rho * u * fluid
    p.jy = p.jy + p.rho * v * fluid
    return p


def _members(case):
    """(kind, nx, ny) of a batch's members: thirds of channel, cavity and
    porous, sides log-uniform, as workloads.batch_mix draws them."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for i in range(case["count"]):
        nx, ny = (int(round(float(np.exp(rng.uniform(
            math.log(case["lo"]), math.log(case["hi"])))))) for _ in range(2))
        out.append((workloads.KINDS[i % 3], nx, max(ny, 5)))
    return out


def _problems(case, seed):
    if case["kind"] == "batch":
        return [_problem(k, nx, ny, seed * 1009 + i)
                for i, (k, nx, ny) in enumerate(_members(case))]
    return [_problem(case["geom"], case["nx"], case["ny"], seed)]


def _domain(p, storage):
    return binding.Domain.from_problem(p, stream=stream(), storage=storage)


def prepare(case, seed):
    with torch.cuda.stream(stream()):
        doms = [_domain(p, case["storage"]) for p in _problems(case, seed)]
        st = {"kind": case["kind"], "steps": case["steps"],
              "storage": case["storage"], "doms": doms}
        if case["kind"] == "batch":
            shapes = [(d.nx, d.ny) for d in doms]
            tiles = sum(binding.lbm_tile_count(nx, ny) for nx, ny in shapes)
            b = binding.Batch(len(doms), tiles, stream=stream())
            for d in doms:
                b.add(d)
            b.set_variant(serving.choose_batch_variant(shapes))
            st["batch"] = b
        if case["kind"] == "restart":
            d = doms[0]
            st["load"], st["save"] = (
                [torch.empty((d.ny, d.nx), dtype=torch.float32,
                             pin_memory=True) for _ in range(3)]
                for _ in range(2))
            d.get_state(st["load"])
    return st


# ---- one pass ----

def _fields(d, storage):
    """The state as a device copy: [3, ny, nx] in the storage format (rows
    padded to 32 nodes, planes to 256 bytes)."""
    buf = d.snapshot()
    es = ES[storage]
    pitch = -(-d.nx // 32) * 32
    plane = -(-pitch * d.ny * es // 256) * 256 // es
    return buf.view(DTYPE[storage]).as_strided((3, d.ny, d.nx),
                                               (plane, pitch, 1))


def run(state):
    with torch.cuda.stream(stream()):
        d, n = state["doms"][0], state["steps"]
        if state["kind"] == "batch":
            b = state["batch"]
            b.step(n)
            res, mass, _ = b.residuals()
            return {"residual": res.astype(np.float32),
                    "mass": mass.astype(np.float32),
                    "state": [_fields(m, state["storage"])
                              for m in state["doms"]]}
        if state["kind"] == "monitor":
            hist = []
            for _ in range(n):
                d.step(1)
                hist.append(d.residual())
            f = _fields(d, state["storage"])
            return {"history": np.array(hist, np.float32), "drho": f[0],
                    "jx": f[1], "jy": f[2]}
        if state["kind"] == "restart":
            d.set_state(*state["load"])
            d.step(n)
            d.get_state(state["save"])
            res, mass = d.residual()
            f = state["save"]
        else:
            d.step(n)
            res, mass = d.residual()
            f = _fields(d, state["storage"])
        return {"residual": res, "mass": mass, "drho": f[0], "jx": f[1],
                "jy": f[2]}


def work(case):
    shapes = ([(nx, ny) for _, nx, ny in _members(case)]
              if case["kind"] == "batch" else [(case["nx"], case["ny"])])
    nodes = float(sum(nx * ny for nx, ny in shapes))
    # the state read once and written once, the node types read once; per
    # step where every step's result is asked for
    calls = case["steps"] if case["kind"] == "monitor" else 1
    per = FLOPS + (FLOPS_SC if case.get("geom") == "drop" else 0.0)
    return {"bytes": calls * nodes * (6 * ES[case["storage"]] + 1),
            "flops": case["steps"] * nodes * per}


# ---- the same in 64 bits ----

_E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1),
      (1, -1)]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


class _Exact:
    """Algorithm 1 in FP64 on tensors: sources padded by one node on every
    side (wrapped, or solid)."""

    def __init__(self, p):
        def dev(a):
            return torch.as_tensor(np.ascontiguousarray(a), device="cuda")
        self.per, self.F = p.periodic, p.force
        self.mask = dev(p.mask)
        self.g = p.meta.get("sc_g", 0.0)
        self.r, self.jx, self.jy = (dev(a.astype(np.float64))
                                    for a in (p.rho, p.jx, p.jy))
        self.fluid = self.mask == 0
        self.solid = self._pad((self.mask == 1).to(torch.float64), 1.0) > 0.5

    def _pad(self, a, fill):
        left, right = ((a[:, -1:], a[:, :1]) if self.per[0] else
                       (torch.full_like(a[:, :1], fill),) * 2)
        a = torch.cat([left, a, right], 1)
        low, high = ((a[-1:], a[:1]) if self.per[1] else
                     (torch.full_like(a[:1], fill),) * 2)
        return torch.cat([low, a, high], 0)

    @staticmethod
    def _at(a, e):
        h, w = a.shape
        return a[1 + e[1]:h - 1 + e[1], 1 + e[0]:w - 1 + e[0]]

    def step(self):
        jx, jy = self.jx + self.F[0], self.jy + self.F[1]
        if self.g:
            psi = self._pad((1 - torch.exp(-self.r)) * (self.mask != 1), 0.0)
            own = -self.g * self._at(psi, (0, 0))
            sx, sy = torch.zeros_like(jx), torch.zeros_like(jy)
            for e, w in zip(_E[1:], _W[1:]):
                q = w * self._at(psi, e)
                sx += e[0] * q
                sy += e[1] * q
            jx, jy = jx + own * sx, jy + own * sy
        r = self._pad(self.r, 1.0)
        u, v = self._pad(jx, 0.0) / r, self._pad(jy, 0.0) / r
        k0 = 1 - 1.5 * (u * u + v * v)
        rn, xn, yn = (torch.zeros_like(self.r) for _ in range(3))
        for e, w in zip(_E, _W):
            c = (-e[0], -e[1])
            cu = c[0] * u + c[1] * v
            f = torch.where(self._at(self.solid, e), w * self.r,
                            self._at(w * r * (k0 + 3 * cu + 4.5 * cu * cu), e))
            rn += f
            if c[0]:
                xn += c[0] * f
            if c[1]:
                yn += c[1] * f
        self.old = self.r, self.jx, self.jy
        self.r = torch.where(self.fluid, rn, self.r)
        self.jx = torch.where(self.fluid, xn, self.jx)
        self.jy = torch.where(self.fluid, yn, self.jy)

    def residual(self):
        (r0, x0, y0), w = self.old, self.fluid
        u, v = self.jx / self.r, self.jy / self.r
        num = float((((u - x0 / r0) ** 2 + (v - y0 / r0) ** 2) * w).sum())
        den = float(((u * u + v * v) * w).sum())
        return (math.sqrt(num / den) if den > 0 else math.sqrt(num),
                float((self.r * w).sum()))

    def state(self, storage):
        """As stored: a solid node holds rho - 1 = 0 and j = -F."""
        sd, sj = SCALE[storage]
        s = self.mask == 1
        return [torch.where(s, torch.zeros_like(self.r), (self.r - 1) * sd),
                torch.where(s, torch.full_like(self.r, -self.F[0] * sj),
                            self.jx * sj),
                torch.where(s, torch.full_like(self.r, -self.F[1] * sj),
                            self.jy * sj)]


def exact(case, seed):
    storage, n = case["storage"], case["steps"]
    if storage != "f32" and case["geom"] not in ("channel", "cavity"):
        return None  # undriven: all of it decays into the rounding noise
    # at most about 20 s of 64-bit steps
    if case["kind"] != "batch" and case["nx"] * case["ny"] * n > 8e9:
        return None
    got = []
    for p in _problems(case, seed):
        x = _Exact(p)
        hist = []
        for t in range(n):
            x.step()
            if case["kind"] == "monitor":
                hist.append(x.residual())
        got.append((hist, x.residual(), x.state(storage)))
    if case["kind"] == "batch":
        return {"residual": np.array([g[1][0] for g in got]),
                "mass": np.array([g[1][1] for g in got]),
                "state": [torch.stack(g[2]) for g in got]}
    hist, (res, mass), f = got[0]
    out = {"drho": f[0], "jx": f[1], "jy": f[2]}
    if case["kind"] == "monitor":
        return {"history": np.array(hist), **out}
    mass = torch.tensor(mass, dtype=torch.float64)
    if storage != "f32":
        # the flow's direction is what stands above the noise of rounding at
        # random; the others decay into it, as does the residual
        return {"residual": None, "mass": mass, "drho": None, "jx": f[1],
                "jy": None}
    return {"residual": torch.tensor(res, dtype=torch.float64), "mass": mass,
            **out}
