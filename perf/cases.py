"""The work that a user of this library has it do, as cases that can be timed.

A case is one segment of a simulation through the Python binding: a lattice
that is already set up and started advances some steps, and the fields that
the user's program saves come back. Workloads are those of
``paper_2112_01975_gb300.inputs`` (drops, the coalescence, the impact on
pillars), the channel flow of the layered Poiseuille tests, the parameter
sweep of ``serve`` (many lattices of uneven sizes in one batch, ticks of 50
steps), and the read-back of diagnostics and checkpoints.

Fields of FP64 lattices are returned as the FP64 the library gives. Those of
reduced storage (FP32, FP16/BF16-shifted) are returned as the FP32 frames that
a program saves of them.
"""
import math

import torch

from paper_2112_01975_gb300 import inputs
from paper_2112_01975_gb300 import lbm as L

STORAGE = {"f64": L.F64, "f32": L.F32, "f16s": L.F16S, "bf16s": L.BF16S}
FLUIDS = {"vdw_tr0.8": inputs.DROP_D2Q9_64, "pr_tr0.7": inputs.DROP_D3Q27_128,
          "pr_tr0.45": inputs.COALESCENCE_D3Q27_256, "pr_tr0.5": inputs.IMPACT_D3Q27_384}


def listed():
    # A case of kind "run": nx x ny x nz nodes (nz = 1: D2Q9), a drop (or two)
    # of the fluid, `steps` steps, then rho, u and U. walls: "none"; "pillars":
    # the impact's two-plane wall with 8 x 8 x 16 pillars, the drop moving
    # down; "channel": solid rows at both ends of y and a body force along x.
    # tuned: the user's program has called autotune() once.
    return [
        # The static drop on 64 x 64 in FP64, the library's default storage and
        # the smallest configured run: thousands of tiny steps.
        dict(name="d2q9_drop_64_f64", kind="run", nx=64, ny=64, nz=1, fluid="vdw_tr0.8", storage="f64",
             walls="none", tuned=False, steps=200),
        # A 2D channel of 200 fluid rows driven by a body force, FP64, odd
        # width: the layered Poiseuille flow's set-up.
        dict(name="d2q9_channel_301x202_f64", kind="run", nx=301, ny=202, nz=1, fluid="vdw_tr0.8",
             storage="f64", walls="channel", tuned=False, steps=100),
        # A large 2D drop in FP32, the sweep's largest 2D size, alone.
        dict(name="d2q9_drop_512_f32", kind="run", nx=512, ny=512, nz=1, fluid="vdw_tr0.8", storage="f32",
             walls="none", tuned=False, steps=100),
        # The configured 3D drop in FP64: the reference runs that reduced
        # storage is held against.
        dict(name="d3q27_drop_128_f64", kind="run", nx=128, ny=128, nz=128, fluid="pr_tr0.7", storage="f64",
             walls="none", tuned=False, steps=20),
        # The same drop in FP32, as in the quick start.
        dict(name="d3q27_drop_128_f32", kind="run", nx=128, ny=128, nz=128, fluid="pr_tr0.7", storage="f32",
             walls="none", tuned=False, steps=50),
        # A small ragged box with pillars in FP32: rows that are no multiple of
        # anything, solids that the drop falls on.
        dict(name="d3q27_pillars_97x61x75_f32", kind="run", nx=97, ny=61, nz=75, fluid="pr_tr0.7",
             storage="f32", walls="pillars", tuned=False, steps=100),
        # The 256^3 coalescence of two drops (density ratio 6.6e4) in
        # FP16-shifted storage, the form for long runs at large size.
        dict(name="d3q27_coalescence_256_f16s", kind="run", nx=256, ny=256, nz=256, fluid="pr_tr0.45",
             storage="f16s", walls="none", tuned=False, steps=40),
        # The drop impact on pillars, the largest configured run and the
        # benchmark's workload, FP32, tuned once as the benchmark does.
        dict(name="d3q27_impact_384x384x256_f32", kind="run", nx=384, ny=384, nz=256, fluid="pr_tr0.5",
             storage="f32", walls="pillars", tuned=True, steps=40),
        # One tick of the sweep server: uneven 3D lattices in FP32 in one batch.
        dict(name="sweep_d3q27_64to160_f32", kind="batch", lattice=1, storage="f32", least=64, most=160,
             members=6, steps=50),
        # The same for uneven 2D lattices in FP16-shifted storage.
        dict(name="sweep_d2q9_64to512_f16s", kind="batch", lattice=0, storage="f16s", least=64, most=512,
             members=16, steps=50),
        # Diagnostics of a running FP32 simulation: all fields, the discrete
        # pressure tensor, mass and momentum (no step between).
        dict(name="diagnostics_160_f32", kind="diagnostics", nx=160, ny=160, nz=160, fluid="pr_tr0.7",
             storage="f32", walls="none", steps=8),
        # Restart from and write of a checkpoint: FP64 populations into
        # BF16-shifted storage, some steps, and out again.
        dict(name="checkpoint_128x96x112_bf16s", kind="checkpoint", nx=128, ny=96, nz=112, fluid="pr_tr0.7",
             storage="bf16s", walls="none", steps=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "run", "batch", "diagnostics", "checkpoint"])
    if kind == "batch":
        lattice = rng.choice([0, 1])
        most = rng.choice([96, 128, 160, 192]) if lattice else rng.choice([128, 256, 384, 512])
        return dict(kind="batch", lattice=lattice, storage=rng.choice(["f32", "f16s"]), least=64, most=most,
                    members=rng.randint(2, 6 if lattice else 24), steps=50)
    three = kind != "run" or rng.random() < 0.65
    storage = rng.choice(["f64", "f32", "f32", "f16s", "bf16s"])
    if kind == "checkpoint" and storage == "f64":
        storage = "f32"
    if three:
        # sides from the smallest box that holds a drop to the coalescence's
        # 256 (128 in FP64); the third side lets the proportions vary
        top = 128 if storage == "f64" else 256
        nx, ny, nz = (_log_int(rng, 24, top) for _ in range(3))
        fluid = "pr_tr0.7"
        walls = rng.choice(["none", "none", "pillars"]) if kind == "run" else "none"
        if walls == "pillars":
            nz = max(nz, 48)
    else:
        nx, ny, nz = _log_int(rng, 32, 512), _log_int(rng, 32, 512), 1
        fluid = "vdw_tr0.8"
        walls = rng.choice(["none", "none", "channel"])
    nodes = nx * ny * nz
    # few steps for large lattices, many for small ones
    steps = 10 if kind == "checkpoint" else 8 if kind == "diagnostics" else max(10, min(200, int(4e8 / nodes)))
    if storage == "f64" and three:
        steps = min(steps, 40)
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, fluid=fluid, storage=storage, walls=walls, steps=steps)
    if kind == "run":
        case["tuned"] = False
    return case


# ---- inputs ---------------------------------------------------------------

def _member_sizes(case):
    """Sides of a batch's lattices: multiples of 32 spread over the range."""
    sides = list(range(case["least"], case["most"] + 1, 32))
    return [sides[(5 * k + 2) % len(sides)] for k in range(case["members"])]


def _mask(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["walls"] == "pillars":
        return inputs.pillar_mask(nx, ny, nz, seed=4, wall=2)
    if case["walls"] == "channel":   # one solid row at each end of y
        import numpy as np
        m = np.zeros((nz, ny, nx), dtype=np.uint8)
        m[:, 0] = m[:, -1] = 1
        return m.ravel()
    return None


def _fields(nx, ny, nz, fluid, walls, seed):
    """(rho0, u0) on the GPU in FP64: a drop (two touching ones for the
    coalescence fluid, at rest) of the fluid's coexistence densities, placed
    and sized by the seed, moving, with 1e-4 relative noise."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) + 1))
    r = (torch.rand(4, generator=g, device="cuda", dtype=torch.float64) * 2 - 1).tolist()
    x = torch.arange(nx, device="cuda", dtype=torch.float64)
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    z = torch.arange(nz, device="cuda", dtype=torch.float64)[:, None, None]
    D = 3 if nz > 1 else 2
    side = min(nx, ny, nz) if D == 3 else min(nx, ny)
    R = 0.25 * side * (1 + 0.05 * r[3])
    cx, cy, cz = nx / 2 + 2 * r[0], ny / 2 + 2 * r[1], (nz / 2 + 2 * r[2] if D == 3 else 0.0)
    if walls == "pillars":   # above the pillar tops (z = 17)
        R = min(0.16 * min(nx, ny), 0.25 * (nz - 18)) * (1 + 0.05 * r[3])
        cz = 17 + R + 8
    centres = [(cx, cy, cz)]
    if fluid is FLUIDS["pr_tr0.45"]:
        R = 40.0 / 256.0 * side
        centres = [(cx - R, cy, cz), (cx + R, cy, cz)]
    rho = None
    for a, b, c in centres:
        d = ((x - a) ** 2 + (y - b) ** 2 + ((z - c) ** 2 if D == 3 else 0.0)).sqrt() - R
        d = 0.5 * (fluid.rho_l + fluid.rho_v) - 0.5 * (fluid.rho_l - fluid.rho_v) * torch.tanh(2.0 * d / 5.0)
        rho = d if rho is None else torch.maximum(rho, d)
    rho = rho.expand(nz, ny, nx).contiguous()
    frac = (rho - fluid.rho_v) / (fluid.rho_l - fluid.rho_v)
    u = torch.zeros((D, nz, ny, nx), device="cuda", dtype=torch.float64)
    if walls == "pillars":
        u[2] = -0.05 * frac   # falling
    elif walls != "channel" and len(centres) == 1:
        u[0] = 0.02 * frac    # drifting
    rho = rho * (1 + 1e-4 * (2 * torch.rand(rho.shape, generator=g, device="cuda", dtype=torch.float64) - 1))
    return rho, u


def _fluid_args(fluid, walls):
    """Keyword arguments of LBM for the fluid and the walls."""
    kw = dict(a=fluid.a, b=fluid.b)
    if walls != "none":
        kw["rho_w"] = fluid.rho_v
    if walls == "channel":
        kw["g"] = (1e-6, 0.0)
    return kw


def _lattice(case, seed, stream):
    fluid = FLUIDS[case["fluid"]]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    g = L.LBM(L.D3Q27 if nz > 1 else L.D2Q9, nx, ny, nz, fluid.eos, fluid.t_over_tc, fluid.kappa, fluid.tau,
              storage=STORAGE[case["storage"]], mask=_mask(case), stream=stream,
              **_fluid_args(fluid, case["walls"]))
    rho, u = _fields(nx, ny, nz, fluid, case["walls"], seed)
    torch.cuda.synchronize()   # the fields were made on another stream
    g.init(rho, u)
    return g


def _room(g):
    """Device buffers for rho, u and U."""
    return tuple(torch.empty(k * g.N, dtype=torch.float64, device="cuda") for k in (1, g.D, g.D))


def prepare(case, seed):
    if case["kind"] == "batch":
        members, rooms = [], []
        for k, n in enumerate(_member_sizes(case)):
            sub = dict(nx=n, ny=n, nz=n if case["lattice"] else 1, fluid="vdw_tr0.8", walls="none",
                       storage=case["storage"])
            members.append(_lattice(sub, 100 * seed + k, None))
            rooms.append(_room(members[-1])[:2])
        return dict(kind="batch", steps=case["steps"], members=members, rooms=rooms, batch=L.Batch(members))
    stream = torch.cuda.Stream()
    g = _lattice(case, seed, stream)
    st = dict(kind=case["kind"], steps=case["steps"], g=g, stream=stream, exact=case["storage"] == "f64")
    with torch.cuda.stream(stream):
        if case["kind"] == "checkpoint":
            st["saved"] = g.get_populations(torch.empty(g.Q * g.N, dtype=torch.float64, device="cuda"))
            st["out"] = torch.empty_like(st["saved"])
        else:
            st["out"] = _room(g)
        if case["kind"] == "diagnostics":
            g.step(case["steps"])
            st["P"] = torch.empty((6 if g.D == 3 else 3) * g.N, dtype=torch.float64, device="cuda")
    if case.get("tuned"):
        g.autotune()
    torch.cuda.synchronize()
    return st


# ---- one pass ---------------------------------------------------------------

def _frames(tensors, exact):
    return list(tensors) if exact else [t.float() for t in tensors]


def run(st):
    if st["kind"] == "batch":
        st["batch"].step(st["steps"])
        st["batch"].sync()
        out = []
        for m, (rho, u) in zip(st["members"], st["rooms"]):
            m.moments(out=(rho, u, None))
            out += _frames((rho, u), False)
        # the batch runs on a stream of its own: the frames are made before
        # its next step may change the fields
        torch.cuda.current_stream().synchronize()
        return out
    g = st["g"]
    with torch.cuda.stream(st["stream"]):
        if st["kind"] == "checkpoint":
            g.set_populations(st["saved"])
            g.step(st["steps"])
            g.get_populations(st["out"])
            return _frames((st["out"],), st["exact"])
        if st["kind"] == "diagnostics":
            g.moments(out=st["out"])
            g.pressure_tensor(out=st["P"])
            mass, momentum = g.reduce()
            return _frames((*st["out"], st["P"]), st["exact"]) + [mass, momentum]
        g.step(st["steps"])
        g.moments(out=st["out"])
        return _frames(st["out"], st["exact"])


# ---- what a pass cannot do without ------------------------------------------

# Bytes of one node's state, read or written once per step (populations and,
# in shifted storage, the source density), and arithmetic per node and step
# by the form with the fewest operations that is known here: sums for the
# moments 2 Q, the equation of state 30, the separable force stencils 2
# fields x 2 rings x 13 (2D: 6), collision 4 Q, factors 80.
def _node_bytes(three, storage):
    q = 27 if three else 9
    return q * {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}[storage] + (4 if storage.endswith("16s") else 0)


def _node_flops(three):
    return 6 * 27 + 30 + 52 + 80 if three else 6 * 9 + 30 + 24 + 50


def work(case):
    if case["kind"] == "batch":
        three = bool(case["lattice"])
        nodes = sum(n ** 3 if three else n ** 2 for n in _member_sizes(case))
        fields = (4 if three else 3) * 8
        steps = case["steps"]
    else:
        three = case["nz"] > 1
        nodes = case["nx"] * case["ny"] * case["nz"]
        fields = (7 if three else 5) * 8
        steps = case["steps"]
        if case["kind"] == "diagnostics":   # the state read once, fields and tensor written
            return {"bytes": nodes * (_node_bytes(three, case["storage"]) + fields + (6 if three else 3) * 8),
                    "flops": nodes * (_node_flops(three) + 300)}
        if case["kind"] == "checkpoint":    # FP64 populations in and out
            fields = 2 * 8 * (27 if three else 9)
    state = _node_bytes(three, case["storage"])
    return {"bytes": nodes * (2 * state * steps + state + fields), "flops": nodes * _node_flops(three) * steps}


# ---- the same in 64 bits, plain torch ---------------------------------------

class _Exact:
    """The method's update in FP64 on [direction][z][y][x] arrays."""

    def __init__(self, nx, ny, nz, fluid, walls, mask):
        self.D = 3 if nz > 1 else 2
        self.Q = 3 ** self.D
        self.c = [(i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1 if self.D == 3 else 0) for i in range(self.Q)]
        self.fluid, self.omega = fluid, 1.0 / fluid.tau
        self.g = (1e-6, 0.0, 0.0) if walls == "channel" else (0.0, 0.0, 0.0)
        self.solid = None if mask is None else torch.from_numpy(mask).cuda().bool().view(nz, ny, nx)
        a, b, tr = fluid.a, fluid.b, fluid.t_over_tc
        if fluid.eos == L.EOS_VDW:
            self.RT, self.aalpha = tr * 8.0 * a / (27.0 * b), a
        else:
            m = 0.37464 + 1.54226 * 0.344 - 0.26992 * 0.344 ** 2
            self.RT = tr * (0.0778 / 0.45724) * a / b
            self.aalpha = a * (1.0 + m * (1.0 - math.sqrt(tr))) ** 2

    @staticmethod
    def at(v, dx, dy, dz):
        """v(r + d)."""
        return torch.roll(v, (-dz, -dy, -dx), (-3, -2, -1))

    def axis(self, v, a, s):
        """v one offset s down and up along axis a."""
        d = [0, 0, 0]
        d[a] = s
        return self.at(v, -d[0], -d[1], -d[2]), self.at(v, *d)

    def excess(self, rho):
        b, RT = self.fluid.b, self.RT
        if self.fluid.eos == L.EOS_VDW:
            return rho * RT / (1 - b * rho) - self.aalpha * rho * rho - rho / 3
        return rho * RT / (1 - b * rho) - self.aalpha * rho * rho / (1 + 2 * b * rho - (b * rho) ** 2) - rho / 3

    def sums(self, v, s):
        """sum_i (w_i / cs2) c_i v(r + s c_i), per component."""
        out = []
        for a in range(self.D):
            lo, hi = self.axis(v, a, s)
            t = 0.5 * (hi - lo)
            for b in range(self.D):
                if b != a:
                    lo, hi = self.axis(t, b, s)
                    t = (4.0 * t + lo + hi) / 6.0
            out.append(t)
        return out

    def force(self, rho, d):
        psi, sgn = d.abs().sqrt(), torch.where(d > 0, 1.0, -1.0).double()
        p1, p2, r1, r2 = self.sums(psi, 1), self.sums(psi, 2), self.sums(rho, 1), self.sums(rho, 2)
        return [-2 * sgn * psi * (4 / 3 * p1[a] - p2[a] / 6) - self.fluid.kappa * rho * (2 * r1[a] - r2[a]) +
                rho * self.g[a] for a in range(self.D)]

    def side(self, f):
        """(rho, u) with the solids' virtual density."""
        rho = f.sum(0)
        u = [sum(self.c[i][a] * f[i] for i in range(self.Q) if self.c[i][a]) / rho for a in range(self.D)]
        if self.solid is not None:
            rho = torch.where(self.solid, self.fluid.rho_v, rho)
            u = [torch.where(self.solid, 0.0, v) for v in u]
        return rho, u

    @staticmethod
    def factors(xi, zeta):
        return (zeta - xi) / 2, 1 - zeta, (zeta + xi) / 2

    def product(self, rho, fac, i):
        v = rho
        for a in range(self.D):
            v = v * fac[a][self.c[i][a] + 1]
        return v

    def start(self, rho0, u0):
        rho = rho0 if self.solid is None else torch.where(self.solid, self.fluid.rho_v, rho0)
        F = self.force(rho, self.excess(rho))
        u = [u0[a] - F[a] / (2 * rho) for a in range(self.D)]
        fac = [self.factors(v, 1 / 3 + v * v) for v in u]
        return torch.stack([self.product(rho, fac, i) for i in range(self.Q)])

    def step(self, f):
        rho, u = self.side(f)
        F = self.force(rho, self.excess(rho))
        fe, fs = [], []
        for a in range(self.D):
            lo, hi = self.axis(rho * u[a] ** 3, a, 1)
            phi = -(1 - self.omega / 2) * (hi - lo) / 2
            xs = u[a] + F[a] / rho
            fe.append(self.factors(u[a], 1 / 3 + u[a] ** 2))
            fs.append(self.factors(xs, 1 / 3 + xs * xs + phi / rho))
        del F
        new, kept = torch.empty_like(f), None
        for i in range(self.Q):
            post = self.product(rho, fs, i) + (1 - self.omega) * (f[i] - self.product(rho, fe, i))
            new[i] = self.at(post, *(-v for v in self.c[i]))
            if self.solid is not None:   # halfway bounce-back at the node itself
                back = self.at(self.solid, *self.c[i]) & ~self.solid
                kept = (kept or []) + [(self.Q - 1 - i, back, post[back])]
        for i, back, v in kept or []:
            new[i][back] = v
        return new

    def moments(self, f):
        rho, u = self.side(f)
        F = self.force(rho, self.excess(rho))
        U = [u[a] + F[a] / (2 * rho) for a in range(self.D)]
        if self.solid is not None:
            U = [torch.where(self.solid, 0.0, v) for v in U]
        return rho.reshape(-1), torch.stack(u).reshape(-1), torch.stack(U).reshape(-1)

    def pressure(self, f):
        rho, _ = self.side(f)
        d = self.excess(rho)
        psi, sgn = d.abs().sqrt(), torch.where(d > 0, 1.0, -1.0).double()
        kap, out = self.fluid.kappa, []
        for a, b in [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]:
            p = torch.zeros_like(rho)
            for i, c in enumerate(self.c):
                cc = c[a] * c[b]
                if not cc:
                    continue
                w = 3.0 * cc * math.prod(2 / 3 if v == 0 else 1 / 6 for v in c)
                up, dn, up2 = c, tuple(-v for v in c), tuple(2 * v for v in c)
                p += cc * f[i]
                p += w * sgn * (4 / 3 * psi * self.at(psi, *up) - (psi * self.at(psi, *up2) +
                                                                 self.at(psi, *dn) * self.at(psi, *up)) / 6)
                p += w * kap * (rho * self.at(rho, *up) - (rho * self.at(rho, *up2) +
                                                           self.at(rho, *dn) * self.at(rho, *up)) / 2)
            out.append(p.reshape(-1))
        return torch.cat(out)


def _exact_state(nx, ny, nz, fluid, walls, mask, seed):
    m = _Exact(nx, ny, nz, fluid, walls, mask)
    return m, m.start(*_fields(nx, ny, nz, fluid, walls, seed))


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for k, n in enumerate(_member_sizes(case)):
            m, f = _exact_state(n, n, n if case["lattice"] else 1, FLUIDS["vdw_tr0.8"], "none", None, 100 * seed + k)
            for _ in range(case["steps"]):
                f = m.step(f)
            out += list(m.moments(f)[:2])
        return out
    m, f = _exact_state(case["nx"], case["ny"], case["nz"], FLUIDS[case["fluid"]], case["walls"], _mask(case), seed)
    for _ in range(case["steps"]):
        f = m.step(f)
    if case["kind"] == "checkpoint":
        return [f.reshape(-1)]
    if case["kind"] == "diagnostics":
        mom = torch.stack([sum(m.c[i][a] * f[i].sum() for i in range(m.Q)) for a in range(m.D)])
        return list(m.moments(f)) + [m.pressure(f), float(f.sum()), mom.cpu().numpy()]
    return list(m.moments(f))
