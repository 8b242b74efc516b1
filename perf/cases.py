"""The work that users of this library have it do, as cases that can be timed and compared.

Each case is one call pattern of the public Python binding over ``glbe.h`` / ``glbe2d.h``:

- ``solve``: a steady solve of a small lattice, from a given initial state to a residual or
  a step cap, with the fields read afterwards (3D and 2D);
- ``march``: ten time steps of a resident lattice with its velocity residual evaluated once,
  then the fields (3D and 2D; the step that parameter studies and production runs repeat);
- ``cavity``: the same march of the lid-driven cavity, flow only or on an extended magnetic
  domain;
- ``batch``: many independent ducts marched together in one persistent launch;
- ``adjoint``: the steady adjoint at a state, for a given dL/du;
- ``unrolled``: the gradient through a transient with checkpoints.

Sizes and parameters are those of this repository's benchmark and tests (plane channel,
Hartmann duct and channel, square duct under a varying force, cavity, batched ducts), and
odd sizes beside them.  Walls, rates and couplings are chosen so that every march is stable.

``exact`` is a second statement of the method in plain torch FP64: collision matrix
T^-1 Lambda T in velocity space, roll streaming, autograd for the gradients.
"""
import math
import random

import torch

U_LID = 0.0235


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _case(kind, shape, storage, steps, *, mhd=False, walls="yz", force=0, nu=0.01, gamma=0.1, Ha=10.0, K=0, n=0,
          pick=0):
    nx, ny, nz = shape            # nz = 0: the two-dimensional lattice
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "storage": storage, "steps": steps, "mhd": mhd, "walls": walls,
            "force": force, "nu": nu, "gamma": gamma, "Ha": Ha, "K": K, "n": n, "pick": pick}


def listed():
    def named(name, *a, **kw):
        return {"name": name, **_case(*a, **kw)}

    return [
        # the plane channel of the parity tests: the smallest solve, all launches and latency
        named("channel_4x32x4_f32_solve", "solve", (4, 32, 4), "f32", 200, walls="y"),
        # the Hartmann duct whose time to a residual of 1e-8 is the headline
        named("hartmann_64x64x8_f32c_solve", "solve", (64, 64, 8), "f32c", 200, mhd=True, walls="y"),
        # the 64^3 copy of the square duct that error and time-to-solution studies use
        named("duct_64_f32c_solve", "solve", (64, 64, 64), "f32c", 100, force=1, nu=0.5),
        # a two-dimensional Hartmann cross-section brought to its steady state
        named("hartmann2d_64x64_f32c_solve", "solve", (64, 64, 0), "f32c", 200, mhd=True, walls="y"),
        # the throughput benchmark: the square duct under its varying force, 16-bit storage
        named("duct_512x256x256_bf16", "march", (512, 256, 256), "bf16", 10, force=1, nu=0.5),
        # the coupled duct in FP32
        named("hartmann_128_f32", "march", (128, 128, 128), "f32", 10, mhd=True),
        # the coupled duct in 16-bit storage, on a grid whose sides are odd and share no factor with a block
        named("hartmann_255x127x129_bf16", "march", (255, 127, 129), "bf16", 10, mhd=True),
        # the large two-dimensional coupled channel
        named("hartmann2d_4096_f32", "march", (4096, 4096, 0), "f32", 10, mhd=True, walls="y"),
        # the MHD cavity of 64^3 fluid nodes inside a 16-node magnetic domain
        named("cavity_mhd_64_f32c", "cavity", (98, 98, 98), "f32c", 20, mhd=True, walls="xyz", nu=0.015, Ha=45.0),
        # batched steady solves of uneven ducts, a bounded number of levels
        named("batch_16_ducts_f32c", "batch", (32, 112, 0), "f32c", 50, nu=0.1, n=16, pick=1),
        # backward of a steady flow: dL/du in, dL/dF out
        named("adjoint_128_f32c", "adjoint", (128, 128, 128), "f32c", 50, mhd=True, force=3, nu=0.05),
        # gradient through a transient, checkpoints every 10 steps
        named("unrolled_64_f32c", "unrolled", (64, 64, 64), "f32c", 40, mhd=True, force=3, nu=0.05, K=10),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng: random.Random):
    kind = rng.choice(["solve", "solve2d", "march", "march", "march2d", "cavity", "batch", "adjoint", "unrolled"])
    mhd = rng.random() < 0.5
    if kind == "solve":
        shape = (_log_int(rng, 4, 64), _log_int(rng, 16, 72), _log_int(rng, 4, 64))
        walls = rng.choice(["y", "yz"]) if shape[2] >= 16 else "y"
        return _case("solve", shape, rng.choice(["f32", "f32c"]), 10 * rng.randint(6, 20), mhd=mhd, walls=walls,
                     force=0 if mhd else rng.choice([0, 1]), nu=0.05 if mhd else rng.choice([0.01, 0.1, 0.5]), Ha=5.0)
    if kind == "solve2d":
        return _case("solve", (_log_int(rng, 8, 256), _log_int(rng, 24, 256), 0), rng.choice(["f32", "f32c"]),
                     10 * rng.randint(6, 20), mhd=mhd, walls="y", nu=0.05, Ha=5.0)
    if kind == "march":
        shape = (_log_int(rng, 32, 512), _log_int(rng, 32, 256), _log_int(rng, 32, 256))
        storage = rng.choice(["bf16", "f16", "f32", "f32c"]) if not mhd else rng.choice(["bf16", "f32", "f32c"])
        if mhd:
            shape = tuple(min(s, 160) for s in shape)
        return _case("march", shape, storage, 10, mhd=mhd, walls=rng.choice(["yz", "yz", "y", "xyz"]),
                     force=rng.choice([0, 1, 3]), nu=0.05 if mhd else 0.5)
    if kind == "march2d":
        shape = (_log_int(rng, 128, 4096), _log_int(rng, 128, 4096), 0)
        return _case("march", shape, rng.choice(["bf16", "f32", "f32c"]) if shape[0] * shape[1] < 8_000_000 else "f32",
                     10, mhd=mhd, walls="y", nu=0.05)
    if kind == "cavity":
        w = _log_int(rng, 20, 64)
        n = w + 34 if mhd else w + 2
        return _case("cavity", (n, n, n), rng.choice(["f32", "f32c"]), 20, mhd=mhd, walls="xyz", nu=0.015, Ha=10.0)
    if kind == "batch":
        return _case("batch", (24, _log_int(rng, 40, 104), 0), rng.choice(["f32", "f32c"]), 10 * rng.randint(2, 5),
                     nu=0.1, n=rng.randint(4, 16), pick=rng.randint(2, 1_000_000))
    shape = tuple(_log_int(rng, 20, 120 if kind == "adjoint" else 64) for _ in range(3))
    if kind == "adjoint":
        return _case("adjoint", shape, rng.choice(["f32", "f32c"]), 10 * rng.randint(3, 5), mhd=mhd,
                     walls=rng.choice(["yz", "xyz"]), force=3, nu=0.05, Ha=5.0)
    return _case("unrolled", shape, rng.choice(["f32", "f32c"]), rng.randint(15, 40), mhd=mhd, walls="yz", force=3,
                 nu=0.05, Ha=5.0, K=rng.randint(4, 12))


# ---------------------------------------------------------------------------
# Inputs: everything a case needs, from the case and the seed alone
# ---------------------------------------------------------------------------
def _walls(case):
    return tuple(int(c in case["walls"]) for c in ("xy" if case["nz"] == 0 else "xyz"))


def _physics(case, rng):
    """Keyword arguments of the context (uniform force, rates, coupling) for one lattice."""
    two_d = case["nz"] == 0
    d = 2 if two_d else 3
    g, nu = case["gamma"], case["nu"]
    kw = {"wall_lo": _walls(case), "wall_hi": _walls(case), "gamma": g, "nu": nu, "storage": case["storage"],
          "F": [0.0] * d}
    if case["kind"] == "cavity":
        kw["U_lid"] = (U_LID * rng.uniform(0.8, 1.0), 0.002 * rng.random(), 0.0)
        width = case["nx"] - 2
        if case["mhd"]:
            width = case["nx"] - 34
            kw["box"] = ((17, 17, 17), (16 + width,) * 3)
    else:
        width = case["ny"] - 2
        if not case["force"]:
            kw["F"][0] = 1e-6 * rng.uniform(0.8, 1.2)
    if case["mhd"]:
        kw.update(induction=1, gamma_m=g, eta=nu, chi=0.01, mu=1.0, B0=[0.0] * d)
        kw["B0"][1] = case["Ha"] * nu / (0.5 * width)
    if case["force"]:
        kw["force_field"] = 2 if two_d else case["force"]
    return kw


def _duct_sizes(case):
    """(edge, gamma, Ha) of each duct.  The Lorentz force is lagged by a step, so a march is stable only while the
    magnetic damping per step, Ha^2 nu / (L^2 gamma), stays well below 1: Ha is held to a quarter of that."""
    r, out = random.Random(case["pick"]), []
    for _ in range(case["n"]):
        edge, gamma, Ha = r.randint(case["nx"], case["ny"]), r.choice([1.0, 0.1, 0.05]), r.choice([0.0, 5.0, 10.0])
        out.append((edge, gamma, min(Ha, 0.5 * (edge - 2) / 2 * math.sqrt(gamma / case["nu"]))))
    return out


def _batch_physics(case, rng):
    """One keyword set per duct: cubic, x periodic, walls y and z, with its own gamma and Hartmann number."""
    out = []
    for edge, gamma, Ha in _duct_sizes(case):
        one = _case("march", (edge, edge, edge), case["storage"], 0, mhd=Ha > 0, nu=case["nu"], gamma=gamma, Ha=Ha)
        out.append((edge, _physics(one, rng)))
    return out


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fields_in(case, kw, seed):
    """Initial deviations (df, dg), force field and objective weights as FP32 tensors on the device: a
    smooth velocity and density disturbance of a few long waves plus small noise in every population."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(seed)
    rng = random.Random(seed + 1)
    E, w, _, E5, W5, _ = _lattice(case["nz"] == 0)
    nx, ny, nz = case["nx"], case["ny"], max(case["nz"], 1)
    c = [torch.arange(n, device=dev, dtype=torch.float32) * (2 * math.pi / n) for n in (nx, ny, nz)]

    def wave(scale):
        v = torch.zeros(nz, ny, nx, device=dev)
        for _ in range(3):
            k = [rng.randint(0, 2), rng.randint(1, 2), rng.randint(0, 2)]
            ph = [rng.uniform(0, 2 * math.pi) for _ in range(3)]
            a = scale * rng.uniform(0.3, 1.0)
            v += a * (torch.cos(k[2] * c[2] + ph[2])[:, None, None] * torch.cos(k[1] * c[1] + ph[1])[None, :, None] *
                      torch.cos(k[0] * c[0] + ph[0])[None, None, :])
        return v

    rho, u = wave(1e-4), [wave(1e-3) for _ in range(2 if case["nz"] == 0 else 3)]
    df = torch.empty(len(w), nz, ny, nx, device=dev)
    for a, e in enumerate(E):
        df[a] = w[a] * (rho + 3 * sum(ei * ui for ei, ui in zip(e, u) if ei))
        df[a] += 1e-6 * (2 * torch.rand(nz, ny, nx, device=dev, generator=gen) - 1)
    got = {"df": df.reshape(len(w), -1)}
    del df
    if case["mhd"]:
        b0 = kw["B0"][1]
        dg = torch.empty(len(u), len(W5), nz, ny, nx, device=dev)
        for j in range(len(u)):
            b = wave(0.02 * b0)
            for a in range(len(W5)):
                dg[j, a] = W5[a] * b
                dg[j, a] += 1e-4 * b0 * (2 * torch.rand(nz, ny, nx, device=dev, generator=gen) - 1)
        got["dg"] = dg.reshape(len(u) * len(W5), -1)
        got["FL"] = torch.zeros(len(u), nz * ny * nx, device=dev)
    if case["force"]:
        n = case["force"]
        F = 1e-6 * 0.2 * torch.randn(n, nz, ny, nx, device=dev, generator=gen)
        y, z = c[1][None, :, None], c[2][:, None, None]
        F[0] += 1e-6 * (1 + 0.5 * torch.sin(y) * torch.cos(z))
        got["F"] = F.reshape(n, -1)
    if case["kind"] in ("adjoint", "unrolled"):
        got["w"] = 1e-3 * torch.randn(3, nz * ny * nx, device=dev, generator=gen)
    return got


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_0809_4730_gb300 import glbe
    rng = random.Random(seed)
    if case["kind"] == "batch":
        doms = [glbe.make_params(e, e, e, **kw) for e, kw in _batch_physics(case, rng)]
        return {"case": case, "batch": glbe.Batch(doms)}
    kw = _physics(case, rng)
    if case["nz"] == 0:
        S = glbe.Solver2D(case["nx"], case["ny"], **kw)
    else:
        S = glbe.Solver(case["nx"], case["ny"], case["nz"], **kw)
    st = {"case": case, "solver": S}
    if case["kind"] == "cavity":       # a cavity starts from rest under its lid
        return st
    got = _fields_in(case, kw, seed)
    if case["force"]:
        S.set_force(got["F"])
    S.set_state(got["df"], got.get("dg"), got.get("FL"), 0)
    if case["kind"] == "solve":        # a solve starts from the given state on every pass
        st.update(df=got["df"], dg=got.get("dg"), FL=got.get("FL"))
    st["w"] = got.get("w")
    return st


def _named_fields(f):
    return {k: v for k, v in zip(("rho", "u", "B"), f) if v is not None}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        b.reset()
        _, res, _ = b.solve(1e-8, case["steps"])
        return {"fields": [_named_fields(b.fields(d)) for d in range(b.n)], "r": [x["r"] for x in res]}
    S = state["solver"]
    if case["kind"] == "solve":
        S.set_state(state["df"], state["dg"], state["FL"], 0)
        _, steps, r = S.solve(1e-10, case["steps"])
        return {**_named_fields(S.fields()), "steps": steps, "r": r}
    if case["kind"] == "adjoint":
        dF, _, it, r = S.adjoint_steady(state["w"], 1e-12, case["steps"])
        return {"dF": dF, "iterations": it, "r": r}
    if case["kind"] == "unrolled":
        dF = S.adjoint_unrolled(case["steps"], case["K"], state["w"])
        return {"dF": dF, **_named_fields(S.fields())}
    S.step(case["steps"])
    return _named_fields(S.fields())


# ---------------------------------------------------------------------------
# What one pass cannot do without
# ---------------------------------------------------------------------------
_VALUE = {"f32": 4, "bf16": 2, "f16": 2, "f32c": 6}


def _lattice_work(case, edge=None, mhd=None):
    """(bytes of one time step, bytes of the fields read, flops of one time step): every population of a
    fluid node read and written once a step, the lagged Lorentz force likewise, the force field read."""
    two_d = case["nz"] == 0 and edge is None
    mhd = case["mhd"] if mhd is None else mhd
    n = [edge] * 3 if edge else [case["nx"], case["ny"], max(case["nz"], 1)]
    w = (0, 1, 1) if edge else _walls(case) + ((0,) if two_d else ())
    nodes = math.prod(a - 2 * b for a, b in zip(n, w))
    flow = nodes
    if case["kind"] == "cavity" and mhd:
        flow = (case["nx"] - 34) ** 3
    d, qf, qg = (2, 9, 10) if two_d else (3, 19, 21)
    v = _VALUE[case["storage"]]
    step = 2 * qf * v * flow + 4 * (d if two_d and case["force"] else case["force"]) * flow
    fields = qf * v * flow + 4 * (1 + d) * nodes
    flops = (20 * qf) * flow
    if mhd:
        step += 2 * qg * v * nodes + 2 * 4 * d * flow
        fields += qg * v * nodes + 4 * d * nodes
        flops += 10 * qg * nodes
    return step, fields, flops, nodes


def work(case):
    steps = case["steps"]
    if case["kind"] == "batch":
        by, fl = 0, 0
        for edge, _, Ha in _duct_sizes(case):
            s, f, o, _ = _lattice_work(case, edge, Ha > 0)
            by, fl = by + steps * s + f, fl + steps * o
        return {"bytes": by, "flops": fl}
    s, f, o, nodes = _lattice_work(case)
    if case["kind"] in ("adjoint", "unrolled"):
        q = 43 if case["mhd"] else 19
        lam = 4 * (2 * q + 3) * nodes                # cotangents in and out, gradient out
        if case["kind"] == "adjoint":
            # the state enters through the forward quantities that the update is linearised at
            return {"bytes": steps * (lam + 4 * (16 if case["mhd"] else 7) * nodes), "flops": 1.2 * steps * o}
        # a forward march, and a backward one that reads every level's state again
        return {"bytes": steps * (s + lam + s // 2) + f, "flops": 3.2 * steps * o}
    return {"bytes": steps * s + f, "flops": steps * o}


# ---------------------------------------------------------------------------
# The same results in 64 bits: plain torch
# ---------------------------------------------------------------------------
def _lattice(two_d):
    """(E, w, rows of T, E of the vector lattice, W, theta_m), the orderings of glbe.h and glbe2d.h."""
    if two_d:
        E = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4

        def rows(x, y, z):
            c = x * x + y * y
            return [1, -4 + 3 * c, 4 - 10.5 * c + 4.5 * c * c, x, (3 * c - 5) * x, y, (3 * c - 5) * y, x * x - y * y,
                    x * y]
        E5 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0)]
        W5, theta = [1 / 3] + [1 / 6] * 4, 1 / 3
    else:
        E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
             (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1), (-1, 0, -1),
             (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12

        def rows(x, y, z):
            c = x * x + y * y + z * z
            p, q = 3 * x * x - c, y * y - z * z
            return [1, 19 * c - 30, (21 * c * c - 53 * c + 24) / 2, x, (5 * c - 9) * x, y, (5 * c - 9) * y, z,
                    (5 * c - 9) * z, p, (3 * c - 5) * p, q, (3 * c - 5) * q, x * y, y * z, x * z, q * x,
                    (z * z - x * x) * y, (x * x - y * y) * z]
        E5 = E[:7]
        W5, theta = [1 / 4] + [1 / 8] * 6, 1 / 4
    return E, w, [list(r) for r in zip(*(rows(*e) for e in E))], E5, W5, theta


class _Plain:
    """The method in FP64 on one lattice: state (f, g, F_L) before collision, full populations."""

    def __init__(self, nx, ny, nz, two_d, kw, F):
        dev = _device()
        self.E, self.w, T, self.E5, self.W5, self.theta = _lattice(two_d)
        self.shape = (max(nz, 1), ny, nx)
        self.d = 2 if two_d else 3
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
        T = t(T)
        snu = 1 / (3 * kw["nu"] / kw["gamma"] + 0.5)
        if two_d:
            s = [1, 1.63, 1.14, 1, 1.92, 1, 1.92, snu, snu]
        else:
            s = [1, 1.19, 1.4, 1, 1.2, 1, 1.2, 1, 1.2, snu, 1.4, snu, 1.4, snu, snu, snu, 1.98, 1.98, 1.98]
        self.C = torch.linalg.inv(T) @ torch.diag(t(s)) @ T
        self.half = torch.eye(len(self.w), dtype=torch.float64, device=dev) - 0.5 * self.C
        self.ig, self.mhd = 1 / kw["gamma"], bool(kw.get("induction"))
        self.Fu = [float(torch.tensor(v, dtype=torch.float32)) for v in list(kw["F"]) + [0.0] * (3 - self.d)]
        self.F = F                       # [n, nodes] FP64 field added to the uniform force, or None
        if self.mhd:
            self.tau = kw["eta"] / (kw["gamma_m"] * self.theta) + 0.5
            self.cm, self.mc = kw["chi"] / kw["gamma_m"], kw["mu"] * kw["chi"]
            self.B0 = list(kw["B0"]) + [0.0] * (3 - self.d)
        # wall planes bound both lattices, the box the flow alone
        wall = torch.zeros(self.shape, dtype=torch.bool, device=dev)
        for axis, (lo, hi) in enumerate(zip(kw["wall_lo"], kw["wall_hi"])):
            v = wall.movedim(2 - axis, 0)
            v[0] |= bool(lo)
            v[-1] |= bool(hi)
        self.wall, self.solid, top = wall, wall.clone(), self.shape[0] - 1 - int(kw["wall_hi"][-1] and not two_d)
        if kw.get("box"):
            lo, hi = kw["box"]
            self.solid |= True
            self.solid[lo[2]:hi[2] + 1, lo[1]:hi[1] + 1, lo[0]:hi[0] + 1] = False
            self.solid |= wall
            top = hi[2]
        U = kw.get("U_lid", (0.0, 0.0, 0.0))
        self.lid = [6 * w * sum(a * b for a, b in zip(e, U)) for e, w in zip(self.E, self.w)]
        self.top = torch.zeros(self.shape, dtype=torch.bool, device=dev)
        self.top[top] = True
        opp = lambda E: [E.index(tuple(-v for v in e)) for e in E]  # noqa: E731
        self.opp, self.opp5 = opp(self.E), opp(self.E5)
        self.blocked = [self._from(self.solid, e) for e in self.E]      # the link's source is not fluid
        self.blocked5 = [self._from(self.wall, e) for e in self.E5]

    @staticmethod
    def _from(v, e):
        return torch.roll(v, shifts=(e[2], e[1], e[0]), dims=(0, 1, 2))

    def start(self, df=None, dg=None):
        dev = _device()
        w = torch.tensor(self.w, dtype=torch.float64, device=dev)[:, None, None, None]
        f = w.expand(-1, *self.shape).clone() if df is None else w + df.double().reshape(-1, *self.shape)
        if not self.mhd:
            return f, None, None
        g = torch.tensor([[W * b for W in self.W5] for b in self.B0], dtype=torch.float64, device=dev)
        g = g[:, :, None, None, None].expand(-1, -1, *self.shape).clone()
        if dg is not None:
            g[:self.d] += dg.double().reshape(self.d, len(self.W5), *self.shape)
        return f, g, torch.zeros(3, *self.shape, dtype=torch.float64, device=dev)

    def force(self, F):
        out = [torch.full(self.shape, v, dtype=torch.float64, device=_device()) for v in self.Fu]
        if F is not None:
            for k in range(F.shape[0]):
                out[k] = out[k] + F[k].reshape(self.shape)
        return out

    def macro(self, s, F):
        """rho, u, total force, B, g^eq at the collision of state s."""
        f, g, FL = s
        rho = f.sum(0)
        m = [sum(e[k] * f[a] for a, e in enumerate(self.E) if e[k]) for k in range(self.d)]
        m += [torch.zeros_like(rho)] * (3 - self.d)
        F = self.force(F)
        B = geq = fl = None
        if self.mhd:
            u = [(m[k] + 0.5 * self.ig * (F[k] + FL[k])) / rho for k in range(3)]
            u = [torch.where(self.solid, 0.0, v) for v in u]
            B = [g[j].sum(0) for j in range(3)]
            geq = []
            for j in range(3):
                for a, e in enumerate(self.E5):
                    conv = sum(e[k] * (u[k] * B[j] - B[k] * u[j]) for k in range(3) if e[k])
                    geq.append(self.W5[a] * (B[j] + conv * (self.cm / self.theta)))
            geq = torch.stack(geq).reshape(3, len(self.W5), *self.shape)
            q = g - geq
            L = [[sum(e[k] * q[j, a] for a, e in enumerate(self.E5) if e[k]) for j in range(3)] for k in range(self.d)]
            L += [[torch.zeros_like(rho)] * 3] * (3 - self.d)
            c = -1 / (self.mc * self.tau * self.theta)
            J = [c * (L[1][2] - L[2][1]), c * (L[2][0] - L[0][2]), c * (L[0][1] - L[1][0])]
            fl = [J[1] * B[2] - J[2] * B[1], J[2] * B[0] - J[0] * B[2], J[0] * B[1] - J[1] * B[0]]
            fl = [torch.where(self.solid, 0.0, v) for v in fl]
            F = [F[k] + fl[k] for k in range(3)]
        u = [(m[k] + 0.5 * self.ig * F[k]) / rho for k in range(3)]
        return rho, u, F, B, geq, fl

    def step(self, s, F):
        """The state one time step later."""
        f, g, _ = s
        rho, u, F, _, geq, fl = self.macro(s, F)
        ig = self.ig
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        neq, S = [], []
        for a, e in enumerate(self.E):
            eu = sum(e[k] * u[k] for k in range(3) if e[k]) if any(e) else 0.0 * uu
            eF = sum(e[k] * F[k] for k in range(3) if e[k]) if any(e) else 0.0 * uu
            neq.append(f[a] - self.w[a] * rho * (1 + 3 * eu + ig * (4.5 * eu * eu - 1.5 * uu)))
            S.append(self.w[a] * ig * (3 * (eF - ig * uF) + 9 * ig * eu * eF))
        mix = lambda M, v: (M @ torch.stack(v).reshape(len(v), -1)).reshape(len(v), *self.shape)  # noqa: E731
        out = f - mix(self.C, neq) + mix(self.half, S)
        new = []
        for a, e in enumerate(self.E):
            back = out[self.opp[a]]
            if self.lid[a] and e[2] < 0:
                back = back + torch.where(self.top, self.lid[a], 0.0)
            new.append(torch.where(self.blocked[a], back, self._from(out[a], e)))
        f2 = torch.stack(new)
        f2 = torch.where(self.solid, f, f2)
        if not self.mhd:
            return f2, None, None
        og = g - (g - geq) / self.tau
        new = [torch.where(self.blocked5[a], 2 * self.W5[a] * self.B0[j] - og[j, self.opp5[a]], self._from(og[j, a], e))
               for j in range(3) for a, e in enumerate(self.E5)]
        g2 = torch.where(self.wall, g, torch.stack(new).reshape(g.shape))
        return f2, g2, torch.stack(fl)

    def fields(self, s, F):
        rho, u, _, B, _, _ = self.macro(s, F)
        out = {"rho": torch.where(self.solid, 0.0, rho).reshape(-1),
               "u": torch.stack([torch.where(self.solid, 0.0, v).reshape(-1) for v in u[:self.d]])}
        if self.mhd:
            out["B"] = torch.stack([torch.where(self.wall, 0.0, v).reshape(-1) for v in B[:self.d]])
        return out

    def march(self, s, F, steps):
        """The state after `steps` steps from level 0, and the last residual r(t) on the way."""
        last, r = None, None
        for t in range(steps):
            if t % 10 == 0:
                u = self.fields(s, F)["u"]
                if last is not None:
                    r = float((u - last).norm() / u.norm())
                last = u
            s = self.step(s, F)
        return s, r


def _vjp(M, s, F, lam, w):
    """One reverse step at state s: cotangent of (f, g, F_L) and of F for lam on the next state (or None)
    plus the objective sum w.u of s (w None: no objective)."""
    leaf = [v.detach().requires_grad_(True) for v in s if v is not None]
    Fx = F.detach().requires_grad_(True)
    full = tuple(leaf) if M.mhd else (leaf[0], None, None)
    total = 0.0
    if lam is not None:
        total = sum((a * b).sum() for a, b in zip([v for v in M.step(full, Fx) if v is not None], lam))
    if w is not None:
        total = total + (M.fields(full, Fx)["u"] * w).sum()
    got = torch.autograd.grad(total, leaf + [Fx])
    return list(got[:-1]), got[-1]


def exact(case, seed):
    with torch.no_grad():
        rng = random.Random(seed)
        if case["kind"] == "batch":
            out = {"fields": [], "r": []}
            for e, kw in _batch_physics(case, rng):
                M = _Plain(e, e, e, False, kw, None)
                s, r = M.march(M.start(), None, case["steps"])
                out["fields"].append(M.fields(s, None))
                out["r"].append(r)
            return out
        kw = _physics(case, rng)
        M = _Plain(case["nx"], case["ny"], case["nz"], case["nz"] == 0, kw, None)
        if case["kind"] == "cavity":
            s, _ = M.march(M.start(), None, case["steps"])
            return M.fields(s, None)
        got = _fields_in(case, kw, seed)
        F = got["F"].double() if case["force"] else None
        s = M.start(got["df"], got.get("dg"))
        if case["kind"] == "solve":
            s, r = M.march(s, F, case["steps"])
            return {**M.fields(s, F), "steps": None, "r": r}
        if case["kind"] == "march":
            s, _ = M.march(s, F, case["steps"])
            return M.fields(s, F)
        w = got["w"].double()
        fluid = (~M.solid).reshape(-1)
    with torch.enable_grad():
        if case["kind"] == "adjoint":
            lam, kept, r = None, None, None
            for k in range(case["steps"]):
                new, dF = _vjp(M, s, F, lam, w)
                if k % 10 == 0:
                    now = dF * fluid
                    r = float((now - kept).norm() / now.norm()) if kept is not None else None
                    kept = now
                lam = new
            return {"dF": dF * fluid, "iterations": None, "r": r}
        states = [s]
        with torch.no_grad():
            for _ in range(case["steps"]):
                states.append(M.step(states[-1], F))
            out = M.fields(states[-1], F)
        lam, grad = _vjp(M, states[-1], F, None, w)
        for s in reversed(states[:-1]):
            lam, dF = _vjp(M, s, F, lam, None)
            grad = grad + dF
        return {"dF": grad * fluid, **out}
