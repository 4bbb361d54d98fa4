"""What the performance of this library is measured on: lattices, closure training and restart
work as a user's program has the library do them, through the public entry points.

Families (key "kind"):
  flow     steps of one lattice (any stencil, storage, streaming, collision, closure and
           boundary set), then the density and velocity fields on the device; with "stats" the
           plane statistics are sampled inside the steps and read back
  refined  coarse steps of a box whose middle planes are refined 2:1, then both levels'
           post-collision populations
  samples  closure-training samples and box-filtered fields of a fine lattice
  train    one minibatch of the closure training: loss, gradient, Adam update
  restart  a checkpoint read back, two steps, the monitored sums and statistics, a checkpoint
           written

Sizes come from the library's configurations (64x32x32 Poiseuille, 512x256x256 and 1024x512x512
channels, 768x384x384 D3Q27 tunnel, 256x128x128 learned closure and refined box), its tests, and
ragged sizes between them.  `exact` restates the method in float64 with plain torch.
"""
import math

import numpy as np
import torch

from paper_2305_09910_gb300 import lbm, refine

CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
TUNNEL = ("inflow", "outflow", "freeslip", "freeslip", "freeslip", "freeslip")
PERIODIC = ("periodic",) * 6
FACES = {"channel": CHANNEL, "tunnel": TUNNEL, "poiseuille": PERIODIC, "box": PERIODIC}
CS = 0.1
U_BULK = 0.05
RATES = (1.19, 1.4, 1.2, 1.4, 1.98)
MLP_SCALE = (600.0, 3000.0)
MLP_FLOOR = 0.05
NPARAM = 1345


# ---- the cases --------------------------------------------------------------------------------

def _flow(name, nx, ny, nz, steps, q=19, prec="f32", stream="pull", closure="smag", coll="trt",
          geom="channel", stats=0):
    c = {"kind": "flow", "nx": nx, "ny": ny, "nz": nz, "steps": steps, "q": q, "prec": prec,
         "stream": stream, "closure": closure, "coll": coll, "geom": geom, "stats": stats}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest configured run, where launches and latency count: a laminar channel with
        # the default settings (in-place streaming), some hundred steps between two looks at it
        _flow("poiseuille64", 64, 32, 32, 100, stream="aa", closure="none", geom="poiseuille"),
        # a lattice between the small and the large ones, as used to tune a set-up before the
        # large run: ragged rows, the multiple-relaxation-time collision of the wind-tunnel runs
        _flow("channel120_mrt", 120, 64, 63, 50, coll="mrt"),
        # the main job: the turbulent channel, profiles sampled every 10th step
        _flow("channel512_stats", 512, 256, 256, 20, stats=10),
        # the largest lattice (268 million cells), populations stored as shifted half floats
        _flow("channel1024_f16", 1024, 512, 512, 10, prec="f16"),
        # the landing-gear tunnel with 27 velocities, inflow, outflow, free-slip sides and a body
        _flow("tunnel768_q27_f16", 768, 384, 384, 10, q=27, prec="f16", geom="tunnel"),
        # the same at a size that fits no tile, float32, in place (one population array)
        _flow("tunnel375_q27_aa", 375, 190, 187, 10, q=27, stream="aa", geom="tunnel"),
        # in-place half storage, ragged: the smallest memory per cell
        _flow("channel251_bf16_aa", 251, 130, 121, 10, prec="bf16", stream="aa"),
        # the learned closure inside the step, at its configured size
        _flow("channel256_mlp", 256, 128, 128, 10, closure="mlp"),
        # a refined box: both levels step, the transfer kernels run between them
        {"name": "refined256", "kind": "refined", "nx": 256, "ny": 128, "nz": 128, "z0": 32, "z1": 96,
         "steps": 3, "prec": "f32"},
        # one minibatch of the closure training at the size the training test uses
        {"name": "train_122880", "kind": "train", "n": 122880, "nbatch": 64},
        # the closure's training data and reference fields from a fine lattice
        {"name": "samples512", "kind": "samples", "nx": 512, "ny": 256, "nz": 256, "stream": "aa",
         "prec": "f32", "steps": 2},
        # what a long run does between its stretches of steps: restart, monitor, checkpoint
        {"name": "restart256", "kind": "restart", "nx": 256, "ny": 128, "nz": 130, "q": 19, "stream": "pull",
         "prec": "f32"},
    ]


def _size(rng, lo, hi):
    """Sizes of a box of lo .. hi cells (logarithmic), x longest, odd and ragged ones among them."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ax, ay = rng.uniform(1.0, 2.5), rng.uniform(0.7, 1.4)
    nz = (n / (ax * ay)) ** (1.0 / 3.0)
    nx, ny, nz = int(nz * ax), int(nz * ay), int(nz)
    if rng.random() < 0.4:
        nx = max(32, nx // 32 * 32)
    return max(nx, 17), max(ny, 12), max(nz, 9)


def draw(rng):
    kind = rng.choice(["flow"] * 6 + ["mlp", "refined", "samples", "train", "restart"])
    if kind == "train":
        return {"kind": "train", "n": int(math.exp(rng.uniform(math.log(300), math.log(1000000)))),
                "nbatch": rng.choice([1, 16, 64])}
    if kind == "refined":
        nx, ny, nz = _size(rng, 5e3, 3e6)
        z0 = rng.randint(2, max(2, nz // 3))
        return {"kind": "refined", "nx": nx, "ny": ny, "nz": nz, "z0": z0,
                "z1": rng.randint(z0 + 2, nz - 2), "steps": rng.randint(1, 4),
                "prec": rng.choice(["f32", "f32", "f16", "bf16"])}
    if kind == "samples":
        nx, ny, nz = _size(rng, 2e4, 3e7)
        return {"kind": "samples", "nx": 2 * (nx // 2), "ny": 2 * (ny // 2), "nz": 2 * (nz // 2),
                "stream": rng.choice(["aa", "pull"]), "prec": rng.choice(["f32", "f32", "f16"]),
                "steps": rng.randint(2, 3)}
    if kind == "restart":
        nx, ny, nz = _size(rng, 2e4, 3e7)
        return {"kind": "restart", "nx": nx, "ny": ny, "nz": nz, "q": rng.choice([19, 27]),
                "stream": rng.choice(["aa", "pull"]), "prec": rng.choice(["f32", "f32", "f16"])}
    if kind == "mlp":
        nx, ny, nz = _size(rng, 1e5, 1.5e7)
        return _flow(None, nx, ny, nz, rng.randint(4, 16), closure="mlp", stream=rng.choice(["pull", "aa"]))
    geom = rng.choice(["channel", "channel", "tunnel", "box"])
    q = rng.choice([19, 19, 27])
    nx, ny, nz = _size(rng, 3e4, 4e7)
    if geom == "tunnel" and nx % 32 == 1:
        nx += 1  # the outflow face does not take such rows
    coll = rng.choice(["trt", "trt", "trt", "mrt" if q == 19 else "reg", "reg"])
    steps = rng.randint(10, 20) if nx * ny * nz > 2e6 else rng.randint(20, 80)
    return _flow(None, nx, ny, nz, steps, q=q, prec=rng.choice(["f32", "f32", "f16", "bf16"]),
                 stream=rng.choice(["pull", "pull", "aa"]), closure=rng.choice(["smag", "smag", "none"]),
                 coll=coll, geom=geom, stats=rng.choice([0, 0, 10]) if geom != "tunnel" else 0)


# ---- inputs -----------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _fluid(case, geom):
    """Relaxation time and body force of a case."""
    ny = case["ny"]
    if geom == "poiseuille":
        return 0.8, 1e-6
    if geom == "tunnel":
        nu = U_BULK * 80 * max(case["nx"], 96) / 768 / 1e4
        return 0.5 + 3 * (max(nu, 0.02) if case["closure"] == "none" else nu), 0.0
    delta = ny / 2.0
    nu = max(2.0 * delta * U_BULK / (180.0 / 0.09) ** (1.0 / 0.88), 2e-3)
    if case.get("closure") == "none":  # no subgrid model: a viscosity that resolves the flow
        nu = max(nu, 0.02)
    u_tau = 180.0 * nu / delta
    return 3.0 * nu + 0.5, min(u_tau * u_tau / delta, 1e-6)


def _velocity(nx, ny, nz, geom, seed):
    """The initial velocity: a perturbed laminar profile (channel, box), a uniform stream with
    noise (tunnel), slow noise (Poiseuille)."""
    g = _gen(seed)
    u = torch.rand((3, nz, ny, nx), generator=g, device="cuda", dtype=torch.float32)
    u.sub_(0.5)
    if geom == "poiseuille":
        return u.mul_(1e-4)
    if geom == "tunnel":
        u.mul_(0.02 * U_BULK)
        u[0] += U_BULK
        return u
    u.mul_(0.1 * U_BULK)
    ph = (torch.rand(4, generator=g, device="cuda") * 2 * math.pi).double()
    x = torch.arange(nx, device="cuda", dtype=torch.float64)
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny
    z = torch.arange(nz, device="cuda", dtype=torch.float64)
    u[0] += (6.0 * U_BULK * y * (1.0 - y)).float()[None, :, None]
    env = (0.1 * U_BULK * torch.sin(math.pi * y)).float()[None, :, None]
    sx = torch.sin(2 * math.pi * 4 * x / nx + ph[0]).float()[None, None, :]
    cx = torch.cos(2 * math.pi * 4 * x / nx + ph[2]).float()[None, None, :]
    u[1] += sx * env * torch.cos(2 * math.pi * 2 * z / nz + ph[1]).float()[:, None, None]
    u[2] += cx * env * torch.sin(2 * math.pi * 2 * z / nz + ph[3]).float()[:, None, None]
    return u


def _flags(nx, ny, nz, geom, seed):
    """Cell flags: solid rows (Poiseuille), a landing-gear-like body (tunnel), else None."""
    if geom == "poiseuille":
        f = torch.zeros((nz, ny, nx), dtype=torch.uint8, device="cuda")
        f[:, 0] = 1
        f[:, ny - 1] = 1
        return f
    if geom != "tunnel":
        return None
    s = nx / 768.0
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5 - nx / 4)[None, None, :]
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5 - ny / 2)[None, :, None]
    z = (torch.arange(nz, device="cuda", dtype=torch.float64) + 0.5 - nz / 2)[:, None, None]
    solid = ((x * x + y * y) <= (12 * s) ** 2) & (z >= 0)
    solid = solid | (((x * x + z * z) <= (6 * s) ** 2) & (y.abs() <= 50 * s))
    for side in (-35 * s, 35 * s):
        solid |= ((x * x + z * z) <= (40 * s) ** 2) & ((y - side).abs() <= 15 * s)
    r = np.random.RandomState(seed & 0x7FFFFFFF).rand(6, 6)
    for b in r[: 3 + int(r[0, 0] * 4)]:
        e, c = (5 + 15 * b[:3]) * s / 2, (2 * b[3:] - 1) * 60 * s
        solid |= ((x - c[0]).abs() <= e[0]) & ((y - c[1]).abs() <= e[1]) & ((z - c[2]).abs() <= e[2])
    return solid.to(torch.uint8)


def _network(seed):
    """Parameters of the 7-32-32-1 closure network (hidden layers scaled by fan-in, a small
    output layer, as after some training)."""
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    p = np.zeros(NPARAM, dtype=np.float32)
    p[:224] = r.normal(0, 1 / math.sqrt(7), 224)
    p[224:256] = r.normal(0, 0.1, 32)
    p[256:1280] = r.normal(0, 1 / math.sqrt(32), 1024)
    p[1280:1312] = r.normal(0, 0.1, 32)
    p[1312:] = r.normal(0, 0.1, 33)
    return p


def _lattice(case, seed, q, geom, closure, stream, prec, coll="trt"):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    tau, force = _fluid(case, geom)
    lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=tau, precision=prec, streaming=stream, closure=closure,
                      cs_smag=CS, faces=FACES[geom], u_inflow=(U_BULK, 0.0, 0.0), collision=coll)
    flags = _flags(nx, ny, nz, geom, seed)
    if flags is not None:
        lat.set_flags(flags)
    lat.set_force(force)
    if closure == "mlp":
        lbm.lbm_set_closure_f32(lat.h, _network(seed), *MLP_SCALE)
        lbm.lbm_set_closure_floor(lat.h, MLP_FLOOR)
    return lat


def _train_inputs(case, seed):
    g = _gen(seed)
    n = case["n"] * case["nbatch"]
    x = torch.randn((n, 7), generator=g, device="cuda").clamp_(-8, 8)
    smag = torch.rand(n, generator=g, device="cuda").mul_(3).sub_(7).exp_()  # 1e-3 .. 2e-2
    target = torch.rand(n, generator=g, device="cuda").mul_(2 * CS * CS).mul_(smag)
    return x, target, smag, smag * smag, torch.from_numpy(_network(seed)).cuda()


class State:
    def __init__(self, case, **kw):
        self.case = case
        self.__dict__.update(kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, target, smag, weight, p = _train_inputs(case, seed)
        z = torch.zeros(NPARAM, dtype=torch.float32, device="cuda")
        return State(case, samples=(x, target, smag, weight), p=p, g=z.clone(), m=z.clone(), v=z.clone(), t=0)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    new = lambda *s: torch.empty(s, dtype=torch.float32, device="cuda")  # noqa: E731
    if kind == "refined":
        tau, force = _fluid(case, "box")
        box = refine.RefinedSlab(nx, ny, nz, case["z0"], case["z1"], stencil=19, tau=tau, force=(force, 0.0, 0.0),
                                 closure="smag", cs_smag=CS, precision=case["prec"])
        uc, uf = _refined_velocity(case, seed)
        for lat, planes in zip(box.coarse, box.planes):
            lat.init_equilibrium(None, uc[:, torch.tensor(planes, device="cuda")].contiguous())
        box.fine.init_equilibrium(None, uf)
        lats = box.coarse + box.fines
        return State(case, box=box, lats=lats, out=[new(19, t.nz, t.ny, t.nx) for t in lats])
    if kind == "flow":
        lat = _lattice(case, seed, case["q"], case["geom"], case["closure"], case["stream"], case["prec"], case["coll"])
        lat.init_equilibrium(None, _velocity(nx, ny, nz, case["geom"], seed))
        if case["stats"]:
            lbm.lbm_stats_reset(lat.h)
        return State(case, lat=lat, rho=new(nz, ny, nx), u=new(3, nz, ny, nx))
    if kind == "samples":
        lat = _lattice(case, seed, 19, "channel", "smag", case["stream"], case["prec"])
        lat.init_equilibrium(None, _velocity(nx, ny, nz, "channel", seed))
        lat.step(case["steps"])
        s = (nz // 2, ny // 2, nx // 2)
        return State(case, lat=lat, tau_c=_coarse_tau(lat), x=new(*s, 7), scalars=[new(*s) for _ in range(3)],
                     rho=new(*s), u=new(3, *s))
    # restart: the checkpoint is a state some steps after the start (non-equilibrium parts in it)
    lat = _lattice(case, seed, case["q"], "channel", "smag", case["stream"], case["prec"])
    lbm.lbm_stats_reset(lat.h)
    return State(case, lat=lat, df=_checkpoint(case, seed), out=new(case["q"], nz, ny, nx), rho=new(nz, ny, nx),
                 u=new(3, nz, ny, nx))


def _coarse_tau(lat_or_case):
    tau = _fluid({"ny": lat_or_case.ny}, "channel")[0]
    return 0.5 + (tau - 0.5) / 2


def _refined_velocity(case, seed):
    """Velocities of both levels: a seeded smooth field plus noise; the fine one 2x finer."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    uc = _velocity(nx, ny, nz, "box", seed)
    uf = _velocity(nx, ny, nz, "box", seed + 1)[:, case["z0"]:case["z1"]]
    uf = uf.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3).contiguous()
    return uc, uf


def _checkpoint(case, seed):
    """Shifted populations: equilibrium of the initial velocity plus a non-equilibrium part."""
    nx, ny, nz, q = case["nx"], case["ny"], case["nz"], case["q"]
    u = _velocity(nx, ny, nz, "channel", seed)
    g = _gen(seed + 7)
    c, w = _stencil(q)
    df = torch.rand((q, nz, ny, nx), generator=g, device="cuda", dtype=torch.float32).sub_(0.5).mul_(2e-3)
    usq = (u * u).sum(0)
    for i in range(q):
        cu = torch.zeros_like(usq)
        for a in range(3):
            if c[i][a]:
                cu.add_(u[a], alpha=float(c[i][a]))
        df[i].add_(3 * cu + 4.5 * cu * cu - 1.5 * usq).mul_(float(w[i]))
    return df


# ---- one pass ---------------------------------------------------------------------------------

def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "flow":
        h = s.lat.h
        if case["stats"]:
            lbm.lbm_step_stats(h, case["steps"], case["stats"])
        else:
            lbm.lbm_step(h, case["steps"])
        lbm.lbm_moments(h, s.rho, s.u)
        if case["stats"]:
            return {"rho": s.rho, "u": s.u, "stats": lbm.lbm_stats_get(h, case["ny"])[0]}
        return {"rho": s.rho, "u": s.u}
    if kind == "refined":
        s.box.step(case["steps"])
        for lat, df in zip(s.lats, s.out):
            lbm.lbm_get_post_collision(lat.h, df)
        return {"coarse": s.out[:-1], "fine": s.out[-1]}
    if kind == "train":
        s.t += 1
        b = (s.t - 1) % case["nbatch"]
        # the loss is a mean over residuals computed in float32
        loss = np.float32(lbm.lbm_closure_loss_grad(s.p, *s.samples, case["n"], b, case["nbatch"], CS, s.g))
        lbm.lbm_adam_step(s.p, s.g, s.m, s.v, 2e-3, s.t)
        return {"loss": loss, "grad": s.g, "params": s.p, "m": s.m, "v": s.v}
    if kind == "samples":
        lbm.lbm_closure_samples(s.lat.h, s.tau_c, CS, MLP_SCALE, s.x, *s.scalars)
        lbm.lbm_filter2(s.lat.h, s.rho, s.u)
        return {"x": s.x, "target": s.scalars[0], "smag": s.scalars[1], "weight": s.scalars[2], "rho": s.rho, "u": s.u}
    h = s.lat.h
    lbm.lbm_set_populations(h, s.df)
    lbm.lbm_step(h, 2)
    sums = lbm.lbm_reduce(h)
    lbm.lbm_stats_reset(h)
    lbm.lbm_stats_sample(h)
    lbm.lbm_moments(h, s.rho, s.u)
    lbm.lbm_get_populations(h, s.out)
    return {"sums": sums, "stats": lbm.lbm_stats_get(h, case["ny"])[0], "rho": s.rho, "u": s.u, "df": s.out}


# ---- what a pass cannot do without --------------------------------------------------------------

def work(case):
    """Bytes and operations.  A step reads and writes every population once and reads a class
    byte per cell (the roofline of the paper's Sec. 5.2, a step taken by itself)."""
    kind = case["kind"]
    if kind == "train":
        return {"bytes": case["n"] * 40.0 + 8 * 4 * NPARAM, "flops": case["n"] * 3.0 * 2 * 1280}
    n = float(case["nx"] * case["ny"] * case["nz"])
    size = 4.0 if case.get("prec") == "f32" else 2.0
    q = case.get("q", 19)
    ops = {19: 300.0, 27: 430.0}[q]
    if kind == "flow":
        ops += 2560.0 if case["closure"] == "mlp" else 0.0
        ops += 400.0 if case["coll"] == "mrt" else 0.0
        return {"bytes": n * (case["steps"] * (2 * q * size + 1) + q * size + 17), "flops": n * case["steps"] * ops}
    if kind == "refined":
        nf = 8.0 * case["nx"] * case["ny"] * (case["z1"] - case["z0"])
        nc = n - nf / 8
        upd = case["steps"] * (nc + 2 * nf)
        return {"bytes": upd * (2 * q * size + 1) + (nc + nf) * q * (size + 4), "flops": upd * ops}
    if kind == "samples":
        return {"bytes": n * (q * size + 1) + n / 8 * 4 * (7 + 3 + 4), "flops": n * 120.0}
    # restart: import, two steps, then sums, statistics, fields and populations of the state
    return {"bytes": n * (q * (4 + size) + 2 * (2 * q * size + 1) + q * size + 16 + 4 * q), "flops": n * (2 * ops + 150)}


# ---- the method in float64 ----------------------------------------------------------------------

_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
      (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
      (0, -1, 1), (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]


def _stencil(q):
    table = {19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[q]
    c = _C[:q]
    return c, [table[sum(v * v for v in d)] for d in c]


def _opp(i):
    return 0 if i == 0 else (i + 1 if i % 2 else i - 1)


class Exact:
    """A lattice in float64: f holds post-streaming (pre-collision) populations."""

    def __init__(self, nx, ny, nz, q, tau, force, faces, closure="none", coll="trt", flags=None, params=None):
        self.shape, self.q, self.tau, self.faces = (nz, ny, nx), q, tau, faces
        self.closure, self.coll, self.flags = closure, coll, flags
        self.c, self.w = _stencil(q)
        dev = {"device": "cuda", "dtype": torch.float64}
        self.cm, self.wv = torch.tensor(self.c, **dev), torch.tensor(self.w, **dev)
        self.F = torch.tensor([force, 0.0, 0.0], **dev)
        self.params = None if params is None else torch.from_numpy(params).cuda().to(torch.bfloat16).double()
        if coll == "mrt":
            self.M, self.rate_of = _mrt(self.c)

    def equilibrium(self, u):
        """f^eq of density 1 and velocity u, as the starting state."""
        usq = (u.double() ** 2).sum(0)
        self.f = torch.empty((self.q,) + self.shape, device="cuda", dtype=torch.float64)
        for i, (d, w) in enumerate(zip(self.c, self.w)):
            cu = sum(float(d[a]) * u[a].double() for a in range(3))
            self.f[i] = w * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)

    def macro(self, f):
        rho = f.sum(0)
        j = self.cm.t() @ f + 0.5 * self.F[:, None]
        return rho, j / rho

    def stress(self, f, rho, u):
        """Non-equilibrium second moments xx, yy, zz, xy, xz, yz."""
        cc = torch.stack([self.cm[:, a] * self.cm[:, b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
        pi = cc @ f
        for k, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            pi[k] -= rho * u[a] * u[b] + (rho / 3 if a == b else 0)
        return pi

    def collide_cells(self, f):
        """Post-collision populations of a batch of cells f[q, n]."""
        rho, u = self.macro(f)
        usq, cu = (u * u).sum(0), self.cm @ u
        feq = self.wv[:, None] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)
        cF, uF = (self.cm @ self.F)[:, None], (u * self.F[:, None]).sum(0)
        guo = self.wv[:, None] * (3 * (cF - uF) + 9 * cu * cF)
        tau = torch.full_like(rho, self.tau)
        pi = self.stress(f, rho, u) if self.closure != "none" or self.coll == "reg" else None
        if self.closure != "none":
            qn = pi[0] ** 2 + pi[1] ** 2 + pi[2] ** 2 + 2 * (pi[3] ** 2 + pi[4] ** 2 + pi[5] ** 2)
            cs2 = CS * CS if self.closure == "smag" else self.learned(pi, rho)
            tau = 0.5 * (self.tau + torch.sqrt(self.tau ** 2 + 18 * math.sqrt(2) * cs2 * torch.sqrt(qn) / rho))
        om = 1 / tau
        if self.coll == "mrt":
            s = [1.0 if g == -1 else om if g == -2 else RATES[g] for g in self.rate_of]
            m, mf = self.M @ (f - feq), self.M @ guo
            dm = torch.stack([-r * m[k] + (1 - 0.5 * r) * mf[k] for k, r in enumerate(s)])
            return f + self.M.t() @ (dm / (self.M ** 2).sum(1)[:, None])
        if self.coll == "reg":
            g2 = f - feq + 0.5 * guo
            out = feq + 0.5 * guo
            H = torch.stack([self.cm[:, a] * self.cm[:, b] - (1 / 3 if a == b else 0)
                             for a in range(3) for b in range(3)])
            return out + (1 - om) * 4.5 * self.wv[:, None] * (H.t() @ (H @ g2))
        opp = torch.tensor([_opp(i) for i in range(self.q)], device=f.device)
        omm = 1 / (3.0 / 16.0 / (tau - 0.5) + 0.5)
        neq = f - feq
        even, odd = 0.5 * (neq + neq[opp]), 0.5 * (neq - neq[opp])
        ge, go = 0.5 * (guo + guo[opp]), 0.5 * (guo - guo[opp])
        return f - om * even - omm * odd + (1 - 0.5 * om) * ge + (1 - 0.5 * omm) * go

    def learned(self, pi, rho):
        x = torch.cat([MLP_SCALE[0] * pi, MLP_SCALE[1] * (rho - 1)[None]]).clamp(-8, 8)
        y = _net(self.params, x.t())
        return (torch.nn.functional.softplus(y) * CS * CS / math.log(2)).clamp_min(MLP_FLOOR ** 2)

    def collide(self):
        """In place, some planes at a time."""
        nz, ny, nx = self.shape
        step = max(1, (1 << 21) // (ny * nx))
        for z in range(0, nz, step):
            b = self.f[:, z:z + step]
            b.copy_(self.collide_cells(b.reshape(self.q, -1)).reshape(b.shape))

    def segments(self, a, ca):
        """(destination, source, face) ranges of axis a (0 x, 1 y, 2 z) for velocity component ca."""
        n = self.shape[2 - a]
        if ca == 0:
            return [(slice(0, n), slice(0, n), None)]
        if ca > 0:
            inner, edge, far = (slice(1, n), slice(0, n - 1), None), slice(0, 1), slice(n - 1, n)
        else:
            inner, edge, far = (slice(0, n - 1), slice(1, n), None), slice(n - 1, n), slice(0, 1)
        face = self.faces[2 * a + (0 if ca > 0 else 1)]
        return [inner, (edge, far if face == "periodic" else edge, face)]

    def stream(self):
        fs, fl = self.f, self.flags
        out = torch.empty_like(fs)
        for i, d in enumerate(self.c):
            o, term = _opp(i), 6 * self.w[i] * U_BULK * d[0]
            for zd, zs, zt in self.segments(2, d[2]):
                for yd, ys, yt in self.segments(1, d[1]):
                    for xd, xs, xt in self.segments(0, d[0]):
                        kinds = (xt, yt, zt)
                        if "outflow" in kinds and "wall" not in kinds:
                            continue
                        if "wall" in kinds or "inflow" in kinds:
                            out[i][zd, yd, xd] = fs[o][zd, yd, xd] + (0 if "wall" in kinds else term)
                            continue
                        e = tuple(-v if k == "freeslip" else v for v, k in zip(d, kinds))
                        v = fs[self.c.index(e)][zs, ys, xs]
                        if fl is not None:
                            v = torch.where(fl[zs, ys, xs] != 0, fs[o][zd, yd, xd], v)
                        out[i][zd, yd, xd] = v
            if self.faces[1] == "outflow" and d[0] < 0:
                v = out[i][:, :, -2]
                out[i][:, :, -1] = v if fl is None else torch.where(fl[:, :, -2] != 0, fs[o][:, :, -1], v)
        self.f = out

    def step(self, n=1):
        for _ in range(n):
            self.collide()
            self.stream()

    def fields(self):
        rho, u = torch.empty(self.shape, device="cuda", dtype=torch.float64), None
        u = torch.empty((3,) + self.shape, device="cuda", dtype=torch.float64)
        for z in range(self.shape[0]):
            r, v = self.macro(self.f[:, z].reshape(self.q, -1))
            rho[z], u[:, z] = r.reshape(rho[z].shape), v.reshape(u[:, z].shape)
        if self.flags is not None:
            rho[self.flags != 0] = 0
            u[:, self.flags != 0] = 0
        return rho, u

    def plane_sums(self, rho, u):
        """count, u, u_a^2, u_x u_y, u_x u_z, u_y u_z summed over each y plane."""
        prod = [u[0] * u[0], u[1] * u[1], u[2] * u[2], u[0] * u[1], u[0] * u[2], u[1] * u[2]]
        cols = [torch.ones_like(rho), u[0], u[1], u[2]] + prod
        return torch.stack([v.sum(dim=(0, 2)) for v in cols], 1)


def _mrt(c):
    rows, rate = [], [-1, 0, 1, -1, 2, -1, 2, -1, 2, -2, 3, -2, 3, -2, -2, -2, 4, 4, 4]
    for x, y, z in c:
        n = x * x + y * y + z * z
        rows.append([1, 19 * n - 30, (21 * n * n - 53 * n + 24) / 2, x, (5 * n - 9) * x, y, (5 * n - 9) * y, z,
                     (5 * n - 9) * z, 3 * x * x - n, (3 * n - 5) * (3 * x * x - n), y * y - z * z,
                     (3 * n - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x,
                     (z * z - x * x) * y, (x * x - y * y) * z])
    return torch.tensor(rows, device="cuda", dtype=torch.float64).t().contiguous(), rate


def _net(p, x):
    gelu = torch.nn.functional.gelu
    h = gelu(x @ p[:224].reshape(32, 7).t() + p[224:256])
    h = gelu(h @ p[256:1280].reshape(32, 32).t() + p[1280:1312])
    return h @ p[1312:1344] + p[1344]


def _exact_lattice(case, seed, q, geom, closure, coll="trt"):
    tau, force = _fluid(case, geom)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    params = _network(seed) if closure == "mlp" else None
    return Exact(nx, ny, nz, q, tau, force, FACES[geom], closure, coll, _flags(nx, ny, nz, geom, seed), params)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if kind == "refined":
        return _exact_refined(case, seed)
    if kind == "flow":
        e = _exact_lattice(case, seed, case["q"], case["geom"], case["closure"], case["coll"])
        e.equilibrium(_velocity(nx, ny, nz, case["geom"], seed))
        stats = 0
        for k in range(case["steps"]):
            if case["stats"] and k % case["stats"] == 0:
                stats = stats + e.plane_sums(*e.fields())
            e.step()
        rho, u = e.fields()
        return {"rho": rho, "u": u, "stats": stats} if case["stats"] else {"rho": rho, "u": u}
    if kind == "samples":
        e = _exact_lattice(case, seed, 19, "channel", "smag")
        e.equilibrium(_velocity(nx, ny, nz, "channel", seed))
        e.step(case["steps"])
        return _exact_samples(e, case)
    e = _exact_lattice(case, seed, case["q"], "channel", "smag")
    e.f = _checkpoint(case, seed).double()
    if case["prec"] != "f32":
        e.f = e.f.half().double()
    e.f += e.wv[:, None, None, None]
    e.step(2)
    rho, u = e.fields()
    mom = torch.stack([rho.sum()] + [(rho * u[a]).sum() for a in range(3)])
    return {"sums": mom, "stats": e.plane_sums(rho, u), "rho": rho, "u": u, "df": e.f - e.wv[:, None, None, None]}


def _exact_train(case, seed):
    x, target, smag, weight, p = _train_inputs(case, seed)
    k = case["nbatch"]
    x, target, smag, weight = (t[::k].double() for t in (x, target, smag, weight))
    p = p.double().requires_grad_(True)
    loss, step, total = 0.0, 1 << 18, float(weight.sum())
    for a in range(0, x.shape[0], step):
        b = slice(a, a + step)
        nu = torch.nn.functional.softplus(_net(p, x[b])) * CS * CS / math.log(2) * smag[b]
        part = (weight[b] * (nu - target[b]) ** 2).sum() / total
        part.backward()
        loss += float(part.detach())
    g = p.grad
    m, v = 0.1 * g, 0.001 * g * g
    new = p.detach() - 2e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return {"loss": loss, "grad": g, "params": new, "m": m, "v": v}


def _exact_samples(e, case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    out = {k: [] for k in ("x", "target", "smag", "weight", "rho", "u")}
    tau_c = _coarse_tau(type("L", (), {"ny": ny}))
    for z in range(0, nz, 2):
        f = e.f[:, z:z + 2].reshape(19, -1)
        rho, u = e.macro(f)
        pi = e.stress(f, rho, u)
        qn = pi[0] ** 2 + pi[1] ** 2 + pi[2] ** 2 + 2 * (pi[3] ** 2 + pi[4] ** 2 + pi[5] ** 2)
        tau = 0.5 * (e.tau + torch.sqrt(e.tau ** 2 + 18 * math.sqrt(2) * CS * CS * torch.sqrt(qn) / rho))
        S, nut = -3 / (2 * rho * tau) * pi, (tau - e.tau) / 3
        mean = lambda v: v.reshape(-1, 2, ny // 2, 2, nx // 2, 2).mean(dim=(1, 3, 5))  # noqa: E731
        rb = mean(rho)
        ub = mean(rho * u) / rb
        uu = mean(torch.stack([rho * u[a] * u[b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])) / rb
        ubb = torch.stack([ub[a] * ub[b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
        sg = uu - ubb - 2 * mean(nut * S)
        Sc = 2 * mean(S)
        sg[:3] = sg[:3] - sg[:3].mean(0)
        mult = torch.tensor([1, 1, 1, 2, 2, 2], device="cuda", dtype=torch.float64)[:, None, None]
        num, den = (mult * sg * Sc).sum(0), (mult * Sc * Sc).sum(0)
        smag = torch.sqrt(2 * den)
        nu = torch.where(smag > 1e-10, -num / (2 * den), torch.zeros_like(num)).clamp_min(0)
        tc = tau_c + 3 * CS * CS * smag
        x = torch.cat([MLP_SCALE[0] * (-(2 * rb / 3) * tc * Sc), MLP_SCALE[1] * (rb - 1)]).clamp(-8, 8)
        vals = (x.permute(1, 2, 0), nu, smag, smag ** 2, rb[0], ub)
        for k, v in zip(("x", "target", "smag", "weight", "rho", "u"), vals):
            out[k].append(v)
    return {k: torch.stack(v, 1 if k == "u" else 0) for k, v in out.items()}


def _exact_refined(case, seed):
    """Volumetric 2:1 transfer on post-collision states, one coarse piece (planes z1 .. nz-1, 0
    .. z0-1) and one fine slab, each with a ghost plane on both sides."""
    nx, ny, nz, z0, z1 = (case[k] for k in ("nx", "ny", "nz", "z0", "z1"))
    tau, force = _fluid(case, "box")
    planes = list(range(z1, nz)) + list(range(z0))
    uc, uf = _refined_velocity(case, seed)
    C = Exact(nx, ny, len(planes), 19, tau, force, PERIODIC, "smag")
    F = Exact(2 * nx, 2 * ny, 2 * (z1 - z0), 19, 0.5 + 2 * (tau - 0.5), force / 2, PERIODIC, "smag")
    C.equilibrium(uc[:, torch.tensor(planes, device="cuda")])
    F.equilibrium(uf)
    C.collide()
    F.collide()

    def pull(e, lo, hi):
        """Streams with the ghost planes lo (below) and hi (above), [q, ny, nx] each, then collides."""
        out = torch.empty_like(e.f)
        for i, (cx, cy, cz) in enumerate(e.c):
            g = torch.roll(e.f[i], (cy, cx), (1, 2))
            if cz == 0:
                out[i] = g
            elif cz > 0:
                out[i][1:], out[i][0] = g[:-1], torch.roll(lo[i], (cy, cx), (0, 1))
            else:
                out[i][:-1], out[i][-1] = g[1:], torch.roll(hi[i], (cy, cx), (0, 1))
        e.f = out
        e.collide()

    def ghost(plane, s):
        """Fine ghost plane in substep s from the coarse interface plane [q, ny, nx]."""
        up = plane.repeat_interleave(2, 1).repeat_interleave(2, 2)
        return torch.stack([torch.roll(up[i], (s * c[1], s * c[0]), (0, 1)) for i, c in enumerate(F.c)])

    def merge(new, old):
        """Coarse ghost plane: mean of the 8 fine values that reach each coarse cell's volume."""
        out = []
        for i, (cx, cy, _) in enumerate(F.c):
            v = torch.roll(new[i], (cy, cx), (0, 1)) + torch.roll(old[i], (2 * cy, 2 * cx), (0, 1))
            out.append(torch.roll(v.reshape(ny, 2, nx, 2).mean(dim=(1, 3)) / 2, (-cy, -cx), (0, 1)))
        return torch.stack(out)

    for _ in range(case["steps"]):
        below, above = C.f[:, -1].clone(), C.f[:, 0].clone()  # coarse planes under and over the slab
        old = F.f[:, [0, -1]].clone()
        pull(F, ghost(below, 0), ghost(above, 0))
        g_hi, g_lo = merge(F.f[:, 0], old[:, 0]), merge(F.f[:, -1], old[:, 1])
        pull(F, ghost(below, 1), ghost(above, 1))
        pull(C, g_lo, g_hi)
    w = C.wv[:, None, None, None]
    return {"coarse": [C.f - w], "fine": F.f - w}
