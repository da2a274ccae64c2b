"""Cases of this framework's use, for timing: what a user's program has in hand
before a call, one pass through the public entry points, and the same results
in 64 bits from plain torch and numpy.

A case is a dict of plain values.  "kind" says what the program does:
  steps    lbm_step on a context whose distributions live in the caller's own
           CUDA tensor (lbm_create_with_buffer); the tensor comes back
  droplet  a whole small study: lbm_init_droplets, lbm_step, then the contact
           angle, the mass, the largest speed and the density
  host     a density field from pinned host memory through lbm_set_rho,
           lbm_step, and the density back to pinned memory with lbm_get_rho
  measure  the contact angle of every droplet of a large domain, the mass and
           the largest speed
  fields   distributions in through lbm_set_f, every field the library derives
           from them out (velocity, density, psi, U, force, Eq. 17 tensor, f)
  batch    lbm_batch_step over many droplet instances, then their angles and
           densities
  adjoint  the gradient of a weighted final density in the bottom wall's
           angles and T, through final_density(...).backward()
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1501_05430_gb300 import adjoint as ADJ
from paper_1501_05430_gb300 import lbm as L

# Eq. 11 parameters of the paper's Table 1 by density ratio: rho1, rho2,
# theta_v, theta_m, theta_l
TABLE1 = {10: (1.122, 9.54, 0.25, -0.02, 0.3), 100: (1.486, 94.65, 0.1633, -0.02, 0.33333),
          1000: (1.325, 971.1017, 0.2, -0.01, 0.33333)}
CS_A, CS_B, CS_R = 0.25, 4.0, 1.0  # Carnahan-Starling constants of the droplet workloads
# the relaxation rates that go with the low Carnahan-Starling temperatures
MRT = dict(s_e=0.8, s_eps=0.8, s_j=1.0, s_q=1.1)
MIXED = ((128, 64), (256, 128), (384, 192), (512, 256))  # grid sizes of the batched sweep


def listed():
    cs = dict(eos="cs", wetting="geometric", walls=True, n_iter=4)
    pw = dict(eos="pw", tau=1.0, rates="bgk", wetting="geometric", walls=True, n_iter=4)
    return [
        # the small domains of angle inversion and parameter studies: launches and latency count
        dict(cs, name="steps_256x128", kind="steps", nx=256, ny=128, precision=32, t=0.7, tau=1.0, rates="bgk",
             drops=1, steps=200),
        # the accuracy workload as the README's quick start runs it, from droplets to the measured angle
        dict(cs, name="droplet_400x200", kind="droplet", nx=400, ny=200, precision=32, t=0.6, tau=0.8, rates="mrt",
             drops=1, steps=400, check=100, stream=False),
        # the throughput workload: density ratio 724, general relaxation rates, 12 droplets a wall
        dict(cs, name="steps_4096x2048", kind="steps", nx=4096, ny=2048, precision=32, t=0.5, tau=0.6, rates="mrt",
             drops=12, steps=32),
        # the paper's own model (Table 1 at ratio 1000, all rates 1) on a domain just past the L2
        dict(pw, name="steps_table1_2048x1026", kind="steps", nx=2048, ny=1026, precision=32, ratio=1000, drops=6,
             steps=64),
        # a width that is no multiple of four, with the compared wetting rule (Martys-Chen, ratio 10)
        dict(pw, name="steps_odd_1001x501", kind="steps", nx=1001, ny=501, precision=32, ratio=10,
             wetting="martys_chen", drops=3, steps=64),
        # the double-precision workload that is compared with the oracle bit for bit
        dict(cs, name="steps_f64_100x60", kind="steps", nx=100, ny=60, precision=64, t=0.8, tau=1.0, rates="bgk",
             drops=1, steps=100),
        # the batched sweep: 256 instances of four sizes and four temperatures
        dict(name="batch_256", kind="batch", eos="cs", sizes="mixed", count=256, steps=256, tuned=True),
        # one of the paper's figures: six angles at ratio 100, 300 x 100, in one batch of the default shape
        dict(name="batch_figure_6x300x100", kind="batch", eos="pw", ratio=100, sizes="300x100", count=6, steps=200,
             tuned=False),
        # the wall-angle inversion's gradient (256 wall angles and T)
        dict(cs, name="adjoint_256x128", kind="adjoint", nx=256, ny=128, precision=32, t=0.7, tau=1.0, rates="bgk",
             drops=1, steps=400, every=100, stream=False),
        # end to end from and to host memory on the throughput workload
        dict(cs, name="host_4096x2048", kind="host", nx=4096, ny=2048, precision=32, t=0.5, tau=0.6, rates="mrt",
             drops=12, steps=20),
        # what is measured at the end of a throughput run
        dict(cs, name="measure_4096x2048", kind="measure", nx=4096, ny=2048, precision=32, t=0.5, tau=0.6,
             rates="mrt", drops=12, steps=4),
        # every field of a stored state, as a plotting or analysis program reads them
        dict(cs, name="fields_800x400", kind="fields", nx=800, ny=400, precision=32, t=0.6, tau=0.8, rates="mrt",
             drops=2, steps=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps"] * 6 + ["droplet", "droplet", "host", "measure", "fields", "batch", "batch",
                                       "adjoint", "adjoint"])
    c = dict(kind=kind, eos=rng.choice(["cs", "cs", "pw"]))
    if c["eos"] == "cs":
        c.update(t=rng.choice([0.5, 0.6, 0.7, 0.8]))
    else:
        c.update(ratio=rng.choice([10, 100, 1000]))
    if kind == "batch":
        c.update(sizes=rng.choice(["mixed", "%dx%d" % (4 * _log(rng, 8, 128), _log(rng, 24, 200))]),
                 count=_log(rng, 2, 200), steps=rng.randrange(20, 100), tuned=rng.random() < 0.5)
        return c
    big = kind in ("steps", "host", "measure")
    nx = _log(rng, 64, 4096 if big else 800)
    ny = max(32, min(2048 if big else 500, int(nx * rng.uniform(0.25, 1.0))))
    if rng.random() < 0.7:
        nx -= nx % 4  # widths are mostly multiples of four, the others any
    if c["eos"] == "cs":
        c.update(tau=round(rng.uniform(0.6, 1.0), 3), rates="mrt" if c["t"] < 0.7 else rng.choice(["mrt", "bgk"]))
    else:
        c.update(tau=1.0, rates="bgk")
    mc = c["eos"] == "pw" and c["ratio"] == 10 and rng.random() < 0.5
    c.update(nx=nx, ny=ny, wetting="martys_chen" if mc else "geometric", n_iter=rng.choice([0, 4, 4, 4]),
             walls=kind != "steps" or rng.random() < 0.85, precision=32,
             drops=max(1, min(12, nx // 300)), steps=20)
    if kind == "steps":
        if nx <= 800 and rng.random() < 0.25:
            c.update(precision=64)
        c.update(steps=2 * max(4, min(100, 4_000_000 // (nx * ny))))
    elif kind == "droplet":
        c.update(steps=rng.randrange(40, 400), stream=rng.random() < 0.5)
    elif kind == "adjoint":
        nx = min(nx, 400)
        c.update({"t": max(c["t"], 0.7)} if c["eos"] == "cs" else {"ratio": 10})
        c.update(nx=nx, ny=min(ny, 200), steps=rng.randrange(20, 200), every=rng.randrange(10, 100), n_iter=4,
                 wetting="geometric", stream=rng.random() < 0.5)
    elif kind in ("measure", "fields"):
        c.update(steps=4 if kind == "measure" else 0, precision=rng.choice([32, 32, 64]) if nx <= 800 else 32)
    return c


# ---- the physics of a case: numbers from the seed alone --------------------------

def _bisect(g, a, b):
    neg = g(a) < 0
    for _ in range(200):
        m = 0.5 * (a + b)
        if (g(m) < 0) == neg:
            a = m
        else:
            b = m
    return 0.5 * (a + b)


def _cs_critical():
    e = 0.13
    for _ in range(60):  # packing fraction at which dp/drho and d2p/drho2 vanish
        e -= (((((e - 5) * e + 4) * e + 20) * e + 5) * e - 1) / ((((5 * e - 20) * e + 12) * e + 40) * e + 5)
    return 8 * CS_A / (CS_B * CS_R * (8 + 20 * e - 4 * e * e) / (1 - e) ** 5), 4 * e / CS_B


def _coexistence(p):
    """(rho_v, rho_l, rho_max): equal pressure and chemical potential, and the
    density above rho_l at which the pressure is rho/3."""
    if p["eos"] == "cs":
        T, rc, top = p["T"], _cs_critical()[1], 4.0 / CS_B * (1 - 1e-13)

        def pr(r):
            e = CS_B * r / 4
            return r * CS_R * T * (1 + e + e * e - e ** 3) / (1 - e) ** 3 - CS_A * r * r

        def dp(r):
            e = CS_B * r / 4
            return CS_R * T * (1 + 4 * e + 4 * e * e - 4 * e ** 3 + e ** 4) / (1 - e) ** 4 - 2 * CS_A * r

        def mu(r):
            e = CS_B * r / 4
            return CS_R * T * (math.log(e) + e * (8 - 9 * e + 3 * e * e) / (1 - e) ** 3) - 2 * CS_A * r

        sv, sl = _bisect(dp, 1e-14 * rc, rc), _bisect(dp, rc, top)
        vap = lambda ps: _bisect(lambda r: pr(r) - ps, 1e-300, sv)  # noqa: E731
        liq = lambda ps: _bisect(lambda r: pr(r) - ps, sl, top)  # noqa: E731
        ps = _bisect(lambda q: mu(liq(q)) - mu(vap(q)), max(pr(sl), 0.0) + 1e-300, pr(sv) * (1 - 1e-15))
        rl = liq(ps)
        return vap(ps), rl, _bisect(lambda r: pr(r) - r / 3, rl, top)
    r1, r2, tv, tm, tl = p["pw"]
    liq = lambda v: r2 - ((r1 - v) * tv + (r2 - r1) * tm) / tl  # noqa: E731
    v = _bisect(lambda v: tv * math.log(r1 / v) + tm * math.log(r2 / r1) + tl * math.log(liq(v) / r2), r1 * 1e-12,
                r1 * (1 - 1e-14))
    rl, slope = liq(v), tl - 1.0 / 3.0
    root = r2 - (r1 * tv + (r2 - r1) * tm - r2 / 3) / slope if slope > 0 else math.inf
    return v, rl, root if root > rl else math.inf


def _problem(c, rng, nx=None, ny=None, t=None):
    """Model numbers, wall angles and droplets of one domain."""
    nx, ny = nx or c["nx"], ny or c["ny"]
    p = dict(nx=nx, ny=ny, eos=c["eos"], kappa=0.5, wetting=c.get("wetting", "geometric"), n_iter=c.get("n_iter", 4),
             walls=c.get("walls", True), tau=c.get("tau", 1.0), G_w=-1.43 if c.get("wetting") == "martys_chen" else 0.0)
    if c["eos"] == "cs":
        p.update(A=-0.9, t=t or c["t"], T=(t or c["t"]) * _cs_critical()[0])
    else:
        p.update(A=-0.6, T=0.0, pw=TABLE1[c["ratio"]])
    inv = 1.0 / p["tau"]
    r = dict(s_e=inv, s_eps=inv, s_j=inv, s_q=inv)
    p["rates"] = dict(r, **MRT) if c.get("rates") == "mrt" else r
    p["width"] = 10.0 if c["eos"] == "pw" or p["t"] < 0.6 else 3.0
    p["rho_v"], p["rho_l"], p["rho_max"] = _coexistence(p)
    # droplets side by side on each wall, one angle for each one's stretch of the wall
    n = c.get("drops", 1)
    walls = (0, 1) if n > 1 else (0,)
    p["theta"] = np.full((2, nx), np.pi / 2)
    p["drops"], p["regions"] = [], []
    cuts = [round(k * nx / n) for k in range(n + 1)]
    for w in walls:
        for a, b in zip(cuts[:-1], cuts[1:]):
            most = min(120.0, 0.36 * (b - a), 0.4 * ny)
            p["drops"].append((0.5 * (a + b) + rng.uniform(-2, 2), most * rng.uniform(0.7, 1.0), w))
            p["theta"][w, a:b] = math.radians(rng.uniform(60.0, 120.0))
            p["regions"].append((w, a, b))
    if c["kind"] == "adjoint":  # an angle of its own for every wall node
        p["theta"][0] = np.radians(rng.uniform(45.0, 135.0, nx))
    return p


def _problems(c, seed):
    rng = np.random.default_rng(seed)
    if c["kind"] != "batch":
        return [_problem(c, rng)]
    out, sizes = [], np.random.default_rng(42).integers(0, 4, c["count"])  # the same mix for every seed
    for i in range(c["count"]):
        nx, ny = MIXED[sizes[i]] if c["sizes"] == "mixed" else map(int, c["sizes"].split("x"))
        if c["eos"] == "cs":
            t = (0.5, 0.6, 0.7, 0.8)[rng.integers(0, 4)]
            d = dict(c, tau=float(rng.uniform(0.6, 1.0)), rates="mrt" if t < 0.7 else "bgk")
        else:
            t, d = None, dict(c, tau=1.0, rates="bgk")
        out.append(_problem(d, rng, nx, ny, t))
    return out


# ---- a user's program ------------------------------------------------------------

def _lib(p, precision, every=0):
    """Arguments of a context: (nx, ny, eos, T, tau), theta, walls, params."""
    eos = L.carnahan_starling(CS_A, CS_B, CS_R) if p["eos"] == "cs" else L.piecewise(*p["pw"][2:], *p["pw"][:2])
    theta = np.full((p["ny"], p["nx"]), np.pi / 2)
    theta[0], theta[-1] = p["theta"]
    params = L.lbm_params_default(
        A=p["A"], kappa=p["kappa"], G_w=p["G_w"], n_iter=p["n_iter"], precision=precision, check_every=every,
        wetting=L.LBM_WET_MARTYS_CHEN if p["wetting"] == "martys_chen" else L.LBM_WET_GEOMETRIC, **p["rates"])
    return (p["nx"], p["ny"], eos, p["T"], p["tau"]), theta, p["walls"], params


def _drop_args(p):
    x, r, w = zip(*p["drops"])
    return np.array(x), np.array(r), np.array(w), p["width"]


class _Own:
    """A context whose distributions live in this program's CUDA tensor."""

    def __init__(self, p, precision, stream):
        args, theta, walls, params = _lib(p, precision)
        dtype = torch.float32 if precision == 32 else torch.float64
        self.stream = stream
        self.buf = torch.empty((2, 9, p["ny"], p["nx"]), dtype=dtype, device="cuda")
        self.ctx = L.lbm_create_with_buffer(*args, self.buf.data_ptr(), self.buf.numel() * self.buf.element_size(),
                                            theta, walls, params, stream)

    def __del__(self):
        L.lbm_destroy(self.ctx)


_streams = []


def _stream(c):
    """The one stream on which a program queues its solvers' work, or None: the default stream."""
    if not c.get("stream", True):
        return None
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    c, ps = case, _problems(case, seed)
    p, s = ps[0], dict(c=case, p=ps[0])
    kind = c["kind"]
    if kind == "adjoint":
        args, theta, _, params = _lib(p, c["precision"])
        s.update(stream=_stream(c), f0=_f0(p), args=args, params=params,
                 theta=torch.tensor(p["theta"][0], device="cuda"), T=torch.tensor(p["T"], dtype=torch.float64),
                 weights=_weights(c, seed))
        return s
    stream = _stream(c)
    if kind == "steps":
        s["own"] = _Own(p, c["precision"], stream)
        L.lbm_init_droplets(s["own"].ctx, *_drop_args(p))
        return s
    if kind == "batch":
        descs = []
        for q in ps:
            args, theta, _, params = _lib(q, 32)
            descs.append(dict(nx=args[0], ny=args[1], eos=args[2], T=args[3], tau=args[4], theta=theta, params=params))
        cfg = None
        if c["tuned"]:  # a shape the autotuner picks, with graphs
            cfg = L.lbm_batch_config_default(threads=256, stages=3, band_rows=[64] * 4, steps_per_launch=32,
                                             graph_launches=2)
        s["batch"] = L.LbmBatch(descs, cfg, stream=stream)
        for q, inst in zip(ps, s["batch"].instances):
            inst.init_droplets(*_drop_args(q))
        s["rho"] = torch.empty(sum(q["nx"] * q["ny"] for q in ps), dtype=torch.float64, pin_memory=True)
        return s
    args, theta, walls, params = _lib(p, c["precision"], every=c.get("check", 0))
    sim = s["sim"] = L.Lbm(*args, theta=theta, walls=walls, params=params, stream=stream)
    if kind == "host":
        s["rho"] = torch.empty((p["ny"], p["nx"]), dtype=torch.float64, pin_memory=True)
        s["rho"].copy_(_rho0([p])[0])
        s["out"] = torch.empty((p["ny"], p["nx"]), dtype=torch.float64, pin_memory=True)
    elif kind == "measure":
        sim.init_droplets(*_drop_args(p))
        sim.step(c["steps"])
    elif kind == "fields":
        f = _f0(p)
        s["f"] = f * (1.0 + 0.02 * np.random.default_rng(seed + 1).uniform(-1.0, 1.0, f.shape))
    return s


def _angle(sim, wall, a, b):
    try:
        return list(sim.contact_angle(wall, a, b))
    except L.LbmError:  # no contact line there
        return [math.nan] * 3


def run(s):
    c, p, kind = s["c"], s["p"], s["c"]["kind"]
    if kind == "steps":
        # an even number of steps: the state is in the array it started in
        L.lbm_step(s["own"].ctx, c["steps"])
        return s["own"].buf[0]
    if kind == "droplet":
        sim = s["sim"]
        sim.init_droplets(*_drop_args(p))
        sim.step(c["steps"])
        return dict(angle=_angle(sim, *p["regions"][0]), mass=sim.mass(), speed=sim.max_speed(), rho=sim.rho())
    if kind == "host":
        sim = s["sim"]
        sim.set_rho(s["rho"].numpy())
        sim.step(c["steps"])
        L.lbm_get_rho(sim.ctx, s["out"].numpy())
        return s["out"]
    if kind == "measure":
        sim = s["sim"]
        return dict(angles=np.array([_angle(sim, *r) for r in p["regions"]]), mass=sim.mass(), speed=sim.max_speed())
    if kind == "fields":
        sim = s["sim"]
        sim.set_f(s["f"])
        ux, uy = sim.u()
        return dict(sim.fields(), ux=ux, uy=uy, f=sim.f())
    if kind == "batch":
        b, at = s["batch"], 0
        b.step(c["steps"])
        theta, H, Lb, status = b.contact_angles(0)
        rho = s["rho"].numpy()
        for inst in b.instances:
            n = inst.nx * inst.ny
            L.lbm_get_rho(inst.ctx, rho[at:at + n].reshape(inst.ny, inst.nx))
            at += n
        return dict(theta=theta, H=H, L=Lb, status=status, rho=s["rho"])
    theta, T = s["theta"].clone().requires_grad_(), s["T"].clone().requires_grad_()
    nx, ny, eos, _, tau = s["args"]
    rho = ADJ.final_density(theta, T, nx=nx, ny=ny, eos=eos, tau=tau, params=s["params"], f0=s["f0"],
                            steps=c["steps"], checkpoint_every=c["every"], theta_top=p["theta"][1],
                            stream=s["stream"])
    (rho * s["weights"]).sum().backward()
    return dict(rho=rho.detach(), theta=theta.grad, T=T.grad)


def work(case):
    """A step reads a state of nine populations a node and writes one, and takes
    about 260 operations a node; a readback reads the populations and writes
    what it returns."""
    ps, k = _problems(case, 0), case["kind"]
    n = float(sum(q["nx"] * q["ny"] for q in ps))
    real = case.get("precision", 32) / 8.0
    step = dict(bytes=18.0 * real * n, flops=260.0 * n)
    if k == "measure":
        return dict(bytes=9.0 * real * n, flops=140.0 * n)
    if k == "fields":
        return dict(bytes=n * (9.0 * 8.0 + 19.0 * 8.0), flops=140.0 * n)
    times = case["steps"] * (4.0 if k == "adjoint" else 1.0)  # forward, replay, reverse (twice the work)
    extra = {"droplet": 8.0, "batch": 8.0, "host": 16.0, "adjoint": 8.0}.get(k, 0.0) * n
    return dict(bytes=times * step["bytes"] + extra, flops=times * step["flops"])


# ---- the same in 64 bits ---------------------------------------------------------

EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
SHAPE = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def _rho0(ps):
    """Initial densities [B, ny, nx]: the largest of the droplets' tanh profiles."""
    out = []
    for p in ps:
        nx, ny = p["nx"], p["ny"]
        x = torch.arange(nx, dtype=torch.float64, device="cuda")
        y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
        rho = torch.full((ny, nx), p["rho_v"], dtype=torch.float64, device="cuda")
        for xc, R, w in p["drops"]:
            dx = x - xc
            dx = dx - nx * torch.floor((dx + 0.5 * nx) / nx)
            r = torch.sqrt(dx * dx + (y - (1.0 if w == 0 else ny - 2.0)) ** 2)
            v = 0.5 * (p["rho_l"] + p["rho_v"]) - 0.5 * (p["rho_l"] - p["rho_v"]) * torch.tanh(2 * (r - R) / p["width"])
            rho = torch.maximum(rho, v)
        out.append(rho)
    return torch.stack(out)


def _f0(p):
    rho = _rho0([p])[0].cpu().numpy()
    f = SHAPE[:, None, None] * rho
    if p["walls"]:
        f[:, 0] = f[:, -1] = 0.0
    return f


def _weights(c, seed):
    w = np.random.default_rng(seed + 7).uniform(-1.0, 1.0, (c["ny"], c["nx"]))
    return torch.tensor(w, device="cuda")


class _Exact:
    """The step of same-sized domains [B, 9, ny, nx] in 64 bits."""

    def __init__(self, ps, theta_bottom=None, T=None):
        p = self.p = ps[0]
        self.B, self.nx, self.ny, self.walls = len(ps), p["nx"], p["ny"], p["walls"]
        col = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda").reshape(-1, 1, 1)  # noqa: E731
        self.T = col([q["T"] for q in ps]) if T is None else T
        self.A, self.kappa, self.Gw = col([q["A"] for q in ps]), p["kappa"], p["G_w"]
        self.top = col([q["rho_max"] for q in ps])
        for k in ("s_e", "s_eps", "s_q"):
            setattr(self, k, col([q["rates"][k] for q in ps]))
        self.s_nu = col([1.0 / q["tau"] for q in ps])
        th = torch.tensor(np.stack([q["theta"] for q in ps]), device="cuda")
        bottom = th[:, 0] if theta_bottom is None else theta_bottom[None]
        self.half = [math.pi / 2 - bottom, math.pi / 2 - th[:, 1]]

    def psi_U(self, rho):
        p = self.p
        if p["eos"] == "cs":
            e = CS_B * rho / 4
            pr = rho * CS_R * self.T * (1 + e + e * e - e ** 3) / (1 - e) ** 3 - CS_A * rho * rho
        else:
            r1, r2, tv, tm, tl = p["pw"]
            pr = torch.where(rho <= r1, rho * tv, torch.where(rho <= r2, r1 * tv + (rho - r1) * tm,
                                                              r1 * tv + (r2 - r1) * tm + (rho - r2) * tl))
        U = pr - rho / 3
        return self.root(-2 * U), U

    @staticmethod
    def root(s):  # sqrt, with value and slope 0 where the argument is not positive
        pos = s > 0
        return torch.where(pos, torch.sqrt(torch.where(pos, s, torch.ones_like(s))), torch.zeros_like(s))

    def state(self, f):
        """rho, psi, U at every node, the solid rows' ghost values included."""
        rho = f.sum(1)
        if not self.walls:
            return (rho,) + self.psi_U(rho)
        if self.p["wetting"] == "martys_chen":
            psi, U = self.psi_U(rho[:, 1:-1])
            z = torch.zeros_like(rho[:, :1])
            return tuple(torch.cat([z, v, z], 1) for v in (rho[:, 1:-1], psi, U))
        ghost = []
        for w, (a, b) in enumerate(((1, 2), (-2, -3))):
            r1, r2 = rho[:, a], rho[:, b]
            da = torch.roll(r1, -1, 1) - torch.roll(r1, 1, 1)
            if self.p["n_iter"] == 0:
                g = r2 + torch.tan(self.half[w]) * da.abs()
            else:
                d = 2 * (r2 - r1)
                for _ in range(self.p["n_iter"]):
                    g = r2 + torch.sin(self.half[w]) * self.root(da * da + d * d)
                    d = r2 - g
            ghost.append(torch.minimum(g.clamp(min=0.0), self.top[:, 0])[:, None])
        rho = torch.cat([ghost[0], rho[:, 1:-1], ghost[1]], 1)
        psi, U = self.psi_U(rho)
        low = torch.ones_like(rho, dtype=torch.bool)
        low[:, 0], low[:, -1] = rho[:, 0] < self.top[:, 0], rho[:, -1] < self.top[:, 0]
        return rho, torch.where(low, psi, torch.zeros_like(psi)), torch.where(low, U, torch.zeros_like(U))

    def force(self, psi, U):
        """Eq. 9 (and Eq. 14) force and the Eq. 17 tensor."""
        P = [torch.roll(psi, (-EY[a], -EX[a]), (1, 2)) for a in range(9)]
        V = [torch.roll(U, (-EY[a], -EX[a]), (1, 2)) for a in range(9)]
        w = [0.0] + [1 / 3] * 4 + [1 / 12] * 4
        s = lambda e, X: sum(w[a] * e[a] * X[a] for a in range(1, 9) if e[a])  # noqa: E731
        Fx = -self.A * s(EX, V) + (1 - self.A) * psi * s(EX, P)
        Fy = -self.A * s(EY, V) + (1 - self.A) * psi * s(EY, P)
        if self.p["wetting"] == "martys_chen" and self.walls:
            solid = torch.zeros((self.ny, 1), dtype=torch.float64, device="cuda")
            solid[0], solid[-1] = 1.0, 1.0
            Fy = Fy - self.Gw * psi * 0.5 * (torch.roll(solid, -1, 0) - torch.roll(solid, 1, 0))
        D = [(1 - self.A) * psi * (P[a] - psi) + 0.5 * self.A * (P[a] ** 2 - psi ** 2) for a in range(9)]
        q = lambda e, g: -0.5 * self.kappa * sum(w[a] * e[a] * g[a] * D[a] for a in range(1, 9) if e[a] * g[a])  # noqa: E731,E501
        return Fx, Fy, q(EX, EX), q(EY, EY), q(EX, EY)

    def step(self, f):
        rho, psi, U = self.state(f)
        Fx, Fy, Qxx, Qyy, Qxy = self.force(psi, U)
        if self.walls:  # the solid rows hold no fluid; any finite density does there
            rho = torch.cat([rho[:, 1:2], rho[:, 1:-1], rho[:, -2:-1]], 1)
        f0, f1, f2, f3, f4, f5, f6, f7, f8 = f.unbind(1)
        ax, dg = f1 + f2 + f3 + f4, f5 + f6 + f7 + f8
        jx, jy = f1 - f3 + f5 - f6 - f7 + f8, f2 - f4 + f5 + f6 - f7 - f8
        vx, vy = (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho
        v2, vF = vx * vx + vy * vy, vx * Fx + vy * Fy
        rel = lambda s, m, eq, S, C: m - s * (m - eq) + (1 - 0.5 * s) * S + C  # noqa: E731
        me = rel(self.s_e, -4 * f0 - ax + 2 * dg, rho * (3 * v2 - 2), 6 * vF, 1.5 * self.s_e * (Qxx + Qyy))
        mp = rel(self.s_eps, 4 * f0 - 2 * ax + dg, rho * (1 - 3 * v2), -6 * vF, 0.0)
        mx = rel(self.s_q, -2 * (f1 - f3) + f5 - f6 - f7 + f8, -rho * vx, -Fx, 0.0)
        my = rel(self.s_q, -2 * (f2 - f4) + f5 + f6 - f7 - f8, -rho * vy, -Fy, 0.0)
        mn = rel(self.s_nu, f1 - f2 + f3 - f4, rho * (vx * vx - vy * vy), 2 * (vx * Fx - vy * Fy),
                 -self.s_nu * (Qxx - Qyy))
        mo = rel(self.s_nu, f5 - f6 + f7 - f8, rho * vx * vy, vx * Fy + vy * Fx, -self.s_nu * Qxy)
        r, e, q = rho / 9, me / 36, mp / 36
        jx, jy, mx, my, mn, mo = (jx + Fx) / 6, (jy + Fy) / 6, mx / 12, my / 12, mn / 4, mo / 4
        out = [r - 4 * e + 4 * q]
        for a in range(1, 9):
            if a < 5:
                g = r - e - 2 * q + EX[a] * (jx - 2 * mx) + EY[a] * (jy - 2 * my) + (EX[a] ** 2 - EY[a] ** 2) * mn
            else:
                g = r + 2 * e + q + EX[a] * (jx + mx) + EY[a] * (jy + my) + EX[a] * EY[a] * mo
            out.append(g)
        new = [torch.roll(g, (EY[a], EX[a]), (1, 2)) for a, g in enumerate(out)]
        if self.walls:  # half-way bounce-back
            for a in range(9):
                rows = [new[a][:, 1:2], new[a][:, 2:-2], new[a][:, -2:-1]]
                if EY[a] > 0:
                    rows[0] = out[OPP[a]][:, 1:2]
                if EY[a] < 0:
                    rows[2] = out[OPP[a]][:, -2:-1]
                z = torch.zeros_like(rows[0])
                new[a] = torch.cat([z] + rows + [z], 1)
        return torch.stack(new, 1)

    def start(self, ps):
        f = torch.tensor(SHAPE, device="cuda")[None, :, None, None] * _rho0(ps)[:, None]
        if self.walls:
            f[:, :, 0] = f[:, :, -1] = 0.0
        return f

    def rho(self, f):
        return f.sum(1)

    def u(self, f):
        rho, psi, U = self.state(f)
        Fx, Fy = self.force(psi, U)[:2]
        e = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda").reshape(1, 9, 1, 1)  # noqa: E731
        u = [((f * e(d)).sum(1) + 0.5 * F) / rho for d, F in ((EX, Fx), (EY, Fy))]
        return [self.fluid(v) for v in u]

    def fluid(self, v):
        if self.walls:
            v = v.clone()
            v[:, 0] = v[:, -1] = 0.0
        return v


def _exact_angle(rho, wall, a, b, mid):
    """Circular-cap angle, height and base width of the droplet on a wall."""
    ny = rho.shape[0]
    rows = rho[1:ny // 2] if wall == 0 else rho[ny // 2:ny - 1][::-1]
    xc = a + int(np.argmax(rows[:, a:b].sum(0)))
    row = rows[0]
    vl = [x for x in range(a, xc) if row[x] < mid]
    vr = [x for x in range(xc + 1, b) if row[x] < mid]
    up = [k for k in range(1, rows.shape[0]) if rows[k, xc] < mid]
    if row[xc] < mid or not vl or not vr or not up:
        return [math.nan] * 3
    x, z, k = vl[-1], vr[0], up[0]
    left = x + (mid - row[x]) / (row[x + 1] - row[x])
    right = z - 1 + (row[z - 1] - mid) / (row[z - 1] - row[z])
    H = k - 1 + (rows[k - 1, xc] - mid) / (rows[k - 1, xc] - rows[k, xc])
    return [2 * math.atan2(2 * H, right - left), H, right - left]


def exact(case, seed):
    c, ps = case, _problems(case, seed)
    p, kind = ps[0], c["kind"]
    if kind == "adjoint":
        from torch.utils.checkpoint import checkpoint

        tb = torch.tensor(p["theta"][0], device="cuda", requires_grad=True)
        T = torch.tensor(p["T"], dtype=torch.float64, device="cuda", requires_grad=True)
        m = _Exact(ps, tb, T)
        f, left = m.start(ps), c["steps"]

        def some(f, k):
            for _ in range(k):
                f = m.step(f)
            return f

        while left:
            k = min(left, 20)
            f, left = checkpoint(some, f, k, use_reentrant=False), left - k
        rho = f.sum(1)[0]
        g = torch.autograd.grad((rho * _weights(c, seed)).sum(), [tb, T], allow_unused=True)
        g = [torch.zeros_like(x) if y is None else y for x, y in zip((tb, T), g)]
        return dict(rho=rho.detach(), theta=g[0], T=g[1])
    with torch.no_grad():
        if kind == "batch":
            rho, sized = [None] * len(ps), {}
            for i, q in enumerate(ps):
                sized.setdefault((q["nx"], q["ny"]), []).append(i)
            for at in sized.values():
                qs = [ps[i] for i in at]
                m = _Exact(qs)
                f = m.start(qs)
                for _ in range(c["steps"]):
                    f = m.step(f)
                for i, r in zip(at, m.rho(f).cpu()):
                    rho[i] = r.reshape(-1)
            t = [_exact_angle(r.numpy().reshape(q["ny"], q["nx"]), 0, 0, q["nx"], 0.5 * (q["rho_v"] + q["rho_l"]))
                 for q, r in zip(ps, rho)]
            t = np.array(t)
            return dict(theta=t[:, 0], H=t[:, 1], L=t[:, 2], status=None, rho=torch.cat(rho))
        m = _Exact(ps)
        if kind == "fields":
            f = _f0(p)
            f = f * (1.0 + 0.02 * np.random.default_rng(seed + 1).uniform(-1.0, 1.0, f.shape))
            f = torch.tensor(f, device="cuda")[None]
        else:
            f = m.start(ps)
            for _ in range(c["steps"]):
                f = m.step(f)
        rho = m.rho(f)
        if kind == "steps":
            return f[0]
        if kind == "host":
            return rho[0]
        ux, uy = m.u(f)
        if kind == "fields":
            full, psi, U = m.state(f)
            Fs = [m.fluid(v)[0] for v in m.force(psi, U)]
            return dict(dict(zip(("Fx", "Fy", "Qxx", "Qyy", "Qxy"), Fs)), rho=full[0], psi=psi[0], U=U[0], ux=ux[0],
                        uy=uy[0], f=f[0])
        r, mid = rho[0].cpu().numpy(), 0.5 * (p["rho_v"] + p["rho_l"])
        mass, speed = float(rho.sum()), float(torch.sqrt(ux * ux + uy * uy).max())
        if kind == "droplet":
            return dict(angle=_exact_angle(r, *p["regions"][0], mid), mass=mass, speed=speed, rho=rho[0])
        return dict(angles=np.array([_exact_angle(r, *q, mid) for q in p["regions"]]), mass=mass, speed=speed)
