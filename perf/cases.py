"""The work a user of the simulator has it do, as measurable cases.

Each case is one pass through the public Python entry points (SnakeSim, rollout,
WarmStartMLP, FemSim): stepping batches of soft snakes at a fixed number of Jacobi updates
or to a residual tolerance, cold, from the previous multipliers, from the network's
prediction or with Newton + PCR; the differentiable calibration rollout with its gradient;
a training step and a forward pass of the warm-start network; frames of tetrahedral soft
links.  Inputs come from the seed alone.  `exact` computes the same outputs in 64 bits with
plain torch, from the method's definitions, wherever a pass has one well-defined value (a
solve that stops at a tolerance has not: the pass it stops in depends on the rounding).
"""
import ctypes
import math

import numpy as np
import torch

from paper_1904_02833_gb300.calib import rollout
from paper_1904_02833_gb300.fem import FemSim
from paper_1904_02833_gb300.mlp import WarmStartMLP
from paper_1904_02833_gb300.sim import SnakeSim

DT, N_SUB, OMEGA, GRAV = 1.0 / 60.0, 20, 1.0 / 3.0, 9.81
FIELDS = ("L0", "mass", "alpha_s", "alpha_b", "gain", "tau_inf", "tau_def", "mu", "damping", "radius",
          "gait_amp", "gait_freq", "gait_lag", "gait_offset", "gait_scale", "gait_alternate", "x0", "y0",
          "z0", "yaw0", "mu_side")
# lanes and nodes per lane that sim_autotune settles on for these lengths (throughput runs
# set them from a saved tuning; the others keep the library's defaults)
TUNED = {21: (32, 1), 31: (32, 1), 41: (32, 2), 51: (32, 2), 61: (32, 2), 71: (32, 3), 81: (32, 3)}
FLOP_NODE_PASS = 216   # FP32 operations of one Jacobi pass per node
FLOP_NODE_PCR = 130    # of one Newton + PCR product with its vector updates per node
FLOP_ELEMENT = 363     # of one soft-link product with its vector updates per element
FLOP_LINEARISE = 1130  # linearisation and final update of a soft-link substep per element
FLOP_ROW_INFER, FLOP_ROW_TRAIN = 39168, 3 * 39168
N_PARAMS = 19841


def listed():
    return [
        # one 41-node snake in a control loop at 60 Hz: a captured env-step per call
        dict(name="step_single_41", kind="fixed", n=1, lo=4, hi=4, seg=10, iters=10, warm=0, aniso=0, law=0,
             contact=1, graph=1, tuned=0, steps=1),
        # the batched locomotion of 4096 uneven snakes at ten updates per substep
        dict(name="step_fleet_4096", kind="fixed", n=4096, lo=2, hi=8, seg=10, iters=10, warm=0, aniso=0, law=0,
             contact=1, graph=1, tuned=1, steps=1),
        # a sweep of 256 clamped actuators over pressure and compliance, relaxing to 1e-6
        dict(name="sweep_static_256", kind="static", n=256, damping=20.0, tol=1e-6),
        # wheeled snakes (anisotropic friction) solved to 1e-4 from the previous multipliers,
        # an odd batch size in the library's default layouts
        dict(name="loco_previous_1500", kind="tol", n=1500, lo=2, hi=8, seg=10, warm=1, beta=0.75, aniso=1,
             tuned=0, settle=30),
        # a large batch solved to 1e-4 from cold multipliers: the plain solver
        dict(name="loco_plain_8192", kind="tol", n=8192, lo=2, hi=8, seg=10, warm=0, beta=1.0, aniso=0, tuned=1,
             settle=30),
        # the learned warm start: the network on the stretch rows at every third substep
        dict(name="loco_learned_4096", kind="learned", n=4096, lo=2, hi=8, seg=10, rows=2, every=3, tuned=1,
             settle=20),
        # contact-free snakes with the paper's own solver, Newton + PCR
        dict(name="fall_newton_pcr_4096", kind="pcr", n=4096, lo=2, hi=8, seg=10, tol=1e-4, tuned=0),
        # calibration: tip trajectories and their gradient in five parameters per snake
        dict(name="calibrate_1024x20", kind="calib", n=1024, lo=4, hi=4, seg=10, iters=10, steps=20, ckpt=10,
             contact=1),
        # one Adam step of the warm-start network on a minibatch of logged rows
        dict(name="train_16384", kind="train", rows=16384),
        # the network on every row of a 4096-snake batch
        dict(name="infer_1261356", kind="infer", rows=1261356),
        # a frame of a large batch of soft links, and of one link
        dict(name="fem_frame_1216", kind="fem", links=1216, m=8, sections=13, n_sub=2, iters=21, pcr=20),
        dict(name="fem_frame_1", kind="fem", links=1, m=8, sections=13, n_sub=2, iters=21, pcr=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fixed", "fixed", "tol", "learned", "pcr", "static", "calib", "train", "infer", "fem"])
    if kind in ("fixed", "tol", "learned", "pcr"):
        seg = rng.choice([5, 7, 10, 10])
        lo = rng.randint(1, 4)
        c = dict(kind=kind, lo=lo, hi=rng.randint(lo, 8), seg=seg)
    if kind == "fixed":
        return dict(c, n=_log_int(rng, 1, 4096), iters=rng.randint(4, 12), warm=rng.randint(0, 1),
                    aniso=rng.randint(0, 1), law=rng.randint(0, 1), contact=rng.randint(0, 1),
                    graph=rng.randint(0, 1), tuned=0, steps=rng.randint(1, 3))
    if kind == "tol":
        warm = rng.randint(0, 1)
        return dict(c, n=_log_int(rng, 16, 8192), warm=warm, beta=0.75 if warm else 1.0, aniso=rng.randint(0, 1),
                    tuned=rng.randint(0, 1), settle=20)
    if kind == "learned":
        return dict(c, n=_log_int(rng, 64, 4096), rows=rng.randint(0, 2), every=rng.randint(1, 4),
                    tuned=rng.randint(0, 1), settle=10)
    if kind == "pcr":
        return dict(c, n=_log_int(rng, 1, 4096), tol=rng.choice([1e-4, 1e-5]), tuned=0)
    if kind == "static":
        return dict(kind=kind, n=_log_int(rng, 9, 256), damping=rng.choice([0.05, 20.0]), tol=rng.choice([1e-5, 1e-6]))
    if kind == "calib":
        lo = rng.randint(1, 4)
        return dict(kind=kind, n=_log_int(rng, 3, 1024), lo=lo, hi=rng.randint(lo, 6), seg=10,
                    iters=rng.randint(5, 12), steps=rng.randint(1, 12), ckpt=rng.randint(1, 10),
                    contact=rng.randint(0, 1))
    if kind == "train":
        return dict(kind=kind, rows=_log_int(rng, 100, 131072))
    if kind == "infer":
        return dict(kind=kind, rows=_log_int(rng, 100, 1261356))
    return dict(kind=kind, links=_log_int(rng, 1, 1216), m=rng.choice([4, 8, 8]), sections=rng.randint(2, 13),
                n_sub=rng.randint(1, 2), iters=rng.choice([11, 21, 42]), pcr=rng.choice([10, 20, 20]))


# ------------------------------------------------------------------ inputs
def _rng(seed):
    return np.random.default_rng([1904, int(seed)])


def _base(n):
    w = dict(L0=0.02, mass=0.01, alpha_s=1e-8, alpha_b=1e-4, gain=20.0, tau_inf=0.15, tau_def=0.25, mu=0.5,
             damping=0.05, radius=0.01, gait_amp=1.0, gait_freq=1.0, gait_lag=math.pi / 2, gait_offset=0.0,
             gait_scale=1.0, gait_alternate=0.0, x0=0.0, y0=0.0, z0=0.01, yaw0=0.0, mu_side=0.0)
    w = {k: np.full(n, w[k]) for k in FIELDS}
    for k, d in (("n_links", 4), ("seg_per_link", 10), ("n_fixed", 0)):
        w[k] = np.full(n, d, np.int32)
    return w


def _snakes(c, rng):
    """Uneven snakes with the paper's gait, as the locomotion workload draws them: link counts
    uniform over the range, in an order of the seed's (the total is the case's)."""
    n = c["n"]
    w = _base(n)
    w["n_links"][:] = rng.permutation(c["lo"] + np.arange(n) % (c["hi"] - c["lo"] + 1))
    w["seg_per_link"][:] = c["seg"]
    w["gait_amp"][:] = rng.uniform(0.3, 1.0, size=n)
    w["gait_freq"][:] = rng.uniform(0.5, 2.0, size=n)
    w["gait_lag"][:] = rng.uniform(math.pi / 4, math.pi, size=n)
    w["mu"][:] = rng.uniform(0.3, 0.8, size=n)
    w["yaw0"][:] = rng.uniform(0.0, 2 * math.pi, size=n)
    if c.get("aniso"):
        w["mu_side"][:] = w["mu"] * rng.uniform(1.5, 4.0, size=n)
    return w


def _settings(**kw):
    s = dict(dt=DT, n_sub=N_SUB, iters=10, tol=0.0, omega=OMEGA, gravity=(0.0, 0.0, -GRAV), contact=True, warm=0)
    s.update(kw)
    return s


def _tune(sim, c):
    if c.get("tuned"):
        for nodes in sorted(set(np.diff(sim.node_off).tolist())):
            if nodes in TUNED:
                sim.set_layout(nodes, *TUNED[nodes])


def _fixed_input(c, seed):
    rng = _rng(seed)
    w = _snakes(c, rng)
    if not c["contact"]:
        w["z0"][:] = 2.0
    s = _settings(iters=c["iters"], warm=c["warm"], beta=0.75 if c["warm"] else 1.0, latency=c["law"],
                  contact=bool(c["contact"]))
    return w, s, int(rng.integers(0, 600))


def _static_input(c, seed):
    rng = _rng(seed)
    w = _base(c["n"])
    w["n_links"][:] = 1
    w["n_fixed"][:] = 2
    w["alpha_b"][:] = 10.0 ** rng.uniform(-5.0, -3.0, size=c["n"])
    w["gait_offset"][:] = np.arange(c["n"]) % 16 / 15.0
    w["gait_scale"][:] = 0.0
    w["gait_freq"][:] = 0.0
    w["z0"][:] = 1.0
    w["damping"][:] = c["damping"]
    return w


def _calib_input(c, seed):
    """Guessed parameters and the recorded tip trajectories they are calibrated against: the
    resting tip swaying by centimetres."""
    rng = _rng(seed)
    n = c["n"]
    w = _snakes(dict(c, aniso=0), rng)
    w["alpha_b"][:] = 10.0 ** rng.uniform(-5.0, -3.0, size=n)
    w["damping"][:] = rng.uniform(0.01, 0.2, size=n)
    w["tau_inf"][:] = rng.uniform(0.05, 0.4, size=n)
    w["tau_def"][:] = rng.uniform(0.05, 0.4, size=n)
    w["gain"][:] = rng.uniform(10.0, 30.0, size=n)
    theta = np.stack([w[k] for k in ("alpha_b", "damping", "tau_inf", "tau_def", "gain")], 1)
    ell = w["n_links"] * w["seg_per_link"] * w["L0"]
    tip = np.stack([ell * np.cos(w["yaw0"]), ell * np.sin(w["yaw0"]), w["z0"]], 1)
    t = np.arange(1, c["steps"] + 1)[:, None, None] * DT
    sway = rng.uniform(0.005, 0.03, (1, n, 3)) * np.sin(2 * math.pi * rng.uniform(0.5, 2.0, (1, n, 3)) * t)
    sway[..., 2] = np.abs(sway[..., 2]) * 0.1
    return w, theta.astype(np.float32), (tip[None] + sway).astype(np.float32), int(rng.integers(0, 60))


def _net_params(seed, out_scale=1.0):
    """A 24-128-128-1 network with scaled normal weights: W1, b1, W2, b2, w3, b3."""
    g = _rng(seed + 7)
    parts = [g.normal(0, math.sqrt(2 / 24), 128 * 24), g.normal(0, 0.1, 128), g.normal(0, math.sqrt(2 / 128), 128 * 128),
             g.normal(0, 0.1, 128), out_scale * g.normal(0, math.sqrt(1 / 128), 128), out_scale * g.normal(0, 0.1, 1)]
    return np.concatenate(parts).astype(np.float32)


def _rows_input(c, seed):
    """Logged rows: row kind one-hot, geometry of order one, small velocities, a multiplier."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    n = c["rows"]
    f = torch.zeros(n, 32, device="cuda")
    f[:, 6:24] = torch.randn(n, 18, device="cuda", generator=g) * 0.5
    f[:, 13:22] *= 0.2
    kind = torch.randint(0, 6, (n,), device="cuda", generator=g)
    f.scatter_(1, kind[:, None], 1.0)
    target = (0.7 * f[:, 7] - 0.4 * f[:, 23] + 0.3 * f[:, 8] * f[:, 9] + 0.1 * kind
              + 0.05 * torch.randn(n, device="cuda", generator=g))
    return f.to(torch.bfloat16), target.contiguous()


def _mesh(m, sections, length=0.1, radius=0.0125):
    """The radially symmetric link mesh: per cross-section a centre and two rings of m
    particles, every prism between sections cut into three tetrahedra; centre-layer,
    perimeter and actuation rows; the first section held."""
    per = 1 + 2 * m
    pid = lambda s, ring, k: s * per + (0 if ring == 0 else 1 + (ring - 1) * m + k % m)  # noqa: E731
    phi = 2.0 * math.pi * np.arange(m) / m
    side = np.round(np.cos(phi), 12)
    X = np.zeros((sections * per, 3))
    for s in range(sections):
        X[s * per: (s + 1) * per, 0] = length * s / (sections - 1)
        for ring, rho in ((1, 0.5 * radius), (2, radius)):
            for k in range(m):
                X[pid(s, ring, k), 1:] = rho * math.cos(phi[k]), rho * math.sin(phi[k])
    tris = [t for k in range(m) for t in ((pid(0, 0, 0), pid(0, 1, k), pid(0, 1, k + 1)),
                                          (pid(0, 1, k), pid(0, 2, k), pid(0, 2, k + 1)),
                                          (pid(0, 1, k), pid(0, 2, k + 1), pid(0, 1, k + 1)))]
    tets = []
    for s in range(sections - 1):
        for tri in tris:
            a, b, d = sorted(v + s * per for v in tri)
            for t in ((a, b, d, a + per), (b, d, a + per, b + per), (d, a + per, b + per, d + per)):
                vol = np.dot(np.cross(X[t[1]] - X[t[0]], X[t[2]] - X[t[0]]), X[t[3]] - X[t[0]])
                tets.append(t if vol > 0 else (t[0], t[2], t[1], t[3]))
    rows = []
    for s in range(sections - 1):
        for p in [pid(s, 0, 0)] + [pid(s, r, k) for r in (1, 2) for k in range(m) if side[k] == 0.0]:
            rows.append((p, p + per, 0))
    for s in range(sections):
        rows += [(pid(s, 2, k), pid(s, 2, k + 1), 1) for k in range(m)]
    for s in range(sections - 1):
        for sg, kind in ((1.0, 2), (-1.0, 3)):
            rows += [(pid(s, r, k), pid(s + 1, r, k), kind) for r in (1, 2) for k in range(m) if side[k] * sg > 0]
    rows = np.asarray(rows, np.int32)
    fixed = np.zeros(sections * per, np.int32)
    fixed[:per] = 1
    return dict(X=X, tets=np.asarray(tets, np.int32), rows=rows[:, :2].copy(), kinds=rows[:, 2].copy(), fixed=fixed)


def _fem_input(c, seed):
    rng = _rng(seed)
    n = c["links"]
    w = dict(youngs=66243.0 * rng.uniform(0.8, 1.2, n), poisson=np.full(n, 0.4999), density=np.full(n, 1070.0),
             damping=np.full(n, 1.0), alpha_inext=np.zeros(n), alpha_perim=np.zeros(n), alpha_act=np.full(n, 1e-3),
             press_amp=6894.76 * rng.uniform(1.0, 3.0, n), press_freq=rng.uniform(0.5, 2.0, n),
             press_phase=rng.uniform(0.0, 2 * math.pi, n), press_offset=np.zeros(n))
    s = dict(dt=DT, n_sub=c["n_sub"], iters=c["iters"], tol=0.0, pcr_iters=c["pcr"], gravity=(0.0, 0.0, 0.0))
    return _mesh(c["m"], c["sections"]), w, s, int(rng.integers(0, 600))


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "fixed":
        w, s, at = _fixed_input(c, seed)
        sim = SnakeSim(w, s)
        _tune(sim, c)
        sim.step_index = at
        return dict(kind=kind, sim=sim, steps=c["steps"], graph=bool(c["graph"]))
    if kind == "static":
        w = _static_input(c, seed)
        sim = SnakeSim(w, _settings(iters=20000, tol=c["tol"], contact=False))
        sim.set_state(press=np.stack([w["gait_offset"], np.zeros(c["n"])], 1).astype(np.float32))
    elif kind in ("tol", "learned"):
        # into locomotion: a third to half a second from the straight resting pose
        w = _snakes(c, _rng(seed))
        sim = SnakeSim(w, _settings(iters=5000, tol=1e-4, warm=1, beta=0.75))
        _tune(sim, c)
        sim.step_index = int(_rng(seed + 1).integers(0, 600))
        sim.step(c["settle"])
        if kind == "tol":
            sim.set_config(warm=c["warm"], beta=c["beta"])
        else:
            sim.set_mlp(WarmStartMLP(_net_params(seed, out_scale=0.02)))
            sim.set_config(warm=2, beta=0.8, beta_net=0.5, net_rows=c["rows"], net_every=c["every"])
    elif kind == "pcr":
        w = _snakes(c, _rng(seed))
        w["z0"][:] = 2.0
        sim = SnakeSim(w, _settings(iters=5000, tol=c["tol"], contact=False, solver=1, pcr_iters=20))
        _tune(sim, c)
        sim.step_index = int(_rng(seed + 1).integers(0, 600))
        sim.step(4)
    elif kind == "calib":
        w, theta, target, at = _calib_input(c, seed)
        sim = SnakeSim(w, _settings(iters=c["iters"], contact=bool(c["contact"])))
        sim.step_index = at
        sim.snapshot_save()
        return dict(kind=kind, sim=sim, theta=torch.tensor(theta, device="cuda", requires_grad=True),
                    target=torch.tensor(target, device="cuda"), steps=c["steps"], ckpt=c["ckpt"])
    elif kind in ("train", "infer"):
        feat, target = _rows_input(c, seed)
        return dict(kind=kind, net=WarmStartMLP(_net_params(seed)), feat=feat, target=target,
                    params=torch.empty(N_PARAMS, device="cuda"))
    else:
        mesh, w, s, at = _fem_input(c, seed)
        sim = FemSim(mesh, w, s)
        sim.set_frame(at)
        return dict(kind=kind, sim=sim)
    sim.snapshot_save()
    return dict(kind=kind, sim=sim)


def run(state):
    kind = state["kind"]
    if kind == "fixed":  # stepping on, and reading the state
        state["sim"].step(state["steps"], graph=state["graph"])
        return dict(state["sim"].state(), lam=state["sim"].lam())
    if kind in ("static", "tol", "learned", "pcr"):  # a planner's look ahead from a saved state
        sim = state["sim"]
        sim.snapshot_restore()
        sim.step(1)
        return dict(sim.state(), lam=sim.lam())
    if kind == "calib":
        state["sim"].snapshot_restore()
        tips = rollout(state["sim"], state["theta"], state["steps"], state["ckpt"])
        loss = ((tips - state["target"]) ** 2).sum(-1).mean(0)
        grad, = torch.autograd.grad(loss.sum(), state["theta"])
        return dict(tips=tips.detach(), loss=loss.detach(), grad=grad)
    if kind == "train":
        net = state["net"]
        loss = net.train_step(state["feat"], state["target"], 1e-3)
        net.lib.mlp_get_params(net.h, ctypes.c_void_p(state["params"].data_ptr()), 1)
        return dict(loss=loss, params=state["params"])
    if kind == "infer":
        return dict(y=state["net"].forward(state["feat"]))
    state["sim"].step(1)
    x, v, resid, products = state["sim"].state_device()
    return dict(x=x, v=v, resid=resid, products=products)


# ------------------------------------------------------------------ work
def work(case):
    c, kind = case, case["kind"]
    if kind in ("train", "infer"):
        b = c["rows"] * (64 + 4) + 4 * N_PARAMS * (7 if kind == "train" else 1)
        return dict(bytes=b, flops=c["rows"] * (FLOP_ROW_TRAIN if kind == "train" else FLOP_ROW_INFER))
    if kind == "fem":
        per, tets = 1 + 2 * c["m"], 9 * c["m"] * (c["sections"] - 1)
        state = c["links"] * per * c["sections"] * 24
        return dict(bytes=2 * state + c["links"] * 52,
                    flops=c["links"] * c["n_sub"] * tets * (c["iters"] * FLOP_ELEMENT + FLOP_LINEARISE))
    links = c["n"] * (1 if kind == "static" else (c["lo"] + c["hi"]) / 2)
    nodes = links * (10 if kind == "static" else c["seg"]) + c["n"]
    state = nodes * (12 + 12 + 24) + links * 8
    if kind == "calib":  # forward, and the reverse sweep at about four times its arithmetic
        passes = c["steps"] * N_SUB * c["iters"]
        return dict(bytes=state + c["n"] * (40 + c["steps"] * 36), flops=5 * nodes * passes * FLOP_NODE_PASS)
    # updates per substep: fixed, or what a solve to the tolerance takes on average
    per_sub = dict(fixed=c.get("iters", 0) + 1, static=800, tol=100 if c.get("warm") else 170, learned=100, pcr=22)[kind]
    flop = FLOP_NODE_PCR if kind == "pcr" else FLOP_NODE_PASS
    return dict(bytes=2 * state + c["n"] * 104, flops=nodes * c.get("steps", 1) * N_SUB * per_sub * flop)


# ------------------------------------------------------------------ the same in 64 bits
class _Snakes64:
    """The substep map on padded [snakes, nodes] arrays in 64 bits: fixed Jacobi updates."""

    def __init__(self, w, s):
        t = lambda a: torch.tensor(np.asarray(np.asarray(a, np.float32), np.float64), device="cuda")  # noqa: E731
        self.p = {k: t(w[k])[:, None] for k in FIELDS}
        self.s = s
        self.h = s["dt"] / s["n_sub"]
        links, seg = np.asarray(w["n_links"]), np.asarray(w["seg_per_link"])
        N = links * seg + 1
        M = int(N.max())
        i = np.arange(M)[None]
        b = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
        self.node = b(i < N[:, None])
        self.seg_on = b(i[:, :-1] + 1 < N[:, None])
        self.bend_on = b((i >= 1) & (i + 1 < N[:, None]))[:, 1:-1]
        self.free = self.node & b(i >= np.asarray(w["n_fixed"])[:, None])
        self.link = b(np.minimum(i // seg[:, None], links[:, None] - 1))
        self.bends = b((i % seg[:, None] != 0))
        self.link_on = b(np.arange(int(links.max()))[None] < links[:, None])
        self.k = torch.arange(int(links.max()), device="cuda")[None]
        self.wi = torch.where(self.free, 1.0 / self.p["mass"], torch.zeros((), device="cuda", dtype=torch.float64))
        d = torch.arange(M, device="cuda")[None] * self.p["L0"]
        yaw = self.p["yaw0"]
        x = torch.stack([self.p["x0"] + d * yaw.cos(), self.p["y0"] + d * yaw.sin(), self.p["z0"].expand_as(d)], -1)
        self.x = x.float().double()
        self.v = torch.zeros_like(x)
        self.press = torch.zeros(len(N), self.link_on.shape[1], 2, device="cuda", dtype=torch.float64)
        self.lam = torch.zeros(len(N), M, 6, device="cuda", dtype=torch.float64)
        self.resid = torch.zeros(len(N), device="cuda", dtype=torch.float64)
        g = [float(np.float32(a)) for a in s["gravity"]]
        self.g = torch.tensor(g, device="cuda", dtype=torch.float64)

    def pressures(self, press, substep, th):
        s, p, h = self.s, self.p, self.h
        law = s.get("latency", 0) == 1
        every = max(1, int(round(float(np.float32(0.0083)) / h)))
        if law and substep % every:
            return press
        cyc = (p["gait_freq"] * ((substep + (every if law else 1)) * h)) % 1.0
        a = p["gait_offset"] + p["gait_scale"] * torch.sin(2 * math.pi * cyc + self.k * p["gait_lag"])
        a = a.clamp(-1.0, 1.0) * p["gait_amp"]
        a = torch.where((p["gait_alternate"] != 0) & (self.k % 2 == 1), -a, a)
        tg = torch.stack([a.clamp(min=0.0), (-a).clamp(min=0.0)], -1)
        if law:
            ki = kd = float(np.float32(0.23))
            up = torch.minimum(tg, press + (tg - press) ** 2 * ki)
            down = torch.maximum(tg, press - (press * kd).clamp(max=float(np.float32(0.085))))
            return torch.where(tg > press, up, torch.where(tg < press, down, press))
        tau = torch.where(tg > press, th["tau_inf"][..., None], th["tau_def"][..., None])
        return tg + (press - tg) * torch.exp(-h / tau)

    def rows(self, x, L0):
        """Segment vectors, values and gradients of the stretch, yaw and pitch rows."""
        e = x[:, 1:] - x[:, :-1]
        dummy = torch.tensor([1.0, 0.0, 0.0], device="cuda", dtype=torch.float64)
        e = torch.where(self.seg_on[..., None], e, dummy)
        h2 = e[..., 0] ** 2 + e[..., 1] ** 2
        l2 = h2 + e[..., 2] ** 2
        hh, ln = h2.sqrt(), l2.sqrt()
        n = e / ln[..., None]
        L = L0[..., None]
        gy = L * torch.stack([-e[..., 1] / h2, e[..., 0] / h2, torch.zeros_like(h2)], -1)
        gp = L * torch.stack([-e[..., 2] * e[..., 0] / (l2 * hh), -e[..., 2] * e[..., 1] / (l2 * hh), hh / l2], -1)
        el = torch.atan2(e[..., 2], hh)
        a, b = e[:, :-1], e[:, 1:]
        yaw = torch.atan2(a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0], a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1])
        return ln, n, gy, gp, yaw, el[:, 1:] - el[:, :-1]

    def limit(self, px, py, ln, bx, by):
        """The friction pair limited to the Coulomb disc, or the ellipse of the body frame."""
        p = self.p
        if float(p["mu_side"].max()) > 0:
            a, b = px * bx + py * by, py * bx - px * by
            u, v = a / p["mu"], b / p["mu_side"]
            n2, rad = u * u + v * v, ln
        else:
            n2, rad = px * px + py * py, p["mu"] * ln
        out = n2 > rad * rad
        safe = torch.where(out, n2, torch.ones_like(n2)).sqrt()
        sc = torch.where(out, rad.clamp(min=0.0) / safe, torch.ones_like(n2))
        return px * sc, py * sc

    def spread(self, x, gr, d):
        """w J^T d, the displacement of the nodes by the row multipliers d [.., 6]."""
        ln, n, gy, gp, _, _ = gr
        out = torch.zeros_like(x)
        out[..., 2] += d[..., 3]
        out[..., 0] += d[..., 4]
        out[..., 1] += d[..., 5]
        f = n * d[:, :-1, :1]
        pad = torch.nn.functional.pad
        out = out + pad(f, (0, 0, 1, 0)) - pad(f, (0, 0, 0, 1))
        for g, k in ((gy, 1), (gp, 2)):
            dd = d[:, 1:-1, k:k + 1]
            lo, hi = g[:, :-1] * dd, g[:, 1:] * dd
            out = out + pad(lo, (0, 0, 0, 2)) - pad(lo + hi, (0, 0, 1, 1)) + pad(hi, (0, 0, 2, 0))
        return self.wi[..., None] * out

    def weights(self, gr):
        _, _, gy, gp, _, _ = gr
        wi = self.wi
        out = [wi[:, :-1] + wi[:, 1:]]
        for g in (gy, gp):
            q = lambda a: (a * a).sum(-1)  # noqa: E731
            out.append(wi[:, :-2] * q(g[:, :-1]) + wi[:, 1:-1] * q(g[:, :-1] + g[:, 1:]) + wi[:, 2:] * q(g[:, 1:]))
        return out

    def bilateral(self, gr, lam, th, rest):
        """Values c + alpha~ lambda and diagonals of the three bilateral row kinds."""
        ln, _, _, _, yaw, pitch = gr
        h2, L0 = self.h ** 2, self.p["L0"]
        at_s, at_b = self.p["alpha_s"] / h2, th["alpha_b"] / h2
        W = self.weights(gr)
        c = [ln - L0 + at_s * lam[:, :-1, 0], L0 * (yaw - rest[:, 1:-1]) + at_b * lam[:, 1:-1, 1],
             L0 * pitch + at_b * lam[:, 1:-1, 2]]
        on = [self.seg_on & (W[0] > 0), self.bend_on & (W[1] > 0), self.bend_on & (W[2] > 0)]
        return c, [W[0] + at_s, W[1] + at_b, W[2] + at_b], on

    def body(self, xs):
        """Horizontal body direction of every node at the substep start."""
        M = xs.shape[1]
        i = torch.arange(M, device="cuda")[None]
        last = self.node.sum(1, keepdim=True) - 1
        at = lambda j: torch.gather(xs[..., :2], 1, j[..., None].expand(-1, -1, 2))  # noqa: E731
        t = at(torch.minimum(i + 1, last)) - at((torch.minimum(i, last) - 1).clamp(min=0))
        n = t.norm(dim=-1, keepdim=True)
        t = torch.where(n > 0, t / n.clamp(min=1e-300), torch.tensor([1.0, 0.0], device="cuda", dtype=torch.float64))
        return t[..., 0], t[..., 1]

    def update(self, x, xs, lam, th, rest, frame):
        om, m, p = self.s["omega"], self.p["mass"], self.p
        om = float(np.float32(om))
        gr = self.rows(x, p["L0"])
        c, D, on = self.bilateral(gr, lam, th, rest)
        z = torch.zeros((), device="cuda", dtype=torch.float64)
        pad = torch.nn.functional.pad
        d = [pad(torch.where(on[0], -om * c[0] / D[0], z), (0, 1))]
        d += [pad(torch.where(on[k], -om * c[k] / D[k], z), (1, 1)) for k in (1, 2)]
        if self.s["contact"]:
            ln = lam[..., 3]
            nl = (ln - om * m * (x[..., 2] - p["radius"])).clamp(min=0.0)
            tx, ty = lam[..., 4] - om * m * (x[..., 0] - xs[..., 0]), lam[..., 5] - om * m * (x[..., 1] - xs[..., 1])
            tx, ty = self.limit(tx, ty, ln, *frame)
            d += [torch.where(self.free, a, z) for a in (nl - ln, tx - lam[..., 4], ty - lam[..., 5])]
        else:
            d += [torch.zeros_like(d[0])] * 3
        d = torch.stack(d, -1)
        return x + self.spread(x, gr, d), lam + d

    def measure(self, x, xs, lam, th, rest, frame):
        p, wi = self.p, self.wi
        c, _, on = self.bilateral(self.rows(x, p["L0"]), lam, th, rest)
        r = torch.stack([torch.where(o, v.abs(), torch.zeros_like(v)).amax(1) for v, o in zip(c, on)]).amax(0)
        if self.s["contact"]:
            cn, b = x[..., 2] - p["radius"], wi * lam[..., 3]
            fb = (cn + b - (cn * cn + b * b).sqrt()).abs()
            ax, ay = wi * lam[..., 4], wi * lam[..., 5]
            px, py = self.limit(ax - (x[..., 0] - xs[..., 0]), ay - (x[..., 1] - xs[..., 1]), b, *frame)
            q = ((ax - px) ** 2 + (ay - py) ** 2).sqrt()
            r = torch.maximum(r, torch.where(self.free, torch.maximum(fb, q), torch.zeros_like(q)).amax(1))
        return r / p["L0"][:, 0]

    def substep(self, x, v, press, lam, substep, th, resid=None):
        s, h = self.s, self.h
        press = self.pressures(press, substep, th)
        dp = torch.gather(press[..., 0] - press[..., 1], 1, self.link)
        rest = torch.where(self.bends, th["gain"] * dp * self.p["L0"], torch.zeros_like(dp))
        free = self.free[..., None].to(x.dtype)
        xs = x
        x = x + free * h * (v + h * self.g)
        frame = self.body(xs) if float(self.p["mu_side"].max()) > 0 else (None, None)
        if s["warm"] == 0:
            lam = torch.zeros_like(lam)
        else:
            gr = self.rows(x, self.p["L0"])
            _, _, on = self.bilateral(gr, lam, th, rest)
            pad = torch.nn.functional.pad
            cf = self.free if s["contact"] else torch.zeros_like(self.free)
            keep = torch.stack([pad(on[0], (0, 1)), pad(on[1], (1, 1)), pad(on[2], (1, 1)), cf, cf, cf], -1)
            lam = float(np.float32(s["beta"])) * lam * keep
            x = x + self.spread(x, gr, lam)
        for _ in range(s["iters"]):
            x, lam = self.update(x, xs, lam, th, rest, frame)
        if resid is not None:
            resid = torch.maximum(resid, self.measure(x, xs, lam, th, rest, frame))
        v = free * (x - xs) * (torch.exp(-th["damping"] * h) / h)[..., None]
        return x, v, press, lam, resid

    def step(self, steps, at):
        th = {k: self.p[k] for k in ("alpha_b", "damping", "tau_inf", "tau_def", "gain")}
        x, v, press, lam = self.x, self.v, self.press, self.lam
        for k in range(steps):
            resid = self.resid * 0
            for sub in range(self.s["n_sub"]):
                x, v, press, lam, resid = self.substep(x, v, press, lam, (at + k) * self.s["n_sub"] + sub, th, resid)
        return dict(pos=x[self.node], vel=v[self.node], press=press[self.link_on], resid=resid, iters=None,
                    lam=lam[self.node])

    def calibrate(self, theta, target, steps, at):
        from torch.utils.checkpoint import checkpoint
        theta = torch.tensor(theta, device="cuda").double().requires_grad_(True)
        cols = ("alpha_b", "damping", "tau_inf", "tau_def", "gain")
        last = (self.node.sum(1) - 1)[:, None, None].expand(-1, 1, 3)
        x, v, press, tips = self.x, self.v, self.press, []
        for k in range(steps):
            for sub in range(self.s["n_sub"]):
                def one(x, v, press, theta, at=(at + k) * self.s["n_sub"] + sub):
                    th = {c: theta[:, i:i + 1] for i, c in enumerate(cols)}
                    return self.substep(x, v, press, self.lam, at, th)[:3]
                x, v, press = checkpoint(one, x, v, press, theta, use_reentrant=False)
            tips.append(torch.gather(x, 1, last)[:, 0])
        tips = torch.stack(tips)
        loss = ((tips - torch.tensor(target, device="cuda").double()) ** 2).sum(-1).mean(0)
        grad, = torch.autograd.grad(loss.sum(), theta)
        return dict(tips=tips.detach(), loss=loss.detach(), grad=grad)


def _net64(params):
    p = torch.tensor(params, device="cuda").double()
    cut = np.cumsum([0, 128 * 24, 128, 128 * 128, 128, 128, 1])
    W1, b1, W2, b2, w3, b3 = (p[a:b].clone().requires_grad_(True) for a, b in zip(cut[:-1], cut[1:]))
    return W1, b1, W2, b2, w3, b3


def _forward64(P, f):
    W1, b1, W2, b2, w3, b3 = P
    silu = torch.nn.functional.silu
    h = silu(f @ W1.view(128, 24).T + b1)
    return silu(h @ W2.view(128, 128).T + b2) @ w3 + b3


def _fem64(mesh, w, s, at):
    """One frame of the soft links: Newton steps of PCR iterations on all rows, in 64 bits."""
    t = lambda a: torch.tensor(np.asarray(np.asarray(a, np.float32), np.float64), device="cuda")  # noqa: E731
    p = {k: t(v) for k, v in w.items()}
    n = len(w["youngs"])
    X = torch.tensor(mesh["X"], device="cuda")
    tet = torch.tensor(mesh["tets"], device="cuda").long()
    row = torch.tensor(mesh["rows"], device="cuda").long()
    kind = torch.tensor(mesh["kinds"], device="cuda")
    P, h = len(X), s["dt"] / s["n_sub"]
    Dm = (X[tet[:, 1:]] - X[tet[:, :1]]).transpose(1, 2)
    B = torch.linalg.inv(Dm)
    G = torch.cat([-B.sum(1, keepdim=True), B], 1)  # [T, 4, 3] shape-function gradients
    vol = torch.linalg.det(Dm) / 6
    vn = torch.zeros(P, dtype=torch.float64, device="cuda").index_add_(0, tet.reshape(-1), (vol / 4).repeat_interleave(4))
    wn = 1.0 / (p["density"][:, None] * vn[None])
    wn = wn * (torch.tensor(mesh["fixed"], device="cuda") == 0)
    rest0 = (X[row[:, 1]] - X[row[:, 0]]).norm(dim=1)
    nu = p["poisson"][:, None, None]
    sc = (1.0 / (vol[None] * p["youngs"][:, None] * h * h))[..., None]

    def comply(v):
        a, b = v[..., :3], v[..., 3:]
        return torch.cat([(1 + nu) * a - nu * a.sum(-1, keepdim=True), (1 + nu) * b], -1)

    def voigt(M):
        o = lambda i, j: 0.5 * (M[..., i, j] + M[..., j, i])  # noqa: E731
        return torch.stack([o(0, 0), o(1, 1), o(2, 2), o(1, 2), o(0, 2), o(0, 1)], -1)

    def spread(R, nd, ve, vd):  # M^-1 J^T v
        S = torch.stack([torch.stack([ve[..., 0], ve[..., 5] / 2, ve[..., 4] / 2], -1),
                         torch.stack([ve[..., 5] / 2, ve[..., 1], ve[..., 3] / 2], -1),
                         torch.stack([ve[..., 4] / 2, ve[..., 3] / 2, ve[..., 2]], -1)], -2)
        c = torch.einsum("ntij,taj->ntai", R @ S, G)
        u = torch.zeros(n, P, 3, dtype=torch.float64, device="cuda")
        u.index_add_(1, tet.reshape(-1), c.reshape(n, -1, 3))
        f = nd * vd[..., None]
        u.index_add_(1, row[:, 1], f)
        u.index_add_(1, row[:, 0], -f)
        return u * wn[..., None]

    def apply(R, nd, at_d, on, ve, vd):
        u = spread(R, nd, ve, vd)
        H = torch.einsum("ntai,taj->ntij", u[:, tet], G)
        ye = voigt(R.transpose(-1, -2) @ H) + sc * comply(ve)
        yd = torch.where(on, (nd * (u[:, row[:, 1]] - u[:, row[:, 0]])).sum(-1) + at_d * vd, torch.zeros_like(vd))
        return ye, yd

    x = X[None].float().double().expand(n, -1, -1).clone()
    v = torch.zeros_like(x)
    worst = torch.zeros(n, dtype=torch.float64, device="cuda")
    products = 0
    dot = lambda a, b: (a[0] * b[0]).sum((1, 2)) + (a[1] * b[1]).sum(1)  # noqa: E731
    for sub in range(s["n_sub"]):
        tp = (at * s["n_sub"] + sub + 1) * h
        pres = p["press_amp"] * (torch.sin(2 * math.pi * p["press_freq"] * tp + p["press_phase"]) + p["press_offset"]).clamp(-1, 1)
        act = torch.where(pres > 0, 3, torch.where(pres < 0, 2, -1))
        eps = 1 + pres.abs() / p["youngs"]
        xs = x
        x = x + h * v
        on = ((kind[None] <= 1) | (kind[None] == act[:, None])) & (wn[:, row[:, 0]] + wn[:, row[:, 1]] > 0)
        alpha = torch.where(kind[None] == 0, p["alpha_inext"][:, None], torch.where(kind[None] == 1, p["alpha_perim"][:, None],
                                                                                  p["alpha_act"][:, None]))
        at_d = alpha / (h * h)
        rest = torch.where(kind[None] >= 2, rest0[None] * eps[:, None], rest0[None])
        le = torch.zeros(n, len(tet), 6, dtype=torch.float64, device="cuda")
        ld = torch.zeros(n, len(row), dtype=torch.float64, device="cuda")
        left = s["iters"]
        while True:
            F = torch.einsum("ntai,taj->ntij", x[:, tet], G)
            R = F
            for _ in range(12):
                inv = torch.linalg.inv(R).transpose(-1, -2)
                R = 0.5 * (R + inv)
            M = R.transpose(-1, -2) @ F
            ce = voigt(M) - torch.tensor([1.0, 1, 1, 0, 0, 0], device="cuda", dtype=torch.float64)
            e = x[:, row[:, 1]] - x[:, row[:, 0]]
            ln = e.norm(dim=-1)
            nd = e / ln[..., None]
            g2 = (G * G)[None]
            wa = wn[:, tet][..., None]
            q = (wa * g2).sum(2)
            dg = torch.stack([q[..., 0], q[..., 1], q[..., 2], (q[..., 1] + q[..., 2]) / 4, (q[..., 0] + q[..., 2]) / 4,
                              (q[..., 0] + q[..., 1]) / 4], -1)
            ckk = torch.cat([torch.ones_like(dg[..., :3]), (1 + nu) * torch.ones_like(dg[..., :3])], -1)
            ie = 1.0 / (dg + sc * ckk)
            idd = torch.where(on, 1.0 / (wn[:, row[:, 0]] + wn[:, row[:, 1]] + at_d), torch.zeros_like(ln))
            be = -(ce + sc * comply(le))
            bd = torch.where(on, -(ln - rest + at_d * ld), torch.zeros_like(ln))
            r = torch.maximum(be.abs().amax((1, 2)), (bd.abs() / rest0).amax(1))
            if left <= 0:
                break
            z = (be * ie, bd * idd)
            pp, dl = z, (torch.zeros_like(be), torch.zeros_like(bd))
            az = apply(R, nd, at_d, on, *z)
            qq = az
            left -= 1
            products += 1
            zaz = dot(z, az)
            for _ in range(min(s["pcr_iters"], left)):
                qs = (qq[0] ** 2 * ie).sum((1, 2)) + (qq[1] ** 2 * idd).sum(1)
                al = zaz / qs
                dl = (dl[0] + al[:, None, None] * pp[0], dl[1] + al[:, None] * pp[1])
                z = (z[0] - al[:, None, None] * qq[0] * ie, z[1] - al[:, None] * qq[1] * idd)
                az = apply(R, nd, at_d, on, *z)
                left -= 1
                products += 1
                new = dot(z, az)
                be_ = new / zaz
                zaz = new
                pp = (z[0] + be_[:, None, None] * pp[0], z[1] + be_[:, None] * pp[1])
                qq = (az[0] + be_[:, None, None] * qq[0], az[1] + be_[:, None] * qq[1])
            le, ld = le + dl[0], ld + dl[1]
            x = x + spread(R, nd, *dl)
        worst = torch.maximum(worst, r)
        v = torch.exp(-p["damping"] * h)[:, None, None] / h * (x - xs)
    return dict(x=x, v=v, resid=worst, products=None)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "fixed":
        w, s, at = _fixed_input(c, seed)
        return _Snakes64(w, s).step(c["steps"], at)
    if kind == "calib":
        w, theta, target, at = _calib_input(c, seed)
        s = _settings(iters=c["iters"], contact=bool(c["contact"]))
        return _Snakes64(w, s).calibrate(theta, target, c["steps"], at)
    if kind in ("train", "infer"):
        f, target = _rows_input(c, seed)
        P = _net64(_net_params(seed))
        if kind == "infer":
            with torch.no_grad():
                return dict(y=torch.cat([_forward64(P, q[:, :24].double()) for q in f.split(131072)]))
        loss = ((_forward64(P, f[:, :24].double()) - target.double()) ** 2).mean()
        grads = torch.autograd.grad(loss, P)
        new = [p.detach() - 1e-3 * g / (g.abs() + 1e-8) for p, g in zip(P, grads)]  # Adam's first step
        return dict(loss=loss.detach().reshape(1), params=torch.cat(new))
    if kind == "fem":
        mesh, w, s, at = _fem_input(c, seed)
        return _fem64(mesh, w, s, at)
    return None  # a solve that stops at a tolerance
