"""The calibration adjoint (reverse mode through the executed solver map) through the
C-ABI and torch.autograd, against the oracle's forward-mode dual-number gradient and
central finite differences.

Tolerance: the adjoint runs in FP32 through 20 substeps x 10 Jacobi updates per env-step;
the oracle's gradient is exact in FP64.  Relative agreement is bounded by the FP32
forward's own sensitivity (~1e-6 relative per substep amplified through the iterations):
2e-2 of each parameter's largest gradient magnitude over the snakes.
"""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1904_02833_gb300.build import build
    build()
    torch.cuda.set_device(0)


def setup_case(n, contact, steps, settle=2, seed=5):
    from paper_1904_02833_gb300.calib import theta_of
    truth, guess = W.calibration(n=n, seed=seed)
    s = W.solver_settings(iters=10, contact=contact)
    ot = oracle.OracleSim(truth, s)
    ot.step(settle)
    target = ot.step(steps, tip=True)
    return truth, guess, s, target, theta_of(guess)


def gpu_grad(guess, s, target, theta, steps, ckpt, settle=2):
    from paper_1904_02833_gb300.calib import rollout
    from paper_1904_02833_gb300.sim import SnakeSim
    sim = SnakeSim(guess, s)
    sim.step(settle)
    th = theta.clone().cuda().requires_grad_(True)
    tips = rollout(sim, th, steps, ckpt)
    tg = torch.tensor(target, dtype=torch.float32, device="cuda")
    loss = ((tips - tg) ** 2).sum(-1).mean(0)
    loss.sum().backward()
    return loss.detach().cpu().numpy(), th.grad.cpu().numpy(), tips.detach().cpu().numpy()


@pytest.mark.parametrize("contact", [False, True])
def test_adjoint_matches_oracle_dual_gradient(contact):
    steps = 6
    truth, guess, s, target, theta = setup_case(6, contact, steps)
    loss, g, tips = gpu_grad(guess, s, target, theta, steps, ckpt=2)
    og = oracle.OracleSim(guess, s)
    og.step(2)
    loss_o, g_o = og.calib_grad(steps, target)
    tips_o = og.step(steps, tip=True)
    # FP32 trajectories of 10-update substeps drift ~1e-5 m from FP64 over the window;
    # the loss measures centimetre-scale tip errors, so it agrees to ~1e-2 relative
    assert np.abs(tips - tips_o).max() < 1e-4
    assert np.allclose(loss, loss_o, rtol=1e-2)
    for k in range(5):
        scale = np.abs(g_o[:, k]).max()
        assert np.abs(g[:, k] - g_o[:, k]).max() <= 2e-2 * scale, (k, g[:, k], g_o[:, k])


def test_checkpoint_spacing_does_not_change_the_gradient():
    steps = 6
    _, guess, s, target, theta = setup_case(4, True, steps)
    _, g1, t1 = gpu_grad(guess, s, target, theta, steps, ckpt=1)
    _, g6, t6 = gpu_grad(guess, s, target, theta, steps, ckpt=6)
    assert np.array_equal(t1, t6)
    # the same arithmetic; only the grouping of the per-segment parameter sums differs
    assert np.allclose(g1, g6, rtol=1e-5, atol=1e-6 * np.abs(g6).max())


def test_adjoint_matches_central_differences_without_contact():
    """Central differences (step 1e-3 relative) of the same loss evaluated in FP64 by the
    oracle (differences of the FP32 loss itself are dominated by its rounding)."""
    steps = 4
    _, guess, s, target, theta = setup_case(3, False, steps)
    _, g, _ = gpu_grad(guess, s, target, theta, steps, ckpt=2)
    names = ["alpha_b", "damping", "tau_inf", "tau_def", "gain"]

    def loss_of(wd):
        # the window starts from the unperturbed settled state; only the window's
        # parameters move (as in the differentiated rollout)
        o = oracle.OracleSim(guess, s)
        o.step(2)
        o.prm = oracle.pack_params(wd)
        tips = o.step(steps, tip=True)
        return np.mean(np.sum((tips - target) ** 2, -1), 0)

    for k, nm in enumerate(names):
        hstep = 1e-3 * guess[nm]
        wp = {a: b.copy() for a, b in guess.items()}
        wm = {a: b.copy() for a, b in guess.items()}
        wp[nm] += hstep
        wm[nm] -= hstep
        fd = (loss_of(wp) - loss_of(wm)) / (2 * hstep)
        scale = np.abs(fd).max()
        assert np.abs(g[:, k] - fd).max() <= 3e-2 * scale + 1e-12, (k, g[:, k], fd)


def test_calibration_batch_runs_and_matches_oracle_on_samples():
    """1024 4-link snakes, 20 env-steps with checkpoints every 5 (the calibration batch
    over a shortened horizon); 3 sampled snakes against the oracle alone."""
    steps = 20
    truth, guess = W.calibration(n=1024, seed=5)
    s = W.solver_settings(iters=10)
    ot = oracle.OracleSim(W.subset(truth, [0, 511, 1023]), s)
    ot.step(1)
    tgt3 = ot.step(steps, tip=True)
    from paper_1904_02833_gb300.calib import rollout, theta_of
    from paper_1904_02833_gb300.sim import SnakeSim
    gt = SnakeSim(truth, s)
    gt.step(1)
    with torch.no_grad():
        target = rollout(gt, theta_of(truth).cuda(), steps, 5)
    sim = SnakeSim(guess, s)
    sim.step(1)
    th = theta_of(guess).cuda().requires_grad_(True)
    tips = rollout(sim, th, steps, 5)
    loss = ((tips - target) ** 2).sum(-1).mean(0)
    loss.sum().backward()
    g = th.grad.cpu().numpy()
    assert np.isfinite(g).all()
    sel = [0, 511, 1023]
    og = oracle.OracleSim(W.subset(guess, sel), s)
    og.step(1)
    _, g_o = og.calib_grad(steps, target[:, sel].double().cpu().numpy())
    for k in range(5):
        scale = np.abs(g_o[:, k]).max()
        assert np.abs(g[sel, k] - g_o[:, k]).max() <= 2e-2 * scale, (k, g[sel, k], g_o[:, k])


@pytest.mark.parametrize("iters", [3, 14])
def test_gradient_at_warp_edges_and_off_chip_iterates(iters):
    """Snakes of 2, 32, 33, 64, 65 and 128 nodes in one batch (a thread per node: ends of
    warps, blocks sized for the longest), the iterates of a substep on chip (3 updates) and
    in the global scratch (14 updates of 128 nodes), against the oracle's dual-number
    gradient; a second backward pass over the same rollout gives the same bits."""
    from paper_1904_02833_gb300.calib import rollout, theta_of
    from paper_1904_02833_gb300.sim import SnakeSim
    steps = 3
    truth, guess = W.calibration(n=6, seed=9)
    for w in (truth, guess):
        w["n_links"][:] = [1, 1, 4, 7, 8, 1]
        w["seg_per_link"][:] = [1, 31, 8, 9, 8, 127]
    assert W.n_nodes(guess).tolist() == [2, 32, 33, 64, 65, 128]
    s = W.solver_settings(iters=iters)
    ot = oracle.OracleSim(truth, s)
    target = ot.step(steps, tip=True)
    sim = SnakeSim(guess, s)
    th = theta_of(guess).cuda().requires_grad_(True)
    tips = rollout(sim, th, steps, 2)
    tg = torch.tensor(target, dtype=torch.float32, device="cuda")
    loss = ((tips - tg) ** 2).sum(-1).mean(0).sum()
    g, = torch.autograd.grad(loss, th, retain_graph=True)
    g2, = torch.autograd.grad(loss, th)
    assert torch.equal(g, g2)
    g = g.cpu().numpy()
    og = oracle.OracleSim(guess, s)
    _, g_o = og.calib_grad(steps, target)
    for k in range(5):
        assert np.abs(g[:, k] - g_o[:, k]).max() <= 2e-2 * np.abs(g_o[:, k]).max(), (k, g[:, k], g_o[:, k])


@pytest.mark.parametrize("contact", [False, True])
def test_gradient_of_vertical_two_node_snakes(contact):
    """Two nodes have no bend row, so a segment that stands straight up or hangs straight down
    (no heading, no gradient of its elevation) is differentiable: free and held ones, and one
    that lies flat, against the oracle's dual-number gradient.  In free flight and on a
    contact the only parameter they depend on is the damping."""
    from paper_1904_02833_gb300.calib import rollout, theta_of
    from paper_1904_02833_gb300.sim import SnakeSim
    steps = 4
    w = {k: np.repeat(v, 4) for k, v in W.pendulum(0.125).items()}
    w["damping"][:] = [0.1, 0.2, 0.3, 0.4]
    w["n_fixed"][:] = [1, 0, 0, 1]
    s = W.solver_settings(iters=10, contact=contact)
    o = oracle.OracleSim(w, s)
    o.x[:] = np.float32([[0, 0, 1], [0, 0, 0.9], [0, 0, 0.4], [0, 0, 0.28], [0.5, 0, 0.5], [0.5, 0, 0.625],
                         [0, 0, 1], [0.125, 0, 1]])
    o.v[:] = np.float32([[0, 0, 0], [0, 0, 0], [0, 0, 0.5], [0, 0, 0.25], [0.25, 0, 0], [0.25, 0, 0],
                         [0, 0, 0], [0, 0, 0]])
    sim = SnakeSim(w, s)
    sim.set_state(pos=o.x.astype(np.float32), vel=o.v.astype(np.float32))
    target = np.zeros((steps, 4, 3))
    th = theta_of(w).cuda().requires_grad_(True)
    tips = rollout(sim, th, steps, 2)
    ((tips - torch.tensor(target, dtype=torch.float32, device="cuda")) ** 2).sum(-1).mean(0).sum().backward()
    loss_o, g_o = o.calib_grad(steps, target)
    tips_o = o.step(steps, tip=True)
    assert np.abs(tips.detach().cpu().numpy() - tips_o).max() < 1e-4
    g = th.grad.cpu().numpy()
    assert np.array_equal(g[:, [0, 2, 3, 4]], np.zeros((4, 4)))
    assert np.abs(g[:, 1] - g_o[:, 1]).max() <= 2e-2 * np.abs(g_o[:, 1]).max(), (g, g_o)


@pytest.mark.parametrize("rho", [2e-10, 1e-20])
def test_nearly_vertical_segments(rho):
    """A falling chain whose segments stand `rho` off the vertical: their fourth power (2e-10)
    or square (1e-20) is below the smallest normal number, where the gradient's (2e-10) and
    the forward pass's quotients still have values.  The chain falls as it stands, so the
    gradient is the damping's alone."""
    from paper_1904_02833_gb300.calib import rollout, theta_of
    from paper_1904_02833_gb300.sim import SnakeSim
    steps, N = 3, 5
    w = W.pendulum(1 / 64)
    w["seg_per_link"][:], w["n_fixed"][:], w["damping"][:] = N - 1, 0, 0.2
    s = W.solver_settings(iters=6, contact=False)
    x = np.float32(np.stack([rho * np.arange(N), np.zeros(N), 1 - np.arange(N) / 64], 1))
    o = oracle.OracleSim(w, s)
    o.x[:] = x
    sim = SnakeSim(w, s)
    sim.set_state(pos=x, vel=np.zeros((N, 3), np.float32))
    target = np.zeros((steps, 1, 3))
    th = theta_of(w).cuda().requires_grad_(True)
    tips = rollout(sim, th, steps, 2)
    g, = torch.autograd.grad((tips ** 2).sum(-1).mean(0).sum(), th)
    _, g_o = o.calib_grad(steps, target)
    assert np.abs(tips.detach().cpu().numpy() - o.step(steps, tip=True)).max() < 1e-5
    if rho > 1e-12:
        g = g.cpu().numpy()
        assert np.isfinite(g).all(), g
        assert abs(g[0, 1] - g_o[0, 1]) <= 2e-2 * abs(g_o[0, 1]), (g, g_o)


def test_gradient_of_micrometre_snakes():
    """Segments of 2^-22 m (a quarter of a micrometre; their sixth power is a subnormal number)
    with compliances and gains that bend them like the usual ones, weightless, against the
    oracle's dual-number gradient."""
    from paper_1904_02833_gb300.calib import rollout, theta_of
    from paper_1904_02833_gb300.sim import SnakeSim
    steps, n = 4, 6
    _, w = W.calibration(n=n, seed=12)
    w["gain"][:] *= w["L0"] * 2.0 ** 22
    w["L0"][:] = 2.0 ** -22
    w["z0"][:] = 0.0
    s = W.solver_settings(iters=6, contact=False, gravity=(0.0, 0.0, 0.0))
    sim = SnakeSim(w, s)
    th = theta_of(w).cuda().requires_grad_(True)
    tips = rollout(sim, th, steps, 2)
    scale = 1e10  # a loss of order one
    g, = torch.autograd.grad(((scale * tips) ** 2).sum(-1).mean(0).sum(), th)
    g = g.cpu().numpy()
    o = oracle.OracleSim(w, s)
    _, g_o = o.calib_grad(steps, np.zeros((steps, n, 3)))
    g_o *= scale ** 2
    for k in range(5):
        assert np.abs(g[:, k] - g_o[:, k]).max() <= 2e-2 * np.abs(g_o[:, k]).max(), (k, g[:, k], g_o[:, k])


def test_checkpoint_interval_beyond_the_rollout():
    """A checkpoint interval longer than the rollout is one segment of the rollout's length,
    also where its substeps are more than an int counts (214748365 x 20 = 4 modulo 2^32): the
    same tips and gradient, and no more memory than the rollout takes."""
    steps = 3
    _, guess, s, target, theta = setup_case(4, True, steps)
    _, g, t = gpu_grad(guess, s, target, theta, steps, ckpt=steps)
    for ckpt in (steps + 1, 100, 214748365, 2 ** 31 - 1):
        _, g1, t1 = gpu_grad(guess, s, target, theta, steps, ckpt=ckpt)
        assert np.array_equal(t, t1) and np.array_equal(g, g1), ckpt


@pytest.mark.parametrize("n,steps,grad", [(512, 20, False), (4096, 14, True)])
def test_rollouts_take_no_records_without_a_gradient_or_beyond_a_gibibyte(n, steps, grad):
    """A rollout no gradient can be asked for (200 MB of substep states), and one whose single
    segment's states exceed 1 GiB, take the device memory of their states and checkpoints alone
    (here below 64 MB); the gradient of either form is the one of short segments."""
    from paper_1904_02833_gb300.calib import rollout, theta_of
    from paper_1904_02833_gb300.sim import SnakeSim
    _, guess = W.calibration(n=n, seed=6)
    s = W.solver_settings(iters=2)
    assert n * steps * s["n_sub"] * (6 * 41 + 2 * 4) * 4 > (2 ** 30 if grad else 2e8)
    sim, ref = SnakeSim(guess, s), SnakeSim(guess, s)
    th = theta_of(guess).cuda().requires_grad_(grad)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    tips = rollout(sim, th, steps, steps)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 64e6
    th2 = th.detach().clone().requires_grad_(True)
    tips2 = rollout(ref, th2, steps, 2)
    assert torch.equal(tips.detach(), tips2.detach())
    if grad:
        g, = torch.autograd.grad((tips ** 2).sum(), th)
        g2, = torch.autograd.grad((tips2 ** 2).sum(), th2)
        assert torch.allclose(g, g2, rtol=1e-4, atol=1e-5 * g2.abs().max().item())
