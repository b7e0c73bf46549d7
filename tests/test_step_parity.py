"""Reconstruction step (Algorithm 2) through gpair_step against the oracle's Algorithm 2 on the
same seeded tiny problem, plus checkpoint/resume of the solver state."""
import os

import numpy as np
import pytest
import torch

import oracle
from gpair_testutil import TAU, device_inputs, oracle_gaussians, rel_l2
from paper_2602_03893_gb300 import _lib, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def problem():
    oracle.set_threads(os.cpu_count() or 1)
    w = synth.tiny(1)
    G = oracle_gaussians(w)
    y = oracle.forward(G, w.sensors, w.v, w.fs, w.t0, w.Nt, k=w.k)
    b = synth.add_noise(y.astype(np.float32), 30.0, seed=101)
    b = (b / np.abs(b).max()).astype(np.float32)   # measured data scaled to max|b| = 1
    return w, G, b


def _gpu_ir(w, b, iters, params):
    gs, arr = device_inputs(w)
    s = _lib.Solver(gs, arr, params)
    bt = torch.as_tensor(b, device="cuda")
    hist = [s.gpair_step(bt) for _ in range(iters)]
    x = s.gpair_solver_image().cpu().numpy()
    s.close()
    return x, np.array([h[0] for h in hist]), np.array([h[1] for h in hist])


def test_adam_npc_cawr_matches_oracle(problem):
    w, G, b = problem
    iters, eta = 20, 0.05
    p = _lib.StepParams(rule=_lib.RULE_ADAM, npc=1, npc_eps=1e-8, eta_max=eta, eta_min=0.0, T0=iters,
                        T_mult=1.0, adam_eps=1e-20)
    x, loss, resid = _gpu_ir(w, b, iters, p)
    xo, lo, ro = oracle.ir(G, w.sensors, w.v, w.fs, w.t0, w.Nt, b, iters, k=w.k, rule="adam", npc=True,
                           npc_eps=1e-8, eta_max=eta, eta_min=0.0, T0=iters, adam_eps=1e-20)
    print("loss gpu", loss[[0, 5, 10, 19]], "oracle", lo[[0, 5, 10, 19]], "x rel", rel_l2(x, xo))
    assert loss[-1] < loss[0]
    # FP64 loss of the first iterate: the reduction itself, |y - b|^2 / N with y = F((0 + eps)^2)
    assert abs(loss[0] - lo[0]) <= 1e-6 * lo[0]
    assert np.max(np.abs(loss - lo) / lo) < 2e-3
    assert rel_l2(x, xo) < 2e-3


def test_cawr_restarts_and_resume_match_oracle(problem):
    """The device step schedule (CAWR step size and Adam's bias corrections, from the device step
    count) against the oracle's Algorithm 2 over 12 Adam steps with T0 = 3, T_mult = 2 and
    eta_min > 0, so that the step size restarts at t = 3 and t = 9 inside the run.  A second solver
    resumes from a checkpoint taken at t = 5 (set_state), continues on the graph-replay path, and
    must land on the same iterate as the oracle at t = 12."""
    w, G, b = problem
    iters, eta, eta_min = 12, 0.05, 0.005
    p = _lib.StepParams(rule=_lib.RULE_ADAM, npc=1, npc_eps=1e-8, eta_max=eta, eta_min=eta_min, T0=3,
                        T_mult=2.0, adam_eps=1e-20)
    x, loss, resid = _gpu_ir(w, b, iters, p)
    xo, lo, ro = oracle.ir(G, w.sensors, w.v, w.fs, w.t0, w.Nt, b, iters, k=w.k, rule="adam", npc=True,
                           npc_eps=1e-8, eta_max=eta, eta_min=eta_min, T0=3, Tmult=2.0, adam_eps=1e-20)
    assert [oracle.cawr(t, eta, eta_min, 3, 2.0) for t in (0, 3, 9)] == pytest.approx([eta] * 3)
    assert np.max(np.abs(loss - lo) / lo) < 2e-3
    assert rel_l2(x, xo) < 2e-3
    # checkpoint at t = 5, resumed in a fresh solver
    gs, arr = device_inputs(w)
    bt = torch.as_tensor(b, device="cuda")
    s1 = _lib.Solver(gs, arr, p)
    for _ in range(5):
        s1.gpair_step(bt, want_loss=False)
    z, m, v, t = s1.gpair_solver_get_state()
    s1.close()
    assert t == 5
    s2 = _lib.Solver(gs, arr, p)
    s2.gpair_solver_set_state(z, m, v, t)
    l5, _ = s2.gpair_step(bt)                   # the loss entering iteration 6 (index 5)
    s2.gpair_solver_steps(bt, iters - 6, want_loss=False)
    _, _, _, t2 = s2.gpair_solver_get_state()
    x2 = s2.gpair_solver_image().cpu().numpy()
    s2.close()
    assert t2 == iters
    assert abs(l5 - lo[5]) <= 2e-3 * lo[5]
    assert rel_l2(x2, xo) < 2e-3


def test_line_search_matches_oracle(problem):
    w, G, b = problem
    iters = 8
    p = _lib.StepParams(rule=_lib.RULE_GD_LINESEARCH, npc=0)
    x, loss, resid = _gpu_ir(w, b, iters, p)
    xo, lo, ro = oracle.ir(G, w.sensors, w.v, w.fs, w.t0, w.Nt, b, iters, k=w.k, rule="linesearch", npc=False)
    assert np.all(np.diff(loss) < 0)
    assert np.max(np.abs(resid - ro) / ro) < 1e-4
    assert rel_l2(x, xo) < 1e-3


def test_adam_on_assa_operator_matches_oracle(problem):
    """gpair_step with the discretised operator (op = ASSA, Algorithm 1) against the oracle's
    Algorithm 2 built on its own ASSA forward and adjoint."""
    w, G, b = problem
    iters, eta = 20, 0.05
    p = _lib.StepParams(rule=_lib.RULE_ADAM, npc=1, npc_eps=1e-8, eta_max=eta, eta_min=0.0, T0=iters,
                        T_mult=1.0, adam_eps=1e-20, op=_lib.OP_ASSA, n_min=25)
    x, loss, resid = _gpu_ir(w, b, iters, p)
    xo, lo, ro = oracle.ir_assa(G, G.sigma[0], w.sensors, w.v, w.fs, w.t0, w.Nt, b, iters, n_min=25, rule="adam",
                                npc=True, npc_eps=1e-8, eta_max=eta, eta_min=0.0, T0=iters, adam_eps=1e-20)
    print("loss gpu", loss[[0, 5, 10, 19]], "oracle", lo[[0, 5, 10, 19]], "x rel", rel_l2(x, xo))
    assert loss[-1] < loss[0]
    assert abs(loss[0] - lo[0]) <= 1e-6 * lo[0]
    assert np.max(np.abs(loss - lo) / lo) < 2e-3
    assert rel_l2(x, xo) < 2e-3


def test_line_search_on_assa_operator_matches_oracle(problem):
    w, G, b = problem
    iters = 8
    p = _lib.StepParams(rule=_lib.RULE_GD_LINESEARCH, npc=0, op=_lib.OP_ASSA, n_min=25)
    x, loss, resid = _gpu_ir(w, b, iters, p)
    xo, lo, ro = oracle.ir_assa(G, G.sigma[0], w.sensors, w.v, w.fs, w.t0, w.Nt, b, iters, n_min=25,
                                rule="linesearch", npc=False)
    assert np.all(np.diff(loss) < 0)
    assert np.max(np.abs(resid - ro) / ro) < 1e-4
    assert rel_l2(x, xo) < 1e-3


def test_assa_solver_profile_records_its_kernels(problem):
    w, G, b = problem
    gs, arr = device_inputs(w)
    s = _lib.Solver(gs, arr, _lib.StepParams(op=_lib.OP_ASSA))
    bt = torch.as_tensor(b, device="cuda")
    s.gpair_solver_profile(True)
    for _ in range(3):
        s.gpair_step(bt, want_loss=False)
    ms, n = s.gpair_solver_timings()
    s.close()
    assert n == 3 and ms[0] > 0 and ms[1] > 0 and ms[2] >= ms[0] + ms[1]


def test_checkpoint_resume(problem):
    w, G, b = problem
    p = _lib.StepParams(rule=_lib.RULE_ADAM, npc=1, eta_max=0.02, T0=20, adam_eps=1e-20)
    gs, arr = device_inputs(w)
    bt = torch.as_tensor(b, device="cuda")
    s1 = _lib.Solver(gs, arr, p)
    for _ in range(6):
        s1.gpair_step(bt, want_loss=False)
    z, m, v, t = s1.gpair_solver_get_state()
    for _ in range(4):
        s1.gpair_step(bt, want_loss=False)
    xa = s1.gpair_solver_image().cpu().numpy()
    s2 = _lib.Solver(gs, arr, p)
    s2.gpair_solver_set_state(z, m, v, t)
    for _ in range(4):
        s2.gpair_step(bt, want_loss=False)
    xb = s2.gpair_solver_image().cpu().numpy()
    assert t == 6
    assert rel_l2(xb, xa) < 1e-5
    s1.close()
    s2.close()


def test_reduce_f64_against_numpy():
    rng = np.random.default_rng(0)
    a = rng.normal(size=1_000_003).astype(np.float32)
    bb = rng.normal(size=a.size).astype(np.float32)
    c = rng.normal(size=a.size).astype(np.float32)
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    _lib.gpair_reduce_f64(torch.as_tensor(a, device="cuda"), torch.as_tensor(bb, device="cuda"),
                          torch.as_tensor(c, device="cuda"), out)
    o = out.cpu().numpy()
    ref0 = float(np.sum((a.astype(np.float64) - bb) ** 2))
    ref1 = float(np.sum(a.astype(np.float64) * c))
    assert abs(o[0] - ref0) <= 1e-12 * ref0
    assert abs(o[1] - ref1) <= 1e-12 * np.sum(np.abs(a.astype(np.float64) * c))


def test_bounded_wait_times_out_and_context_survives():
    """Failure detection without a fault: a device wait that nothing completes gives up after its
    bound, the host reads the timeout from the status word, and the next operator call runs
    normally on the same context."""
    import torch

    from gpair_testutil import gpu_forward

    assert _lib.gpair_last_device_status() == 0
    _lib.gpair_wait_selftest(4096)
    torch.cuda.synchronize()
    assert _lib.gpair_last_device_status() == 4            # GPAIR_ERR_TIMEOUT
    assert _lib.gpair_last_device_status() == 0            # reading clears the word
    w = synth.tiny(1)
    assert np.abs(gpu_forward(w)).max() > 0
    with pytest.raises(_lib.GpairError):
        _lib.gpair_wait_selftest(0)                         # rejected on the host, nothing launched



def test_paper_scale_first_step_in_the_benchmark_configuration():
    """gpair_step on the benchmark's problem (8.4 M Gaussians, 1024 x 4096 data) from z = 0.
    With NPC, x0 = eps^2 ~ 1e-16, so y0 ~ 0, the entering loss is |b|^2 / N, and the latent
    gradient is g_z = 2 eps F^T (-2 b / N) to relative 1e-12.  The oracle computes it for 2000
    sampled Gaussians and applies its own Adam (first step, bias-corrected: close to -eta sign(g_z),
    less by the fraction adam_eps / |g_z|).  Entries are compared where |g_z| is at least 1e-3 of
    the sample's RMS, where the GPU's relative 1e-4 gradient error changes the step by < 1e-4."""
    w = synth.paper_scale(3)
    rng = np.random.default_rng(51)
    b = rng.normal(size=(w.Nd, w.Nt)).astype(np.float32)
    eta = 0.02
    p = _lib.StepParams(rule=_lib.RULE_ADAM, npc=1, npc_eps=1e-8, eta_max=eta, eta_min=0.0, T0=10, T_mult=1.0,
                        adam_eps=1e-20)
    gs, arr = device_inputs(w)
    s = _lib.Solver(gs, arr, p)
    bt = torch.as_tensor(b, device="cuda")
    loss0, resid0 = s.gpair_step(bt)
    z1, _, _, t = s.gpair_solver_get_state()
    z1 = z1.cpu().numpy()
    s.close()
    N = w.Nd * w.Nt
    bb = float(np.sum(b.astype(np.float64) ** 2))
    assert t == 1
    assert abs(loss0 - bb / N) <= 1e-6 * bb / N
    assert abs(resid0 - np.sqrt(bb)) <= 1e-6 * np.sqrt(bb)
    idx = np.sort(rng.choice(w.M, 2000, replace=False))
    G = oracle_gaussians(w, A=np.ones(w.M, np.float32))
    Gs = oracle.Gaussians(G.c[idx], G.sigma[idx], G.A[idx])
    gx = oracle.adjoint(Gs, w.sensors, w.v, w.fs, w.t0, w.Nt, -2.0 * b.astype(np.float64) / N, k=w.k)["A"]
    gz = np.ascontiguousarray(gx * 2.0 * (0.0 + 1e-8))
    z, m, v = np.zeros(gz.size), np.zeros(gz.size), np.zeros(gz.size)
    oracle.adam(z, m, v, gz, 1, oracle.cawr(0, eta, 0.0, 10), eps=1e-20)
    sure = np.abs(gz) >= 1e-3 * np.sqrt(np.mean(gz * gz))
    assert sure.sum() > 1500
    assert np.all(np.abs(np.abs(z[sure]) - eta) < 0.05 * eta)
    np.testing.assert_allclose(z1[idx][sure], z[sure], rtol=1e-4, atol=0)


@pytest.mark.parametrize("kind", ["adam", "linesearch", "assa", "vcr"])
def test_graph_replayed_steps_equal_single_steps(problem, kind):
    """gpair_solver_steps (one step captured as a CUDA graph, replayed) gives the iterates of the
    same number of gpair_step calls; the step counter and a checkpoint set between the two paths
    carry over.  The launches are the same; the forward's within-bin order (atomic ranks) makes
    two runs agree to FP32 rounding rather than bit for bit."""
    w, G, b = problem
    kw = dict(rule=_lib.RULE_ADAM, npc=1, eta_max=0.03, T0=5, T_mult=2.0, adam_eps=1e-20)
    if kind == "linesearch":
        kw = dict(rule=_lib.RULE_GD_LINESEARCH, npc=0)
    elif kind == "assa":
        kw.update(op=_lib.OP_ASSA, n_min=25)
    elif kind == "vcr":
        kw.update(vcr_lambda=1e-6, vcr_beta=0.5)
    p = _lib.StepParams(**kw)
    gs, arr = device_inputs(w)
    bt = torch.as_tensor(b, device="cuda")
    s1, s2 = _lib.Solver(gs, arr, p), _lib.Solver(gs, arr, p)
    losses = [s1.gpair_step(bt)[0] for _ in range(7)]
    l2, _ = s2.gpair_solver_steps(bt, 3)
    l2b, _ = s2.gpair_solver_steps(bt, 4)
    z1, m1, v1, t1 = s1.gpair_solver_get_state()
    z2, m2, v2, t2 = s2.gpair_solver_get_state()
    assert t1 == t2 == 7
    for a, c in ((z1, z2), (m1, m2), (v1, v2)):
        assert rel_l2(c.cpu().numpy(), a.cpu().numpy()) < 1e-5
    assert abs(l2 - losses[2]) <= 1e-6 * losses[2] and abs(l2b - losses[6]) <= 1e-6 * losses[6]
    # a checkpoint taken on the step path resumes on the graph path
    s3 = _lib.Solver(gs, arr, p)
    s3.gpair_solver_set_state(z1, m1, v1, t1)
    s1.gpair_step(bt)
    s3.gpair_solver_steps(bt, 1)
    za, _, _, _ = s1.gpair_solver_get_state()
    zb, _, _, tb = s3.gpair_solver_get_state()
    assert tb == 8 and rel_l2(zb.cpu().numpy(), za.cpu().numpy()) < 1e-5
    for s in (s1, s2, s3):
        s.close()


@pytest.mark.parametrize("kind", ["step", "steps"])
def test_captured_state_and_captured_steps_mix_with_eager_ones(problem, kind):
    """A set_state recorded in a graph changes the iterate when the graph runs, not when it is recorded, and so do
    recorded steps: whatever comes after works on the iterate that the device then has.  Losses of the
    iterates tell which amplitudes a step used."""
    w, G, b = problem
    p = _lib.StepParams(rule=_lib.RULE_ADAM, npc=1, eta_max=0.03, T0=50, adam_eps=1e-20)
    gs, arr = device_inputs(w)
    bt = torch.as_tensor(b, device="cuda")
    z0 = torch.as_tensor(np.random.default_rng(5).uniform(0.2, 1.0, w.M).astype(np.float32), device="cuda")
    zero = torch.zeros_like(z0)

    def eager(s):
        return s.gpair_step(bt)[0] if kind == "step" else s.gpair_solver_steps(bt, 1)[0]

    ref = _lib.Solver(gs, arr, p)
    ref.gpair_solver_set_state(z0, zero, zero, 0)
    want = [eager(ref) for _ in range(3)]
    z_ref = ref.gpair_solver_get_state()[0]
    s = _lib.Solver(gs, arr, p)
    eager(s)
    graph, steps = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s.gpair_solver_set_state(z0, zero, zero, 0)
    eager(s)
    graph.replay()
    got = [eager(s)]
    with torch.cuda.graph(steps):
        s.gpair_step(bt, want_loss=False)
    graph.replay()                       # the recorded step has not run: back to z0
    steps.replay()
    got += [eager(s), eager(s)]
    z = s.gpair_solver_get_state()[0]
    assert np.allclose(got, want, rtol=1e-5), (got, want)
    assert rel_l2(z.cpu().numpy(), z_ref.cpu().numpy()) < 1e-5
    ref.close()
    s.close()
