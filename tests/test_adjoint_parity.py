"""Adjoint and parameter gradients: CUDA path against the FP64 oracle (relative L2 1e-4 plus
the weight of window-ambiguous terms), and the adjoint identity on the GPU itself."""
import os

import numpy as np
import pytest

import oracle
from gpair_testutil import TAU, edge_workload, gpu_adjoint, gpu_forward, oracle_gaussians, rel_l2
from paper_2602_03893_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _threads():
    oracle.set_threads(os.cpu_count() or 1)


def _assert_grad(g_gpu, g_ora, amb, tol=1e-4):
    g_gpu = np.asarray(g_gpu, np.float64)
    assert np.all(np.isfinite(g_gpu))
    err = np.linalg.norm(g_gpu - g_ora)
    bound = tol * np.linalg.norm(g_ora) + np.linalg.norm(amb)
    assert err <= bound, f"rel err {err / np.linalg.norm(g_ora):.3e}"
    return err / np.linalg.norm(g_ora)


def _check(w, delta, full, k=None, A=None, gauss_idx=None):
    k = w.k if k is None else k
    out = gpu_adjoint(w, delta, full, A=A, k=k)
    G = oracle_gaussians(w, A)
    if gauss_idx is not None:
        G = oracle.Gaussians(G.c[gauss_idx], G.sigma[gauss_idx], G.A[gauss_idx])
    ref = oracle.adjoint(G, w.sensors, w.v, w.fs, w.t0, w.Nt, delta, k=k,
                         want=("A", "c", "sigma") if full else ("A",), tau=TAU, want_amb=True)
    pick = (lambda a: a) if gauss_idx is None else (lambda a: a[..., gauss_idx])
    rels = {"A": _assert_grad(pick(out["A"]), ref["A"], ref["ambA"])}
    if full:
        rels["c"] = _assert_grad(pick(out["c"]), ref["c"], ref["ambC"])
        rels["sigma"] = _assert_grad(pick(out["sigma"]), ref["sigma"], ref["ambS"])
    return rels


@pytest.mark.parametrize("k", [3.0, 6.0])
def test_tiny_amplitude_gradient(k):
    w = synth.tiny(1)
    delta = np.random.default_rng(2).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    _check(w, delta, full=False, k=k)


@pytest.mark.parametrize("sigma_scale", [1.01, 1.02])
def test_window_edge_position_in_and_out_of_expansion(sigma_scale):
    w = edge_workload(sigma_scale)
    delta = np.random.default_rng(12).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    _check(w, delta, full=False, A=w.A)


@pytest.mark.parametrize("h", [0.2e-3, 0.08e-3])
def test_moment_expansion_with_seven_and_eight_terms(h):
    g = synth.centred_grid(16, 16, 12, h)
    A = np.random.default_rng(13).uniform(0.0, 1.0, g.M).astype(np.float32)
    w = synth.Workload("terms", g, synth.cap_sensors(64, 20e-3, 160.0), 1024, A=A)
    delta = np.random.default_rng(14).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    _check(w, delta, full=False, A=w.A)


def test_adjoint_identity_on_gpu():
    w = synth.tiny(1)
    rng = np.random.default_rng(4)
    x = rng.uniform(0, 1, w.M).astype(np.float32)
    delta = rng.normal(size=(w.Nd, w.Nt)).astype(np.float32)
    Fx = gpu_forward(w, A=x).astype(np.float64)
    FTd = gpu_adjoint(w, delta, False)["A"].astype(np.float64)
    lhs, rhs = float(np.sum(Fx * delta)), float(x.astype(np.float64) @ FTd)
    assert abs(lhs - rhs) <= 1e-5 * np.linalg.norm(Fx) * np.linalg.norm(delta)


@pytest.mark.parametrize("k", [3.0, 6.0])
def test_free_gaussians_full_gradient(k):
    g = synth.centred_grid(16, 16, 12, 0.1e-3)
    free = synth.free_gaussians(g, 41, A=np.random.default_rng(6).uniform(0.2, 1.0, g.M))
    w = synth.Workload("free-grad", g, synth.cap_sensors(48, 25e-3, 170.0), 2048, free=free)
    delta = np.random.default_rng(7).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    _check(w, delta, full=True, k=k)


def test_grid_full_gradient_ragged():
    g = synth.centred_grid(13, 9, 6, 0.15e-3)
    A = np.random.default_rng(9).uniform(0.1, 1.0, g.M).astype(np.float32)
    w = synth.Workload("ragged-grad", g, synth.cap_sensors(37, 15e-3, 160.0), 1501, A=A, t0=3.3e-6)
    delta = np.random.default_rng(10).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    _check(w, delta, full=True)


def test_paper_scale_full_launch_sampled_gaussians():
    """The benchmark's launch (8.4 M Gaussians x 1024 sensors); 3000 sampled Gaussians are
    recomputed by the oracle over all sensors (each gradient entry is independent)."""
    w = synth.paper_scale(3)
    rng = np.random.default_rng(11)
    delta = rng.normal(size=(w.Nd, w.Nt)).astype(np.float32)
    idx = np.sort(rng.choice(w.M, 3000, replace=False))
    rels = _check(w, delta, full=False, gauss_idx=idx)
    assert rels["A"] < 1e-4


@pytest.mark.parametrize("nd", [1, 15, 16, 33, 97, 130])
@pytest.mark.parametrize("sides", [(3, 2, 1), (11, 9, 6)])
def test_moment_adjoint_few_tiles(nd, sides):
    """One to eight CTAs share a brick's sensors: a lone sensor, the last count without a split, counts that
    leave the last CTA short, and chunks of 64 with a remainder; records that end before the last windows."""
    g = synth.centred_grid(*sides, 0.1e-3)
    w = synth.Workload("few", g, synth.cap_sensors(nd, 15e-3, 150.0), 405, A=np.ones(g.M, np.float32))
    delta = np.random.default_rng(nd).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    _check(w, delta, full=False, A=w.A)


@pytest.mark.parametrize("assa", [False, True])
@pytest.mark.parametrize("nd", [3, 130])
def test_sensor_on_a_node_with_a_record_that_begins_later(assa, nd):
    """Sensors on lattice nodes add nothing to the nodes' gradients where their records do not reach back to the
    time of flight 0; the parts of the others stay.  Coordinates that are exact in FP32, so that the distance of
    node and sensor comes out as 0, or its square just below it."""
    import torch
    from gpair_testutil import device_inputs
    from paper_2602_03893_gb300 import _lib

    h = 2.0 ** -13
    g = synth.Grid(17, 9, 10, h, h, 0.0, 0.0, 0.0)
    on = np.random.default_rng(1).choice(g.M, 40, replace=False)
    nodes = (np.stack([on % g.nx, on // g.nx % g.ny, on // (g.nx * g.ny)], axis=1) + 0.5) * h
    far = synth.cap_sensors(nd, 12e-3, 140.0) + np.float32(1e-3)
    xyz = np.concatenate([nodes, far]).astype(np.float32)
    w = synth.Workload("on-a-node", g, xyz, 400, A=np.ones(g.M, np.float32), t0=4e-6)
    delta = np.random.default_rng(nd).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    # 4 us is 6 mm, beyond the lattice: these sensors see nothing of it
    wf = synth.Workload("far", g, xyz[40:], 400, A=w.A, t0=4e-6)

    def grad(work, d):
        if not assa:
            return gpu_adjoint(work, d, False, A=work.A)["A"]
        gs, arr = device_inputs(work)
        gA = torch.full((work.M,), float("nan"), device="cuda")
        _lib.gpair_assa_adjoint(gs, arr, torch.as_tensor(d, device="cuda"), gA)
        return gA.cpu().numpy()

    got, want = grad(w, delta), grad(wf, np.ascontiguousarray(delta[40:]))
    assert np.all(np.isfinite(got)), np.flatnonzero(~np.isfinite(got))
    # the same terms, summed in chunks of 32 that begin elsewhere
    assert rel_l2(got, want) < 1e-6


@pytest.mark.parametrize("sides,nds", [((35, 33, 18), (31, 64, 70)), ((50, 44, 30), (40, 130)), ((62, 55, 31), (15, 16, 130)),
                                       ((60, 60, 47), (299, 300, 512))])
def test_moment_adjoint_more_tiles(sides, nds):
    """The rule that divides a brick's sensors over CTAs, at its lines: 125, 336, 448 and 768 bricks."""
    for nd in nds:
        g = synth.centred_grid(*sides, 0.1e-3)
        w = synth.Workload("more", g, synth.cap_sensors(nd, 15e-3, 150.0), 605, A=np.ones(g.M, np.float32))
        delta = np.random.default_rng(nd).normal(size=(w.Nd, w.Nt)).astype(np.float32)
        _check(w, delta, full=False, gauss_idx=np.sort(np.random.default_rng(7).choice(w.M, 400, replace=False)))
