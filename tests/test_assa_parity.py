"""The paper's discretised operator (adaptive supersampling alignment, Algorithm 1): CUDA path
through the C ABI against the FP64 oracle's three-stage evaluation, element by element.

Snapping a time of flight to the fine grid is an integer decision taken from an FP32 phase on the
GPU and an FP64 distance in the oracle; pairs within TAU_SNAP fine samples of a rounding tie may
go either way, and the oracle bounds what either choice changes (`amb`).  Tolerances: signals
relative L2 1e-5, gradients 1e-4, each plus that bound."""
import os

import numpy as np
import pytest

import oracle
from gpair_testutil import device_inputs, oracle_gaussians, rel_l2
from paper_2602_03893_gb300 import synth

pytestmark = pytest.mark.gpu

TAU_SNAP = 1e-4      # fine samples; the FP32 phase resolves ~1e-6 of one


@pytest.fixture(scope="module", autouse=True)
def _threads():
    oracle.set_threads(os.cpu_count() or 1)


def gpu_assa_forward(w, A=None, n_min=25):
    import torch

    from paper_2602_03893_gb300 import _lib

    gs, arr = device_inputs(w, A)
    y = torch.full((w.Nd, w.Nt), float("nan"), device="cuda")
    _lib.gpair_assa_forward(gs, arr, y, n_min=n_min)
    torch.cuda.synchronize()
    assert _lib.gpair_last_device_status() == 0
    return y.cpu().numpy()


def gpu_assa_adjoint(w, delta, A=None, n_min=25):
    import torch

    from paper_2602_03893_gb300 import _lib

    gs, arr = device_inputs(w, A)
    d = torch.as_tensor(np.ascontiguousarray(delta, dtype=np.float32), device="cuda")
    gA = torch.full((w.M,), float("nan"), device="cuda")
    _lib.gpair_assa_adjoint(gs, arr, d, gA, n_min=n_min)
    torch.cuda.synchronize()
    return gA.cpu().numpy()


def _check_forward(w, A=None, n_min=25, sensors_idx=None, tol=1e-5):
    G = oracle_gaussians(w, A)
    sens = w.sensors if sensors_idx is None else w.sensors[sensors_idx]
    y_ora, amb = oracle.assa_forward(G, G.sigma[0], sens, w.v, w.fs, w.t0, w.Nt, n_min=n_min, tau=TAU_SNAP,
                                     want_amb=True)
    y = gpu_assa_forward(w, A, n_min)
    if sensors_idx is not None:
        y = y[sensors_idx]
    assert np.all(np.isfinite(y))
    err = np.linalg.norm(y - y_ora)
    assert np.abs(y_ora).max() > 0
    assert err <= tol * np.linalg.norm(y_ora) + np.linalg.norm(amb), (err / np.linalg.norm(y_ora), np.linalg.norm(amb))
    return err / np.linalg.norm(y_ora)


def _dense(w, seed=8):
    return np.random.default_rng(seed).uniform(0.0, 1.0, w.M).astype(np.float32)


@pytest.mark.parametrize("n_min", [25, 101])
def test_tiny_forward(n_min):
    w = synth.tiny(1)
    _check_forward(w, n_min=n_min)
    _check_forward(w, A=_dense(w), n_min=n_min)


def test_tiny_adjoint_and_identity():
    w = synth.tiny(1)
    rng = np.random.default_rng(3)
    delta = rng.normal(size=(w.Nd, w.Nt)).astype(np.float32)
    G = oracle_gaussians(w)
    g_ora, amb = oracle.assa_adjoint(G, G.sigma[0], w.sensors, w.v, w.fs, w.t0, w.Nt, delta, tau=TAU_SNAP,
                                     want_amb=True)
    g = gpu_assa_adjoint(w, delta)
    assert np.all(np.isfinite(g))
    assert np.linalg.norm(g - g_ora) <= 1e-4 * np.linalg.norm(g_ora) + np.linalg.norm(amb)
    # <F x, d> = <x, F^T d> on the GPU itself
    x = _dense(w, 9)
    Fx = gpu_assa_forward(w, A=x).astype(np.float64)
    lhs, rhs = float(np.sum(Fx * delta)), float(x.astype(np.float64) @ g.astype(np.float64))
    assert abs(lhs - rhs) <= 1e-5 * np.linalg.norm(Fx) * np.linalg.norm(delta)


def test_ragged_grid_without_tma_and_time_origin():
    g = synth.centred_grid(13, 11, 7, 0.15e-3)
    A = np.random.default_rng(5).uniform(0.1, 1.0, g.M).astype(np.float32)
    w = synth.Workload("ragged", g, synth.cap_sensors(13, 12e-3, 170.0), 437, A=A, t0=6.4e-6)
    _check_forward(w)
    delta = np.random.default_rng(6).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    G = oracle_gaussians(w)
    g_ora, amb = oracle.assa_adjoint(G, G.sigma[0], w.sensors, w.v, w.fs, w.t0, w.Nt, delta, tau=TAU_SNAP,
                                     want_amb=True)
    gg = gpu_assa_adjoint(w, delta)
    assert np.linalg.norm(gg - g_ora) <= 1e-4 * np.linalg.norm(g_ora) + np.linalg.norm(amb)


def test_mid_sensor_subset():
    w = synth.mid(2)
    idx = np.random.default_rng(0).choice(w.Nd, 10, replace=False)
    _check_forward(w, A=_dense(w), sensors_idx=idx)


def test_paper_scale_full_launch_sampled_sensors():
    """The benchmark's configuration with a dense iterate-like image; the oracle recomputes 6
    sensors (the forward is separable per sensor)."""
    w = synth.paper_scale(3)
    x = (np.random.default_rng(1).uniform(0.0, 1.0, w.M) ** 2).astype(np.float32)
    _check_forward(w, A=x, sensors_idx=np.array([0, 137, 511, 600, 901, 1023]))


def test_free_gaussians_are_rejected():
    from paper_2602_03893_gb300 import _lib

    g = synth.centred_grid(4, 4, 4, 0.1e-3)
    w = synth.Workload("free", g, synth.cap_sensors(8, 10e-3, 120.0), 256,
                       free=synth.free_gaussians(g, 3, A=np.ones(g.M)))
    with pytest.raises(_lib.GpairError):
        gpu_assa_forward(w)


def test_sensor_inside_a_slab_box_and_wide_amplitude_range():
    """The band adds are 32-bit fixed point scaled per (slab, sensor) by the sensor's distance to
    the slab's box; a sensor inside the box keeps float adds.  Amplitudes spanning six decades
    check that rounding to 2^-19 of the largest scaled mass stays within the tolerance."""
    g = synth.centred_grid(16, 12, 8, 0.1e-3)
    rng = np.random.default_rng(12)
    A = (10.0 ** rng.uniform(-6.0, 0.0, g.M)).astype(np.float32)
    sens = synth.cap_sensors(12, 8e-3, 150.0)
    inside = np.array([[0.23e-3, -0.17e-3, 0.11e-3]], dtype=np.float32)     # within the grid's box
    w = synth.Workload("inside", g, np.concatenate([sens, inside]), 512, A=A)
    _check_forward(w, A=A)


def test_paper_scale_adjoint_sampled_gaussians():
    """The benchmark's launch (8.4 M Gaussians x 1024 sensors, alpha = 2); the oracle recomputes
    2000 sampled Gaussians' gradients over all sensors (each entry is independent)."""
    w = synth.paper_scale(3)
    rng = np.random.default_rng(13)
    delta = rng.normal(size=(w.Nd, w.Nt)).astype(np.float32)
    idx = np.sort(rng.choice(w.M, 2000, replace=False))
    g = gpu_assa_adjoint(w, delta)
    assert np.all(np.isfinite(g))
    G = oracle_gaussians(w)
    Gs = oracle.Gaussians(G.c[idx], G.sigma[idx], G.A[idx])
    g_ora, amb = oracle.assa_adjoint(Gs, G.sigma[0], w.sensors, w.v, w.fs, w.t0, w.Nt, delta, tau=TAU_SNAP,
                                     want_amb=True)
    assert np.linalg.norm(g[idx] - g_ora) <= 1e-4 * np.linalg.norm(g_ora) + np.linalg.norm(amb)


@pytest.mark.parametrize("nd", [11, 12, 33, 130])
@pytest.mark.parametrize("n_min", [1, 25, 61])
@pytest.mark.parametrize("sides", [(8, 8, 4), (17, 9, 10), (35, 20, 17)])
def test_few_sensors_and_slabs(sides, n_min, nd):
    """The last count with a warp to a sensor and the first with a lane to one, a group of 32 with a remainder; fine
    grids of alpha = 1, 2 and 4; one brick, ragged bricks, several slabs of 16; records that end early."""
    g = synth.centred_grid(*sides, 0.1e-3)
    w = synth.Workload("assa-few", g, synth.cap_sensors(nd, 15e-3, 150.0), 410, A=None)
    _check_forward(w, A=_dense(w), n_min=n_min)


def test_sensors_in_the_volume_and_large_amplitudes():
    """Sensors inside a slab's box have no bound on A / r: their lanes add floats beside the others' integers."""
    g = synth.centred_grid(20, 18, 9, 0.1e-3)
    xyz = synth.cap_sensors(40, 12e-3, 120.0)
    xyz[::7] = (np.array([0.21, -0.33, 0.08]) * 1e-3 + np.arange(6)[:, None] * 1.7e-5).astype(np.float32)
    w = synth.Workload("assa-in", g, xyz, 400, A=None)
    _check_forward(w, A=_dense(w) * 1e6)


def test_sparse_slabs():
    """Slabs and bricks without amplitudes."""
    g = synth.centred_grid(40, 33, 40, 0.1e-3)
    A = np.zeros(g.M, np.float32)
    A[np.random.default_rng(3).choice(g.M, 25, replace=False)] = 1.0
    _check_forward(synth.Workload("assa-sparse", g, synth.cap_sensors(40, 20e-3, 120.0), 900, A=None), A=A)


@pytest.mark.parametrize("sides,h,sigma,n_min,off,shells",
                         [((16, 16, 16), 1e-4, 1e-4, 513, 2.0, 1), ((35, 20, 17), 1e-4, 1e-4, 513, 4.0, 1),
                          ((16, 16, 16), 1.2e-5, 1.2e-5, 513, 0.25, 1), ((16, 16, 16), 2.4e-5, 2.4e-5, 129, 2.0, 24)])
def test_lattice_far_from_the_origin(sides, h, sigma, n_min, off, shells):
    """Fine grids of alpha = 32 and 256, lattices so far out that the slabs' boxes, widened by a part of their
    coordinates, start several fine samples before the nearest node: the farthest nodes' masses, seen along
    the diagonals of two bricks, stay in the band.  Only nodes at the bricks' corners have amplitudes."""
    g = synth.centred_grid(*sides, h, sigma=sigma, centre=(off, -off, off))
    ix, iy, iz = (np.arange(n) for n in sides)
    at = [(np.isin(q % b, (0, b - 1)) | (q == n - 1)) for q, b, n in ((iz, 4, sides[2]), (iy, 8, sides[1]), (ix, 8, sides[0]))]
    A = (at[0][:, None, None] & at[1][None, :, None] & at[2][None, None, :]).astype(np.float32).ravel()
    d = np.array([[7.0 * x, 7.0 * y, 3.0 * z] for x in (-1, 1) for y in (-1, 1) for z in (-1, 1)])
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    o = np.array([g.ox, g.oy, g.oz])
    xyz = np.concatenate([o + np.array([4.0, 4.0, 2.0]) * h * (2 * q + 1) + (10e-3 + 1e-5 * r) * d
                          for q in (0, 1) for r in range(shells)])
    w = synth.Workload("assa-far", g, xyz.astype(np.float32), 400, A=A)
    _check_forward(w, A=A, n_min=n_min)


@pytest.mark.parametrize("nd", [33, 65, 230])
@pytest.mark.parametrize("n_min", [1, 25, 61, 101, 257])
@pytest.mark.parametrize("sides", [(35, 20, 17), (40, 24, 40)])
def test_lanes_and_the_other_kernel(sides, n_min, nd):
    """On both sides of the rules that choose the kernel: 150 to 192 and more warps, fine grids of alpha = 1 to 16
    whose bands leave room for many and for few warps, slabs of one and of several bricks."""
    g = synth.centred_grid(*sides, 0.1e-3)
    w = synth.Workload("assa-rules", g, synth.cap_sensors(nd, 15e-3, 150.0), 410, A=None)
    _check_forward(w, A=_dense(w), n_min=n_min)


def test_lanes_with_sensors_in_the_volume():
    """Lanes without a bound on A / r beside lanes with one, and a brick without amplitudes."""
    g = synth.centred_grid(24, 24, 12, 0.1e-3)
    xyz = synth.cap_sensors(300, 12e-3, 120.0)
    xyz[::29] = (np.array([0.21, -0.33, 0.08]) * 1e-3 + np.arange(len(xyz[::29]))[:, None] * 1.7e-5).astype(np.float32)
    w = synth.Workload("assa-in-lanes", g, xyz, 400, A=None)
    A = _dense(w) * 1e6
    A.reshape(12, 24, 24)[:4, :8, :8] = 0.0
    _check_forward(w, A=A)


@pytest.mark.parametrize("nd", [1, 15, 16, 33, 63, 130])
@pytest.mark.parametrize("n_min", [1, 25, 61])
@pytest.mark.parametrize("sides", [(3, 2, 1), (17, 9, 10), (62, 55, 31)])
def test_adjoint_few_tiles(sides, n_min, nd):
    """One, two, four and eight CTAs to a brick's sensors, counts that leave the last CTA short; fine grids of alpha =
    1, 2 and 4 whose residual is correlated residue by residue; records that end before the last windows."""
    g = synth.centred_grid(*sides, 0.1e-3)
    w = synth.Workload("assa-adj-few", g, synth.cap_sensors(nd, 15e-3, 150.0), 405, A=np.ones(g.M, np.float32))
    delta = np.random.default_rng(nd).normal(size=(w.Nd, w.Nt)).astype(np.float32)
    idx = np.sort(np.random.default_rng(7).choice(w.M, min(w.M, 1500), replace=False))
    G = oracle_gaussians(w)
    Gs = oracle.Gaussians(G.c[idx], G.sigma[idx], G.A[idx])
    g_ora, amb = oracle.assa_adjoint(Gs, G.sigma[0], w.sensors, w.v, w.fs, w.t0, w.Nt, delta, n_min=n_min, tau=TAU_SNAP,
                                     want_amb=True)
    gg = gpu_assa_adjoint(w, delta, n_min=n_min)
    assert np.all(np.isfinite(gg))
    assert np.linalg.norm(gg[idx] - g_ora) <= 1e-4 * np.linalg.norm(g_ora) + np.linalg.norm(amb)


def test_short_of_memory_takes_the_plan_with_fewer_rows():
    """The benchmark's size with 640 MB left on the device: the lanes' rows (784 MB) do not fit, the other kernel's do,
    in the operator and in a solver.  Signals against the oracle at this file's tolerance; the solver's first loss
    against that of the signals themselves (data 0: the mean of their squares), which two forwards within 1e-5 of the
    exact one give to 4e-5."""
    import torch

    from paper_2602_03893_gb300 import _lib

    w = synth.paper_scale(3)
    x = (np.random.default_rng(1).uniform(0.0, 1.0, w.M) ** 2).astype(np.float32)
    gs, arr = device_inputs(w, A=x)
    y, zero = (torch.zeros((w.Nd, w.Nt), device="cuda") for _ in range(2))
    p = _lib.StepParams(rule=_lib.RULE_ADAM, npc=0, op=_lib.OP_ASSA)

    def loss():
        s = _lib.Solver(gs, arr, p)
        try:
            s.gpair_solver_set_state(gs.A, t=0)
            return s.gpair_step(zero)[0]
        finally:
            s.close()

    _lib.gpair_assa_forward(gs, arr, y)
    loss()                                               # every kernel is loaded
    _lib.gpair_release_scratch()
    torch.cuda.empty_cache()
    left = 640 << 20
    hog = []
    try:
        while True:                                     # in pieces: the driver rounds large blocks up
            free = torch.cuda.mem_get_info()[0]
            if free <= left + (64 << 20):
                break
            hog.append(torch.empty(max(free - left - (32 << 20), 32 << 20) // 4 * 4, dtype=torch.uint8, device="cuda"))
        y.fill_(float("nan"))
        _lib.gpair_assa_forward(gs, arr, y)
        torch.cuda.synchronize()
        assert _lib.gpair_last_device_status() == 0
        _lib.gpair_release_scratch()
        got = loss()
    finally:
        hog.clear()
        _lib.gpair_release_scratch()
        torch.cuda.empty_cache()
    want = float((y.double() ** 2).mean())
    assert abs(got - want) <= 4e-5 * want
    idx = np.array([0, 137, 511, 600, 901, 1023])
    G = oracle_gaussians(w, x)
    y_ora, amb = oracle.assa_forward(G, G.sigma[0], w.sensors[idx], w.v, w.fs, w.t0, w.Nt, n_min=25, tau=TAU_SNAP,
                                     want_amb=True)
    err = np.linalg.norm(y.cpu().numpy()[idx] - y_ora)
    assert err <= 1e-5 * np.linalg.norm(y_ora) + np.linalg.norm(amb)
