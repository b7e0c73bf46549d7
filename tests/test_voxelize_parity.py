"""Voxelisation (Eq. 2 sampled on a grid): CUDA path against the FP64 oracle, relative L2 1e-4."""
import numpy as np
import pytest
import torch

import oracle
from gpair_testutil import device_inputs, oracle_gaussians, rel_l2
from paper_2602_03893_gb300 import _lib, synth

pytestmark = pytest.mark.gpu


def _gpu_vox(w, og: synth.Grid, k):
    gs, _ = device_inputs(w)
    vol = torch.full((og.nz, og.ny, og.nx), float("nan"), device="cuda")
    _lib.gpair_voxelize(gs, _lib.Grid(og.nx, og.ny, og.nz, og.ox, og.oy, og.oz, og.h, og.sigma), k, vol)
    torch.cuda.synchronize()
    return vol.cpu().numpy()


def _ora_vox(w, og, k):
    return oracle.voxelize(oracle_gaussians(w), k, og.nx, og.ny, og.nz, og.ox, og.oy, og.oz, og.h)


@pytest.mark.parametrize("k", [3.0, 2.0])
def test_lattice_tiny(k):
    w = synth.tiny(1)
    v = _gpu_vox(w, w.grid, k)
    assert rel_l2(v, _ora_vox(w, w.grid, k)) < 1e-4


def test_lattice_mid():
    w = synth.mid(2)
    v = _gpu_vox(w, w.grid, 3.0)
    assert rel_l2(v, _ora_vox(w, w.grid, 3.0)) < 1e-4


def test_lattice_ragged_dims():
    g = synth.centred_grid(13, 7, 5, 0.1e-3)
    A = np.random.default_rng(1).uniform(0, 1, g.M).astype(np.float32)
    w = synth.Workload("ragged", g, synth.cap_sensors(1, 5e-3, 10.0), 16, A=A)
    assert rel_l2(_gpu_vox(w, g, 3.0), _ora_vox(w, g, 3.0)) < 1e-4


@pytest.mark.parametrize("k", [1.5, 4.2, 5.5, 6.0, 7.5])
def test_lattice_tap_counts_ragged(k):
    """Tap counts 1, 4, 5 and 6 a side (the fused three-axis kernel) and 7 (the separate passes)
    on a lattice whose sides are not multiples of the fused kernel's 32 x 8 x 16 block."""
    g = synth.centred_grid(37, 19, 21, 0.1e-3)
    A = np.random.default_rng(4).uniform(0, 1, g.M).astype(np.float32)
    w = synth.Workload("ragged-taps", g, synth.cap_sensors(1, 5e-3, 10.0), 16, A=A)
    assert rel_l2(_gpu_vox(w, g, k), _ora_vox(w, g, k)) < 1e-4


def test_free_gaussians_scatter_path():
    g = synth.centred_grid(24, 20, 16, 0.1e-3)
    free = synth.free_gaussians(g, 3, A=np.random.default_rng(2).uniform(0, 1, g.M))
    w = synth.Workload("free", g, synth.cap_sensors(1, 5e-3, 10.0), 16, free=free)
    og = synth.centred_grid(30, 26, 20, 0.08e-3)
    assert rel_l2(_gpu_vox(w, og, 3.0), _ora_vox(w, og, 3.0)) < 1e-4


def test_grid_gaussians_onto_other_grid():
    w = synth.tiny(1)
    og = synth.centred_grid(20, 18, 22, 0.15e-3)
    assert rel_l2(_gpu_vox(w, og, 3.0), _ora_vox(w, og, 3.0)) < 1e-4


def test_lattice_paper_scale_sampled_crops():
    """The benchmark's call (256 x 256 x 128 Gaussians onto their own lattice, k = 3: three
    separable passes with 4-output runs and compile-time taps) against the oracle on 14 crops of
    6 x 6 x 6 voxels, including faces, edges and corners of the volume.  Each crop's oracle sum
    takes every Gaussian within k sigma of it (a lattice margin of 4 nodes at sigma = h)."""
    w = synth.paper_scale(3)
    g = w.grid
    A = (np.random.default_rng(31).uniform(0.0, 1.0, g.M) ** 2).astype(np.float32)
    ww = synth.Workload(w.name, g, w.sensors[:1], 16, A=A)
    v = _gpu_vox(ww, g, 3.0)
    rng = np.random.default_rng(32)
    C, R = 6, 4
    starts = [(0, 0, 0), (g.nx - C, g.ny - C, g.nz - C), (0, g.ny - C, 0), (g.nx - C, 0, g.nz // 2),
              (g.nx // 2, 0, 0), (0, g.ny // 2, g.nz - C)]
    starts += [tuple(int(rng.integers(0, n - C + 1)) for n in (g.nx, g.ny, g.nz)) for _ in range(8)]
    A3 = A.reshape(g.nz, g.ny, g.nx)
    for (x0, y0, z0) in starts:
        xa, ya, za = max(0, x0 - R), max(0, y0 - R), max(0, z0 - R)
        xb, yb, zb = min(g.nx, x0 + C + R), min(g.ny, y0 + C + R), min(g.nz, z0 + C + R)
        # the crop's Gaussians and voxels share one lattice whose origin is 0 (voxelization depends
        # on differences only), so that offsets of exactly k sigma stay exact ties, as on the full
        # lattice; the crop's interior then has every Gaussian that reaches it
        nx, ny, nz = xb - xa, yb - ya, zb - za
        Gs = oracle.gaussians_from_grid(nx, ny, nz, 0.0, 0.0, 0.0, g.h, g.sigma,
                                        np.ascontiguousarray(A3[za:zb, ya:yb, xa:xb]).reshape(-1))
        full = oracle.voxelize(Gs, 3.0, nx, ny, nz, 0.0, 0.0, 0.0, g.h)
        ref = full[z0 - za:z0 - za + C, y0 - ya:y0 - ya + C, x0 - xa:x0 - xa + C]
        got = v[z0:z0 + C, y0:y0 + C, x0:x0 + C]
        assert rel_l2(got, ref) < 1e-4, (x0, y0, z0, rel_l2(got, ref))


# One entry, a partial group of 32, the last set that is not sorted, the first that is, and two radix blocks;
# tiles of 8^3: a single voxel, whole tiles and remainders.
@pytest.mark.parametrize("M", [1, 33, 4096, 4097, 9001])
@pytest.mark.parametrize("dims", [(1, 1, 1), (16, 8, 24), (23, 9, 17), (40, 37, 33)])
def test_free_gaussians_tiles(M, dims):
    rng = np.random.default_rng(M + sum(dims))
    dx = 0.07e-3
    ext = np.array(dims) * dx
    c = ((rng.uniform(-0.7, 0.7, (M, 3))) * ext).astype(np.float32)      # some lie outside the volume
    sig = np.exp(rng.uniform(np.log(0.03e-3), np.log(0.2e-3), M)).astype(np.float32)
    A = rng.uniform(0, 1, M).astype(np.float32)
    A[::7] = 0.0
    gs = _lib.Gaussians(A=_cuda(A), cx=_cuda(c[:, 0]), cy=_cuda(c[:, 1]), cz=_cuda(c[:, 2]), sigma=_cuda(sig))
    o = [float(np.float32(-e / 2)) for e in ext]
    og = _lib.Grid(*dims, *o, dx, dx)
    vol = torch.full(dims[::-1], float("nan"), device="cuda")
    _lib.gpair_voxelize(gs, og, 3.0, vol)
    G = oracle.gaussians_from_soa(c[:, 0], c[:, 1], c[:, 2], sig, A)
    ref = oracle.voxelize(G, 3.0, *dims, *o, float(np.float32(dx)))
    got = vol.cpu().numpy()
    # a voxel at a box's edge may count on one side only: a term below e^-4.5 of its amplitude
    bad = np.abs(got - ref) > 1e-4 * max(1e-30, np.abs(ref).max())
    assert bad.mean() < 1e-3 and np.linalg.norm((got - ref)[~bad]) <= 1e-4 * np.linalg.norm(ref) + 1e-30


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_free_gaussians_not_finite_stay_in_their_box(value):
    """An amplitude that is not finite marks the voxels of its own box and no others of the tiles it meets."""
    dx, n = 1e-4, 24
    c = np.array([[0.5, 3.5, -2.5], [-6.5, 1.5, 2.5], [0.5, 0.5, 0.5]], np.float32) * np.float32(dx)
    A = np.array([1.0, value, 2.0], np.float32)
    sig = np.full(3, dx, np.float32)
    gs = _lib.Gaussians(A=_cuda(A), cx=_cuda(c[:, 0]), cy=_cuda(c[:, 1]), cz=_cuda(c[:, 2]), sigma=_cuda(sig))
    o = -n * dx / 2
    vol = torch.zeros((n, n, n), device="cuda")
    _lib.gpair_voxelize(gs, _lib.Grid(n, n, n, o, o, o, dx, dx), 2.5, vol)
    at = np.arange(n) - n / 2 + 0.5
    on = [np.abs(at - q) <= 2.5 for q in (-6.5, 1.5, 2.5)]
    box = on[2][:, None, None] & on[1][None, :, None] & on[0][None, None, :]
    assert np.array_equal(~np.isfinite(vol.cpu().numpy()), box)


def test_free_gaussians_captured():
    """A captured call (the scatter) gives the tiles' result."""
    rng = np.random.default_rng(5)
    M, n, dx = 300, 19, 1e-4
    c = (rng.uniform(-0.5, 0.5, (M, 3)) * n * dx).astype(np.float32)
    sig = rng.uniform(0.5e-4, 2e-4, M).astype(np.float32)
    gs = _lib.Gaussians(A=_cuda(rng.uniform(0, 1, M).astype(np.float32)), cx=_cuda(c[:, 0]), cy=_cuda(c[:, 1]),
                        cz=_cuda(c[:, 2]), sigma=_cuda(sig))
    og = _lib.Grid(n, n, n, -n * dx / 2, -n * dx / 2, -n * dx / 2, dx, dx)
    one, two = torch.empty((n, n, n), device="cuda"), torch.empty((n, n, n), device="cuda")
    _lib.gpair_voxelize(gs, og, 3.0, one)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _lib.gpair_voxelize(gs, og, 3.0, two)
    graph.replay()
    # the same terms in another order: 300 of them, in single precision
    assert torch.allclose(one, two, rtol=300 * 2.0 ** -23, atol=300 * 2.0 ** -23 * float(one.max()))


@pytest.mark.parametrize("dims", [(64, 16, 32), (65, 17, 5), (68, 15, 33), (4, 1, 1), (131, 40, 9)])
@pytest.mark.parametrize("k", [1.5, 3.0, 6.0])
def test_lattice_fused_tiles(dims, k):
    """Whole and ragged 64 x 16 tiles, rows of whole vectors and not, planes fewer and more than a CTA's."""
    g = synth.centred_grid(*dims, 0.1e-3)
    A = np.random.default_rng(4).uniform(0, 1, g.M).astype(np.float32)
    w = synth.Workload("tiles", g, synth.cap_sensors(1, 5e-3, 10.0), 16, A=A)
    assert rel_l2(_gpu_vox(w, g, k), _ora_vox(w, g, k)) < 1e-4


def _set(M, ext, lo, hi, seed, spread=0.55):
    rng = np.random.default_rng(seed)
    c = (rng.uniform(-spread, spread, (M, 3)) * np.asarray(ext)).astype(np.float32)      # some lie outside
    sig = np.exp(rng.uniform(np.log(lo), np.log(hi), M)).astype(np.float32)
    A = rng.uniform(0.2, 1, M).astype(np.float32)
    A[::11] = 0.0
    return c, sig, A


# Sides of the boxes in voxels (6 sigma / dx): all scattered by threads, on both sides of VOX_SMALL's 4, all listed; few
# enough for a warp to each box and enough for the tiles, in one super of 1024 and in several, with whole and ragged
# tiles; sets that go to the tiles as they are (4096 of them at most, M times the tiles up to 2^21).
@pytest.mark.parametrize("M,dims", [(5, (257, 40, 37)), (2048, (88, 80, 77)), (4096, (64, 64, 64)), (4097, (33, 24, 41)),
                                    (2100, (81, 81, 81)), (9000, (64, 17, 40)), (20000, (40, 64, 33))])
@pytest.mark.parametrize("lo,hi", [(1.0, 2.5), (3.0, 5.5), (6.0, 9.0), (2.0, 26.0)])
def test_free_gaussians_small_and_large_boxes(M, dims, lo, hi):
    dx = 0.07e-3
    ext = np.array(dims) * dx
    c, sig, A = _set(M, ext, lo * dx / 6, hi * dx / 6, M)
    gs = _lib.Gaussians(A=_cuda(A), cx=_cuda(c[:, 0]), cy=_cuda(c[:, 1]), cz=_cuda(c[:, 2]), sigma=_cuda(sig))
    o = [float(np.float32(-e / 2)) for e in ext]
    og = _lib.Grid(*dims, *o, dx, dx)
    ref = oracle.voxelize(oracle.gaussians_from_soa(c[:, 0], c[:, 1], c[:, 2], sig, A), 3.0, *dims, *o, float(np.float32(dx)))
    for _ in range(2):                       # the second call finds the first one's scratch
        vol = torch.full(dims[::-1], float("nan"), device="cuda")
        _lib.gpair_voxelize(gs, og, 3.0, vol)
        got = vol.cpu().numpy()
        # a voxel at a box's edge may count on one side only: a term below e^-4.5 of its amplitude
        bad = np.abs(got - ref) > 1e-4 * max(1e-30, np.abs(ref).max())
        assert bad.mean() < 1e-3 and np.linalg.norm((got - ref)[~bad]) <= 1e-4 * np.linalg.norm(ref) + 1e-30


@pytest.mark.parametrize("M", [40, 5000])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e38])
def test_free_gaussians_odd_values_by_either_path(M, value):
    """A few Gaussians with a centre, width or amplitude that is not finite (or not in voxel units) among others: by
    tiles of the set as it is and after the split, the volume of the captured call (all scattered)."""
    dx, n = 1e-4, 40
    c, sig, A = _set(M, [n * dx] * 3, 0.3e-4, 3e-4, 3)
    c[3, 0], A[8], c[9, 2] = value, value, -value
    gs = _lib.Gaussians(A=_cuda(A), cx=_cuda(c[:, 0]), cy=_cuda(c[:, 1]), cz=_cuda(c[:, 2]), sigma=_cuda(sig))
    og = _lib.Grid(n, n, n, -n * dx / 2, -n * dx / 2, -n * dx / 2, dx, dx)
    one, two = torch.empty((n, n, n), device="cuda"), torch.empty((n, n, n), device="cuda")
    _lib.gpair_voxelize(gs, og, 3.0, one)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _lib.gpair_voxelize(gs, og, 3.0, two)
    graph.replay()
    same = torch.isfinite(one) & torch.isfinite(two)
    assert torch.equal(torch.isfinite(one), torch.isfinite(two))
    assert torch.equal(torch.isnan(one), torch.isnan(two))
    lim = M * 2.0 ** -23 * float(two[same].abs().max())
    assert float((one - two)[same].abs().max()) <= lim


def test_allocation_does_not_end_another_threads_capture():
    """A first call on a stream allocates its scratch while another thread records a graph."""
    import threading

    dx, n, M = 1e-4, 64, 20000
    c, sig, A = _set(M, [n * dx] * 3, 0.5e-4, 3e-4, 5)
    gs = _lib.Gaussians(A=_cuda(A), cx=_cuda(c[:, 0]), cy=_cuda(c[:, 1]), cz=_cuda(c[:, 2]), sigma=_cuda(sig))
    og = _lib.Grid(n, n, n, -n * dx / 2, -n * dx / 2, -n * dx / 2, dx, dx)
    vol, x = torch.empty((n, n, n), device="cuda"), torch.zeros(8, device="cuda")
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    err = []

    def call():
        try:
            _lib.gpair_voxelize(gs, og, 3.0, vol, stream=other)
        except Exception as e:               # noqa: BLE001 -- reported below, in the test's own thread
            err.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        x += 1
        t = threading.Thread(target=call)
        t.start()
        t.join()
        x += 1
    graph.replay()
    torch.cuda.synchronize()
    assert not err and float(x[0]) == 2.0
    ref = torch.empty_like(vol)
    _lib.gpair_voxelize(gs, og, 3.0, ref)
    assert torch.allclose(vol, ref, rtol=M * 2.0 ** -23, atol=M * 2.0 ** -23 * float(ref.max()))


def test_scratch_of_the_tiles_gives_way_to_other_calls():
    """A set of eight million leaves 370 MB of scratch on its stream; with 150 MB left on the device, a call that needs
    300 MB has it."""
    rng = np.random.default_rng(2)
    M, n, dx = 8_000_000, 256, 1e-4
    u = lambda lo, hi: _cuda(rng.uniform(lo, hi, M).astype(np.float32))
    gs = _lib.Gaussians(A=u(0.2, 1), cx=u(0, n * dx), cy=u(0, n * dx), cz=u(0, n * dx), sigma=u(2e-5, 3e-5))
    og = _lib.Grid(n, n, n, 0.0, 0.0, 0.0, dx, dx)
    vol = torch.empty((n, n, n), device="cuda")
    w = synth.Workload("long", synth.centred_grid(8, 8, 4, 1e-4), synth.cap_sensors(64, 12e-3, 140.0), 1 << 20)
    gl, arr = device_inputs(w, A=np.ones(w.M, np.float32))
    delta = torch.randn((w.Nd, w.Nt), device="cuda")
    want, got = torch.empty(w.M, device="cuda"), torch.empty(w.M, device="cuda")
    _lib.gpair_assa_adjoint(gl, arr, delta, want, n_min=1)
    _lib.gpair_release_scratch()
    _lib.gpair_voxelize(gs, og, 3.0, vol)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    left, hog = 150 << 20, []
    try:
        while True:
            free = torch.cuda.mem_get_info()[0]
            if free <= left + (64 << 20):
                break
            hog.append(torch.empty(max(free - left - (32 << 20), 32 << 20) // 4 * 4, dtype=torch.uint8, device="cuda"))
        _lib.gpair_assa_adjoint(gl, arr, delta, got, n_min=1)
        torch.cuda.synchronize()
    finally:
        hog.clear()
        _lib.gpair_release_scratch()
        torch.cuda.empty_cache()
    assert torch.equal(got, want)            # the same launches on the same data
