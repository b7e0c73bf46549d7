"""The performance cases: what a user of this library has it do, through its public entry points.

A case is a dict of plain values; `kind` says which call it makes:

  reconstruct  Algorithm 2 through the solver: `steps` iterations from a given iterate and its Adam
               moments (a resumed or warm-started reconstruction), on the windowed closed form
               (op = "exact") or the paper's discretised operator (op = "assa"), with or without
               the vessel continuity regulariser
  simulate     signals of a sparse vessel phantom (gpair_forward), as training data is made
  operator     the differentiable grid operator of a learned pipeline: forward and backward
  fit          the differentiable free-centre operator: signals and all five gradients
  regularise   value and gradient of the vessel continuity regulariser of an image
  evaluate     a reconstruction compared with its reference: voxelised, projected, and the
               MSE / PSNR / SSIM of the volume and of the projection
  render       free Gaussians voxelised on a lattice
  network      the warm start's U-Net on one back-projected volume
  layer        one convolution layer of the U-Net in training: forward, ReLU backward, weight, bias
               and input gradients

Lengths are metres, times seconds; every acquisition is at 40 MHz and 1500 m/s with the 3-sigma
window, the sensors lie on a spherical cap below the volume.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2602_03893_gb300 import _lib, autograd, unet

V, FS, K = 1500.0, 40e6, 3.0
DELTA = V / FS


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # a small reconstruction start to finish of a coarse volume (the repository's tiny workload):
        # launches and latency decide
        {"name": "reconstruct_tiny", "kind": "reconstruct", "op": "exact", "vcr": False, "steps": 20,
         "nx": 16, "ny": 16, "nz": 16, "h": 2e-4, "nd": 128, "nt": 1024, "radius": 0.020, "opening": 180.0},
        # one iteration at the paper's in-vivo scale, the headline workload
        {"name": "reconstruct_paper", "kind": "reconstruct", "op": "exact", "vcr": False, "steps": 1,
         "nx": 256, "ny": 256, "nz": 128, "h": 1e-4, "nd": 1024, "nt": 4096, "radius": 0.080, "opening": 140.0},
        # the paper's own iteration (its discretised operator and its regulariser) on the mid workload
        {"name": "reconstruct_assa_vcr", "kind": "reconstruct", "op": "assa", "vcr": True, "steps": 2,
         "nx": 128, "ny": 128, "nz": 64, "h": 1e-4, "nd": 1024, "nt": 4096, "radius": 0.060, "opening": 120.0},
        # the signals of one training phantom of the warm start (2000 of them make its training set)
        {"name": "simulate_mid", "kind": "simulate",
         "nx": 128, "ny": 128, "nz": 64, "h": 1e-4, "nd": 1024, "nt": 4096, "radius": 0.060, "opening": 120.0},
        # the grid operator as a layer on a small ragged volume: no side a multiple of the tiles
        {"name": "operator_ragged", "kind": "operator",
         "nx": 45, "ny": 37, "nz": 29, "h": 1e-4, "nd": 97, "nt": 1501, "radius": 0.040, "opening": 140.0},
        # one gradient step of a free-Gaussian fit: the repository's differentiation workload
        {"name": "fit_diff", "kind": "fit", "side": 64, "m": 262144, "h": 1e-4, "nd": 512, "nt": 2048,
         "radius": 0.040, "opening": 180.0},
        # the same for a few Gaussians and sensors, as a fit starts
        {"name": "fit_small", "kind": "fit", "side": 12, "m": 1500, "h": 1e-4, "nd": 48, "nt": 1024,
         "radius": 0.020, "opening": 180.0},
        # the regulariser of an image of the in-vivo scale
        {"name": "regularise_paper", "kind": "regularise", "nx": 256, "ny": 256, "nz": 128},
        # Table 1's figures of one reconstruction of that scale
        {"name": "evaluate_paper", "kind": "evaluate", "nx": 256, "ny": 256, "nz": 128, "h": 1e-4, "win": 7},
        # the field of a fitted set, drawn on a lattice of half its spacing
        {"name": "render_free", "kind": "render", "side": 64, "m": 262144, "h": 1e-4, "nx": 128, "ny": 128, "nz": 128,
         "dx": 0.5e-4},
        # the initial image of one reconstruction
        {"name": "network_mid", "kind": "network", "d": 64, "hh": 128, "w": 128},
        # the widest layer of the network at full resolution, in training
        {"name": "layer_d1a", "kind": "layer", "d": 64, "hh": 128, "w": 128, "cin": 48, "cout": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _acquisition(rng, half, nd_lo=32, nd_hi=1024):
    """Sensors and record for a volume of the given half diagonal: most records hold every window, some
    end before the last ones."""
    radius = max(half + 0.010, rng.uniform(0.020, 0.080))
    need = (radius + half + 1e-3) / DELTA
    return {"nd": _log(rng, nd_lo, nd_hi), "nt": int(need * rng.uniform(0.95, 1.4)) + 16,
            "radius": round(radius, 5), "opening": float(rng.choice([90, 120, 140, 180]))}


def _volume(rng, most):
    """A lattice of up to `most` nodes, sides from 9, ragged as often as not."""
    while True:
        n = [_log(rng, 9, 256), _log(rng, 9, 256), _log(rng, 9, 160)]
        if rng.random() < 0.4:
            n = [max(8, q // 8 * 8) for q in n]
        if n[0] * n[1] * n[2] <= most:
            return n


def _pairs_case(rng, kind, most):
    while True:
        nx, ny, nz = _volume(rng, 8388608)
        h = rng.choice([1e-4, 1e-4, 1.25e-4, 2e-4])
        c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "h": h}
        c.update(_acquisition(rng, 0.5 * h * math.sqrt(nx * nx + ny * ny + nz * nz)))
        if 2e5 <= nx * ny * nz * c["nd"] <= most:
            return c


def draw(rng):
    kind = rng.choice(["reconstruct", "reconstruct", "simulate", "operator", "fit", "regularise", "evaluate", "render",
                       "network", "layer"])
    if kind == "reconstruct":
        c = _pairs_case(rng, kind, 2e9)
        c["op"] = rng.choice(["exact", "exact", "assa"])
        c["vcr"] = rng.random() < 0.5
        c["steps"] = max(1, min(_log(rng, 1, 20), int(2e9 / (c["nx"] * c["ny"] * c["nz"] * c["nd"]))))
        return c
    if kind in ("simulate", "operator"):
        return _pairs_case(rng, kind, 2e9)
    if kind in ("fit", "render"):
        m = _log(rng, 500, 262144)
        side = max(4, math.ceil(m ** (1 / 3)))
        c = {"kind": kind, "side": side, "m": m, "h": 1e-4}
        if kind == "fit":
            c.update(_acquisition(rng, 0.9 * side * 1e-4, 16, 512))
        else:
            c["dx"] = rng.choice([0.5e-4, 0.7e-4, 1e-4])
            c.update({a: max(8, int(side * 1e-4 / c["dx"] * rng.uniform(0.7, 1.1))) for a in ("nx", "ny", "nz")})
        return c
    if kind in ("regularise", "evaluate"):
        nx, ny, nz = _volume(rng, 8388608)
        c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz}
        if kind == "evaluate":
            c.update(h=rng.choice([1e-4, 2e-4]), win=rng.choice([5, 7, 7, 9]))
        return c
    if kind == "network":
        return {"kind": kind, **{a: 8 * _log(rng, 1, 16) for a in ("hh", "w")}, "d": 8 * _log(rng, 1, 8)}
    widths = [(s.cin, s.cout) for s in unet.layer_specs().values() if s.taps == 27]
    cin, cout = rng.choice(widths)
    while True:
        c = {"kind": kind, "d": _log(rng, 4, 64), "hh": _log(rng, 4, 128), "w": _log(rng, 4, 128), "cin": cin,
             "cout": cout}
        if c["d"] * c["hh"] * c["w"] * cin * cout <= 64 * 128 * 128 * 48 * 16:
            return c


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(gen, *shape):
    return torch.rand(shape, device="cuda", generator=gen)


def _randn(gen, *shape):
    return torch.randn(shape, device="cuda", generator=gen)


def _cap(n, radius, opening):
    """n point sensors evenly spread (golden-angle spiral) over a cap below the origin."""
    i = np.arange(n, dtype=np.float64)
    cos_t = 1.0 - (1.0 - math.cos(math.radians(opening) / 2.0)) * (i + 0.5) / n
    sin_t = np.sqrt(np.maximum(0.0, 1.0 - cos_t ** 2))
    phi = i * math.pi * (3.0 - math.sqrt(5.0))
    xyz = np.stack([radius * sin_t * np.cos(phi), radius * sin_t * np.sin(phi), -radius * cos_t], 1)
    return torch.as_tensor(xyz.astype(np.float32), device="cuda")


def _array(c):
    return _lib.SensorArray(xyz=_cap(c["nd"], c["radius"], c["opening"]), sound_speed=V, fs=FS, n_samples=c["nt"],
                            window_k=K)


def _grid(nx, ny, nz, h):
    return _lib.Grid(nx, ny, nz, -nx * h / 2, -ny * h / 2, -nz * h / 2, h, h)


def _case_grid(c):
    return _grid(c["nx"], c["ny"], c["nz"], c["h"])


def _axis(n, o, h, dtype=torch.float64):
    """Node centres along one axis from the float32 origin and spacing."""
    o, h = float(np.float32(o)), float(np.float32(h))
    return o + (torch.arange(n, device="cuda", dtype=dtype) + 0.5) * h


def _centres(g):
    """[M, 3] float64 node centres, x fastest."""
    z, y, x = torch.meshgrid(_axis(g.nz, g.oz, g.dx), _axis(g.ny, g.oy, g.dx), _axis(g.nx, g.ox, g.dx), indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)


def _vessels(nx, ny, nz, gen, n=24):
    """A sparse image [nz, ny, nx]: capsules one to three nodes thick, log-normal intensities, zero between."""
    r = torch.rand((n, 8), generator=gen, device="cuda").cpu().numpy()
    ext = np.array([nx, ny, nz], dtype=np.float64)
    A = torch.zeros((nz, ny, nx), device="cuda")
    for q in r:
        p0 = q[:3] * ext
        d = q[3:6] - 0.5
        p1 = p0 + d / (np.linalg.norm(d) + 1e-9) * 0.3 * ext[:2].min()
        rad = 0.7 + 2.3 * q[6]
        lo = np.clip(np.floor(np.minimum(p0, p1) - rad), 0, ext - 1).astype(int)
        hi = np.clip(np.ceil(np.maximum(p0, p1) + rad), 1, ext).astype(int)
        if np.any(hi <= lo):
            continue
        ax = [torch.arange(lo[k], hi[k], device="cuda", dtype=torch.float32) + 0.5 for k in range(3)]
        X, Y, Z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
        s = p1 - p0
        t = ((X - p0[0]) * s[0] + (Y - p0[1]) * s[1] + (Z - p0[2]) * s[2]) / float(s @ s)
        t = t.clamp(0, 1)
        d2 = (X - p0[0] - t * s[0]) ** 2 + (Y - p0[1] - t * s[1]) ** 2 + (Z - p0[2] - t * s[2]) ** 2
        box = A[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
        box.copy_(torch.maximum(box, torch.where(d2 <= rad * rad, float(np.exp(0.4 * (2 * q[7] - 1))), 0.0)))
    return A


def _image(nx, ny, nz, gen):
    """A dense non-negative image [nz, ny, nx], as an iterate is: vessels on a small background."""
    return _vessels(nx, ny, nz, gen) * (0.7 + 0.6 * _rand(gen, nz, ny, nx)) + (0.1 * _rand(gen, nz, ny, nx)) ** 2


def _free_set(c, gen):
    """m Gaussians on a jittered lattice of side^3 nodes: centres, widths log-uniform from 0.05 to 0.2 mm,
    amplitudes as an optimisation's iterate has them."""
    s, m, h = c["side"], c["m"], c["h"]
    at = torch.arange(m, device="cuda")
    ijk = torch.stack([at % s, (at // s) % s, at // (s * s)])
    cen = (ijk + 0.5 - s / 2) * h + (2 * _rand(gen, 3, m) - 1) * 0.5 * h
    sig = torch.exp(math.log(0.05e-3) + math.log(4.0) * _rand(gen, m))
    return [t.contiguous() for t in (_rand(gen, m) ** 2, cen[0], cen[1], cen[2], sig)]


def _reconstruct_inputs(c, seed):
    """The measured signals of some point absorbers with 30 dB noise, and the iterate with its moments."""
    gen = _gen(seed)
    g, xyz = _case_grid(c), _cap(c["nd"], c["radius"], c["opening"])
    M = g.nx * g.ny * g.nz
    src = torch.unique(torch.randint(0, M, (min(256, M // 8),), generator=gen, device="cuda"))
    amp = 0.5 + _rand(gen, src.numel()).double()
    cen = _centres(g)[src]
    sig = float(np.float32(g.sigma))
    b = _signals(cen, amp, torch.full_like(amp, sig), xyz.double(), c["nt"])
    b = (b + b.square().mean().sqrt() * 10 ** -1.5 * _randn(gen, *b.shape).double()).float()
    x = (0.1 * _rand(gen, M)) ** 2
    x[src] = amp.float() * (0.6 + 0.8 * _rand(gen, src.numel()))
    z = torch.sqrt(x)
    # the moments' scale: that of the gradient 2 A^T (2 (y - b) / N) z at a few nodes
    at = torch.randint(0, M, (64,), generator=gen, device="cuda")
    gx = _adjoint(_centres(g)[at], torch.full((64,), sig, device="cuda", dtype=torch.float64), xyz.double(), b.double())[0]
    scale = float(gx.square().mean().sqrt()) * 4.0 / b.numel() * float(z.mean())
    m = 0.3 * scale * _randn(gen, M)
    v = (scale * (0.5 + _rand(gen, M))) ** 2
    return g, xyz, b.contiguous(), z, m, v


STEP0, ETA, T0 = 7, 1e-2, 50      # the iteration the resumed state had reached, the step size, the first restart


def _step_params(c):
    return _lib.StepParams(eta_max=ETA, T0=T0, adam_eps=1e-20, op=_lib.OP_ASSA if c["op"] == "assa" else _lib.OP_EXACT,
                           vcr_lambda=1e-12 if c["vcr"] else 0.0, vcr_beta=0.5 if c["vcr"] else 0.0, vcr_eps=1e-4)


def _layer_inputs(c, seed):
    gen = _gen(seed)
    n, ci, co = c["d"] * c["hh"] * c["w"], c["cin"], c["cout"]
    x = torch.relu(_randn(gen, n, ci)).to(torch.bfloat16)
    w = (_randn(gen, co, 27, ci) * math.sqrt(2.0 / (27 * ci))).to(torch.bfloat16)
    b = 0.1 * _randn(gen, co)
    gy = (1e-3 * _randn(gen, n, co)).to(torch.bfloat16)
    act = torch.relu(_randn(gen, n, co)).to(torch.bfloat16)      # the activations that the backward pass had stored
    return x, w, b, gy, act


def prepare(case, seed):
    c, gen = case, _gen(seed)
    s = {"case": c}
    kind = c["kind"]
    if kind == "reconstruct":
        g, _, s["b"], s["z"], s["m"], s["v"] = _reconstruct_inputs(c, seed)
        s["arr"] = _array(c)
        s["x"] = torch.empty_like(s["z"])
        s["solver"] = _lib.Solver(_lib.Gaussians(A=s["z"], grid=g), s["arr"], _step_params(c))
    elif kind == "simulate":
        s["g"] = _lib.Gaussians(A=_vessels(c["nx"], c["ny"], c["nz"], gen).reshape(-1), grid=_case_grid(c))
        s["arr"] = _array(c)
    elif kind == "operator":
        s["A"] = _image(c["nx"], c["ny"], c["nz"], gen).reshape(-1).requires_grad_(True)
        s["grid"], s["arr"] = _case_grid(c), _array(c)
        s["gy"] = _randn(gen, c["nd"], c["nt"])
    elif kind == "fit":
        s["p"] = [t.requires_grad_(True) for t in _free_set(c, gen)]
        s["arr"] = _array(c)
        s["gy"] = _randn(gen, c["nd"], c["nt"])
    elif kind == "regularise":
        s["x"] = _image(c["nx"], c["ny"], c["nz"], gen).reshape(-1)
    elif kind == "evaluate":
        A = _image(c["nx"], c["ny"], c["nz"], gen)
        s["g"] = _lib.Gaussians(A=A.reshape(-1), grid=_case_grid(c))
        s["ref"] = _reference(c, A, gen)
    elif kind == "render":
        A, cx, cy, cz, sig = _free_set(c, gen)
        s["g"] = _lib.Gaussians(A=A, cx=cx, cy=cy, cz=cz, sigma=sig)
        s["out"] = _grid(c["nx"], c["ny"], c["nz"], c["dx"])
    elif kind == "network":
        s["net"] = unet.UNet3D((c["d"], c["hh"], c["w"]), seed=int(seed) % 1000003)
        s["x"] = _image(c["w"], c["hh"], c["d"], gen).reshape(-1)
    else:
        s["x"], s["w"], s["b"], gy, s["act"] = _layer_inputs(c, seed)
        s["gy"] = gy
        s["out"], s["dx"] = torch.empty_like(gy), torch.empty_like(s["x"])
        s["dw"], s["db"] = torch.empty(s["w"].shape, device="cuda"), torch.empty_like(s["b"])
        s["wt"] = torch.empty_like(s["w"])
    return s


def _reference(c, A, gen):
    """The image that the reconstruction is compared with: the field of its amplitudes, blurred and noisy."""
    ref = F.avg_pool3d(A[None, None], 3, stride=1, padding=1)[0, 0] * 10.0
    return (ref * (0.9 + 0.2 * _rand(gen, c["nz"], c["ny"], c["nx"]))).contiguous()


# ---------------------------------------------------------------- the calls

def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "reconstruct":
        sol = s["solver"]
        sol.gpair_solver_set_state(s["z"], s["m"], s["v"], STEP0)
        # one iteration as a program's own loop makes it, several as one call
        loss, resid = sol.gpair_step(s["b"]) if c["steps"] == 1 else sol.gpair_solver_steps(s["b"], c["steps"])
        x = sol.gpair_solver_image(s["x"])
        z, m, v, _ = sol.gpair_solver_get_state()
        return {"x": x, "z": z, "m": m, "v": v, "loss": loss, "resid": resid}
    if kind == "simulate":
        return _lib.gpair_forward(s["g"], s["arr"], torch.empty((c["nd"], c["nt"]), device="cuda"))
    if kind == "operator":
        y = autograd.grid_signals(s["A"], s["grid"], s["arr"])
        (gA,) = torch.autograd.grad(y, [s["A"]], s["gy"])
        return {"y": y, "gA": gA}
    if kind == "fit":
        y = autograd.gaussian_signals(*s["p"], s["arr"])
        return {"y": y, "g": list(torch.autograd.grad(y, s["p"], s["gy"]))}
    if kind == "regularise":
        grad = torch.zeros_like(s["x"])
        value = _lib.gpair_vcr(s["x"], (c["nz"], c["ny"], c["nx"]), 0.5, 1e-4, 1.0, grad)
        return {"value": value, "grad": grad}
    if kind == "evaluate":
        dims = (c["nz"], c["ny"], c["nx"])
        vol = _lib.gpair_voxelize(s["g"], s["g"].grid, K, torch.empty(dims, device="cuda"))
        volume = _lib.gpair_image_metrics(vol, s["ref"], dims, c["win"], 1.0)
        p, q = _lib.gpair_zmap(vol, dims), _lib.gpair_zmap(s["ref"], dims)
        image = _lib.gpair_image_metrics(p, q, (1, c["ny"], c["nx"]), c["win"], 1.0)
        return {"vol": vol, "map": p, "refmap": q, "volume": volume, "image": image}
    if kind == "render":
        o = s["out"]
        return _lib.gpair_voxelize(s["g"], o, K, torch.empty((o.nz, o.ny, o.nx), device="cuda"))
    if kind == "network":
        return s["net"].forward(s["x"], 2.0)
    dims = (c["d"], c["hh"], c["w"])
    unet.gpair_conv3d_fwd(s["x"], dims, c["cin"], s["w"], s["b"], c["cout"], 27, True, s["out"])
    unet.gpair_relu_bwd(s["act"], s["gy"])
    s["dw"].zero_()
    s["db"].zero_()
    unet.gpair_conv3d_wgrad(s["x"], s["gy"], dims, c["cin"], c["cout"], 27, s["dw"], s["db"])
    unet.gpair_conv3d_dgrad(s["gy"], dims, c["cout"], s["w"], c["cin"], 27, s["wt"], s["dx"])
    return {"out": s["out"], "gy": s["gy"], "dw": s["dw"], "db": s["db"], "dx": s["dx"]}


# ---------------------------------------------------------------- what they cannot do without

def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: the definition's -- 4 (forward) or 5 (adjoint) a
    sample of a pair's window and 10 a pair (discretised operator: 10 a pair), the full gradient 10 a
    sample and 40 a pair, the stencils, box sums and convolutions as defined."""
    c, kind = case, case["kind"]
    n = c.get("nx", 0) * c.get("ny", 0) * c.get("nz", 0)
    if kind in ("reconstruct", "simulate", "operator"):
        pairs, sig = n * c["nd"], 4 * c["nd"] * c["nt"]
        samples = pairs * 2 * K * c["h"] / DELTA
        fwd = 4 * samples + 10 * pairs
        if kind == "simulate":
            return {"bytes": 4 * n + sig, "flops": fwd}
        adj = 5 * samples + 10 * pairs
        if kind == "operator":
            return {"bytes": 8 * n + 2 * sig, "flops": fwd + adj}
        if c["op"] == "assa":
            fwd = adj = 10 * pairs
        return {"bytes": c["steps"] * (6 * 4 * n + sig) + 4 * 4 * n, "flops": c["steps"] * (fwd + adj + 20 * n + (150 * n if c["vcr"] else 0))}
    if kind == "fit":
        pairs = c["m"] * c["nd"]
        samples = pairs * 2 * K * (0.15e-3 / math.log(4.0)) / DELTA       # the mean width of the set
        return {"bytes": 10 * 4 * c["m"] + 8 * c["nd"] * c["nt"], "flops": 14 * samples + 50 * pairs}
    if kind == "regularise":
        return {"bytes": 8 * n, "flops": 150 * n}
    if kind == "evaluate":
        return {"bytes": 12 * n + 8 * c["nx"] * c["ny"], "flops": 80 * n}
    if kind == "render":
        box = (2 * K * (0.15e-3 / math.log(4.0)) / c["dx"]) ** 3
        return {"bytes": 20 * c["m"] + 4 * n, "flops": 2 * c["m"] * box}
    nv = c["d"] * c["hh"] * c["w"]
    if kind == "network":
        lv = {"e1": 0, "d1": 0, "ou": 0, "e2": 1, "d2": 1, "e3": 2, "d3": 2, "b4": 3}
        return {"bytes": 4 * nv + 32 * nv,
                "flops": sum(2 * (nv >> 3 * lv[k[:2]]) * s.cin * s.cout * s.taps for k, s in unet.layer_specs().items())}
    return {"bytes": 2 * nv * (2 * c["cin"] + 4 * c["cout"]) + 8 * 27 * c["cin"] * c["cout"],
            "flops": 3 * 2 * nv * 27 * c["cin"] * c["cout"]}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch

CHUNK = 1 << 24       # pairs at a time
MOST = 4e10           # window samples evaluated at most


def _windows(cen, xyz, sig, nt):
    """For sensors xyz against centres cen: R [nd, M], the first sample of each window, and how many to walk."""
    R = torch.cdist(xyz, cen, compute_mode="donot_use_mm_for_euclid_dist")
    first = torch.ceil((R - K * sig) * (FS / V) - 1e-3).long()
    return R, first, int(float(sig.max()) * 2 * K / DELTA) + 3


def _signals(cen, amp, sig, xyz, nt):
    """y[j][n] = sum_i A_i / 2R d exp(-d^2 / 2 sigma_i^2) over |d| <= k sigma_i, d = R - v n / fs."""
    y = torch.zeros((xyz.shape[0], nt), device="cuda", dtype=torch.float64)
    rows = max(1, CHUNK // cen.shape[0])
    for j in range(0, xyz.shape[0], rows):
        R, n, W = _windows(cen, xyz[j:j + rows], sig, nt)
        w = amp / (2 * R)
        row = torch.arange(R.shape[0], device="cuda")[:, None] * nt
        out = y[j:j + rows].reshape(-1)
        for _ in range(W):
            d = R - n.double() * DELTA
            on = (d.abs() <= K * sig) & (n >= 0) & (n < nt)
            val = torch.where(on, w * d * torch.exp(-d * d / (2 * sig * sig)), 0.0)
            out.scatter_add_(0, (row + n.clamp(0, nt - 1)).reshape(-1), val.reshape(-1))
            n = n + 1
    return y


def _adjoint(cen, sig, xyz, dl, amp=None):
    """gA, and with amp also the gradients with respect to the centres and widths."""
    nt = dl.shape[1]
    M = cen.shape[0]
    out = [torch.zeros(M, device="cuda", dtype=torch.float64) for _ in range(5 if amp is not None else 1)]
    rows = max(1, CHUNK // M)
    for j in range(0, xyz.shape[0], rows):
        R, n, W = _windows(cen, xyz[j:j + rows], sig, nt)
        S = [torch.zeros_like(R) for _ in range(4 if amp is not None else 1)]
        row = torch.arange(R.shape[0], device="cuda")[:, None] * nt
        flat = dl[j:j + rows].reshape(-1)
        for _ in range(W):
            d = R - n.double() * DELTA
            on = (d.abs() <= K * sig) & (n >= 0) & (n < nt)
            u = torch.where(on, flat[row + n.clamp(0, nt - 1)] * torch.exp(-d * d / (2 * sig * sig)), 0.0)
            if amp is not None:
                S[1] += u
                S[2] += u * d * d
                S[3] += u * d ** 3
            S[0] += u * d
            n = n + 1
        out[0] += (S[0] / (2 * R)).sum(0)
        if amp is not None:
            w = amp / (2 * R)
            gR = w * (S[1] - S[2] / sig ** 2) - w * S[0] / R
            for k in range(3):
                out[1 + k] += (gR / R * (cen[:, k][None] - xyz[j:j + rows, k][:, None])).sum(0)
            out[4] += (w * S[3] / sig ** 3).sum(0)
    return out


class _Exact:
    """The closed form on a lattice."""

    def __init__(self, g, xyz, nt):
        self.cen, self.xyz, self.nt = _centres(g), xyz.double(), nt
        self.sig = torch.full((self.cen.shape[0],), float(np.float32(g.sigma)), device="cuda", dtype=torch.float64)

    def forward(self, A):
        return _signals(self.cen, A, self.sig, self.xyz, self.nt)

    def adjoint(self, dl):
        return _adjoint(self.cen, self.sig, self.xyz, dl)[0]


class _Assa:
    """The discretised operator (Algorithm 1) at the paper's minimum pulse length of 25."""

    def __init__(self, g, xyz, nt):
        s = float(np.float32(g.sigma))
        nh = max(1, math.ceil(3 * s / DELTA))
        self.al = max(1, math.ceil(12 / nh))
        self.K = self.al * nh
        d = -DELTA / self.al * torch.arange(self.K, -self.K - 1, -1, device="cuda", dtype=torch.float64)
        self.h = (0.5 * d * torch.exp(-d * d / (2 * s * s)))[None, None]
        self.cen, self.xyz, self.nt = _centres(g), xyz.double(), nt

    def _pairs(self):
        n = self.al * self.nt
        rows = max(1, CHUNK // self.cen.shape[0])
        for j in range(0, self.xyz.shape[0], rows):
            R = torch.cdist(self.xyz[j:j + rows], self.cen, compute_mode="donot_use_mm_for_euclid_dist")
            k = torch.floor(R / V * self.al * FS + 0.5).long()
            row = torch.arange(R.shape[0], device="cuda")[:, None] * n
            yield j, j + R.shape[0], 1 / R, (row + k.clamp(0, n - 1)), (k >= 0) & (k < n)

    def forward(self, A):
        imp = torch.zeros((self.xyz.shape[0], self.al * self.nt), device="cuda", dtype=torch.float64)
        for a, b, inv, at, on in self._pairs():
            imp[a:b].reshape(-1).scatter_add_(0, at.reshape(-1), torch.where(on, A * inv, 0.0).reshape(-1))
        return F.conv1d(imp[:, None], self.h, padding=self.K, stride=self.al)[:, 0]

    def adjoint(self, dl):
        n = self.al * self.nt
        up = torch.zeros((dl.shape[0], n), device="cuda", dtype=torch.float64)
        up[:, ::self.al] = dl
        conv = F.conv1d(up[:, None], self.h.flip(-1), padding=self.K)[:, 0]
        g = torch.zeros(self.cen.shape[0], device="cuda", dtype=torch.float64)
        for a, b, inv, at, on in self._pairs():
            g += torch.where(on, conv[a:b].reshape(-1)[at] * inv, 0.0).sum(0)
        return g


def _vcr(x, beta, eps):
    """R_VCR of an image [nz, ny, nx] and its gradient."""
    x = x.detach().requires_grad_(True)
    p = F.pad(x[None, None], (1,) * 6, mode="replicate")[0, 0]

    def at(dz, dy, dx):
        return p[1 + dz:p.shape[0] - 1 + dz, 1 + dy:p.shape[1] - 1 + dy, 1 + dx:p.shape[2] - 1 + dx]

    e = [(0, 0, 1), (0, 1, 0), (1, 0, 0)]
    sh, st = 0, 0
    for q in range(3):
        a = e[q]
        n = tuple(-t for t in a)
        st = st + ((at(*a) - at(*n)) / 2) ** 2
        sh = sh + (at(*a) - 2 * at(0, 0, 0) + at(*n)) ** 2
        for r in range(q):
            b = e[r]
            pp, pm = tuple(s + t for s, t in zip(a, b)), tuple(s - t for s, t in zip(a, b))
            mixed = (at(*pp) - at(*pm) - at(*(-t for t in pm)) + at(*(-t for t in pp))) / 4
            sh = sh + 2 * mixed ** 2
    value = torch.sqrt(sh + eps).sum() + beta * torch.sqrt(st + eps).sum()
    (grad,) = torch.autograd.grad(value, [x])
    return value.detach(), grad


def _metrics(x, y, win, peak):
    mse = (x - y).square().mean()
    win = (win if x.shape[0] > 1 else 1, win, win)
    n = win[0] * win[1] * win[2]

    def box(q):
        return F.avg_pool3d(q[None, None], win, stride=1)[0, 0]

    mx, my = box(x), box(y)
    vx, vy, vxy = (n / (n - 1) * (box(a * b) - box(a) * box(b)) for a, b in ((x, x), (y, y), (x, y)))
    c1, c2 = (0.01 * peak) ** 2, (0.03 * peak) ** 2
    ssim = ((2 * mx * my + c1) * (2 * vxy + c2)) / ((mx * mx + my * my + c1) * (vx + vy + c2))
    return {"mse": mse, "psnr": 10 * torch.log10(peak * peak / mse), "ssim": ssim.mean()}


def _smooth(A, h):
    """The field of a lattice's Gaussians (sigma = h) at its nodes, each to 3 sigma an axis."""
    t = torch.exp(-0.5 * torch.arange(-3, 4, device="cuda", dtype=torch.float64) ** 2)
    v = A[None, None]
    for k in range(3):
        shape, pad = [1, 1, 1, 1, 1], [0, 0, 0]
        shape[2 + k], pad[k] = 7, 3
        v = F.conv3d(v, t.reshape(shape), padding=tuple(pad))
    return v[0, 0]


def _render(g, o):
    f = lambda t: t.double()[:, None]
    sig = f(g.sigma)
    W = int(float(g.sigma.max()) * 2 * K / o.dx) + 3
    ax = []
    for cen, org, n in ((g.cx, o.ox, o.nx), (g.cy, o.oy, o.ny), (g.cz, o.oz, o.nz)):
        org, dx = float(np.float32(org)), float(np.float32(o.dx))
        at = torch.ceil((f(cen) - K * sig - org) / dx - 0.5 - 1e-3).long() + torch.arange(W, device="cuda")
        d = org + (at.double() + 0.5) * dx - f(cen)
        on = (d.abs() <= K * sig) & (at >= 0) & (at < n)
        ax.append((at.clamp(0, n - 1), torch.where(on, torch.exp(-d * d / (2 * sig * sig)), 0.0)))
    vol = torch.zeros(o.nx * o.ny * o.nz, device="cuda", dtype=torch.float64)
    (ix, fx), (iy, fy), (iz, fz) = ax
    for a in range(W):
        for b in range(W):
            w = f(g.A) * fz[:, a:a + 1] * fy[:, b:b + 1] * fx
            vol.scatter_add_(0, ((iz[:, a:a + 1] * o.ny + iy[:, b:b + 1]) * o.nx + ix).reshape(-1), w.reshape(-1))
    return vol.reshape(o.nz, o.ny, o.nx)


def _conv64(x, w, dims, b=None):
    """[nv, ci] and [co, taps, ci] -> [nv, co], zero padding."""
    s = round(w.shape[1] ** (1 / 3))
    k = w.double().reshape(w.shape[0], s, s, s, -1).permute(0, 4, 1, 2, 3)
    v = x.double().reshape(1, *dims, -1).permute(0, 4, 1, 2, 3)
    y = F.conv3d(v, k, None if b is None else b.double(), padding=s // 2)
    return y[0].permute(1, 2, 3, 0).reshape(-1, w.shape[0])


def _network64(net, x, dims):
    def conv(name, v, q):
        y = _conv64(v, net.wbf[name], [d >> q for d in dims], net.b32[name])
        return torch.relu(y) if net.convs[name].relu else y

    def grid(v, q):
        return v.reshape(1, *[d >> q for d in dims], -1).permute(0, 4, 1, 2, 3)

    def flat(v):
        return v[0].permute(1, 2, 3, 0).reshape(-1, v.shape[1])

    v = torch.zeros((x.numel(), unet.CIN_PAD), device="cuda", dtype=torch.float64)
    v[:, 0] = x
    skip = []
    for q in range(3):
        v = conv("e%db" % (q + 1), conv("e%da" % (q + 1), v, q), q)
        skip.append(v)
        v = flat(F.avg_pool3d(grid(v, q), 2))
    v = conv("b4b", conv("b4a", v, 3), 3)
    for q in (2, 1, 0):
        v = torch.cat([flat(F.interpolate(grid(v, q + 1), scale_factor=2, mode="nearest")), skip[q]], 1)
        v = conv("d%db" % (q + 1), conv("d%da" % (q + 1), v, q), q)
    return conv("out", v, 0)


def _reconstruct64(c, seed):
    g, xyz, b, z, m, v = (t.double() if isinstance(t, torch.Tensor) else t for t in _reconstruct_inputs(c, seed))
    p = _step_params(c)
    f32 = lambda q: float(np.float32(q))
    b1, b2, eps = f32(p.beta1), f32(p.beta2), f32(p.npc_eps)
    op = (_Assa if c["op"] == "assa" else _Exact)(g, xyz, c["nt"])
    N = b.numel()
    loss = resid = None
    for t in range(STEP0, STEP0 + c["steps"]):
        x = (z + eps) ** 2
        r = op.forward(x) - b
        gx = op.adjoint(2 * r / N)
        loss, resid = r.square().sum() / N, r.square().sum().sqrt()
        if c["vcr"]:
            value, gr = _vcr(x.reshape(g.nz, g.ny, g.nx), f32(p.vcr_beta), f32(p.vcr_eps))
            loss, gx = loss + f32(p.vcr_lambda) * value, gx + f32(p.vcr_lambda) * gr.reshape(-1)
        gz = gx * 2 * (z + eps)
        m = b1 * m + (1 - b1) * gz
        v = b2 * v + (1 - b2) * gz * gz
        eta = 0.5 * f32(p.eta_max) * (1 + math.cos(math.pi * t / T0))
        z = z - eta * (m / (1 - b1 ** (t + 1))) / (torch.sqrt(v / (1 - b2 ** (t + 1))) + f32(p.adam_eps))
    return {"x": (z + eps) ** 2, "z": z, "m": m, "v": v, "loss": loss, "resid": resid}


def exact(case, seed):
    c, gen, kind = case, _gen(seed), case["kind"]
    if kind in ("reconstruct", "simulate", "operator"):
        walk = 1 if c.get("op") == "assa" else int(2 * K * c["h"] / DELTA) + 3
        if c["nx"] * c["ny"] * c["nz"] * c["nd"] * walk * c.get("steps", 1) > MOST:
            return None
    if kind == "reconstruct":
        return _reconstruct64(c, seed)
    if kind in ("simulate", "operator"):
        op = _Exact(_case_grid(c), _cap(c["nd"], c["radius"], c["opening"]), c["nt"])
        make = _vessels if kind == "simulate" else _image
        y = op.forward(make(c["nx"], c["ny"], c["nz"], gen).double().reshape(-1))
        return y if kind == "simulate" else {"y": y, "gA": op.adjoint(_randn(gen, c["nd"], c["nt"]).double())}
    if kind == "fit":
        A, cx, cy, cz, sig = (t.double() for t in _free_set(c, gen))
        gy = _randn(gen, c["nd"], c["nt"]).double()
        xyz, cen = _cap(c["nd"], c["radius"], c["opening"]).double(), torch.stack([cx, cy, cz], 1)
        return {"y": _signals(cen, A, sig, xyz, c["nt"]), "g": _adjoint(cen, sig, xyz, gy, A)}
    if kind == "regularise":
        value, grad = _vcr(_image(c["nx"], c["ny"], c["nz"], gen).double(), 0.5, float(np.float32(1e-4)))
        return {"value": value, "grad": grad.reshape(-1)}
    if kind == "evaluate":
        A = _image(c["nx"], c["ny"], c["nz"], gen)
        ref, vol = _reference(c, A, gen).double(), _smooth(A.double(), c["h"])
        p, q = vol.amax(0), ref.amax(0)
        return {"vol": vol, "map": p, "refmap": q, "volume": _metrics(vol, ref, c["win"], 1.0),
                "image": _metrics(p[None], q[None], c["win"], 1.0)}
    if kind == "render":
        A, cx, cy, cz, sig = _free_set(c, gen)
        return _render(_lib.Gaussians(A=A, cx=cx, cy=cy, cz=cz, sigma=sig), _grid(c["nx"], c["ny"], c["nz"], c["dx"]))
    dims = [c["d"], c["hh"], c["w"]]
    if kind == "network":
        net = unet.UNet3D(dims, seed=int(seed) % 1000003)
        x = _image(c["w"], c["hh"], c["d"], gen).reshape(-1)
        return _network64(net, (x * 2.0).to(torch.bfloat16).double(), dims)
    x, w, b, gy, act = (t.double() for t in _layer_inputs(c, seed))
    w.requires_grad_(True)
    x.requires_grad_(True)
    b.requires_grad_(True)
    y, gy = _conv64(x, w, dims, b), gy * (act > 0)
    dx, dw, db = torch.autograd.grad(y, [x, w, b], gy)
    return {"out": torch.relu(y.detach()), "gy": gy, "dw": dw, "db": db, "dx": dx}
