"""Performance cases of the cone-beam library: what its users run, through the public entry points.

A user of this library simulates scans, projects and backprojects volumes (alone or under
autograd), reconstructs them (FDK, PDHG-TV, the learned primal-dual) and trains the learned
blocks. The listed cases cover that over the sizes of the repository's own workloads
(`paper_2512_21180_gb300.inputs.geometry`): the 16^3 and 64^3 test sizes, where launches and
host work count, the 128^3 learned workload, the clinical 256 x 256 x 192 scan, and an odd-sized
anisotropic scan between them. The learned primal-dual is covered by its parts (projector pair at
its size, dual and primal convolutions, input and weight gradients) and by one iteration of its LIRE
form through the model's own call, not by a whole unrolled network: every BF16 rounding of an
activation is a discrete decision, so after eight iterations the FP32 output has moved by 1e-3 when
its inputs change by 1e-7, and by 6e-7 after one LIRE iteration (measured).

`draw` gives cases of the same kinds with other sizes. All inputs come from the seed alone:
ellipsoid phantoms and their analytic line integrals, in plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2512_21180_gb300 import _lib, inputs, lpd, ops, projector

SLOPE = 0.2  # LeakyReLU slope of the learned blocks

# ---- cases ----------------------------------------------------------------------------------


def _scan(workload: str, **kw) -> dict:
    """One of the repository's named scans as plain values."""
    g = inputs.geometry(workload)
    c = dict(nx=g["n"][0], ny=g["n"][1], nz=g["n"][2], vx=g["vox"][0], vy=g["vox"][1], vz=g["vox"][2],
             nu=g["nu"], nv=g["nv"], du=g["du"], dv=g["dv"], uoff=g["u_offset"], voff=0.0, na=g["n_angles"], batch=1)
    c.update(kw)
    return c


def listed() -> list[dict]:
    return [
        # the gradcheck / unit-test size: one forward and one adjoint, all launch and host latency
        _scan("tiny16", name="pair_tiny16", kind="pair"),
        # a small scan, as in tests and quick experiments: forward and adjoint
        _scan("small64", name="pair_small64", kind="pair"),
        # a training step's data term: y = P x for two volumes, then dL/dx = P^T dL/dy by autograd
        _scan("diff128", name="autograd_diff128", kind="autograd", batch=2),
        # odd sizes, anisotropic voxels, shifted panel in both directions: forward and adjoint
        dict(name="pair_ragged", kind="pair", nx=181, ny=167, nz=93, vx=2.5, vy=2.75, vz=3.1, nu=371, nv=213,
             du=1.1, dv=1.3, uoff=71.5, voff=-9.0, na=150, batch=1),
        # the clinical scan, the benchmark's workload: forward and adjoint, one step of any iterative method
        _scan("clinical", name="pair_clinical", kind="pair"),
        # FDK_w of the clinical scan: the start of every reconstruction
        _scan("clinical", name="fdk_clinical", kind="fdk"),
        # the iterative baseline at the learned workload's size (a whole reconstruction runs 50-100 of these iterations)
        _scan("lpd128", name="pdhg_lpd128", kind="pdhg", iters=20),
        # polychromatic detector readings with Poisson noise, ten energy bins: training-data generation
        _scan("lpd128", name="poly_lpd128", kind="poly", bins=10, noise=True, counts=False),
        # one iteration of the learned LIRE network through its own call: projections of two volumes, 3-D dual convolutions
        # over (angle, v, u), backprojections of two items, primal convolutions, output convolution
        _scan("lpd128", name="lire_iteration_lpd128", kind="lire"),
        # the learned dual block's hidden layer: 3x3, 32 -> 32 channels over 200 projections of 192 x 256, LeakyReLU
        dict(name="conv_dual_lpd128", kind="conv", nimg=200, D=1, H=192, W=256, cin=32, cout=32, taps3d=0, grad=False),
        # the primal block's hidden layer in the backward: 3x3x3 input gradient with the LeakyReLU mask, 128^3
        dict(name="conv_primal_dgrad_lpd128", kind="conv", nimg=1, D=128, H=128, W=128, cin=32, cout=32, taps3d=1,
             grad=True),
        # its weight and bias gradient
        dict(name="wgrad_primal_lpd128", kind="wgrad", nimg=1, D=128, H=128, W=128, cin=32, cout=32, taps3d=1),
    ]


def _log_int(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scan(rng: random.Random, samples: float) -> dict:
    """A scan of random size whose projector pair costs at most `samples` samples per operator."""
    while True:
        n = _log_int(rng, 14, 270)
        nx, ny = (max(9, int(n * rng.uniform(0.75, 1.2))) for _ in range(2))
        nz = max(7, int(n * rng.uniform(0.5, 1.1)))
        ext = rng.uniform(240.0, 520.0)  # mm, as the repository's volumes (256 ... 512)
        vx = round(ext / nx, 3)
        vy = round(vx * rng.choice([1.0, 1.0, ext / ny / vx]), 3)
        vz = round(vx * rng.choice([1.0, rng.uniform(0.7, 1.5)]), 3)
        nu = max(12, int(n * rng.uniform(1.3, 2.3)))
        nu = rng.choice([nu, nu, (nu + 3) & ~3, 256, 512]) if n > 90 else rng.choice([nu, (nu + 3) & ~3])
        nv = max(9, int(n * rng.uniform(0.8, 1.7)))
        du = round(rng.uniform(350.0, 480.0) / nu, 3)
        dv = round(rng.uniform(0.8, 1.2) * du, 3)
        uoff = rng.choice([0.0, round(rng.uniform(0.1, 0.38) * nu * du, 2), -round(rng.uniform(0.1, 0.3) * nu * du, 2)])
        voff = rng.choice([0.0, 0.0, round(rng.uniform(-20.0, 20.0), 1)])
        na, batch = _log_int(rng, 9, 410), rng.choice([1, 1, 1, 2, 4])
        if 0.9 * max(nx, ny) * nu * nv * na * batch <= samples:
            return dict(nx=nx, ny=ny, nz=nz, vx=vx, vy=vy, vz=vz, nu=nu, nv=nv, du=du, dv=dv, uoff=uoff, voff=voff,
                        na=na, batch=batch)


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["pair", "pair", "forward", "adjoint", "autograd", "fdk", "pdhg", "poly", "conv", "wgrad"])
    if kind in ("pair", "autograd"):
        return dict(_draw_scan(rng, 8e9), kind=kind)
    if kind in ("forward", "adjoint"):
        return dict(_draw_scan(rng, 1.8e10), kind=kind)
    if kind == "fdk":
        return dict(_draw_scan(rng, 1.8e10), kind=kind)
    if kind == "pdhg":
        return dict(_draw_scan(rng, 8e8), kind=kind, iters=rng.choice([1, 5, 10]))
    if kind == "poly":
        noise = rng.random() < 0.8
        return dict(_draw_scan(rng, 1e9), kind=kind, bins=rng.randint(1, 10), noise=noise,
                    counts=noise and rng.random() < 0.5)
    taps3d = rng.choice([0, 1])
    wide = rng.choice([0, 0, 1])
    cin = rng.choice([5, 6, 7, 8, 32, 32]) if not wide else rng.choice([32, 64])
    cout = 64 if wide and rng.random() < 0.7 else rng.choice([32, 32, 5])
    if taps3d:
        nimg, D, H, W = rng.choice([1, 2]), _log_int(rng, 6, 128), _log_int(rng, 8, 128), _log_int(rng, 9, 160)
    else:
        nimg, D, H, W = _log_int(rng, 3, 200), 1, _log_int(rng, 10, 200), _log_int(rng, 11, 260)
    c = dict(kind=kind, nimg=nimg, D=D, H=H, W=W, cin=cin, cout=cout, taps3d=taps3d)
    return dict(c, grad=rng.random() < 0.4 and cin % 8 == 0) if kind == "conv" else c


# ---- inputs ---------------------------------------------------------------------------------


def _geometry_dict(c: dict) -> dict:
    return dict(n=(c["nx"], c["ny"], c["nz"]), vox=(c["vx"], c["vy"], c["vz"]), center=(0.0, 0.0, 0.0), nu=c["nu"],
                nv=c["nv"], du=c["du"], dv=c["dv"], u_offset=c["uoff"], v_offset=c["voff"], sid=inputs.SID_MM,
                sdd=inputs.SDD_MM, n_angles=c["na"], batch=c["batch"])


def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _ellipsoids(c: dict, seed: int, n: int = 12) -> list[tuple]:
    """(centre, semi-axes, rotation, value) rows: a body and random soft-tissue ellipsoids."""
    rng = np.random.default_rng(seed)
    ext = np.array([c["nx"] * c["vx"], c["ny"] * c["vy"], c["nz"] * c["vz"]])
    rows = [(np.zeros(3), 0.5 * ext * np.array([0.75, 0.65, 0.9]), np.eye(3), 0.012)]
    for _ in range(n):
        q = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        rows.append((rng.uniform(-0.28, 0.28, 3) * ext, rng.uniform(0.03, 0.16, 3) * ext.min(), q,
                     rng.uniform(0.002, 0.012)))
    return rows


def _phantom(c: dict, rows) -> torch.Tensor:
    """Voxelised ellipsoids [nz, ny, nx], FP32, 1/mm."""
    ax = [(torch.arange(c["n" + a], device="cuda", dtype=torch.float32) - 0.5 * (c["n" + a] - 1)) * c["v" + a]
          for a in "xyz"]
    vol = torch.zeros((c["nz"], c["ny"], c["nx"]), device="cuda")
    for ctr, axes, R, val in rows:
        q = 0.0
        for i in range(3):
            m = R[i] / axes[i]
            l = (float(m[0]) * (ax[0] - float(ctr[0])) + (float(m[1]) * (ax[1] - float(ctr[1])))[:, None]
                 + (float(m[2]) * (ax[2] - float(ctr[2])))[:, None, None])
            q = q + l * l
        vol += (q <= 1.0).float() * float(val)
    return vol


def _chords(c: dict, rows) -> torch.Tensor:
    """Analytic line integrals of the ellipsoids along the scan's rays [na, nv, nu], FP32."""
    th = (2.0 * math.pi / c["na"]) * np.arange(c["na"])
    u = torch.as_tensor((np.arange(c["nu"]) - 0.5 * (c["nu"] - 1)) * c["du"] + c["uoff"], device="cuda").float()
    v = torch.as_tensor((np.arange(c["nv"]) - 0.5 * (c["nv"] - 1)) * c["dv"] + c["voff"], device="cuda").float()
    ln = torch.sqrt(u[None, :] ** 2 + v[:, None] ** 2 + inputs.SDD_MM ** 2)
    out = torch.zeros((c["na"], c["nv"], c["nu"]), device="cuda")
    for ctr, axes, R, val in rows:
        M = R / axes[:, None]
        src = np.stack([inputs.SID_MM * np.cos(th), inputs.SID_MM * np.sin(th), 0 * th], 1) - ctr
        d0 = np.stack([-inputs.SDD_MM * np.cos(th), -inputs.SDD_MM * np.sin(th), 0 * th], 1)
        eu = np.stack([-np.sin(th), np.cos(th), 0 * th], 1)
        a = b = 0.0
        cc = -1.0
        for i in range(3):
            t = [torch.as_tensor(w @ M[i], device="cuda").float()[:, None, None] for w in (src, d0, eu)]
            r = t[1] + t[2] * u[None, None, :] + float(M[i][2]) * v[None, :, None]
            a, b, cc = a + r * r, b + r * t[0], cc + t[0] * t[0]
        disc = (b * b - a * cc).clamp_(min=0.0)
        out += torch.sqrt(disc).div_(a).mul_(ln[None]).mul_(2.0 * float(val))
    return out


def _volumes(c: dict, seed: int) -> torch.Tensor:
    return torch.stack([_phantom(c, _ellipsoids(c, 1000 * seed + b)) for b in range(c["batch"])])


def _projections(c: dict, seed: int, noise: float = 0.0) -> torch.Tensor:
    p = torch.stack([_chords(c, _ellipsoids(c, 1000 * seed + b)) for b in range(c["batch"])])
    if noise:
        p += noise * torch.randn(p.shape, generator=_gen(seed), device="cuda")
    return p


def _row_blocked(g: torch.Generator, c: dict, slots: int, used: int) -> torch.Tensor:
    """BF16 activations [nimg, D, H, slots / 8, W, 8] after a LeakyReLU, slots >= used zero."""
    x = torch.randn((c["nimg"], c["D"], c["H"], slots // 8, c["W"], 8), generator=g, device="cuda")
    x = torch.where(x > 0, x, SLOPE * x)
    ch = torch.arange(slots, device="cuda").reshape(slots // 8, 1, 8)
    return (x * (ch < used)).to(torch.bfloat16).contiguous()


def _slots(ch: int) -> int:
    return next(s for s in (8, 16, 32, 64) if s >= ch)


def _pdhg_steps(c: dict) -> tuple[float, float]:
    """(gamma, sigma = tau) from the Schur bound on ||P|| in closed form: largest row sum
    (the volume's diagonal) times largest column sum (rays through a voxel times step)."""
    ext = [c["nx"] * c["vx"], c["ny"] * c["vy"], c["nz"] * c["vz"]]
    mag = inputs.SDD_MM / (inputs.SID_MM - 0.5 * math.hypot(ext[0], ext[1]))
    nP = math.sqrt(math.hypot(ext[0], ext[1]) * c["na"] * c["vx"] * c["vy"] * c["vz"] * mag * mag / (c["du"] * c["dv"]))
    gamma = nP / math.sqrt(12.0)
    return gamma, 0.99 / math.hypot(nP, gamma * math.sqrt(12.0))


def prepare(case: dict, seed: int) -> dict:
    c, k = case, case["kind"]
    s = {"case": c}
    if k in ("conv", "wgrad"):
        g = _gen(seed)
        taps = 27 if c["taps3d"] else 9
        s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        if k == "conv":
            src, dst = (c["cout"], c["cin"]) if c["grad"] else (c["cin"], c["cout"])
            s["x"] = _row_blocked(g, c, _slots(src), src)
            s["w"] = torch.randn((c["cout"], taps, c["cin"]), generator=g, device="cuda") * math.sqrt(2.0 / (c["cin"] * taps))
            s["b"] = 0.1 * torch.randn(c["cout"], generator=g, device="cuda")
            s["y"] = torch.zeros((c["nimg"], c["D"], c["H"], _slots(dst) // 8, c["W"], 8), dtype=torch.bfloat16, device="cuda")
            if c["grad"]:
                s["mask"] = _row_blocked(g, c, _slots(dst), dst)
        else:
            s["x"] = _row_blocked(g, c, _slots(c["cin"]), c["cin"])
            s["dy"] = _row_blocked(g, c, _slots(c["cout"]), c["cout"])
            s["dw"] = torch.empty((c["cout"], taps, c["cin"]), device="cuda")
            s["db"] = torch.empty(c["cout"], device="cuda")
        return s
    if k != "poly":
        s["geom"] = projector.Geometry(_geometry_dict(c))
    if k in ("pair", "forward", "autograd"):
        s["x"] = _volumes(c, seed)
    if k in ("pair", "adjoint", "autograd"):
        s["y"] = _projections(c, seed + 1, noise=0.05)
    if k == "fdk":
        s["y"] = _projections(c, seed, noise=0.01)
    if k == "pdhg":
        s["y"] = _projections(c, seed, noise=0.01)
        s["x0"] = 0.8 * _volumes(c, seed)
        s["gamma"], s["step"] = _pdhg_steps(c)
    if k == "lire":
        s["net"] = lpd.LPD(s["geom"], n_iter=1, n_mem=8, lire=True, max_batch=c["batch"])
        s["y"], s["x0"] = _projections(c, seed, noise=0.01), 0.8 * _volumes(c, seed)
    if k == "poly":
        E, mw, mb, _ = inputs.poly_tables()
        n = c["bins"]
        s["tables"] = (E[:n], mw[:n], mb[:n])
        s["I0"] = torch.as_tensor(inputs.poly_intensity(_geometry_dict(c))[:n], device="cuda").contiguous()
        water = _projections(c, seed) * (1.0 / inputs.MU_WATER_60)
        bone = torch.stack([_chords(c, _ellipsoids(c, 1000 * seed + b + 500, 3)[1:]) for b in range(c["batch"])]) * 40.0
        s["L"] = torch.stack([water, bone], 1).contiguous()
        s["seed"] = seed
    return s


# ---- one pass -------------------------------------------------------------------------------


def run(s: dict):
    c, k = s["case"], s["case"]["kind"]
    if k == "forward":
        return projector.forward_project(s["geom"], s["x"])
    if k == "adjoint":
        return projector.back_project(s["geom"], s["y"])
    if k == "pair":
        return projector.forward_project(s["geom"], s["x"]), projector.back_project(s["geom"], s["y"])
    if k == "autograd":
        x = s["x"].requires_grad_(True)
        p = projector.project(s["geom"], x)
        return p.detach(), torch.autograd.grad(p, x, s["y"])[0]
    if k == "fdk":
        return ops.fdk(s["geom"], s["y"])
    if k == "pdhg":
        return ops.pdhg(s["geom"], s["y"], s["x0"], c["iters"], 0.5, s["gamma"], s["step"], s["step"])
    if k == "lire":
        return s["net"].forward(s["y"], s["x0"])
    if k == "poly":
        reading, y, counts = ops.poly_reading(s["L"], s["I0"], *s["tables"], s["seed"], noise=c["noise"],
                                              want_counts=c["counts"])
        return (reading, y) if counts is None else (reading, y, counts)
    st = torch.cuda.current_stream().cuda_stream
    lib = _lib.load()
    if k == "conv":
        g = c["grad"]
        _lib.check(lib.cbct_conv(s["x"].data_ptr(), c["nimg"], c["D"], c["H"], c["W"], 8 * s["x"].shape[3], c["taps3d"],
                                 s["w"].data_ptr(), None if g else s["b"].data_ptr(), c["cin"], c["cout"], int(g),
                                 2 if g else 0, SLOPE, s["y"].data_ptr(), 8 * s["y"].shape[3],
                                 s["mask"].data_ptr() if g else None, None, 0, s["status"].data_ptr(), st), "cbct_conv")
        return s["y"]
    _lib.check(lib.cbct_conv_wgrad(s["x"].data_ptr(), 8 * s["x"].shape[3], c["cin"], s["dy"].data_ptr(),
                                   8 * s["dy"].shape[3], c["cout"], c["nimg"], c["D"], c["H"], c["W"], c["taps3d"],
                                   s["dw"].data_ptr(), s["db"].data_ptr(), 0, s["status"].data_ptr(), st),
               "cbct_conv_wgrad")
    return s["dw"], s["db"]


# ---- what a pass cannot do without ----------------------------------------------------------


def _samples(c: dict) -> float:
    """(ray, plane) pairs with a nonzero bilinear footprint, from an even subset of the rays."""
    ks = np.unique(np.linspace(0, c["na"] - 1, min(c["na"], 24)).astype(int))
    us = np.unique(np.linspace(0, c["nu"] - 1, min(c["nu"], 48)).astype(int))
    vs = np.unique(np.linspace(0, c["nv"] - 1, min(c["nv"], 16)).astype(int))
    n, vox = np.array([c["nx"], c["ny"], c["nz"]]), np.array([c["vx"], c["vy"], c["vz"]])
    tot = 0
    for k in ks:
        th = 2.0 * math.pi * k / c["na"]
        S, D0, EU, EV = _frame(c, th)
        R = D0 + us[:, None, None] * EU + vs[None, :, None] * EV
        ax = (np.abs(R[..., 0]) < np.abs(R[..., 1])).astype(int)
        for a in (0, 1):
            r = R[ax == a]
            if not len(r):
                continue
            t = (np.arange(n[a])[None, :] - S[a]) / r[:, a:a + 1]
            qb, qz = S[1 - a] + t * r[:, 1 - a:2 - a], S[2] + t * r[:, 2:3]
            tot += np.count_nonzero((t > 0) & (t < 1) & (qb > -1) & (qb < n[1 - a]) & (qz > -1) & (qz < n[2]))
    return tot * (c["na"] / len(ks)) * (c["nu"] / len(us)) * (c["nv"] / len(vs))


def work(case: dict) -> dict:
    c, k = case, case["kind"]
    if k in ("conv", "wgrad"):
        taps, npix = (27 if c["taps3d"] else 9), c["nimg"] * c["D"] * c["H"] * c["W"]
        act = 2.0 * npix * (_slots(c["cin"]) + _slots(c["cout"]) + (_slots(c["cin"]) if c.get("grad") else 0))
        return {"bytes": act + 4.0 * taps * c["cin"] * c["cout"], "flops": 2.0 * npix * taps * c["cin"] * c["cout"]}
    vol, ray = 4.0 * c["batch"] * c["nx"] * c["ny"] * c["nz"], 4.0 * c["batch"] * c["na"] * c["nv"] * c["nu"]
    if k == "poly":
        # per draw: the exponential of the mean and one uniform pair
        return {"bytes": 2 * ray + 2 * ray + (c["bins"] * ray if c["counts"] else 0) + 4.0 * c["bins"] * c["nu"] * c["nv"],
                "flops": 20.0 * c["bins"] * ray / 4}
    if k == "fdk":
        nue = c["nu"] + math.ceil(2 * abs(c["uoff"]) / c["du"] - 1e-9)
        ramp = c["batch"] * c["na"] * c["nv"] * 10.0 * nue * math.log2(2 * nue)
        return {"bytes": vol + ray, "flops": ramp + 10.0 * c["na"] * vol / 4}
    if k == "lire":  # two projections and two backprojections; dual and primal blocks 8 -> 32 -> 32 -> 4, 3x3x3
        mac = 27 * (8 * 32 + 32 * 32 + 32 * 4)
        return {"bytes": 3 * ray + 4 * vol, "flops": 32.0 * c["batch"] * _samples(c) + 2.0 * mac * (vol + ray) / 4}
    s = c["batch"] * _samples(c)  # a bilinear sample (or its transpose): eight operations
    passes = {"forward": 1, "adjoint": 1, "pair": 2, "autograd": 2, "pdhg": 2 * c.get("iters", 1)}[k]
    byt = passes * (vol + ray)
    if k == "pdhg":  # per iteration also: z1 and x read and written, three dual components read and written
        byt += c["iters"] * (3 * ray + 10 * vol)
    return {"bytes": byt, "flops": 8.0 * s * passes}


# ---- the same in 64 bits --------------------------------------------------------------------


def _frame(c: dict, th: float):
    """Source, pixel (0, 0) direction, column and row steps in voxel-index coordinates."""
    co, si = math.cos(th), math.sin(th)
    vox = np.array([c["vx"], c["vy"], c["vz"]])
    a = -0.5 * (c["nu"] - 1) * c["du"] + c["uoff"]
    b = -0.5 * (c["nv"] - 1) * c["dv"] + c["voff"]
    S = np.array([inputs.SID_MM * co, inputs.SID_MM * si, 0.0]) / vox + 0.5 * (np.array([c["nx"], c["ny"], c["nz"]]) - 1)
    D0 = np.array([-inputs.SDD_MM * co - a * si, -inputs.SDD_MM * si + a * co, b]) / vox
    return S, D0, np.array([-c["du"] * si, c["du"] * co, 0.0]) / vox, np.array([0.0, 0.0, c["dv"]]) / vox


def _planes(c: dict, k: int):
    """For each principal axis at angle k: the columns of that axis, the in-plane coordinate
    q_b [planes, columns], q_z [planes, columns, rows], validity [planes, columns] and the
    step length [columns, rows], in 64 bits."""
    n, vox = (c["nx"], c["ny"], c["nz"]), (c["vx"], c["vy"], c["vz"])
    S, D0, EU, EV = _frame(c, 2.0 * math.pi * k / c["na"])
    iu = np.arange(c["nu"])
    # the principal axis is decided on the FP32 direction (one rounding of each column's sum)
    r32 = [(iu * np.float64(np.float32(EU[i])) + np.float64(np.float32(D0[i]))).astype(np.float32) for i in (0, 1)]
    isx = np.abs(r32[0]) >= np.abs(r32[1])
    rz = torch.as_tensor(D0[2] + np.arange(c["nv"]) * EV[2], device="cuda")
    for a in (0, 1):
        cols = np.nonzero(isx if a == 0 else ~isx)[0]
        if not len(cols):
            continue
        ra = torch.as_tensor(D0[a] + cols * EU[a], device="cuda")
        rb = torch.as_tensor(D0[1 - a] + cols * EU[1 - a], device="cuda")
        t = (torch.arange(n[a], device="cuda", dtype=torch.float64)[:, None] - S[a]) / ra
        qb, qz = S[1 - a] + t * rb, S[2] + t[:, :, None] * rz
        step = torch.sqrt(vox[a] ** 2 + (vox[1 - a] * rb / ra)[:, None] ** 2 + (vox[2] * rz / ra[:, None]) ** 2)
        yield a, torch.as_tensor(cols, device="cuda"), qb, qz, (t > 0) & (t < 1), step


def _split(q: torch.Tensor, n: int):
    """Cell index into an array padded by one on both sides, clamped outside, and the fraction."""
    f = torch.floor(q)
    ok = (f >= -1) & (f <= n - 1)
    return torch.where(ok, f + 1, torch.full_like(f, n + 1)).long(), q - f


def _forward64(c: dict, vol: torch.Tensor) -> torch.Tensor:
    """Joseph projection of [B, nz, ny, nx] in 64 bits."""
    n = (c["nx"], c["ny"], c["nz"])
    out = torch.zeros((vol.shape[0], c["na"], c["nv"], c["nu"]), device="cuda", dtype=torch.float64)
    for b in range(vol.shape[0]):
        v = vol[b].double()
        pl = [torch.nn.functional.pad(v.permute(2, 1, 0), (1, 2, 1, 2)), torch.nn.functional.pad(v.permute(1, 2, 0), (1, 2, 1, 2))]
        for k in range(c["na"]):
            for a, cols, qb, qz, ok, step in _planes(c, k):
                P, nb = pl[a], n[1 - a]  # [plane, b + pad, z + pad]
                jb, fb = _split(qb, nb)
                i = torch.arange(n[a], device="cuda")[:, None]
                row = (P[i, jb] * (1 - fb)[..., None] + P[i, jb + 1] * fb[..., None]) * ok[..., None]
                jz, fz = _split(qz, n[2])
                s = torch.gather(row, 2, jz) * (1 - fz) + torch.gather(row, 2, jz + 1) * fz
                out[b, k][:, cols] = (s.sum(0) * step).T
    return out


def _adjoint64(c: dict, proj: torch.Tensor) -> torch.Tensor:
    """The transpose of _forward64 on [B, na, nv, nu]."""
    n = (c["nx"], c["ny"], c["nz"])
    out = torch.zeros((proj.shape[0], c["nz"], c["ny"], c["nx"]), device="cuda", dtype=torch.float64)
    for b in range(proj.shape[0]):
        acc = [torch.zeros((n[a] * (n[1 - a] + 3), n[2] + 3), device="cuda", dtype=torch.float64) for a in (0, 1)]
        for k in range(c["na"]):
            for a, cols, qb, qz, ok, step in _planes(c, k):
                pw = proj[b, k].double()[:, cols].T * step  # [columns, rows]
                jz, fz = _split(qz, n[2])
                row = torch.zeros((n[a], len(cols), n[2] + 3), device="cuda", dtype=torch.float64)
                row.scatter_add_(2, jz, pw * (1 - fz))
                row.scatter_add_(2, jz + 1, pw * fz)
                row *= ok[..., None]
                jb, fb = _split(qb, n[1 - a])
                at = (torch.arange(n[a], device="cuda")[:, None] * (n[1 - a] + 3) + jb).reshape(-1)
                acc[a].index_add_(0, at, (row * (1 - fb)[..., None]).reshape(-1, n[2] + 3))
                acc[a].index_add_(0, at + 1, (row * fb[..., None]).reshape(-1, n[2] + 3))
        vx, vy = (acc[a].reshape(n[a], n[1 - a] + 3, n[2] + 3)[:, 1:n[1 - a] + 1, 1:n[2] + 1] for a in (0, 1))
        out[b] = vx.permute(2, 1, 0) + vy.permute(2, 0, 1)
    return out


def _fdk64(c: dict, proj: torch.Tensor) -> torch.Tensor:
    nu, nv, uoff = c["nu"], c["nv"], c["uoff"]
    u = (np.arange(nu) - 0.5 * (nu - 1)) * c["du"] + uoff
    v = (np.arange(nv) - 0.5 * (nv - 1)) * c["dv"] + c["voff"]
    D = 0.5 * nu * c["du"] - abs(uoff)
    us = u if uoff > 0 else -u
    w = np.full(nu, 0.5) if uoff == 0 else np.where(us < -D, 0.0, np.where(us > D, 1.0, np.sin(0.25 * math.pi * (us + D) / D) ** 2))
    pad = math.ceil(2 * abs(uoff) / c["du"] - 1e-9)
    nue, lo = nu + pad, (pad if uoff > 0 else 0)
    cosw = w[None, :] * inputs.SDD_MM / np.sqrt(inputs.SDD_MM ** 2 + u[None, :] ** 2 + v[:, None] ** 2)
    tau = c["du"] * inputs.SID_MM / inputs.SDD_MM
    d = np.arange(nue)[:, None] - np.arange(nue)[None, :]
    h = np.where(d == 0, 1 / (4 * tau), np.where(d % 2 != 0, -1.0 / (math.pi ** 2 * np.where(d == 0, 1, d) ** 2.0 * tau), 0.0))
    H, C = torch.as_tensor(h, device="cuda"), torch.as_tensor(cosw, device="cuda")
    x, y, z = (torch.as_tensor((np.arange(c["n" + a]) - 0.5 * (c["n" + a] - 1)) * c["v" + a], device="cuda") for a in "xyz")
    out = torch.zeros((proj.shape[0], c["nz"], c["ny"], c["nx"]), device="cuda", dtype=torch.float64)
    for b in range(proj.shape[0]):
        for k in range(c["na"]):
            q0 = torch.zeros((nv, nue), device="cuda", dtype=torch.float64)
            q0[:, lo:lo + nu] = proj[b, k].double() * C
            q = torch.nn.functional.pad(q0 @ H, (1, 2, 1, 2))
            th = 2.0 * math.pi * k / c["na"]
            co, si = math.cos(th), math.sin(th)
            U = inputs.SID_MM - (x[None, :] * co + y[:, None] * si)
            m = inputs.SDD_MM / U
            fu = (m * (-x[None, :] * si + y[:, None] * co) - uoff) / c["du"] + 0.5 * (nu - 1) + lo
            ju, au = _split(fu, nue)
            jv, av = _split((m[None] * z[:, None, None] - c["voff"]) / c["dv"] + 0.5 * (nv - 1), nv)
            flat, at = q.reshape(-1), jv * (nue + 3) + ju[None]
            s = (flat[at] * (1 - au) + flat[at + 1] * au) * (1 - av)
            s += (flat[at + nue + 3] * (1 - au) + flat[at + nue + 4] * au) * av
            out[b] += (inputs.SID_MM / U) ** 2 * s * (U > 0)
    return out * (2.0 * math.pi / c["na"])


def _pdhg64(c: dict, s: dict) -> torch.Tensor:
    def grad(x):
        g = torch.zeros((3,) + x.shape, device="cuda", dtype=torch.float64)
        g[0][..., :-1] = x[..., 1:] - x[..., :-1]
        g[1][..., :-1, :] = x[..., 1:, :] - x[..., :-1, :]
        g[2][..., :-1, :, :] = x[..., 1:, :, :] - x[..., :-1, :, :]
        return g

    def div(z):
        d = torch.zeros_like(z[0])
        for i, dim in enumerate((-1, -2, -3)):
            n = z[i].shape[dim]
            f = z[i].narrow(dim, 0, n - 1)
            d.narrow(dim, 0, n - 1).add_(f)
            d.narrow(dim, 1, n - 1).sub_(f)
        return d

    gamma, step, rad = s["gamma"], s["step"], 0.5 / s["gamma"]
    y, x = s["y"].double(), s["x0"].double()
    xb, z1, z2 = x.clone(), torch.zeros_like(y), torch.zeros((3,) + x.shape, device="cuda", dtype=torch.float64)
    for _ in range(c["iters"]):
        z1 = (z1 + step * (_forward64(c, xb) - y)) / (1 + step)
        z2 = z2 + step * gamma * grad(xb)
        nrm = torch.sqrt((z2 * z2).sum(0))
        z2 = z2 * torch.where(nrm > rad, rad / nrm, torch.ones_like(nrm))
        xn = (x - step * (_adjoint64(c, z1) - gamma * div(z2))).clamp(min=0.0)
        xb, x = 2 * xn - x, xn
    return x


def _channels(x: torch.Tensor) -> torch.Tensor:
    """Row-blocked [nimg, D, H, slots / 8, W, 8] -> zero-padded [nimg, D + 2, H + 2, W + 2, slots], FP64."""
    y = x.double().transpose(-3, -2)
    y = y.reshape(y.shape[:-2] + (-1,))
    return torch.nn.functional.pad(y, (0, 0, 1, 1, 1, 1, 1, 1))


def _taps(c: dict):
    for t in range(27 if c["taps3d"] else 9):
        yield t, (t // 9 if c["taps3d"] else 1), (t // 3) % 3, t % 3


def _conv64(c: dict, s: dict) -> torch.Tensor:
    x, w = _channels(s["x"]), s["w"].to(torch.bfloat16).double()
    D, H, W = c["D"], c["H"], c["W"]
    src, dst = (c["cout"], c["cin"]) if c["grad"] else (c["cin"], c["cout"])
    out = torch.zeros((c["nimg"], D, H, W, 8 * s["y"].shape[3]), device="cuda", dtype=torch.float64)
    for t, d, h, q in _taps(c):
        m = w[:, -1 - t] if c["grad"] else w[:, t].T  # [source channels, output channels]
        out[..., :dst] += x[:, d:d + D, h:h + H, q:q + W, :src] @ m
    if c["grad"]:
        mask = _channels(s["mask"])[:, 1:-1, 1:-1, 1:-1]
        out = torch.where(mask > 0, out, SLOPE * out)
    else:
        out[..., :dst] += s["b"].double()
        out = torch.where(out > 0, out, SLOPE * out)
    return out.reshape(out.shape[:-1] + (-1, 8)).transpose(-3, -2).contiguous()


def _wgrad64(c: dict, s: dict):
    x, dy = _channels(s["x"]), _channels(s["dy"])[:, 1:-1, 1:-1, 1:-1, :c["cout"]].reshape(-1, c["cout"])
    D, H, W = c["D"], c["H"], c["W"]
    dw = torch.zeros_like(s["dw"], dtype=torch.float64)
    for t, d, h, q in _taps(c):
        dw[:, t] = dy.T @ x[:, d:d + D, h:h + H, q:q + W, :c["cin"]].reshape(-1, c["cin"])
    return dw, dy.sum(0)


def exact(case: dict, seed: int):
    c, k = case, case["kind"]
    if k == "lire" or (k == "poly" and c["noise"]):
        return None  # BF16 roundings inside, random draws: no value in 64 bits
    s = prepare(c, seed)
    if k == "forward":
        return _forward64(c, s["x"])
    if k == "adjoint":
        return _adjoint64(c, s["y"])
    if k in ("pair", "autograd"):
        return _forward64(c, s["x"]), _adjoint64(c, s["y"])
    if k == "fdk":
        return _fdk64(c, s["y"])
    if k == "pdhg":
        return _pdhg64(c, s)
    if k == "conv":
        return _conv64(c, s)
    if k == "wgrad":
        return _wgrad64(c, s)
    E, mw, mb = s["tables"]
    resp = np.interp(E, [20.0, 60.0, 120.0], [5.0, 20.0, 10.0])
    reading = torch.zeros_like(s["L"][:, 0], dtype=torch.float64)
    air = torch.zeros_like(s["I0"][0], dtype=torch.float64)
    for j in range(len(E)):
        i0 = s["I0"][j].double()
        reading += resp[j] * i0 * torch.exp(-(mw[j] * s["L"][:, 0].double() + mb[j] * s["L"][:, 1].double()))
        air += resp[j] * i0
    return reading, -torch.log((reading.clamp(min=resp.min()) / air).clamp(max=1.0))
