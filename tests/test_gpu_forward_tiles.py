"""Staged forward projection at the edges of its tiling: every box configuration, rows that span
two and more z-cells, rows and columns past the panel, volumes whose rows do not start on 16
bytes, planes cut by the panel, small calls on the direct kernel, and non-finite voxels. The
reference is the FP64 instantiation, an independent kernel with one thread per ray."""
import ctypes

import pytest
import torch

from paper_2512_21180_gb300 import _lib
from paper_2512_21180_gb300 import inputs as I
from paper_2512_21180_gb300 import projector as P

pytestmark = pytest.mark.gpu

T = I.geometry("tiny16")


def scan(n, vox, nu, nv, du, dv, na=9, **kw):
    return I.scaled(T, n=n, vox=(vox, vox, 4.0 if vox > 2 else 2.0), nu=nu, nv=nv, du=du, dv=dv, n_angles=na, **kw)


# name -> (geometry, box configuration chosen for it)
CASES = {
    "box0": (scan((64, 60, 40), 4.0, 130, 70, 1.2, 1.2), 0),
    "box1_ragged": (scan((61, 63, 41), 4.0, 121, 50, 1.6, 1.6, u_offset=30.0, v_offset=5.0), 1),
    "box2": (scan((60, 64, 40), 4.0, 101, 45, 2.4, 2.7), 2),
    "box3": (scan((60, 66, 40), 4.0, 81, 45, 3.2, 3.4), 3),
    "box5_four_cells": (scan((67, 64, 40), 4.0, 61, 33, 4.5, 5.0, 15), 5),
    "box6_five_cells": (scan((67, 64, 40), 2.5, 61, 33, 4.5, 6.0, 15), 6),
    "direct": (scan((64, 64, 40), 2.0, 61, 33, 7.0, 7.0, 15), -1),
    "panel_cuts_volume": (scan((96, 96, 24), 12.0, 150, 40, 4.0, 4.0, 15), 5),
    "nv_one": (scan((64, 60, 40), 4.0, 1030, 1, 0.4, 1.2, 20), None),
}
TOL = 1e-5  # the FP32 projector pair's bar against 64 bits


def check(got, ref):
    assert float((got.double() - ref).norm()) <= TOL * float(ref.norm())
    assert float((got.double() - ref).abs().max()) <= TOL * float(ref.abs().max())


@pytest.mark.parametrize("batch", [1, 2])
@pytest.mark.parametrize("name", list(CASES))
def test_boxes_match_fp64(name, batch):
    g, cfg = CASES[name]
    geom = P.Geometry(g)
    c = ctypes.c_int()
    _lib.check(_lib.load().cbct_forward_config(geom.handle, ctypes.byref(c), None, None))
    assert cfg is None or c.value == cfg
    x = torch.as_tensor(I.random_volume((batch,) + geom.vol_shape, 17), device="cuda")
    got = P.forward_project(geom, x)
    check(got, P.forward_project(geom, x.double()))
    acc = P.forward_project(geom, x, out=torch.ones_like(got), accumulate=True)
    assert float((acc - 1.0 - got).abs().max()) <= 4e-7 * (1.0 + float(got.abs().max()))
    assert torch.equal(got, P.forward_project(geom, x))
    assert geom.device_status() == 0


@pytest.mark.parametrize("nx", [16, 17])
@pytest.mark.parametrize("du,cfg", [(3.2, None), (4.5, 4)])
def test_more_slices_than_a_grid_holds(du, cfg, nx):
    """257 volumes of 256 slices (65,792): more than a grid's z extent, on a fine panel and on one
    whose box is among the coarse ones; items against the FP64 instantiation."""
    geom = P.Geometry(I.scaled(T, n=(nx, 16, 256), vox=(4.0, 4.0, 4.0), nu=31, nv=33, du=du, dv=1.1 * du, n_angles=5))
    c = ctypes.c_int()
    _lib.check(_lib.load().cbct_forward_config(geom.handle, ctypes.byref(c), None, None))
    assert c.value >= 0 and (cfg is None or c.value == cfg)
    x = torch.as_tensor(I.random_volume((257,) + geom.vol_shape, 23), device="cuda")
    got = P.forward_project(geom, x)
    for b in (0, 128, 255, 256):
        check(got[b:b + 1], P.forward_project(geom, x[b:b + 1].double()))


def test_threads_with_geometries_of_one_box():
    """Two volumes of different length share a kernel whose shared memory follows the length."""
    import threading
    geoms = [P.Geometry(scan((n, 60, 40), 4.0, 130, 70, 1.2, 1.2)) for n in (64, 66)]
    xs = [torch.as_tensor(I.random_volume((1,) + g.vol_shape, 3), device="cuda") for g in geoms]
    want = [P.forward_project(g, x) for g, x in zip(geoms, xs)]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                outs = [P.forward_project(geoms[i], xs[i]) for _ in range(100)]
                torch.cuda.current_stream().synchronize()
                if not all(torch.equal(o, want[i]) for o in outs):
                    bad.append(i)
        except Exception as e:  # (a refused launch)
            bad.append(e)

    ts = [threading.Thread(target=work, args=(i % 2,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad


def test_volume_rows_off_16_bytes():
    """A contiguous volume at an odd element offset of a larger buffer (x rows of 64 voxels)."""
    geom = P.Geometry(CASES["box0"][0])
    n = 64 * 60 * 40
    buf = torch.as_tensor(I.random_volume((n + 3,), 4), device="cuda")
    want = P.forward_project(geom, buf[3:].clone().reshape((1,) + geom.vol_shape))
    assert torch.equal(P.forward_project(geom, buf[3:].reshape((1,) + geom.vol_shape)), want)


@pytest.mark.parametrize("name", ["box0", "box1_ragged", "box5_four_cells", "panel_cuts_volume"])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
def test_non_finite_voxels_reach_only_their_rays(name, value):
    """The rays whose bilinear footprint holds the voxel (the FP64 projection of that voxel alone)
    become non-finite, every other ray keeps its value."""
    geom = P.Geometry(CASES[name][0])
    x = torch.as_tensor(I.random_volume((1,) + geom.vol_shape, 8), device="cuda")
    clean = P.forward_project(geom, x)
    at = (0,) + tuple(n // 2 for n in geom.vol_shape)
    one = torch.zeros_like(x, dtype=torch.float64)
    one[at] = 1.0
    w = P.forward_project(geom, one)
    x[at] = value
    got = P.forward_project(geom, x)
    touched = w > 1e-4 * w.max()
    assert int(touched.sum()) >= 9
    assert not bool(torch.isfinite(got[touched]).any())
    far = w == 0
    assert bool(torch.isfinite(got[far]).all())
    assert float((got[far] - clean[far]).abs().max()) <= TOL * float(clean.abs().max())


@pytest.mark.parametrize("name", ["box0", "box1_ragged", "box2", "box3", "box5_four_cells", "box6_five_cells"])
@pytest.mark.parametrize("value", [1e2, 1e4, 1e6, 1e9])
def test_large_voxels_leave_other_rays_alone(name, value):
    """Large finite voxels (alternate z-slices of a block, so that rows which share levels lie on both
    sides of them): a ray that gives them no weight keeps its value to a rounding of its own sum,
    whatever they hold."""
    geom = P.Geometry(CASES[name][0])
    x = torch.as_tensor(I.random_volume((1,) + geom.vol_shape, 8), device="cuda").abs() + 0.1
    clean = P.forward_project(geom, x)
    nz, ny, nx = geom.vol_shape
    hot = torch.zeros_like(x)
    hot[0, nz // 4:3 * nz // 4:5, ny // 3:ny // 3 + 3, nx // 2:nx // 2 + 5] = 1.0
    w = P.forward_project(geom, hot)      # the same sample positions
    got = P.forward_project(geom, torch.where(hot > 0, torch.full_like(x, value), x))
    far, near = w == 0, w > 0
    assert int(near.sum()) > 100 and int(far.sum()) > 1000
    # about a hundred positive samples, each rounded to 2^-24 of its value: the two sums may be grouped alike
    assert float(((got[far] - clean[far]).abs() - 1e-6 * clean[far]).max()) <= 0.0


@pytest.mark.parametrize("name", ["box0", "box1_ragged", "box2", "box3", "box5_four_cells", "nv_one"])
def test_smooth_volumes_to_a_few_roundings(name):
    """On a smooth volume the positions' rounding hardly shows, and a ray is a short sum of FP32 samples:
    measured 1e-7 to 4e-7 of the norm on scans; 1e-6 tells a longer sum or a lost bit."""
    geom = P.Geometry(CASES[name][0])
    z, y, x = (torch.linspace(-1, 1, n, device="cuda", dtype=torch.float64) for n in geom.vol_shape)
    v = torch.exp(-2.0 * (x[None, None] ** 2 + (y[None, :, None] - 0.2) ** 2 + (z[:, None, None] + 0.1) ** 2))
    v = (0.02 * v * (1.0 + 0.3 * torch.cos(3.0 * x + 1.0))).float()[None]
    got, ref = P.forward_project(geom, v), P.forward_project(geom, v.double())
    assert float((got.double() - ref).norm()) <= 1e-6 * float(ref.norm())
