"""Segment-gather backprojection at the edges of its tiling: footprints of several tiles in
columns and rows, parts of more angles than one list holds, panels smaller than a tile, odd
sizes, batches, and non-finite pixels. The reference is the FP64 instantiation, an independent
kernel that visits every row of every column."""
import numpy as np
import pytest
import torch

from paper_2512_21180_gb300 import inputs as I
from paper_2512_21180_gb300 import projector as P

pytestmark = pytest.mark.gpu

T = I.geometry("tiny16")
CASES = {
    # 30 pixels per voxel: a brick sees about 500 columns x 300 rows (5 x 6 tiles)
    "fine_panel": I.scaled(T, n=(20, 18, 11), vox=(8.0, 8.0, 8.0), nu=601, nv=333, du=0.41, dv=0.43, n_angles=3),
    # one part of more than 128 angles (16 parts)
    "many_angles": I.scaled(T, n=(17, 16, 9), n_angles=2100),
    # 64 bricks and more: parts of eight angles and a last one of fewer
    "eight_per_part": I.scaled(T, n=(64, 52, 60), vox=(4.0, 4.0, 4.0), nu=90, nv=60, du=2.9, dv=4.1, n_angles=61),
    # panels of one row, one column, and widths around a multiple of 4
    "one_row": I.scaled(T, nv=1, nu=31, n_angles=5),
    "one_column": I.scaled(T, nu=1, nv=29, n_angles=5),
    "nu_113": I.scaled(T, n=(33, 31, 17), nu=113, nv=53, du=1.3, dv=1.9, u_offset=11.0, v_offset=-7.0, n_angles=11),
    # coarse panel: less than one row per voxel
    "coarse_panel": I.scaled(T, n=(40, 44, 24), vox=(2.0, 2.0, 2.0), nu=22, nv=9, du=7.0, dv=9.0, n_angles=7),
    # volume reaching close to the source: strongly varying magnification
    "near_source": I.scaled(T, n=(48, 48, 8), vox=(28.0, 28.0, 10.0), nu=200, nv=24, du=4.0, dv=4.0, n_angles=9),
}
TOL = 1e-5  # the FP32 projector pair's bar against 64 bits


@pytest.mark.parametrize("batch", [1, 3])
@pytest.mark.parametrize("name", list(CASES))
def test_tiles_match_fp64(name, batch):
    geom = P.Geometry(CASES[name])
    y = torch.as_tensor(I.random_volume((batch,) + geom.proj_shape, 31), device="cuda")
    got = P.back_project(geom, y)
    ref = P.back_project(geom, y.double())
    assert float((got.double() - ref).norm()) <= TOL * float(ref.norm())
    assert float((got.double() - ref).abs().max()) <= TOL * float(ref.abs().max())
    acc = P.back_project(geom, y, out=torch.ones_like(got), accumulate=True)
    assert float((acc - 1.0 - got).abs().max()) <= 4e-7 * (1.0 + float(got.abs().max()))
    assert torch.equal(got, P.back_project(geom, y))
    assert geom.device_status() == 0


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf"), 3e38])
def test_non_finite_pixels_reach_only_their_voxels(value):
    """One bad pixel: the voxels its ray touches (FP64 backprojection of that pixel alone)
    become non-finite (or huge, for a finite pixel whose column sums overflow), every other
    voxel keeps its value."""
    g = I.scaled(T, n=(20, 20, 20), vox=(4.0, 4.0, 4.0), nu=61, nv=57, du=1.6, dv=1.6, n_angles=6)
    geom = P.Geometry(g)
    y = torch.as_tensor(I.random_volume((1,) + geom.proj_shape, 5), device="cuda")
    clean = P.back_project(geom, y)
    at = (0, 2, 30, 33)
    one = torch.zeros_like(y, dtype=torch.float64)
    one[at] = 1.0
    w = P.back_project(geom, one)
    y[at] = value
    if value == 3e38:
        y[0, 2, 31, 33] = value  # the two add up to more than FP32 holds
        one[0, 2, 31, 33] = 1.0
        w = P.back_project(geom, one)
    got = P.back_project(geom, y)
    touched, untouched = w > 1e-4 * w.max(), w == 0
    assert int(touched.sum()) > 20 and int(untouched.sum()) > 1000
    if value == 3e38:
        assert bool((got[touched].abs() > 1e30).all())
    else:
        assert not bool(torch.isfinite(got[touched]).any())
    assert float((got[untouched] - clean[untouched]).abs().max()) <= TOL * float(clean.abs().max())


def test_empty_projection_gives_exact_zeros():
    geom = P.Geometry(CASES["nu_113"])
    assert float(P.back_project(geom, torch.zeros((1,) + geom.proj_shape, device="cuda")).abs().max()) == 0.0
    y = torch.zeros((1,) + geom.proj_shape, device="cuda")
    y[0, 3, 20, 50] = 1e6
    got, ref = P.back_project(geom, y), P.back_project(geom, y.double())
    assert bool((got[ref == 0] == 0).all())


@pytest.mark.parametrize("name", ["fine_panel", "eight_per_part", "nu_113", "coarse_panel", "near_source"])
@pytest.mark.parametrize("value", [1e2, 1e3, 1e4, 1e6, 1e9])
def test_large_pixels_leave_other_voxels_alone(name, value):
    """Large finite pixels on a positive background: a voxel that their rays give no weight keeps
    its value. Columns that span more than a factor of 1024 (windows of up to four rows) are summed row by
    row: 1e-5, the projector pair's bar, for 1e4 and more; so is 1e2 by its size. Just below the factor, a
    prefix sum of 1024 windows rounds to 2^-24 of itself, 6e-5 of the smallest window, with a lever arm of up
    to 26 rows in the interval's first moment: 1e-4 once the columns and angles of a voxel average it."""
    geom = P.Geometry(CASES[name])
    na, nv, nu = geom.proj_shape
    y = torch.as_tensor(I.random_volume((1,) + geom.proj_shape, 9), device="cuda").abs() + 0.1
    clean = P.back_project(geom, y)
    hot = torch.zeros_like(y)
    hot[0, :, nv // 4::max(1, nv // 3), nu // 5::max(1, nu // 4)] = 1.0
    w = P.back_project(geom, hot)
    got = P.back_project(geom, torch.where(hot > 0, torch.full_like(y, value), y))
    far = (w == 0) & (P.back_project(geom, hot.double()) == 0) & (clean > 0.05 * clean.max())
    assert int(far.sum()) > 300 and int((w > 0).sum()) > 50
    tol = 1e-4 if value == 1e3 else 1e-5
    assert float(((got[far] - clean[far]).abs() / clean[far]).max()) <= tol


@pytest.mark.parametrize("name", ["many_angles", "eight_per_part", "nu_113", "near_source"])
def test_smooth_projections_to_a_few_roundings(name):
    """On smooth projections a voxel is a sum of short FP32 sums: measured 1.6e-7 to 3.5e-7 of the norm on
    scans; 1e-6 tells a longer sum or a lost bit."""
    geom = P.Geometry(CASES[name])
    na, nv, nu = geom.proj_shape
    k, v, u = (torch.linspace(-1, 1, n, device="cuda", dtype=torch.float64) for n in (na, nv, nu))
    p = 3.0 * torch.exp(-u[None, None] ** 2 - v[None, :, None] ** 2) * (1.0 + 0.2 * torch.cos(9.0 * k))[:, None, None]
    p = p.float()[None].contiguous()
    got, ref = P.back_project(geom, p), P.back_project(geom, p.double())
    assert float((got.double() - ref).norm()) <= 1e-6 * float(ref.norm())


@pytest.mark.parametrize("name", ["fine_panel", "eight_per_part", "nu_113"])
@pytest.mark.parametrize("rows", [(0, 1), (2, 3), (-2, -1), (-4, -3)])
def test_large_pixels_near_the_panel_edges(name, rows):
    """A large pixel in one of the last rows of the panel (or of a tile of a finer panel) has no full window
    of rows behind it; the voxels that only see those rows keep their value all the same."""
    geom = P.Geometry(CASES[name])
    na, nv, nu = geom.proj_shape
    y = torch.as_tensor(I.random_volume((1,) + geom.proj_shape, 9), device="cuda").abs() + 0.1
    clean = P.back_project(geom, y)
    step = 52 if name == "fine_panel" else nv     # (tiles of 52 rows)
    for row in rows:
        hot = torch.zeros_like(y)
        hot[0, :, row % step::step, nu // 5::max(1, nu // 4)] = 1.0
        got = P.back_project(geom, torch.where(hot > 0, torch.full_like(y, 1e6), y))
        far = (P.back_project(geom, hot) == 0) & (P.back_project(geom, hot.double()) == 0) & (clean > 0.01 * clean.max())
        assert int(far.sum()) > 300
        assert float(((got[far] - clean[far]).abs() / clean[far]).max()) <= 1e-5
