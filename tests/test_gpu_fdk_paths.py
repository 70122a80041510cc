"""FDK_w over its row filters (direct, transforms of 1024, 2048 and 4096 points) and angle splits,
against the FP64 oracle: odd row counts (a last row without a partner), batches, accumulation, and
rows with a non-finite value, which must not reach the rows they share a transform with."""
import numpy as np
import pytest
import torch

from paper_2512_21180_gb300 import _lib
from paper_2512_21180_gb300 import inputs as I
from paper_2512_21180_gb300 import ops
from paper_2512_21180_gb300 import projector as P

from gpu_util import rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu

B = I.geometry("small64")
CASES = {
    "direct_wide": I.scaled(B, n=(20, 18, 9), nu=2050, nv=3, du=0.2, dv=8.0, n_angles=8),
    "direct_small_split": I.scaled(B, n=(23, 21, 17), nu=90, nv=31, du=3.0, dv=5.0, n_angles=70, u_offset=30.0),
    "fft1024": I.scaled(B, n=(24, 26, 19), nu=300, nv=41, du=1.1, dv=4.0, n_angles=30),
    "fft1024_edge": I.scaled(B, n=(24, 26, 19), nu=512, nv=35, du=0.6, dv=4.0, n_angles=30, v_offset=9.0),
    "fft2048_offset": I.scaled(B, n=(24, 26, 19), nu=400, nv=37, du=0.9, dv=4.0, n_angles=30, u_offset=-110.0),
    "fft4096": I.scaled(B, n=(24, 26, 19), nu=1300, nv=35, du=0.25, dv=4.0, n_angles=30, u_offset=60.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_paths_match_oracle(O, name):
    g = CASES[name]
    G, geom = O.Geom(g), P.Geometry(g)
    y = np.stack([O.forward(G, O.phantom(G, I.ellipsoids(g, 3 + b, n_soft=6, axes_mm=(8.0, 50.0)))) for b in range(2)])
    y = y.astype(np.float32)
    got = ops.fdk(geom, to_gpu(y))
    for b in range(2):
        assert rel_l2(to_np(got[b]), O.fdk(G, y[b].astype(np.float64))) <= 1e-4  # the FDK bar (positions in FP32)
    assert torch.equal(ops.fdk(geom, to_gpu(y)), got)
    acc, yg = torch.ones_like(got), to_gpu(y)
    _lib.check(_lib.load().cbct_fdk(geom.handle, yg.data_ptr(), acc.data_ptr(), 2, 1,
                                    torch.cuda.current_stream().cuda_stream))
    assert float((acc - 1.0 - got).abs().max()) <= 1e-6 * (1.0 + float(got.abs().max()))


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 3e38])
@pytest.mark.parametrize("name", ["fft1024", "direct_small_split"])
def test_non_finite_row_stays_in_its_row(O, name, value):
    g = CASES[name]
    geom = P.Geometry(g)
    y = to_gpu(I.random_volume((1,) + geom.proj_shape, 6))
    clean = ops.fdk(geom, y)
    k, iv = 5, 12
    y[0, k, iv, 40:44] = value
    got = ops.fdk(geom, y)
    # detector row of every voxel at that angle
    z, yy, x = (torch.arange(n, device="cuda", dtype=torch.float64) - 0.5 * (n - 1) for n in geom.vol_shape)
    th = 2 * np.pi * k / g["n_angles"]
    U = 1000.0 - 4.0 * (x[None, :] * np.cos(th) + yy[:, None] * np.sin(th))
    fv = (1536.0 / U)[None] * (4.0 * z)[:, None, None] / g["dv"] + 0.5 * (g["nv"] - 1)
    far = ((fv - iv).abs() > 1.01)[None]
    assert float((got[far] - clean[far]).abs().max()) <= 1e-6 * float(clean.abs().max())
    near = ((fv - iv).abs() < 0.9)[None]
    assert int(near.sum()) > 100
    if value != 3e38:
        assert int((~torch.isfinite(got[near])).sum()) > 50


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 3e38])
@pytest.mark.parametrize("rows", [(12,), (13,), (12, 13)])
def test_a_bad_row_leaves_its_partner_alone(O, rows, value):
    """Rows 12 and 13 share a transform: one of them with four bad pixels, or both. Every voxel whose
    detector row lies a row away from the bad ones keeps its bits, the partner's own band included."""
    g = CASES["fft1024"]
    geom = P.Geometry(g)
    y = to_gpu(I.random_volume((1,) + geom.proj_shape, 6))
    k = 5
    # the other angles, and the bad rows, contribute nothing: what is left is the partner's band
    y[0, :k] = 0.0
    y[0, k + 1:] = 0.0
    for iv in rows:
        y[0, k, iv] = 0.0
    clean = ops.fdk(geom, y)
    for iv in rows:
        y[0, k, iv, 40:44] = value
    got = ops.fdk(geom, y)
    z, yy, x = (torch.arange(n, device="cuda", dtype=torch.float64) - 0.5 * (n - 1) for n in geom.vol_shape)
    th = 2 * np.pi * k / g["n_angles"]
    U = 1000.0 - 4.0 * (x[None, :] * np.cos(th) + yy[:, None] * np.sin(th))
    fv = ((1536.0 / U)[None] * (4.0 * z)[:, None, None] / g["dv"] + 0.5 * (g["nv"] - 1))[None]
    far = ((fv < min(rows) - 1.01) | (fv > max(rows) + 1.01))
    assert int(far.sum()) > 1000
    if value == 3e38:   # finite, but the transform overflows: the partner is summed tap by tap
        assert float((got[far] - clean[far]).abs().max()) <= 1e-6 * float(clean.abs().max())
    else:
        assert torch.equal(got[far], clean[far])
        near = torch.zeros_like(far)
        for iv in rows:
            near |= (fv - iv).abs() < 0.9
        assert int((~torch.isfinite(got[near])).sum()) > 50


def detector_rows(geom, g, k):
    """Detector row coordinate of every voxel at angle k."""
    z, yy, x = (torch.arange(n, device="cuda", dtype=torch.float64) - 0.5 * (n - 1) for n in geom.vol_shape)
    th = 2 * np.pi * k / g["n_angles"]
    U = 1000.0 - 4.0 * (x[None, :] * np.cos(th) + yy[:, None] * np.sin(th))
    fv = (1536.0 / U)[None] * (4.0 * z)[:, None, None] - g["v_offset"]
    return (fv / g["dv"] + 0.5 * (g["nv"] - 1))[None]


@pytest.mark.parametrize("name", ["fft1024", "fft2048_offset", "fft4096"])
@pytest.mark.parametrize("large", [12, 13])
@pytest.mark.parametrize("factor", [1e3, 1e6, 1e9, 1e30])
def test_rows_round_to_their_own_size(name, large, factor):
    """Rows 12 and 13 share a transform; one of them is larger by a factor. The voxels on the other
    row's side do not see it and keep what they get beside an empty row, to the transform's rounding of
    their own row (about 11 passes of 2^-24 on values three times the largest output: 2e-6)."""
    g, k = CASES[name], 5
    geom = P.Geometry(g)
    y = torch.zeros((1,) + geom.proj_shape, device="cuda")
    y[0, k] = to_gpu(I.random_volume(geom.proj_shape[1:], 6)).abs() + 0.1
    alone, beside = y.clone(), y.clone()
    alone[0, k, large] = 0.0
    beside[0, k, large] *= factor
    want, got = ops.fdk(geom, alone), ops.fdk(geom, beside)
    fv = detector_rows(geom, g, k)
    far = (fv < large - 1.01) | (fv > large + 1.01)
    other = far & ((fv - (25 - large)).abs() < 0.9)   # voxels that see the partner
    assert int(far.sum()) > 1000 and int(other.sum()) > 50
    assert float((got[far] - want[far]).abs().max()) <= 2e-6 * float(want.abs().max())


@pytest.mark.parametrize("name", ["fft1024", "fft4096"])
def test_an_empty_row_stays_empty_beside_its_partner(name):
    g, k = CASES[name], 5
    geom = P.Geometry(g)
    y = torch.zeros((1,) + geom.proj_shape, device="cuda")
    y[0, k, 12] = to_gpu(I.random_volume((geom.proj_shape[2],), 6)).abs() + 0.1
    got, fv = ops.fdk(geom, y), detector_rows(geom, g, k)
    partner = (fv > 13.01) & (fv < 13.9)
    assert int(partner.sum()) > 100 and int((got != 0).sum()) > 100
    assert bool((got[partner] == 0).all())
