"""Volumes of an odd number of voxels with panels a multiple of 4 wide: the iterative solvers'
scratch projections, and a caller's output off a 16-byte boundary, take the forward projector's
vector stores only where the buffer allows them."""
import math

import numpy as np
import pytest
import torch

from paper_2512_21180_gb300 import inputs as I
from paper_2512_21180_gb300 import ops
from paper_2512_21180_gb300 import projector as P

from gpu_util import rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu

# 45 x 47 x 43 voxels (odd), 64 columns: the staged forward kernel with full-width tiles
G_ODD = I.scaled(I.geometry("tiny16"), n=(45, 47, 43), vox=(4.0, 4.0, 4.0), nu=64, nv=40, du=2.9, dv=3.0, n_angles=12)


def test_solvers_on_odd_volumes(O):
    g = I.scaled(I.geometry("tiny16"), n=(15, 17, 11), nu=32, nv=16, du=3.2, dv=4.0, u_offset=6.0, n_angles=16)
    G, geom = O.Geom(g), P.Geometry(g)
    y = O.forward(G, O.phantom(G, I.ellipsoids(g, 3, n_soft=5, axes_mm=(8.0, 30.0))))
    gam = O.opnorm_P(G) / math.sqrt(12.0)
    sig = 0.99 / O.opnorm_K(G, gamma=gam)
    ref = O.pdhg(G, y, np.zeros(G.vol_shape), 30, 0.05, sig, sig, gamma=gam)
    got = to_np(ops.pdhg(geom, to_gpu(y), torch.zeros((1,) + G.vol_shape, device="cuda"), 30, 0.05, gam, sig, sig))[0]
    assert rel_l2(got, ref) <= 1e-4
    assert abs(ops.opnorm(geom, gamma=5.0, iters=100) / O.opnorm_K(G, iters=100, gamma=5.0) - 1.0) < 1e-4


def test_solver_scratch_on_staged_sizes():
    geom = P.Geometry(G_ODD)
    y = torch.rand((1,) + geom.proj_shape, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    x = torch.zeros((1,) + geom.vol_shape, device="cuda")
    tau = 1.0 / ops.opnorm(geom, iters=10) ** 2
    want = x - tau * P.back_project(geom, P.forward_project(geom, x) - y)
    want = want - tau * P.back_project(geom, P.forward_project(geom, want) - y)
    assert rel_l2(to_np(ops.landweber(geom, y, x, 2, tau)), to_np(want)) <= 1e-6
    z = ops.pdhg(geom, y, x, 3, 0.1, 10.0, 1e-3, 1e-3)
    assert bool(torch.isfinite(z).all()) and float(z.abs().max()) > 0


def test_forward_output_off_16_bytes():
    geom = P.Geometry(G_ODD)
    x = torch.as_tensor(I.random_volume((1,) + geom.vol_shape, 3), device="cuda")
    want = P.forward_project(geom, x)
    buf = torch.ones(want.numel() + 1, device="cuda")
    out = buf[1:].reshape(want.shape)
    P.forward_project(geom, x, out=out)
    assert torch.equal(out, want)
    P.forward_project(geom, x, out=out, accumulate=True)
    assert float((out - 2 * want).abs().max()) <= 1e-6 * float(want.abs().max())
