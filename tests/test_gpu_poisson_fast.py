"""Counts of the FP32-decided Poisson sampler against the FP64 definition of the oracle, at the
means where its branches meet or give up: around 10 (inversion / rejection), next to zero, above
the range FP32 handles, intensities that are not FP32 numbers, rays that absorb everything."""
import numpy as np
import pytest
import torch

from paper_2512_21180_gb300 import inputs as I
from paper_2512_21180_gb300 import ops

from gpu_util import to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("I0,lo,hi", [
    (10.0, 0.0, 1e-4), (10.00001, 0.0, 1e-4), (12.3456789012345, 0.0, 0.5), (1e5, 0.0, 1e-3), (1e5, 9.0, 30.0),
    (3e6, -0.5, 2.0), (5e6, 0.0, 0.3), (1e9, 15.0, 70.0), (1e-3, -8.0, 2.0), (1e13, 30.0, 120.0)])
def test_counts_at_the_edges(O, I0, lo, hi):
    p = I.line_integrals(300_001, 5, lo, hi)
    p[:4] = [lo, hi, np.float32(np.inf), np.float32(np.nan)]
    got = ops.poisson(to_gpu(p), I0, seed=2**40 + 9).cpu().numpy()
    assert np.array_equal(got, O.poisson(p, I0, seed=2**40 + 9))


@pytest.mark.parametrize("n_ang,nv,nu,batch,ne", [(1, 1, 1, 1, 1), (70, 3, 5, 2, 16), (5, 37, 71, 3, 4)])
def test_reading_counts_with_dark_pixels(O, n_ang, nv, nu, batch, ne):
    """Ragged panels and frame groups, pixels of no intensity, line integrals from 0 to opaque."""
    rng = np.random.default_rng(ne)
    E = np.linspace(25.0, 115.0, ne)
    mw, mb = rng.uniform(0.01, 0.04, ne), rng.uniform(0.03, 0.2, ne)
    I0 = rng.uniform(0.0, 5000.0, (ne, nv, nu)).astype(np.float32)
    I0[:, 0, 0] = 0.0
    L = rng.uniform(0.0, 300.0, (batch, 2, n_ang, nv, nu)).astype(np.float32)
    L[:, :, 0] = 0.0
    L[:, 0, -1] = 5000.0
    r, y, c = ops.poly_reading(to_gpu(L), to_gpu(I0), E, mw, mb, seed=3, want_counts=True)
    Lw, Lb = (L[:, i].astype(np.float64)[..., None] for i in (0, 1))
    lam = np.moveaxis(I0.astype(np.float64), 0, -1) * np.exp(-(mw * Lw + mb * Lb))
    ref = O.poisson_lam(lam.reshape(-1), 3).reshape(c.shape)
    assert np.array_equal(c.cpu().numpy(), ref)
    resp = np.array([O.resp(e) for e in E])
    want = (ref * resp).sum(-1)
    np.testing.assert_allclose(r.cpu().numpy(), want, rtol=1e-6, atol=1e-6)
    assert bool(torch.isfinite(y[..., 1:, :] if nv > 1 else y[..., 1:]).all())
