"""The one-launch Jacobi of dk_pca_fit at the sizes where its layout changes: the smallest, odd
feature counts (a padded pair), one CTA against several (between 134 and 136 features), a
shorter last CTA.

Tolerance, derived before the first run: a fit of 10 sweeps applies about 10 p rotations to a
row, each with a relative rounding of 2 u; as a random walk sqrt(10 * 785) * 2 * 6e-8 = 1e-5 of a
row's norm, taken ten times as large for the components' orthonormality and for the residual
C v - lambda v relative to the largest eigenvalue (together they bound every eigenvalue's error
by the same amount). The off-diagonal norm as in test_pca_gpu.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [2, 3, 9, 64, 134, 136, 199, 256, 785])
def test_one_launch_jacobi(p):
    import torch
    from oracle import preprocess as pp
    from paper_2602_01330_gb300 import build, dualk
    build.build()
    ctx = dualk.Context(0)
    rng = np.random.Generator(np.random.PCG64(p))
    basis = np.linalg.qr(rng.normal(size=(p, p)))[0]
    x = (rng.normal(size=(2 * p + 40, p)) * np.sqrt(np.geomspace(4.0, 0.05, p)) @ basis.T).astype(np.float32)
    model = dualk.pca_fit(ctx, torch.from_numpy(x).cuda(), p, sweeps=10)
    ctx.sync_status()
    mean, scale, _, w = pp.pca_fit(x, p)
    z = (x.astype(np.float64) - mean) / scale
    cov = z.T @ z / (x.shape[0] - 1)
    v = model["components"].cpu().numpy().astype(np.float64)
    lam = model["eigenvalues"].cpu().numpy().astype(np.float64)
    assert model["off_norm"].item() < 1e-5
    assert np.abs(v @ v.T - np.eye(p)).max() <= 1e-4
    assert np.abs(v @ cov - lam[:, None] * v).max() <= 1e-4 * w[0]
    again = dualk.pca_fit(ctx, torch.from_numpy(x).cuda(), p, sweeps=10)
    assert all(torch.equal(model[k], again[k]) for k in model)  # deterministic
    ctx.close()
