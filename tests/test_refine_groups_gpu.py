"""The refinement pass with few and ragged hits (bond 4: 8 lanes per chain, four chains a warp;
bond 8: a warp per chain): nearly every entry above tau, counts below, at and past a warp's groups.

Tolerance, set before the first run: 1e-6 on K_q (the FP32 path's), against statevectors; with
and without the norm workspace the bits are the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reps", [2, 3])
@pytest.mark.parametrize("b,m", [(1, 1), (1, 5), (3, 33), (17, 41)])
def test_few_and_ragged_hits(reps, b, m):
    import torch
    from oracle import circuit
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    n = 7
    base = synthetic.uniform_angles(1, n, seed=3, dtype=np.float32)
    xc = synthetic.near_copies(np.repeat(base, m, axis=0), 1e-3, 1e-1, seed=4)
    xr = synthetic.near_copies(np.repeat(base, b, axis=0), 1e-3, 1e-1, seed=5)
    fm = dualk.FeatureMap(reps=reps, chi_max=2 ** reps)
    rows = dualk.mps_build(ctx, torch.from_numpy(xr).cuda(), fm)
    cols = dualk.mps_build(ctx, torch.from_numpy(xc).cuda(), fm)
    ref = circuit.kernel_matrix(xr.astype(np.float64), xc.astype(np.float64), reps)
    assert (ref > 0.02).mean() > 0.9  # nearly all are refined
    got = dualk.dual_kernel_rows(ctx, rows, cols, w=1.0, want=("kq", "logkq"))
    out = dualk.dual_kernel_rows(ctx, rows, cols, w=1.0, want=("kq", "logkq"), refine=None)
    ctx.sync_status()
    assert np.abs(got["kq"].cpu().numpy() - ref).max() <= 1e-6
    dualk._check(dualk._lib().dk_gram_refine(
        ctx.handle, dualk._ptr(rows.data), b, dualk._ptr(cols.data), m, n, fm.chi_max, rows.dtype, 0, b, 0, m,
        dualk._ptr(rows.x), dualk._ptr(cols.x), 1.0 / n, 1.0, 0.02, None, dualk._ptr(out["kq"]), None,
        dualk._ptr(out["logkq"]), m, 0, None, 0, dualk._stream(None)), "dk_gram_refine")
    ctx.sync_status()
    assert torch.equal(got["kq"], out["kq"]) and torch.equal(got["logkq"], out["logkq"])
    ctx.close()
