"""The refinement pass at the edges of its batches of 32 queued entries (a warp's hits below, at and
past 32 and 64, sparse and dense): every refined entry has the bits that it has when it is refined in
a block of its own, with and without the norms' workspace, and the others keep theirs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reps", [2, 3])
@pytest.mark.parametrize("n", [1, 2, 9])
@pytest.mark.parametrize("m,every", [(31, 1), (32, 1), (33, 1), (64, 1), (95, 1), (700, 7), (700, 40)])
def test_batches(reps, n, m, every):
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    P = dualk._ptr
    xc = synthetic.uniform_angles(m, n, seed=6, dtype=np.float32)
    near = synthetic.near_copies(np.repeat(xc[:1], m, axis=0), 1e-3, 1e-1, seed=4)
    xc[::every] = near[::every]
    fm = dualk.FeatureMap(reps=reps, chi_max=2 ** reps)
    rows = dualk.mps_build(ctx, torch.from_numpy(near[:2].copy()).cuda(), fm)
    cols = dualk.mps_build(ctx, torch.from_numpy(xc).cuda(), fm)
    plain = dualk.dual_kernel_rows(ctx, rows, cols, w=0.5, refine=None)

    def refine(out, col0, ncols, ws):
        dualk._check(dualk._lib().dk_gram_refine(
            ctx.handle, P(rows.data), 2, P(cols.data), m, n, fm.chi_max, rows.dtype, 0, 2, col0, ncols, P(rows.x),
            P(cols.x), 1.0 / n, 0.5, 0.02, P(out["k"]), P(out["kq"]), P(out["kc"]), P(out["logkq"]), ncols, 0, P(ws),
            int(ws.numel()) if ws is not None else 0, dualk._stream(None)), "dk_gram_refine")

    alone = {k: v.clone() for k, v in plain.items()}
    for c in range(m):
        one = {k: v[:, c:c + 1].contiguous() for k, v in plain.items()}
        refine(one, c, 1, None)
        for k in alone:
            alone[k][:, c:c + 1] = one[k]
    hits = plain["kq"] > 0.02
    assert hits.sum().item() >= 1.8 * len(range(0, m, every))  # nearly all of the near copies
    for ws in (None, dualk.refine_workspace(2, m, "cuda")):
        got = {k: v.clone() for k, v in plain.items()}
        refine(got, 0, m, ws)
        ctx.sync_status()
        for k in got:
            assert torch.equal(got[k], alone[k]), k
            assert torch.equal(got[k][~hits], plain[k][~hits]), k
    ctx.close()


@pytest.mark.parametrize("n", [2, 9])
def test_more_entries_than_the_gpu_holds_warps_for(n):
    """A symmetric block of 700 x 700 entries (each warp scans several 32s) against the same rows as a
    rectangular block of their own."""
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    m = 700
    x = synthetic.near_copies(np.repeat(synthetic.uniform_angles(7, n, seed=6, dtype=np.float32), m // 7, axis=0),
                              1e-3, 1e-1, seed=4)
    cols = dualk.mps_build(ctx, torch.from_numpy(x).cuda(), dualk.FeatureMap())
    rows = dualk.mps_build(ctx, torch.from_numpy(x[:30].copy()).cuda(), dualk.FeatureMap())
    whole = dualk.gram(ctx, cols, w=0.5)
    part = dualk.dual_kernel_rows(ctx, rows, cols, w=0.5)
    ctx.sync_status()
    upper = torch.triu(torch.ones(30, m, dtype=torch.bool, device="cuda"), 1)
    assert (whole["kq"] > 0.02).sum().item() > 60000
    for k in whole:
        assert torch.equal(whole[k][:30][upper], part[k][upper]), k
        assert torch.equal(whole[k], whole[k].T), k
    ctx.close()
