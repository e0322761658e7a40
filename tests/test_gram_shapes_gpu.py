"""Every complex64 bond-4 tile shape and the built-in choice (narrow shapes, lanes per pair) give
the bits of shape 17, and the built-in bond-8 choice those of tile shape 2: each pair is
contracted by the same arithmetic whatever tile it lands in. Blocks with few and ragged rows,
square and rectangular, aligned features or not. Complex128 blocks on both sides of the rule
(lanes per pair, tiles) agree with each other bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5, 24])
@pytest.mark.parametrize("b,m", [(1, 1), (1, 33), (2, 65), (3, 64), (5, 7), (37, 130), (70, 9)])
def test_shapes_same_bits(b, m, n):
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    x = torch.from_numpy(synthetic.uniform_angles(b + m, n, seed=n, dtype=np.float32)).cuda()
    fm = dualk.FeatureMap()
    rows, cols = dualk.mps_build(ctx, x[:b].contiguous(), fm), dualk.mps_build(ctx, x[b:].contiguous(), fm)

    def both():
        r = dualk.dual_kernel_rows(ctx, rows, cols, refine=None)
        g = dualk.gram(ctx, cols, refine=None)
        return [t for d in (r, g) for t in d.values()]
    ctx.set_gram_config(17)
    ref = both()
    for cid in [0, 19] + list(range(20, dualk.gram_config_count() + 1)):
        ctx.set_gram_config(cid)
        assert all(torch.equal(u, v) for u, v in zip(both(), ref)), cid
    ctx.set_gram_config(0)
    ctx.sync_status()
    ctx.close()


@pytest.mark.parametrize("b,m", [(1, 1), (3, 33), (20, 70)])
def test_bond8_built_in_same_bits(b, m):
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    x = torch.from_numpy(synthetic.uniform_angles(b + m, 11, seed=8, dtype=np.float32)).cuda()
    fm = dualk.FeatureMap(reps=3, chi_max=8)
    rows, cols = dualk.mps_build(ctx, x[:b].contiguous(), fm), dualk.mps_build(ctx, x[b:].contiguous(), fm)
    got = []
    for cid in (0, 2):
        ctx.set_gram_config(cid)
        r = dualk.dual_kernel_rows(ctx, rows, cols, refine=None)
        g = dualk.gram(ctx, cols, refine=None)
        got.append([t for d in (r, g) for t in d.values()])
    ctx.set_gram_config(0)
    ctx.sync_status()
    assert all(torch.equal(u, v) for u, v in zip(*got))
    ctx.close()


def test_complex128_lanes_and_tiles_same_bits():
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    x = torch.from_numpy(synthetic.uniform_angles(260, 6, seed=9, dtype=np.float32)).cuda()
    mps = dualk.mps_build(ctx, x, dualk.FeatureMap(), dtype=dualk.DK_C128)
    whole = dualk.gram(ctx, mps)  # 33930 pairs: tiles
    for r0, c0, nr, nc in ((0, 0, 30, 41), (7, 100, 1, 160), (250, 3, 10, 5)):  # lanes
        part = dualk.gram_tile(ctx, mps, mps, row0=r0, nrows=nr, col0=c0, ncols=nc)
        for k in whole:
            upper = torch.triu(torch.ones(260, 260, dtype=torch.bool, device="cuda"))[r0:r0 + nr, c0:c0 + nc]
            assert torch.equal(part[k][upper], whole[k][r0:r0 + nr, c0:c0 + nc][upper])
    ctx.sync_status()
    ctx.close()
