"""K_c of the tcgen05 block Gram, whose 128 x 128 form sums the squared distances in two extra
warps beside the MMAs (blocks of 9 qubits and more, no split over the blocks), in a kernel of its
own otherwise. Both run the per-pair Kahan sum in feature order of every block Gram kernel, so K_c
has the bits of the mma.sync form: exact equality, set before the first run."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [8, 9, 11])  # own kernel; the extra warps from 9 on
@pytest.mark.parametrize("n,rows,m", [(1, 0, 1), (17, 0, 129), (31, 0, 700), (16, 1300, 1900), (9, 5, 40)])
def test_kc_bits(n, b, rows, m):
    """One pair; one entry past a tile and a feature past the staged 16; several tiles, whole
    passes below the diagonal; a rectangle that isn't split, ragged both ways; a split one."""
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    x = torch.from_numpy(synthetic.uniform_angles(m + rows, n, seed=n, dtype=np.float32)).cuda()
    fm = dualk.FeatureMap(reps=2, block=b)
    states = lambda a: dualk.block_states(ctx, a.contiguous(), fm, dualk.DK_ENT_CHAIN, prec=dualk.DK_PREC_BF16X3)
    cols = states(x[rows:])
    args = (states(x[:rows]), cols) if rows else (cols,)
    got = {}
    for form in (dualk.DK_BLOCK_TCGEN05, dualk.DK_BLOCK_MMA_SYNC):
        ctx.set_block_gram_form(form)
        got[form] = dualk.gram_blocks(ctx, *args, w=0.25, want=("k", "kc", "kq"))
    torch.cuda.synchronize()
    ctx.sync_status()
    a, c = got[dualk.DK_BLOCK_TCGEN05], got[dualk.DK_BLOCK_MMA_SYNC]
    assert torch.equal(a["kc"], c["kc"])
    kq, kc, k = (a[s].double() for s in ("kq", "kc", "k"))
    assert (k - (0.25 * kq + 0.75 * kc)).abs().max() <= 1e-6
    ctx.close()
