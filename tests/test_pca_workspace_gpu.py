"""What a workspace held before does not enter a fit: the words of the one-launch Jacobi lie in
V^T's part and reach back into the end of A's, padding included, and a workspace full of words
that carry the tag of an early round gives the bits of a workspace of zeros."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FIRST_TAG = 0xff800001  # the tag of round 0


@pytest.mark.parametrize("p", [67, 100, 129, 131])  # 4 p^2 is no multiple of 256: A's part is padded
def test_stale_words(p):
    import torch
    from paper_2602_01330_gb300 import build, dualk
    build.build()
    ctx, lib = dualk.Context(0), dualk._lib()
    rng = np.random.Generator(np.random.PCG64(p))
    x = torch.from_numpy((rng.normal(size=(2 * p, p)) @ rng.normal(size=(p, p))).astype(np.float32)).cuda()
    nbytes = int(lib.dk_pca_workspace_bytes(p))

    def fit(tag):
        ws = torch.zeros(nbytes // 4, dtype=torch.int32, device="cuda")
        if tag is not None:
            ws[3::4] = tag - (1 << 32)
        out = [torch.zeros(n, device="cuda") for n in (p, p, p * p, p, 1)]
        st = lib.dk_pca_fit(ctx.handle, dualk._ptr(x), 2 * p, p, p, 2, dualk._ptr(ws), nbytes,
                            *[dualk._ptr(t) for t in out], dualk._stream(None))
        assert st == 0
        ctx.sync_status()
        return out

    clean = fit(None)
    for r in range(4):
        assert all(torch.equal(a, b) for a, b in zip(clean, fit(FIRST_TAG + r)))
    ctx.close()
