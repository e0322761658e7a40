"""The SVM calls' launch rules: class pairs larger than the likely size go to a second launch, and
prediction takes 8, 4 or 1 rows per CTA. The results of a problem do not depend on either: the
same two-class problem among 10 declared classes and alone, and the same rows classified in one
call and one by one, give the same bits (the arithmetic and its order are the same)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n_jobs", [(40, 1), (333, 3), (1300, 2)])
def test_same_bits_whatever_the_launch(m, n_jobs):
    import torch
    from paper_2602_01330_gb300 import build, dualk
    build.build()
    ctx = dualk.Context(0)
    rng = np.random.Generator(np.random.PCG64(m))
    y = (rng.random(m) < 0.4).astype(np.int32)
    x = rng.normal(size=(m, 4)) + 0.8 * y[:, None]
    d2 = ((x[:, None, :] - x[None, :, :]) ** 2).sum(-1)

    def dev(a, dt):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).cuda()
    kq, kc = dev(np.exp(-0.5 * d2), np.float32), dev(np.exp(-0.1 * d2), np.float32)
    w, C = dev(np.linspace(0, 1, n_jobs), np.float32), dev(np.full(n_jobs, 5.0), np.float32)
    idx = dev(np.stack([rng.permutation(m) for _ in range(n_jobs)]), np.int32)
    cnt, lab = dev(np.full(n_jobs, m), np.int32), dev(y, np.int32)
    two = dualk.svm_ovo_train(ctx, kq, kc, w, C, idx, cnt, lab, 2)
    ten = dualk.svm_ovo_train(ctx, kq, kc, w, C, idx, cnt, lab, 10)
    ctx.sync_status()
    assert int(two["iters"].min()) > 0
    for k in two:
        assert torch.equal(two[k][:, 0], ten[k][:, 0])
    pad = torch.zeros((n_jobs * 200, 1), dtype=torch.int32, device="cuda")  # many jobs: more rows per CTA
    many = {k: v.repeat(200, *[1] * (v.dim() - 1)) for k, v in two.items()}
    rows = torch.arange(m, dtype=torch.int32, device="cuda")[:13].repeat(n_jobs * 200, 1).contiguous()
    a = dualk.svm_ovo_predict(ctx, kq, kc, w.repeat(200), many, 2, rows=rows, idx=idx.repeat(200, 1),
                              count=cnt.repeat(200))
    for r in (0, 7, 12):
        b = dualk.svm_ovo_predict(ctx, kq, kc, w, two, 2, rows=pad[:n_jobs] + r, idx=idx, count=cnt)
        assert torch.equal(a["decision"][:n_jobs, r], b["decision"][:, 0])
        assert torch.equal(a["pred"][:n_jobs, r], b["pred"][:, 0])
    ctx.sync_status()
    ctx.close()
