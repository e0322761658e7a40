"""The bond-4 build, whose warps hand each other the sites in chunks of 8: chains that end before,
at and after a chunk (one chunk, both buffers, a buffer used again) with one, two and four samples
a CTA, full and ragged.

Tolerances, set before the first run: 1e-6 on K_q (the FP32 path's, refined) against statevectors up to 9
qubits and against the FP64 complex128 build beyond; log K_q of a sample with itself is exactly 0,
because the build's norm runs the Gram's arithmetic on the stored tensors; the tensors don't depend
on how many samples share a CTA."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reps", [1, 2])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 16, 17, 24, 25, 41])
def test_chunk_edges(n, reps):
    import torch
    from oracle import circuit
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    base = synthetic.uniform_angles(1, n, seed=11, dtype=np.float32)
    x = synthetic.near_copies(np.repeat(base, 611, axis=0), 1e-2, 3e-1, seed=n)
    fm = dualk.FeatureMap(reps=reps, chi_max=4)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    mps = dualk.mps_build(ctx, dev(x), fm)
    got = dualk.gram(ctx, mps, w=1.0, want=("kq", "logkq"))
    kq = got["kq"].cpu().numpy().astype(np.float64)
    assert np.all(np.diag(got["logkq"].cpu().numpy()) == 0.0)
    few = 13
    if n <= 9:
        ref = circuit.kernel_matrix(x[:few].astype(np.float64), x.astype(np.float64), reps)
    else:
        wide = dualk.mps_build(ctx, dev(x), fm, dtype=dualk.DK_C128)
        ref = dualk.gram(ctx, wide, w=1.0, want=("kq",))["kq"].cpu().numpy().astype(np.float64)[:few]
    assert np.abs(kq[:few] - ref).max() <= 1e-6
    for dtype in (dualk.DK_C64, dualk.DK_C128):
        full = dualk.mps_build(ctx, dev(x), fm, dtype=dtype)  # four samples a CTA, the last ragged
        for m in (1, few, 303):  # one a CTA; two, the last ragged
            part = dualk.mps_build(ctx, dev(x[:m]), fm, dtype=dtype)
            assert torch.equal(part.complex_view(), full.complex_view()[:, :m])
            assert torch.equal(part.log_norm, full.log_norm[:m])
    ctx.sync_status()
    ctx.close()
