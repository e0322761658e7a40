"""The forms of dk_pca_fit side by side, through a small library of its own that includes pca.cu:
all rounds in one launch (one CTA below 64 features, several from there on), and one launch per
round. Both apply the same operations in the same order, so they give the same bits at every size;
one launch per round is also what runs beyond what shared memory holds (1373 features on 152 SMs).

A wait that runs out (a launch one CTA short: its words of the first round never come, so every
other CTA gives up there, before it sends a row; the wait's limit is 2 s) is reported by
dk_sync_status, leaves NaN in the outputs, and the next fit is as good as any."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FORMS = r"""
#include "pca.cu"
// form 0: as dk_pca_fit; 1: one launch per round; 2: one launch, its last CTA missing
extern "C" __attribute__((visibility("default"))) int pca_form(dk_ctx* ctx, const float* x, int m, int p, int k,
                                                               int sweeps, void* ws, float* mean, float* scale,
                                                               float* comps, float* eig, float* off, int form,
                                                               int* ctas) {
  using namespace dk::pca;
  PersistPlan plan = plan_of(ctx, p);
  if (form == 1) plan.ctas = 0;
  if (form == 2 && --plan.ctas < 2) return -1;
  *ctas = plan.ctas;
  return fit(ctx, x, m, p, k, sweeps, carve(ws, p), plan, mean, scale, comps, eig, off, nullptr);
}
"""


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    from paper_2602_01330_gb300 import build
    d = tmp_path_factory.mktemp("forms")
    src, so = d / "forms.cu", str(d / "forms.so")
    src.write_text(FORMS)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", "-cudart", "static",
                    "-o", so, str(src)], check=True, capture_output=True)
    lib = ctypes.CDLL(so)
    vp, i32 = ctypes.c_void_p, ctypes.c_int
    lib.pca_form.argtypes = [vp, vp, i32, i32, i32, i32, vp, vp, vp, vp, vp, vp, i32, ctypes.POINTER(i32)]
    return lib


@pytest.fixture(scope="module")
def dk():
    import torch
    from paper_2602_01330_gb300 import build, dualk
    build.build()
    ctx = dualk.Context(0)
    yield dualk, ctx, torch
    ctx.close()


def _fit(dk, forms, x, k, sweeps, form):
    dualk, ctx, torch = dk
    m, p = x.shape
    ws = torch.empty(int(dualk._lib().dk_pca_workspace_bytes(p)), dtype=torch.uint8, device="cuda")
    out = [torch.zeros(n, device="cuda") for n in (p, p, k * p, k, 1)]
    ctas = ctypes.c_int(-1)
    torch.cuda.synchronize()  # the other library's call is on the legacy default stream
    assert forms.pca_form(ctx.handle, dualk._ptr(x), m, p, k, sweeps, dualk._ptr(ws), *[dualk._ptr(t) for t in out],
                          form, ctypes.byref(ctas)) == 0
    torch.cuda.synchronize()
    return out, ctas.value


def _data(torch, p):
    rng = np.random.Generator(np.random.PCG64(p))
    x = rng.normal(size=(p + 40, p)) * np.sqrt(np.geomspace(4.0, 0.05, p))
    return torch.from_numpy((x @ rng.normal(size=(p, p))).astype(np.float32)).cuda()


@pytest.mark.parametrize("p,ctas", [(2, 1), (3, 1), (16, 1), (17, 1), (33, 1), (47, 1), (61, 1), (62, 1),  # one CTA
                                    (63, 11), (65, 11), (67, 12),  # odd: a padded pair; 67: a last CTA of one pair too
                                    (68, 12), (128, 22), (134, 23), (200, 34),  # a last CTA of one pair
                                    (113, 19), (199, 34), (255, 43), (256, 43), (782, 131), (783, 131),
                                    (915, 115), (954, 120), (1372, 138)])  # four and five pairs, more threads
def test_one_launch_and_one_per_round_same_bits(dk, forms, p, ctas):
    dualk, ctx, torch = dk
    x = _data(torch, p)
    one, n = _fit(dk, forms, x, p, 2, 0)
    ctx.sync_status()
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert n == ctas
    per_round, _ = _fit(dk, forms, x, p, 2, 1)
    ctx.sync_status()
    model = dualk.pca_fit(ctx, x, p, sweeps=2)
    for a, b, name in zip(one, per_round, ("mean", "scale", "components", "eigenvalues", "off_norm")):
        assert torch.equal(a, b), name
        assert torch.equal(a.view_as(model[name]), model[name]), name
    ctx.sync_status()


def test_one_launch_per_round_beyond_shared_memory(dk):
    """1373 features, on the launch-per-round form. What holds after any number of sweeps: the
    components V are orthonormal, the eigenvalues are the diagonal of V C V^T, and off_norm is its
    relative off-diagonal norm. Tolerance as derived in test_pca_rounds_gpu.py: at most 10 sweeps of
    1373 rotations of a row, each with a relative rounding of 2 u, as a random walk sqrt(13730) * 2 *
    6e-8 = 1.3e-5 of the row's norm, taken ten times as large."""
    dualk, ctx, torch = dk
    p = 1373
    x = _data(torch, p)
    z = x.double()
    z = (z - z.mean(0)) / z.std(0, correction=0)
    cov = z.T @ z / (x.shape[0] - 1)
    for sweeps in (1, 2, 10):
        model = dualk.pca_fit(ctx, x, p, sweeps=sweeps)
        ctx.sync_status()
        v, lam = model["components"].double(), model["eigenvalues"].double()
        rotated = v @ cov @ v.T
        diag = torch.diag(rotated)
        off = ((rotated - torch.diag(diag)).norm() / rotated.norm()).item()
        assert (v @ v.T - torch.eye(p, device="cuda", dtype=torch.float64)).abs().max().item() <= 1.3e-4
        assert (diag - lam).abs().max().item() <= 1.3e-4 * lam[0].item()
        assert abs(model["off_norm"].item() - off) <= 1.3e-4


def test_wait_that_runs_out(dk, forms):
    dualk, ctx, torch = dk
    x = _data(torch, 67)
    good, _ = _fit(dk, forms, x, 67, 2, 0)
    bad, _ = _fit(dk, forms, x, 67, 2, 2)
    with pytest.raises(RuntimeError, match="wait"):
        ctx.sync_status()
    assert all(torch.isnan(t).all() for t in bad[2:])  # components, eigenvalues, off_norm
    again, _ = _fit(dk, forms, x, 67, 2, 0)
    ctx.sync_status()
    assert all(torch.equal(a, b) for a, b in zip(good, again))
