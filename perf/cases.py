"""Performance cases of the dual-kernel engine: the calls its users make, over the sizes they
make them at, through the public binding (paper_2602_01330_gb300.dualk).

A case is a dict of plain values; its "kind" names the call:

  serve   a request of b test samples against a resident training set: MPS build of the
          request, then its dual-kernel rows (what serving.KernelServer launches per request,
          and, with a large b, the prediction step of the benchmark)
  gram    the symmetric Gram of m samples of n qubits, with or without the MPS build before it
  build   the MPS build of a training set
  wide    the wide-bond forms: bond 8 in FP32, bond 32 in split BF16 on tensor cores
  blocks  a block-structured map: block statevectors, then their exact Gram
  svm     cross-validation of the dual-kernel SVM: the fold x C x w grid trained in one launch,
          the held-out samples voted in another
  pca     the pre-processing: PCA fit on raw pixels, then the training features

Inputs are the package's seeded Fashion-MNIST-shaped samples (synthetic.py); the SVM's kernel
matrices are formed here in 64 bits from such samples, so that its inputs do not depend on the
Gram kernels. exact() restates every call in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2602_01330_gb300 import dualk, synthetic, workload

DEV = "cuda"
W = 0.5                      # mixing weight of the benchmark and the server
ALL = ("k", "kq", "kc", "logkq")


def listed():
    return [
        # one sample to classify against the server's smallest resident set: launch latency
        {"name": "serve_n16_b1", "kind": "serve", "m": 8000, "n": 16, "b": 1, "reps": 2},
        # a ragged request of the server's usual size (1..256 rows) on its largest set
        {"name": "serve_n784_b37", "kind": "serve", "m": 8000, "n": 784, "b": 37, "reps": 2},
        # the benchmark's prediction rows: 500 test samples against 2000
        {"name": "rows_n784_b500", "kind": "serve", "m": 2000, "n": 784, "b": 500, "reps": 2},
        # the tiny study: 8 qubits, 64 samples, complex128
        {"name": "gram_n8_c128", "kind": "gram", "m": 64, "n": 8, "reps": 2, "c128": True, "build": True},
        # a low-dimensional Gram of the feature-dimension sweep, where many K_q are large
        {"name": "gram_n16_m2000", "kind": "gram", "m": 2000, "n": 16, "reps": 2, "c128": False, "build": True},
        # the benchmark's training Gram: 2000 samples of 784 raw pixels
        {"name": "gram_n784_m2000", "kind": "gram", "m": 2000, "n": 784, "reps": 2, "c128": False, "build": False},
        # its MPS build
        {"name": "build_n784_m2000", "kind": "build", "m": 2000, "n": 784, "reps": 2},
        # the precision study at 256 qubits: bond 8 with its build, FP32
        {"name": "chi8_n256_m1000", "kind": "wide", "m": 1000, "n": 256, "reps": 3, "bf16x3": False, "build": True},
        # and bond 32 on tensor cores, on MPS that are kept
        {"name": "chi32_n256_m512", "kind": "wide", "m": 512, "n": 256, "reps": 5, "bf16x3": True, "build": False},
        # the benchmark's samples through all-to-all blocks of 10 qubits, split BF16
        {"name": "blocks10_n784_m2000", "kind": "blocks", "m": 2000, "n": 784, "block": 10, "full": True,
         "bf16x3": True},
        # 5 folds x 4 C x 5 w on 2000 samples of 10 classes
        {"name": "svm_cv_m2000", "kind": "svm", "m": 2000, "n": 16, "classes": 10, "folds": 5, "n_c": 4, "n_w": 5},
        # the whole pixel space of the training set
        {"name": "pca_p784_m2000", "kind": "pca", "m": 2000, "p": 784, "k": 784},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["serve", "serve", "gram", "gram", "build", "wide", "blocks", "svm", "pca"])
    if kind == "serve":
        return {"kind": kind, "m": _log_int(rng, 500, 8000), "n": _log_int(rng, 8, 784), "b": _log_int(rng, 1, 256),
                "reps": rng.choice([1, 2, 2])}
    if kind == "gram":
        if rng.random() < 0.25:
            return {"kind": kind, "m": _log_int(rng, 16, 400), "n": _log_int(rng, 4, 96), "reps": 2, "c128": True,
                    "build": rng.random() < 0.5}
        return {"kind": kind, "m": _log_int(rng, 40, 2000), "n": _log_int(rng, 4, 784), "reps": rng.choice([1, 2, 2]),
                "c128": False, "build": rng.random() < 0.5}
    if kind == "build":
        return {"kind": kind, "m": _log_int(rng, 20, 4000), "n": _log_int(rng, 8, 784), "reps": rng.choice([1, 2, 2])}
    if kind == "wide":
        bf16x3 = rng.random() < 0.5
        m, n = (_log_int(rng, 30, 400), _log_int(rng, 12, 256)) if bf16x3 else (_log_int(rng, 60, 1000), _log_int(rng, 16, 256))
        return {"kind": kind, "m": m, "n": n, "reps": 5 if bf16x3 else 3, "bf16x3": bf16x3,
                "build": rng.random() < 0.5}
    if kind == "blocks":
        bf16x3 = rng.random() < 0.7
        return {"kind": kind, "m": _log_int(rng, 100, 2000 if bf16x3 else 1000), "n": _log_int(rng, 40, 784),
                "block": rng.randint(6, 10), "full": rng.random() < 0.6, "bf16x3": bf16x3}
    if kind == "svm":
        return {"kind": kind, "m": _log_int(rng, 150, 2000), "n": rng.choice([8, 12, 16]), "classes": rng.randint(2, 10),
                "folds": 5, "n_c": rng.randint(1, 4), "n_w": rng.randint(1, 5)}
    p = _log_int(rng, 16, 784)
    return {"kind": kind, "m": rng.randint(max(100, 2 * p), 2000), "p": p, "k": rng.randint(max(2, p // 4), p)}


# ---- inputs ----

def _features(case, seed, b=0):
    d = synthetic.fmnist_like(case["m"], b, case["n"], seed_train=2 * seed + 1000, seed_test=2 * seed + 1001)
    return d


def _fmap(case):
    reps = case["reps"]
    return dualk.FeatureMap(reps=reps, chi_max=max(4, 2 ** reps))


def _pixels(case, seed):
    x, _ = synthetic.images(case["m"], 2 * seed + 1000)
    sel = np.linspace(0, synthetic.N_PIXELS - 1, case["p"]).round().astype(int)
    return np.ascontiguousarray(x[:, sel], dtype=np.float32)


def _svm_grid(case, labels, seed):
    """Stratified folds and the job lists of the fold x C x w grid (as svm.DualKernelSVM lays them out)."""
    folds, cs, ws = case["folds"], (0.1, 1.0, 10.0, 100.0)[: case["n_c"]], (0.0, 0.25, 0.5, 0.75, 1.0)[: case["n_w"]]
    rng = np.random.Generator(np.random.PCG64(seed))
    fold = np.empty(labels.size, dtype=np.int64)
    for c in np.unique(labels):
        sel = np.flatnonzero(labels == c)
        sel = sel[rng.permutation(sel.size)]
        fold[sel] = np.arange(sel.size) % folds
    jobs = [(f, c, w) for c in cs for w in ws for f in range(folds)]
    tr = [np.flatnonzero(fold != f) for f in range(folds)]
    va = [np.flatnonzero(fold == f) for f in range(folds)]
    m_max, r_max = max(t.size for t in tr), max(v.size for v in va)
    g = {"idx": np.zeros((len(jobs), m_max), np.int32), "count": np.zeros(len(jobs), np.int32),
         "rows": np.zeros((len(jobs), r_max), np.int32), "row_count": np.zeros(len(jobs), np.int32)}
    for j, (f, _, _) in enumerate(jobs):
        g["idx"][j, :tr[f].size], g["count"][j] = tr[f], tr[f].size
        # every fold's held-out list is filled to r_max with its own samples, so that all of the output is written
        g["rows"][j], g["row_count"][j] = np.resize(va[f], r_max), r_max
    g = {k: torch.from_numpy(v).to(DEV) for k, v in g.items()}
    g["w"] = torch.tensor([w for _, _, w in jobs], dtype=torch.float32, device=DEV)
    g["C"] = torch.tensor([c for _, c, _ in jobs], dtype=torch.float32, device=DEV)
    g["labels"] = torch.from_numpy(labels.astype(np.int32)).to(DEV)
    return g


def prepare(case, seed):
    ctx = dualk.Context(0)
    kind = case["kind"]
    st = {"case": case, "ctx": ctx}
    if kind == "pca":
        st["x"] = torch.from_numpy(_pixels(case, seed)).to(DEV)
        return st
    if kind == "svm":
        d = _features(case, seed)
        x = torch.from_numpy(d["x_train"]).to(DEV)
        lk = _exact_log_kq(x, x, 2)
        st["kq"] = torch.exp(lk).float().contiguous()
        st["kc"] = _exact_kc(x, x).float().contiguous()
        st.update(_svm_grid(case, (d["y_train"] % case["classes"]).astype(np.int64), seed))
        return st
    d = _features(case, seed, case.get("b", 0))
    x = st["x"] = torch.from_numpy(d["x_train"]).to(DEV)
    if kind == "serve":
        st["fmap"] = _fmap(case)
        st["train"] = dualk.mps_build(ctx, x, st["fmap"])
        st["x_test"] = torch.from_numpy(d["x_test"]).to(DEV)
    elif kind == "blocks":
        st["fmap"] = dualk.FeatureMap(reps=2, block=case["block"])
    else:
        st["fmap"] = _fmap(case)
        st["dtype"] = dualk.DK_C128 if case.get("c128") else dualk.DK_C64
        if kind != "build" and not case["build"]:
            st["mps"] = dualk.mps_build(ctx, x, st["fmap"], dtype=st["dtype"])
    return st


# ---- the calls ----

def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "serve":
        test = dualk.mps_build(ctx, state["x_test"], state["fmap"])
        out = dualk.dual_kernel_rows(ctx, test, state["train"], w=W, want=("k", "kq", "logkq"))
        return {k: v for k, v in out.items() if v is not None}
    if kind == "build":
        mps = dualk.mps_build(ctx, state["x"], state["fmap"])
        return {"mps": mps.complex_view(), "bond_dims": mps.bond_dims, "log_norm": mps.log_norm}
    if kind in ("gram", "wide"):
        mps = dualk.mps_build(ctx, state["x"], state["fmap"], dtype=state["dtype"]) if case["build"] else state["mps"]
        return dualk.gram(ctx, mps, w=W, want=ALL, prec=dualk.DK_PREC_BF16X3 if case.get("bf16x3") else None)
    if kind == "blocks":
        ent = dualk.DK_ENT_FULL if case["full"] else dualk.DK_ENT_CHAIN
        states = dualk.block_states(ctx, state["x"], state["fmap"], ent,
                                    prec=dualk.DK_PREC_BF16X3 if case["bf16x3"] else dualk.DK_PREC_F32)
        return dualk.gram_blocks(ctx, states, w=W, want=ALL)
    if kind == "svm":
        model = dualk.svm_ovo_train(ctx, state["kq"], state["kc"], state["w"], state["C"], state["idx"],
                                    state["count"], state["labels"], case["classes"])
        votes = dualk.svm_ovo_predict(ctx, state["kq"], state["kc"], state["w"], model, case["classes"],
                                      rows=state["rows"], row_count=state["row_count"], idx=state["idx"],
                                      count=state["count"])
        return {**model, **votes}
    model = dualk.pca_fit(ctx, state["x"], case["k"])
    features = dualk.pca_transform(ctx, state["x"], model, fit_range=True)
    return {**model, "features": features}


def work(case):
    kind, m = case["kind"], case["m"]
    if kind == "pca":
        # covariance, a tridiagonal eigensolver's 9 p^3 with all vectors, the projection
        p, k = case["p"], case["k"]
        return {"bytes": 4.0 * (m * p + k * p + 3 * p + k + m * k + 2 * k),
                "flops": 1.0 * m * p * p + 9.0 * p ** 3 + 2.0 * m * p * k}
    if kind == "svm":
        # the kernel matrices read once; 2 rows and 2 passes per step, about 2 steps per sample of a problem
        jobs = case["folds"] * case["n_c"] * case["n_w"]
        c = case["classes"]
        pairs, size = c * (c - 1) // 2, 2.0 * m * (case["folds"] - 1) / case["folds"] / c
        m_max, r_max = m * (case["folds"] - 1) // case["folds"] + c, m // case["folds"] + c
        return {"bytes": 8.0 * m * m + 4.0 * jobs * (pairs * (m_max + 2) + m_max + r_max * (pairs + 2)),
                "flops": jobs * pairs * (2.0 * size * 12.0 * size + 2.0 * r_max * m_max)}
    n = case["n"]
    if kind == "blocks":
        nb, dim = -(-n // case["block"]), 2 ** case["block"]
        pairs = m * (m + 1) / 2
        return {"bytes": 4.0 * m * n + 16.0 * m * m, "flops": 8.0 * dim * nb * pairs + 3.0 * n * pairs}
    reps = case["reps"]
    real = 8 if case.get("c128") else 4
    site = 2.0 * real * max(4, 2 ** reps) ** 2
    per = workload.flops_per_pair(n, reps)
    if kind == "serve":
        b = case["b"]
        return {"bytes": site * m * n + 4.0 * n * (m + b) + 12.0 * b * m, "flops": b * m * (per + 3.0 * n)}
    if kind == "build":
        return {"bytes": site * m * n + 4.0 * m * n, "flops": m * (per + 60.0 * n * 4 ** reps)}
    pairs = m * (m + 1) / 2
    return {"bytes": (0.0 if case["build"] else site * m * n) + 4.0 * m * n + 16.0 * m * m,
            "flops": pairs * (per + 3.0 * n)}


# ---- the same in 64 bits ----

def _exact_kc(xr, xc):
    a, b = xr.double(), xc.double()
    d2 = (a * a).sum(1)[:, None] + (b * b).sum(1)[None, :] - 2.0 * (a @ b.T)
    if xr is xc:
        d2.fill_diagonal_(0.0)
    return torch.exp(-d2.clamp_min(0.0) / xr.shape[1])


def _site_phases(x, reps):
    """Per sample and site in complex128: L[i, k, c], the local factor of the repetition bits c
    (bit rho - 1: the qubit's value after repetition rho), and w[i, k] = exp(-i theta / 2) of the
    bond to the left."""
    x = x.double()
    n = x.shape[1]
    c = torch.arange(2 ** reps)
    pop = sum((c >> q) & 1 for q in range(reps))
    sign = sum(((c & (c >> 1)) >> q) & 1 for q in range(reps)) % 2
    amp = 2.0 ** (-reps / 2.0) * (1.0 - 2.0 * sign.double()).to(x.device)
    e = (reps - 2 * pop).to(x.device).double()
    local = torch.polar(amp.abs().expand(x.shape[0], n, -1).contiguous(), -x[:, :, None] * e)
    local = local * torch.sign(amp)
    theta = torch.zeros_like(x)
    theta[:, 1:] = (math.pi - x[:, :-1]) * (math.pi - x[:, 1:])
    return local, torch.polar(torch.ones_like(theta), -theta)


def _mix(v, axis, same, other):
    """Both values of one bit: out0 = same v0 + other v1, out1 = other v0 + same v1."""
    v0, v1 = v.select(axis, 0), v.select(axis, 1)
    return torch.stack((same * v0 + other * v1, other * v0 + same * v1), axis)


def _exact_log_kq(xr, xc, reps):
    """log K_q of every pair from the closed form of the chain's amplitude: a sum over each
    qubit's bits in both states, carried left to right with the last repetition's bit shared."""
    out = torch.empty((xr.shape[0], xc.shape[0]), dtype=torch.float64, device=xr.device)
    lc, wc = _site_phases(xc, reps)
    per_pair = 16 * 2 ** (2 * reps - 1)
    step = max(1, int(1.2e9 // (per_pair * xc.shape[0])))
    half = 2 ** (reps - 1)
    bits = [2] * (reps - 1)
    for r0 in range(0, xr.shape[0], step):
        lr, wr = _site_phases(xr[r0:r0 + step], reps)
        lr = lr.conj()
        shape = (lr.shape[0], lc.shape[0], 2, *bits, *bits)
        e2 = torch.zeros(shape[:2], dtype=torch.float64, device=xr.device)
        v = None
        for k in range(xr.shape[1]):
            if v is None:
                v = torch.ones((1,), dtype=torch.complex128, device=xr.device)
                v = v.expand(shape[0], shape[1], 2, half, half)
            else:
                one = [1] * (2 * reps - 2)
                a, b = wr[:, k].view(-1, 1, *one), wc[:, k].view(1, -1, *one)
                v = v.reshape(shape)
                for q in range(reps - 1):
                    v = _mix(v, 3 + q, a.conj(), a).reshape(shape)
                for q in range(reps - 1):
                    v = _mix(v, 3 + reps - 1 + q, b, b.conj()).reshape(shape)
                s = a.conj() * b
                v = _mix(v, 2, s, s.conj())
            v = v.reshape(shape[0], shape[1], 2, half, half)
            v = v * lr[:, k].view(-1, 1, 2, half, 1)
            v = v * lc[:, k].view(1, -1, 2, 1, half)
            if k % 16 == 15:
                top = v.abs().amax(dim=(2, 3, 4)).clamp_min(1e-300)
                ex = torch.floor(torch.log2(top))
                v = v * torch.exp2(-ex)[:, :, None, None, None]
                e2 += ex
        amp = v.sum(dim=(2, 3, 4))
        out[r0:r0 + step] = torch.log(amp.real ** 2 + amp.imag ** 2) + 2.0 * math.log(2.0) * e2
    return out


def _exact_gram(lk, kc, want):
    kq = torch.exp(lk).float().double()  # as far as a float32 output reaches: 0 below its range
    full = {"k": W * kq + (1.0 - W) * kc, "kq": kq, "kc": kc, "logkq": lk}
    return {k: full[k] for k in want}


def _exact_states(x, block, full):
    """Block statevectors in complex128: [block][sample][2^b], short last block alone."""
    x = x.double()
    n = x.shape[1]
    states = []
    for s0 in range(0, n, block):
        xb = x[:, s0:s0 + block]
        b = xb.shape[1]
        idx = torch.arange(2 ** b, device=x.device)
        z = torch.stack([1.0 - 2.0 * ((idx >> (b - 1 - q)) & 1) for q in range(b)]).double()
        phi = xb @ z
        for q in range(b):
            for r in range(q + 1, b):
                if full or r == q + 1:
                    phi = phi + ((math.pi - xb[:, q]) * (math.pi - xb[:, r]))[:, None] * (z[q] * z[r])
        ph = torch.polar(torch.ones_like(phi), -phi)
        psi = 2.0 ** (-b / 2.0) * ph
        psi = psi.reshape(x.shape[0], *([2] * b))
        for q in range(b):
            u, v = psi.select(1 + q, 0), psi.select(1 + q, 1)
            psi = torch.stack((u + v, u - v), 1 + q) * math.sqrt(0.5)
        states.append(psi.reshape(x.shape[0], -1) * ph)
    return states


def _exact_pca(x, k):
    x = x.double()
    m = x.shape[0]
    mean = x.mean(0)
    scale = (x - mean).square().mean(0).sqrt()
    scale = torch.where(scale > 0, scale, torch.ones_like(scale))
    z = (x - mean) / scale
    lam = torch.linalg.eigvalsh(z.T @ z / (m - 1))
    # an eigenvector, and what is projected on it, is only as certain in FP32 as its eigenvalue's gap
    # to the next: the noise directions' gaps leave them no 64-bit value to be held to
    return {"mean": mean, "scale": scale, "components": None, "eigenvalues": lam.flip(0)[:k], "off_norm": None,
            "lo": None, "hi": None, "features": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "svm":
        return None  # multipliers of an iteration stopped at a tolerance: no 64-bit value
    if kind == "pca":
        return _exact_pca(torch.from_numpy(_pixels(case, seed)).to(DEV), case["k"])
    d = _features(case, seed, case.get("b", 0))
    x = torch.from_numpy(d["x_train"]).to(DEV)
    if kind == "serve":
        xt = torch.from_numpy(d["x_test"]).to(DEV)
        return _exact_gram(_exact_log_kq(xt, x, case["reps"]), _exact_kc(xt, x), ("k", "kq", "logkq"))
    if kind == "build":
        # no 64-bit value: where a bond's rank drops (a feature at exactly pi) the last column of the
        # gauge is rounding, and the norm's logarithm is the rounding of 1
        return None
    if kind == "blocks":
        lk = 0.0
        for psi in _exact_states(x, case["block"], case["full"]):
            g = psi.conj() @ psi.T
            lk = lk + torch.log(g.real ** 2 + g.imag ** 2)
        return _exact_gram(lk, _exact_kc(x, x), ALL)
    return _exact_gram(_exact_log_kq(x, x, case["reps"]), _exact_kc(x, x), ALL)
