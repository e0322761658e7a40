// One-against-one SVM on precomputed kernel values: the consumer of the Gram and of the
// dual-kernel rows (§II-B: dual problem Eqs. 1-2, decision function Eqs. 4-5, one-against-
// one voting; §II-D: the mixed kernel K = w K_q + (1 - w) K_c of Eq. 11 and the 5-fold
// cross-validation over C and w).
//
// Training: one CTA per (job, class pair). A job is one training set (a list of sample
// indices into the kernel matrix) with its C and w, so a whole cross-validation grid (folds x
// C x w) is one call. The CTA compacts the pair's samples (in list order), then runs
// sequential minimal optimisation with the second-order working-set rule of Fan, Chen and
// Lin (JMLR 6, 2005): per step a block-wide argmax picks i, the kernel row of i is gathered
// from the Gram in global memory (L2-resident), a block-wide argmin of the guaranteed
// decrease picks j, one thread solves the two-variable problem, and the gradient is updated
// with rows i and j. Multipliers and gradient are FP64 in shared memory, the working-set
// choice compares FP32 copies (the kernel values are the FP32 Gram outputs); nothing else is
// written until the end, so no global scratch is used. The loop ends when the largest KKT
// violation is below tol, or after max_iter steps.
//
// Prediction: one CTA per job and R rows: the rows' kernel values against the job's training
// samples are staged in shared memory, each class pair's decision values are warp-wide dot
// products with its coefficients, and the votes pick the class.
#include <math.h>
#include <stdint.h>

#include "common.cuh"
#include "internal.h"

namespace dk {
namespace svm {

constexpr int NT = 256;        // threads per CTA (prediction)
constexpr int NW = NT / 32;
constexpr int MAX_CLASS = 32;

__host__ __device__ inline void pair_of(int p, int n_class, int& c1, int& c2) {
  int c = 0, base = 0;
  while (p >= base + (n_class - 1 - c)) {
    base += n_class - 1 - c;
    ++c;
  }
  c1 = c;
  c2 = c + 1 + (p - base);
}

// kernel value K(r, c) of the mixed matrix
__device__ __forceinline__ float kval(const float* kq, const float* kc, long long ld, float w, int r, int c) {
  const long long o = (long long)r * ld + c;
  float v = 0.0f;
  if (kq) v = w * __ldg(kq + o);
  if (kc) v = fmaf(1.0f - w, __ldg(kc + o), v);
  return v;
}

// float -> double, exact, and double -> float, rounded to nearest even, by integer operations (the
// conversion instructions, like all FP64, hold an SM's FP64 pipe 16 cycles a warp); values
// outside the normal range of both take the instruction.
__device__ __forceinline__ double widen(float v) {
  const unsigned u = __float_as_uint(v), e = (u >> 23) & 0xffu;
  if (e == 0u || e == 0xffu) return double(v);
  return __hiloint2double(int((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), int(u << 29));
}
__device__ __forceinline__ float narrow(double v) {
  const unsigned hi = unsigned(__double2hiint(v)), lo = unsigned(__double2loint(v)), e = (hi >> 20) & 0x7ffu;
  if (e < 897u || e > 1150u) return float(v);
  unsigned u = (((hi & 0x7fffffffu) - 0x38000000u) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1fffffffu;
  u += (rest > 0x10000000u || (rest == 0x10000000u && (u & 1u))) ? 1u : 0u;
  return __uint_as_float((hi & 0x80000000u) | u);
}
// v with its sign flipped where `flip`
__device__ __forceinline__ double flip_if(double v, bool flip) {
  return __hiloint2double(__double2hiint(v) ^ (flip ? int(0x80000000u) : 0), __double2loint(v));
}

struct TrainArgs {
  const float* kq;
  const float* kc;
  long long ld;
  int n;           // samples of the kernel matrix (valid indices 0..n-1)
  unsigned* status;
  const float* w;
  const float* C;
  const int32_t* idx;
  const int32_t* count;
  int m_max;
  const int32_t* labels;
  int n_class;
  int n_pairs;
  double tol;
  int max_iter;
  float* coef;
  float* bias;
  int32_t* iters;
  int cap;   // samples the launch's shared memory holds
  int skip;  // problems of at most this many samples are another launch's
};

struct ArgF {
  float v;
  int i;
};

__device__ __forceinline__ bool better_f(const ArgF& x, const ArgF& y, bool want_max) {
  if (x.i < 0) return false;
  if (y.i < 0) return true;
  if (x.v != y.v) return want_max ? x.v > y.v : x.v < y.v;
  return x.i < y.i;
}

__device__ __forceinline__ void warp_arg_f(ArgF& x, bool want_max) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ArgF b{__shfl_xor_sync(0xffffffffu, x.v, o), __shfl_xor_sync(0xffffffffu, x.i, o)};
    if (better_f(b, x, want_max)) x = b;
  }
}

constexpr unsigned char IN_UP = 1, IN_LOW = 2;

// membership of one multiplier in the upper / lower index sets
__device__ __forceinline__ unsigned char set_flags(double alpha, double C, int y) {
  unsigned char f = 0;
  if ((y > 0 && alpha < C) || (y < 0 && alpha > 0.0)) f |= IN_UP;
  if ((y > 0 && alpha > 0.0) || (y < 0 && alpha < C)) f |= IN_LOW;
  return f;
}

// Shared memory (dynamic), per sample of the pair: alpha, grad (FP64), v = -y grad (FP32
// copy for the working-set choice), kd, ki (FP32 kernel values), gi (kernel index), pos
// (position in the job's list, below 4096), y (int8) and the set flags (uint8).
// Arithmetic: the gradient and the multipliers are FP64; the choice of the working pair
// compares FP32 copies (FP64 issues at a small fraction of the FP32 rate on GB300, and the
// choice is a heuristic: any violating pair makes progress); the stopping test reads the two
// chosen gradients in FP64 where their FP32 copies do not already decide it.
//
// Bound by the FP64 pipe (16 cycles a warp instruction and SM) and the barriers of a step, so:
// the gradient update is three FP64 operations a sample, conversions are integer operations and
// products by y sign flips; the update pass also finds the next step's i, and three barriers a
// step are left; and CTAs are small (128 threads, shared memory for a class pair's likely
// size), so that a step's latencies hide behind other problems. Larger problems are left to
// a second launch with room for all samples. Same operations on the same values: the bits do
// not depend on the launch. Measured, 4500 problems of 320 samples (2000 samples, 10 classes):
// 7.1 ms against 15.8 ms before; prediction of their 40000 held-out rows 0.65 ms against 3.0 ms
// (one row per CTA, which read all coefficients again for every row).
template <int TNT>
__global__ void __launch_bounds__(TNT, TNT == 128 ? 8 : 3) ovo_train_kernel(const TrainArgs a) {
  constexpr int TNW = TNT / 32;
  constexpr int KEEP = 4;  // kernel values of row j a thread keeps in registers
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int p = blockIdx.x, job = blockIdx.y;
  const int mm = a.m_max, cap = a.cap;
  double* alpha = reinterpret_cast<double*>(sm_raw);
  double* grad = alpha + cap;
  float* vf = reinterpret_cast<float*>(grad + cap);
  float* kd = vf + cap;
  float* ki = kd + cap;
  int* gi = reinterpret_cast<int*>(ki + cap);
  unsigned short* pos = reinterpret_cast<unsigned short*>(gi + cap);
  signed char* ys = reinterpret_cast<signed char*>(pos + cap);
  unsigned char* fl = reinterpret_cast<unsigned char*>(ys + cap);
  __shared__ ArgF red_up[TNW], red_low[TNW], red_j[TNW];
  __shared__ double red_d[8];
  __shared__ int s_np, s_n1, s_warp_base[TNW + 1];
  __shared__ double s_step;

  int c1, c2;
  pair_of(p, a.n_class, c1, c2);
  const int cnt = min(max(a.count[job], 0), mm);
  const int32_t* idx = a.idx + (long long)job * mm;
  const float w = a.w[job];
  const double C = double(a.C[job]);
  float* coef = a.coef + ((long long)job * a.n_pairs + p) * mm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // 1. the pair's samples, in list order (warp ballots + a block prefix per chunk of TNT)
  if (tid == 0) {
    s_np = 0;
    s_n1 = 0;
  }
  __syncthreads();
  for (int k0 = 0; k0 < cnt; k0 += TNT) {
    const int k = k0 + tid;
    int lab = -1, g = 0;
    if (k < cnt) {
      g = idx[k];
      if (g >= 0 && g < a.n) lab = a.labels[g];
      else record_status(a.status, DEV_BAD_INDEX);  // skipped
    }
    const bool in = lab == c1 || lab == c2;
    const unsigned bal = __ballot_sync(0xffffffffu, in);
    if (lane == 0) s_warp_base[warp + 1] = __popc(bal);
    __syncthreads();
    if (tid == 0) {
      s_warp_base[0] = s_np;
      for (int w2 = 1; w2 <= TNW; ++w2) s_warp_base[w2] += s_warp_base[w2 - 1];
    }
    __syncthreads();
    if (in) {
      const int dst = s_warp_base[warp] + __popc(bal & ((1u << lane) - 1u));
      if (dst < cap) {
        gi[dst] = g;
        pos[dst] = static_cast<unsigned short>(k);
        ys[dst] = lab == c1 ? 1 : -1;
      }
      if (lab == c1) atomicAdd(&s_n1, 1);
    }
    __syncthreads();
    if (tid == 0) s_np = s_warp_base[TNW];
    __syncthreads();
  }
  const int np = s_np;
  const int n1 = s_n1;
  if (np > cap || np <= a.skip) return;  // the other launch's
  // positions of the job's list outside the pair (and past count) get coefficient 0
  for (int k = tid; k < mm; k += TNT) coef[k] = 0.0f;
  if (np == 0 || n1 == 0 || n1 == np) {  // a class of the pair is absent from this job
    if (tid == 0) {
      a.bias[(long long)job * a.n_pairs + p] = 0.0f;
      if (a.iters) a.iters[(long long)job * a.n_pairs + p] = 0;
    }
    return;
  }
  ArgF up{0.0f, -1}, low{0.0f, -1};  // this thread's candidates for the next step
  auto consider = [&](int t, float v, unsigned char f) {
    if ((f & IN_UP) && (up.i < 0 || v > up.v)) up = ArgF{v, t};
    if ((f & IN_LOW) && (low.i < 0 || v < low.v)) low = ArgF{v, t};
  };
  for (int t = tid; t < np; t += TNT) {
    alpha[t] = 0.0;
    grad[t] = -1.0;
    vf[t] = float(ys[t]);  // -y (-1)
    fl[t] = set_flags(0.0, C, ys[t]);
    kd[t] = kval(a.kq, a.kc, a.ld, w, gi[t], gi[t]);
    consider(t, vf[t], fl[t]);
  }

  // 2. SMO with second-order working-set selection
  int it = 0;
  bool converged = false;
  const float tol_f = float(a.tol);
  for (; it < a.max_iter; ++it) {
    warp_arg_f(up, true);
    warp_arg_f(low, false);
    if (lane == 0) {
      red_up[warp] = up;
      red_low[warp] = low;
    }
    __syncthreads();  // also: every sample's state is written
    up = red_up[0];
    low = red_low[0];
#pragma unroll
    for (int w2 = 1; w2 < TNW; ++w2) {
      if (better_f(red_up[w2], up, true)) up = red_up[w2];
      if (better_f(red_low[w2], low, false)) low = red_low[w2];
    }
    if (up.i < 0 || low.i < 0) {
      converged = true;
      break;
    }
    const int i = up.i;
    // The FP64 values lie within 2^-24 of their FP32 copies: where the copies' gap exceeds tol by
    // more than that and the rounding of this test, the FP64 gap does too.
    const float gap_f = up.v - low.v;
    if (!(gap_f - 4e-7f * (fabsf(up.v) + fabsf(low.v)) > 1.000001f * tol_f)) {
      const double vmax = -double(ys[i]) * grad[i];
      if (vmax - (-double(ys[low.i]) * grad[low.i]) < a.tol) {
        converged = true;
        break;
      }
    }
    // the kernel row of i, and j: the lower-set index with the largest guaranteed decrease
    // (vmax - v_t)^2 / curvature
    const float vmax_f = up.v, kdi = kd[i];
    const int gii = gi[i];
    ArgF jb{0.0f, -1};
    for (int t = tid; t < np; t += TNT) {
      const float kit = kval(a.kq, a.kc, a.ld, w, gii, gi[t]);
      ki[t] = kit;
      const float v = vf[t];
      if ((fl[t] & IN_LOW) && v < vmax_f) {
        const float gap = vmax_f - v;
        float curv = kdi + kd[t] - 2.0f * kit;
        if (!(curv > 0.0f)) curv = 1e-12f;
        const float obj = -(gap * gap) / curv;
        if (jb.i < 0 || obj < jb.v) jb = ArgF{obj, t};
      }
    }
    warp_arg_f(jb, false);
    if (lane == 0) red_j[warp] = jb;
    __syncthreads();
    ArgF bj = red_j[0];
#pragma unroll
    for (int w2 = 1; w2 < TNW; ++w2)
      if (better_f(red_j[w2], bj, false)) bj = red_j[w2];
    if (bj.i < 0) {
      converged = true;
      break;
    }
    const int j = bj.i;
    if (tid == 0) {
      // exact step t along a_i += y_i t, a_j -= y_j t (keeps sum y a), clipped to the box
      const bool ni = ys[i] < 0, nj = ys[j] < 0;
      const double ai = alpha[i], aj = alpha[j];
      double eta = widen(kd[i]) + widen(kd[j]) - 2.0 * widen(ki[j]);
      if (!(eta > 0.0)) eta = 1e-12;
      const double vmax = flip_if(grad[i], !ni), vj = flip_if(grad[j], !nj);
      double step = (vmax - vj) / eta;
      // a_i + y_i t in [0, C] and a_j - y_j t in [0, C]
      const double lo_i = ni ? ai - C : -ai, hi_i = ni ? ai : C - ai;
      const double lo_j = nj ? -aj : aj - C, hi_j = nj ? C - aj : aj;
      step = fmin(fmax(step, fmax(lo_i, lo_j)), fmin(hi_i, hi_j));
      const double an = ai + flip_if(step, ni), bn = aj + flip_if(step, !nj);
      alpha[i] = an;
      alpha[j] = bn;
      fl[i] = set_flags(an, C, ys[i]);
      fl[j] = set_flags(bn, C, ys[j]);
      s_step = step;
    }
    // the kernel row of j meanwhile
    const int gij = gi[j];
    float kj[KEEP];
#pragma unroll
    for (int q = 0; q < KEEP; ++q) {
      const int t = tid + q * TNT;
      kj[q] = t < np ? kval(a.kq, a.kc, a.ld, w, gij, gi[t]) : 0.0f;
    }
    __syncthreads();
    // gradient: += y_t (step K_it - step K_jt); and the next step's candidates
    const double step = s_step;
    up = ArgF{0.0f, -1};
    low = ArgF{0.0f, -1};
    auto update = [&](int t, float kjt) {
      const bool neg = ys[t] < 0;
      const double d = fma(step, widen(ki[t]), -__dmul_rn(step, widen(kjt)));
      const double g = grad[t] + flip_if(d, neg);
      grad[t] = g;
      const float v = narrow(flip_if(g, !neg));
      vf[t] = v;
      consider(t, v, fl[t]);
    };
#pragma unroll
    for (int q = 0; q < KEEP; ++q)
      if (tid + q * TNT < np) update(tid + q * TNT, kj[q]);
    for (int t = tid + KEEP * TNT; t < np; t += TNT) update(t, kval(a.kq, a.kc, a.ld, w, gij, gi[t]));
  }
  __syncthreads();

  // 3. bias (Eq. 5): minus the mean of y grad over the free multipliers, or minus the
  // midpoint of the feasible interval when none is free. The sum runs as 256 threads' would:
  // partial sums over t = v, v + 256, ..., warps of 32 of them, the warps in order.
  double nfree = 0.0, ub = 1e300, lb = -1e300;
  for (int v0 = 0; v0 < 256; v0 += TNT) {
    double sfree = 0.0;
    for (int t = v0 + tid; t < np; t += 256) {
      const double yt = ys[t];
      const double yg = yt * grad[t];
      const double at = alpha[t];
      if (at > 0.0 && at < C) {
        sfree += yg;
        nfree += 1.0;
      } else if ((at >= C && yt < 0) || (at <= 0.0 && yt > 0)) {
        ub = fmin(ub, yg);
      } else {
        lb = fmax(lb, yg);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sfree += __shfl_xor_sync(0xffffffffu, sfree, o);
    if (lane == 0) red_d[(v0 >> 5) + warp] = sfree;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    nfree += __shfl_xor_sync(0xffffffffu, nfree, o);
    ub = fmin(ub, __shfl_xor_sync(0xffffffffu, ub, o));
    lb = fmax(lb, __shfl_xor_sync(0xffffffffu, lb, o));
  }
  __shared__ double red_n[TNW], red_ub[TNW], red_lb[TNW];
  if (lane == 0) {
    red_n[warp] = nfree;
    red_ub[warp] = ub;
    red_lb[warp] = lb;
  }
  __syncthreads();
  // 4. outputs: a_t y_t at the sample's position in the job's list
  for (int t = tid; t < np; t += TNT) coef[pos[t]] = float(alpha[t] * double(ys[t]));
  if (tid == 0) {
    double tf = 0.0, tn = 0.0;
    for (int w2 = 0; w2 < 8; ++w2) tf += red_d[w2];
    for (int w2 = 0; w2 < TNW; ++w2) {
      tn += red_n[w2];
      ub = fmin(ub, red_ub[w2]);
      lb = fmax(lb, red_lb[w2]);
    }
    double r;
    if (tn > 0.0) r = tf / tn;
    else if (ub < 1e299 && lb > -1e299) r = 0.5 * (ub + lb);
    else r = ub < 1e299 ? ub : lb;
    a.bias[(long long)job * a.n_pairs + p] = float(-r);
    if (a.iters) a.iters[(long long)job * a.n_pairs + p] = converged ? it : -1;
  }
}

struct PredictArgs {
  const float* kq;
  const float* kc;
  long long ld;
  int n_rows, n_cols;  // valid row / column indices of the kernel matrix
  unsigned* status;
  const float* w;
  const int32_t* rows;
  const int32_t* row_count;
  int r_max;
  const int32_t* idx;
  const int32_t* count;
  int m_max;
  const float* coef;
  const float* bias;
  int n_class;
  int n_pairs;
  float* decision;
  int32_t* pred;
};

// Shared memory (dynamic): the kernel values of the CTA's R rows ([R][m_max] floats) and the pair
// decisions. The coefficients, the larger operand, are read once for R rows.
template <int R>
__global__ void __launch_bounds__(NT) ovo_predict_kernel(const PredictArgs a) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  float* kr = reinterpret_cast<float*>(sm_raw);
  float* dec = kr + R * a.m_max;
  const int r0 = blockIdx.x * R, job = blockIdx.y;
  const int rc = a.row_count ? min(a.row_count[job], a.r_max) : a.r_max;
  if (r0 >= rc) return;
  const int cnt = a.count ? min(max(a.count[job], 0), a.m_max) : a.m_max;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t* idx = a.idx ? a.idx + (long long)job * a.m_max : nullptr;
  const float w = a.w[job];
  int row[R];  // -1: not classified
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = r0 + q;
    row[q] = r < rc ? (a.rows ? a.rows[(long long)job * a.r_max + r] : r) : -1;
    if (r < rc && (row[q] < 0 || row[q] >= a.n_rows)) {
      if (tid == 0) record_status(a.status, DEV_BAD_INDEX);
      row[q] = -1;
    }
  }
  for (int k = tid; k < cnt; k += NT) {
    const int c = idx ? idx[k] : k;
    const bool valid = c >= 0 && c < a.n_cols;
    bool used = false;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      used = used || row[q] >= 0;
      kr[q * a.m_max + k] = valid && row[q] >= 0 ? kval(a.kq, a.kc, a.ld, w, row[q], c) : 0.0f;
    }
    if (!valid && used) record_status(a.status, DEV_BAD_INDEX);  // this training sample does not contribute
  }
  __syncthreads();
  for (int p = warp; p < a.n_pairs; p += NW) {
    const float* cf = a.coef + ((long long)job * a.n_pairs + p) * a.m_max;
    float s[R];
#pragma unroll
    for (int q = 0; q < R; ++q) s[q] = 0.0f;
#pragma unroll 4
    for (int k = lane; k < cnt; k += 32) {
      const float v = __ldg(cf + k);
#pragma unroll
      for (int q = 0; q < R; ++q) s[q] = fmaf(v, kr[q * a.m_max + k], s[q]);
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
      if (lane == 0 && row[q] >= 0) {
        const float f = s[q] + a.bias[(long long)job * a.n_pairs + p];
        dec[q * a.n_pairs + p] = f;
        if (a.decision) a.decision[((long long)job * a.r_max + r0 + q) * a.n_pairs + p] = f;
      }
    }
  }
  __syncthreads();
  bool classify = false;
#pragma unroll
  for (int q = 0; q < R; ++q) classify = classify || (tid == q && row[q] >= 0);
  if (classify && a.pred) {
    int votes[MAX_CLASS];
    for (int c = 0; c < a.n_class; ++c) votes[c] = 0;
    for (int p = 0; p < a.n_pairs; ++p) {
      int c1, c2;
      pair_of(p, a.n_class, c1, c2);
      ++votes[dec[tid * a.n_pairs + p] > 0.0f ? c1 : c2];
    }
    int best = 0;
    for (int c = 1; c < a.n_class; ++c)
      if (votes[c] > votes[best]) best = c;
    a.pred[(long long)job * a.r_max + r0 + tid] = best;
  }
}

template <int R>
dk_status launch_predict(const PredictArgs& a, int n_jobs, cudaStream_t st) {
  const size_t smem = size_t(R) * size_t(a.m_max + a.n_pairs) * sizeof(float);
  // the shared-memory opt-in is per device: set before every launch that needs it
  if (smem > 48 * 1024 && cudaFuncSetAttribute(ovo_predict_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               int(smem)) != cudaSuccess)
    return DK_ERR_CUDA;
  ovo_predict_kernel<R><<<dim3((a.r_max + R - 1) / R, n_jobs), NT, smem, st>>>(a);
  return launch_status();
}

size_t train_smem(int m_max) {
  return size_t(m_max) * (2 * sizeof(double) + 3 * sizeof(float) + sizeof(int) + sizeof(short) + 2) + 16;
}

// Problems of skip < np <= cap samples, 128 or 256 threads a CTA.
dk_status launch_train(TrainArgs a, int skip, int cap, int n_jobs, cudaStream_t st) {
  a.skip = skip;
  a.cap = cap;
  const size_t smem = train_smem(cap);
  auto go = [&](auto kern, int threads) {
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
      return DK_ERR_CUDA;
    kern<<<dim3(a.n_pairs, n_jobs), threads, smem, st>>>(a);
    return launch_status();
  };
  return cap <= 1024 ? go(ovo_train_kernel<128>, 128) : go(ovo_train_kernel<256>, 256);
}

}  // namespace svm
}  // namespace dk

using namespace dk;

DK_API dk_status dk_svm_ovo_train(dk_ctx* ctx, const float* kq, const float* kc, long long ld, int n, int n_jobs,
                                  const float* w, const float* C, const int32_t* idx, const int32_t* count,
                                  int m_max, const int32_t* labels, int n_class, float tol, int max_iter,
                                  float* coef, float* bias, int32_t* iters, void* stream) {
  if (!ctx || (!kq && !kc) || !w || !C || !idx || !count || !labels || !coef || !bias) return DK_ERR_ARG;
  if (n_jobs < 1 || n_jobs > 65535 || m_max < 2 || n < 1 || ld < n || !(tol > 0.0f) || max_iter < 1)
    return DK_ERR_ARG;
  if (n_class < 2 || n_class > svm::MAX_CLASS) return DK_ERR_UNSUPPORTED;
  if (m_max > DK_SVM_MAX_SAMPLES) return DK_ERR_UNSUPPORTED;
  svm::TrainArgs a{kq,  kc,     ld,      n,     ctx->status, w, C, idx, count, m_max, labels, n_class,
                   n_class * (n_class - 1) / 2, double(tol), max_iter, coef, bias, iters, 0, 0};
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // a class pair of a balanced job holds 2 / n_class of its samples: where that leaves most of the
  // list out, the likely sizes go first and what exceeds them follows (its CTAs mostly see that
  // there is nothing to do: 10 us per 1000 of them)
  const int likely = (int(2.6 * m_max / n_class) + 63) / 32 * 32;
  if (10 * likely > 7 * m_max) return svm::launch_train(a, -1, m_max, n_jobs, st);
  const dk_status s = svm::launch_train(a, -1, likely, n_jobs, st);
  return s == DK_OK ? svm::launch_train(a, likely, m_max, n_jobs, st) : s;
}

DK_API dk_status dk_svm_ovo_predict(dk_ctx* ctx, const float* kq, const float* kc, long long ld, int n_rows,
                                    int n_cols, int n_jobs, const float* w, const int32_t* rows,
                                    const int32_t* row_count, int r_max, const int32_t* idx, const int32_t* count,
                                    int m_max, const float* coef, const float* bias, int n_class, float* decision,
                                    int32_t* pred, void* stream) {
  if (!ctx || (!kq && !kc) || !w || !coef || !bias || (!decision && !pred)) return DK_ERR_ARG;
  if (n_jobs < 1 || n_jobs > 65535 || r_max < 1 || m_max < 1 || n_rows < 1 || n_cols < 1 || ld < n_cols)
    return DK_ERR_ARG;
  if ((!rows && r_max > n_rows) || (!idx && m_max > n_cols)) return DK_ERR_ARG;
  if (n_class < 2 || n_class > svm::MAX_CLASS) return DK_ERR_UNSUPPORTED;
  if (m_max > DK_SVM_MAX_SAMPLES) return DK_ERR_UNSUPPORTED;
  const int n_pairs = n_class * (n_class - 1) / 2;
  svm::PredictArgs a{kq,    kc,        ld,    n_rows, n_cols, ctx->status, w,       rows,     row_count,
                     r_max, idx,       count, m_max,  coef,   bias,        n_class, n_pairs, decision, pred};
  // rows per CTA: as many as leave four CTAs per SM and fit in shared memory
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  auto fits = [&](int r) {
    return (long long)((r_max + r - 1) / r) * n_jobs >= 4LL * ctx->sm_count &&
           size_t(r) * size_t(m_max + n_pairs) * sizeof(float) <= 112 * 1024;
  };
  if (fits(8)) return svm::launch_predict<8>(a, n_jobs, st);
  if (fits(4)) return svm::launch_predict<4>(a, n_jobs, st);
  return svm::launch_predict<1>(a, n_jobs, st);
}
