// Data pre-processing of §II-A on the GPU: standardisation (zero mean, unit variance per
// pixel), PCA (the leading eigenvectors of the covariance of the standardised training rows)
// and min-max scaling of the projected features to [0, range_max].
//
// * Column statistics: two passes per column in FP64 (a constant column gets scale 1).
// * Covariance C = Z^T Z / (m - 1): 32 x 32 output tiles, the standardised rows staged in
//   shared memory 32 at a time, FP32 accumulation.
// * Eigenvectors: parallel cyclic Jacobi (round-robin pairing: every round rotates p/2
//   disjoint index pairs, a sweep is p - 1 rounds). Each 2 x 2 block (i1, j1) x (i2, j2) takes
//   both rotations at once, J1^T B J2, so rows and columns move together; the eigenvector
//   matrix is kept transposed (row i = eigenvector i), so its update is a row update. All
//   rounds run in one cooperative launch with the matrix in shared memory
//   (jacobi_persist_kernel) as long as it fits, one launch per round beyond. A fixed number of
//   sweeps runs without host synchronisation; the remaining relative off-diagonal norm is
//   returned.
// * Selection: eigenvalues ranked in decreasing order (the smaller index first on ties), the
//   leading k rows written with the sign that makes the entry of largest magnitude positive.
// * Transform: y = ((x - mean) / scale) C_k^T by 32 x 32 tiles; min-max scaling fitted on
//   the training rows (or given) and applied with clipping.
//
// Working memory (A and V^T, 2 p^2 floats, plus the rotation table) is a caller-provided
// workspace of dk_pca_workspace_bytes(p) bytes.
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "common.cuh"
#include "internal.h"
#include "jacobi_ring.h"

namespace dk {
namespace pca {

constexpr int T32 = 32;

// 8 columns x 8 row groups per CTA (two warps): FP64 issue bounds it, one warp instruction per 16
// cycles and SM, so the columns are spread over many SMs. 2000 x 784: 68 us (32 columns per CTA,
// eight warps on each of 25 SMs: 100 us). Every sum keeps its order.
__global__ void __launch_bounds__(64) col_stats_kernel(const float* __restrict__ x, int m, int p,
                                                       float* __restrict__ mean, float* __restrict__ scale) {
  constexpr int NC = 8;
  const int lc = threadIdx.x & (NC - 1), c = blockIdx.x * NC + lc, rg = threadIdx.x / NC;
  __shared__ double red[8][NC];
  __shared__ double s_mean[NC];
  double s = 0.0;
  if (c < p) {
#pragma unroll 8
    for (int r = rg; r < m; r += 8) s += double(x[(long long)r * p + c]);
  }
  red[rg][lc] = s;
  __syncthreads();
  if (rg == 0) {
    double t = 0.0;
    for (int g = 0; g < 8; ++g) t += red[g][lc];
    s_mean[lc] = t / m;
  }
  __syncthreads();
  const double mu = s_mean[lc];
  double q = 0.0;
  if (c < p) {
#pragma unroll 8
    for (int r = rg; r < m; r += 8) {
      const double d = double(x[(long long)r * p + c]) - mu;
      q += d * d;
    }
  }
  __syncthreads();
  red[rg][lc] = q;
  __syncthreads();
  if (rg == 0 && c < p) {
    double t = 0.0;
    for (int g = 0; g < 8; ++g) t += red[g][lc];
    const double var = t / m;
    mean[c] = float(mu);
    scale[c] = var > 0.0 ? float(sqrt(var)) : 1.0f;
  }
}

// C[i][j] = sum_r z_ri z_rj / (m - 1), z_rc = (x_rc - mean_c) / scale_c: 32 x 32 tiles on and
// above the diagonal, written to both sides (a product's factors commute, so the two sums are the
// same); the next 32 rows are loaded under the products of these. Bound by the loads' latency and
// the divisions. 2000 x 784: 172 us (every tile, loads and products in turn: 255 us).
__global__ void __launch_bounds__(256) cov_kernel(const float* __restrict__ x, int m, int p,
                                                  const float* __restrict__ mean, const float* __restrict__ scale,
                                                  float* __restrict__ A) {
  __shared__ __align__(16) float zi[T32][T32], zj[T32][T32];
  // tile row ti holds the tiles (ti, ti) .. (ti, nt - 1)
  const int nt = (p + T32 - 1) / T32;
  int ti = 0, tj = blockIdx.x;
  while (tj >= nt - ti) tj -= nt - ti++;
  const int i0 = ti * T32, j0 = (ti + tj) * T32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 8 rows of 4 outputs per thread
  // this thread stages columns i0 + tx and j0 + tx of rows ty, ty + 8, ty + 16, ty + 24
  const int ci = i0 + tx, cj = j0 + tx;
  const float mi = ci < p ? mean[ci] : 0.0f, si = ci < p ? scale[ci] : 1.0f;
  const float mj = cj < p ? mean[cj] : 0.0f, sj = cj < p ? scale[cj] : 1.0f;
  float vi[4], vj[4];
  auto load = [&](int r0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = r0 + ty + 8 * q;
      vi[q] = r < m && ci < p ? x[(long long)r * p + ci] : mi;
      vj[q] = r < m && cj < p ? x[(long long)r * p + cj] : mj;
    }
  };
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  load(0);
  for (int r0 = 0; r0 < m; r0 += T32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      // beyond the data the loads gave the mean itself: a zero
      zi[ty + 8 * q][tx] = r0 + ty + 8 * q < m ? (vi[q] - mi) / si : 0.0f;
      zj[ty + 8 * q][tx] = r0 + ty + 8 * q < m ? (vj[q] - mj) / sj : 0.0f;
    }
    __syncthreads();
    if (r0 + T32 < m) load(r0 + T32);
#pragma unroll 8
    for (int rr = 0; rr < T32; ++rr) {
      const float b = zj[rr][tx];
      const float4 a = *reinterpret_cast<const float4*>(&zi[rr][ty * 4]);
      acc[0] = fmaf(a.x, b, acc[0]);
      acc[1] = fmaf(a.y, b, acc[1]);
      acc[2] = fmaf(a.z, b, acc[2]);
      acc[3] = fmaf(a.w, b, acc[3]);
    }
    __syncthreads();
  }
  const float inv = 1.0f / float(m - 1);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = i0 + ty * 4 + q, j = j0 + tx;
    if (i < p && j < p) {
      A[(long long)i * p + j] = acc[q] * inv;
      if (i0 != j0) A[(long long)j * p + i] = acc[q] * inv;
    }
  }
}

// Vt = identity
__global__ void eye_kernel(float* __restrict__ Vt, int p) {
  const long long n = (long long)p * p;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    Vt[e] = (e / p == e % p) ? 1.0f : 0.0f;
}

// index of round-robin position t in round r (positions 0..pe-1, pe even; 0 stays put)
__device__ __forceinline__ int rr_pos(int t, int r, int pe) { return t == 0 ? 0 : 1 + (t - 1 + r) % (pe - 1); }

// (c, s, t) of the rotation that zeroes a_ij, i < j
__device__ __forceinline__ float4 pair_rotation(float aii, float ajj, float aij) {
  float c = 1.0f, s = 0.0f, t = 0.0f;
  if (fabsf(aij) > 1e-30f) {
    // angle that zeroes a_ij: tau = (a_jj - a_ii) / (2 a_ij), t the smaller root
    const float tau = (ajj - aii) / (2.0f * aij);
    t = (tau >= 0.0f ? 1.0f : -1.0f) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
    c = rsqrt_chain(1.0f + t * t);  // correctly rounded: c^2 + s^2 - 1 stays unbiased
    s = t * c;
  }
  return make_float4(c, s, t, 0.0f);
}

// B' = J1^T B J2 of one 2 x 2 block (J = [[c, s], [-s, c]]); `own`: the block of a pair with
// itself, whose rotation zeroes the off-diagonal and moves the diagonal by -/+ t a_ij, which
// keeps the trace to one rounding
__device__ __forceinline__ void rotate_block(float4 r1, float4 r2, bool own, float& b00, float& b01, float& b10,
                                             float& b11) {
  // explicit fmaf: the same bits wherever a block or one of its elements is computed
  // rows: R0 = c1 B0 - s1 B1, R1 = s1 B0 + c1 B1
  const float q00 = fmaf(r1.x, b00, -__fmul_rn(r1.y, b10)), q01 = fmaf(r1.x, b01, -__fmul_rn(r1.y, b11));
  const float q10 = fmaf(r1.y, b00, __fmul_rn(r1.x, b10)), q11 = fmaf(r1.y, b01, __fmul_rn(r1.x, b11));
  // columns: C0 = c2 R.0 - s2 R.1, C1 = s2 R.0 + c2 R.1
  float n00 = fmaf(r2.x, q00, -__fmul_rn(r2.y, q01)), n01 = fmaf(r2.y, q00, __fmul_rn(r2.x, q01));
  float n10 = fmaf(r2.x, q10, -__fmul_rn(r2.y, q11)), n11 = fmaf(r2.y, q10, __fmul_rn(r2.x, q11));
  if (own) {
    n00 = fmaf(-r1.z, b01, b00);
    n11 = fmaf(r1.z, b01, b11);
    n01 = 0.0f;
    n10 = 0.0f;
  }
  b00 = n00;
  b01 = n01;
  b10 = n10;
  b11 = n11;
}

// rows i, j of V^T under the pair's rotation
__device__ __forceinline__ void rotate_rows(float c, float s, float& u, float& v) {
  const float a = fmaf(c, u, -__fmul_rn(s, v)), b = fmaf(s, u, __fmul_rn(c, v));
  u = a;
  v = b;
}

// rotation angles of pair k of round r: (i, j, c, s) with i < j; a pair holding the
// padding index p (odd p) is the identity
__device__ __forceinline__ void jacobi_pair_params(const float* A, int p, int pe, int r, int k, int2* ij,
                                                   float4* cs) {
  int i = rr_pos(k, r, pe), j = rr_pos(pe - 1 - k, r, pe);
  if (i > j) {
    const int t = i;
    i = j;
    j = t;
  }
  ij[k] = make_int2(i, j);
  cs[k] = j < p ? pair_rotation(A[(long long)i * p + i], A[(long long)j * p + j], A[(long long)i * p + j])
                : make_float4(1.0f, 0.0f, 0.0f, 0.0f);
}

// the rotation angles of round r (the first round of a fit)
__global__ void jacobi_params_kernel(const float* __restrict__ A, int p, int pe, int r, int2* __restrict__ ij,
                                     float4* __restrict__ cs) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < pe / 2) jacobi_pair_params(A, p, pe, r, k, ij, cs);
}

// one round: block (k1) handles the rows of pair k1; thread k2 the 2 x 2 block with the
// columns of pair k2: B' = J1^T B J2 (J = [[c, s], [-s, c]]); the block's pair also rotates
// rows i1, j1 of V^T
//
// One launch per round: the CTA that finishes the round last (a counter each CTA bumps after
// a fence) computes the next round's angles from the finished matrix, so no launch of its
// own and no CTA waits for another; it also resets the counter. r_next < 0: last round.
__global__ void __launch_bounds__(256) jacobi_rotate_kernel(float* __restrict__ A, float* __restrict__ Vt, int p,
                                                            int npairs, int2* __restrict__ ij,
                                                            float4* __restrict__ cs, unsigned* __restrict__ done,
                                                            int pe, int r_next) {
  const int k1 = blockIdx.x;
  const int2 a = ij[k1];
  const float4 r1 = cs[k1];
  const int i1 = a.x, j1 = a.y;
  const bool has_j1 = j1 < p;
  for (int k2 = threadIdx.x; k2 < npairs; k2 += blockDim.x) {
    const int2 b = ij[k2];
    const float4 r2 = cs[k2];
    const int i2 = b.x, j2 = b.y;
    const bool has_j2 = j2 < p;
    float b00 = A[(long long)i1 * p + i2];
    float b01 = has_j2 ? A[(long long)i1 * p + j2] : 0.0f;
    float b10 = has_j1 ? A[(long long)j1 * p + i2] : 0.0f;
    float b11 = (has_j1 && has_j2) ? A[(long long)j1 * p + j2] : 0.0f;
    rotate_block(r1, r2, k1 == k2 && has_j1, b00, b01, b10, b11);
    A[(long long)i1 * p + i2] = b00;
    if (has_j2) A[(long long)i1 * p + j2] = b01;
    if (has_j1) A[(long long)j1 * p + i2] = b10;
    if (has_j1 && has_j2) A[(long long)j1 * p + j2] = b11;
  }
  if (has_j1) {
    for (int col = threadIdx.x; col < p; col += blockDim.x) {
      float u = Vt[(long long)i1 * p + col], v = Vt[(long long)j1 * p + col];
      rotate_rows(r1.x, r1.y, u, v);
      Vt[(long long)i1 * p + col] = u;
      Vt[(long long)j1 * p + col] = v;
    }
  }
  if (r_next < 0) return;
  __shared__ bool last;
  __threadfence();  // this CTA's writes of A are visible before it counts itself done
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(done, 1u) == unsigned(npairs - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();  // every other CTA's writes are visible to this one
  for (int k = threadIdx.x; k < npairs; k += blockDim.x) jacobi_pair_params(A, p, pe, r_next, k, ij, cs);
  if (threadIdx.x == 0) *done = 0u;
}

// ---- the same rounds in one launch, the matrix held in shared memory ----
//
// A round of the launch-per-round form is a few hundred nanoseconds of arithmetic inside 10 us
// of launch, scattered reads and a last-CTA pass. Here one cooperative launch runs every round:
//  * Round-robin positions are a ring: with position 0 fixed, the index at position t moves to
//    t - 1 each round (1 to pe - 1). Pair k holds positions (k, pe - 1 - k). CTA g owns `ppc`
//    consecutive pairs, i.e. the rows of A at 2 ppc positions, whole, in shared memory; per
//    round one row of its upper run goes to CTA g - 1 and one of its lower run to g + 1.
//  * The angle of a pair needs a_ii, a_jj and a_ij. A diagonal element changes only with its own
//    pair's rotation, so every CTA keeps the whole diagonal; the owner of row i computes the
//    pair's a_ij of the next round and its angle first of all and publishes them. A round then
//    costs one trip through L2, under which the rows and the columns of V^T are rotated. V^T is
//    split by columns, which rotations never mix.
//  * Rows stand at their positions in two copies: a round reads one and writes the other, each
//    row where it stands next, so one barrier a round is enough.
//  * Everything in transit is a 16-byte word with a round tag, stored and loaded as one: the tag
//    says that the values are there, so there is no barrier and no fence. Words alternate
//    between two buffers. Every CTA publishes at least one word in every round and every CTA
//    waits for all of them (ring_publishes says why; the pair of an odd p's padding index has
//    its word too, and a last CTA of one pair always sends one, for which a thread of its own
//    waits). A CTA publishes for round q + 1 only when it has read all words of round q, so a
//    CTA that has all words of round q + 1 and writes over those of round q knows that every
//    other one has read them. The rows' words need only that neighbours send to each other in
//    every round. All waits are bounded; the launch is cooperative, so the CTAs run at the same
//    time.
// Below 64 features one CTA does it all (SOLO), and the angles pass through shared memory: 10 sweeps
// take 0.50 ms at p = 48 and 0.66 at 62, several CTAs 0.60 at 48 and 0.69 at 64, and at p = 130, where one
// CTA's rows and V^T take longer than a trip through L2, 1.8 against 9.2 ms.
// The arithmetic and its order are those of jacobi_rotate_kernel: bit-identical results.
// Bound by the latency of a round: the L2 round trip (about 950 cycles from a store to another
// SM's load of it), the angle's divisions and roots (about 700 on one warp) and one barrier.
// Measured, 10 sweeps at p = 784 (131 CTAs of 3 row pairs): 12.7 ms, 1.6 us a round, against
// 79.4 ms with one launch per round (10.1 us).

struct PersistArgs {
  float* A;
  float* Vt;
  uint4* words;  // box memory
  unsigned* done;
  unsigned* failed;
  unsigned* status;
  int p, ppc, vc, rounds;
};

// Round tags are bit patterns of negative signalling NaNs, which no arithmetic result has, so
// nothing that the workspace held before (the covariance) reads as one.
__device__ __forceinline__ unsigned tag_of(int round) { return 0xff800001u + unsigned(round); }

__device__ __forceinline__ void put_word(uint4* w, float v0, float v1, float v2, unsigned tag) {
  asm volatile(
      "{\n\t.reg .b128 x;\n\t.reg .b64 lo, hi;\n\tmov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\t"
      "mov.b128 x, {lo, hi};\n\tst.relaxed.gpu.global.b128 [%0], x;\n\t}" ::"l"(w),
      "r"(__float_as_uint(v0)), "r"(__float_as_uint(v1)), "r"(__float_as_uint(v2)), "r"(tag)
      : "memory");
}
__device__ __forceinline__ uint4 get_word(const uint4* w) {
  unsigned long long lo, hi;
  asm volatile(
      "{\n\t.reg .b128 x;\n\tld.relaxed.gpu.global.b128 x, [%2];\n\tmov.b128 {%0, %1}, x;\n\t}"
      : "=l"(lo), "=l"(hi)
      : "l"(w)
      : "memory");
  return make_uint4(unsigned(lo), unsigned(lo >> 32), unsigned(hi), unsigned(hi >> 32));
}

// Waits (bounded) until the word at `src` carries `tag`; `w` may hold an earlier look at it. The
// clock, a slow read, is looked at every 1024 polls.
__device__ __forceinline__ bool await_word(uint4& w, const uint4* src, unsigned tag) {
  unsigned long long t0 = 0;
  for (unsigned it = 1; w.w != tag; ++it) {
    w = get_word(src);
    if ((it & 1023u) == 0u) {
      const unsigned long long t = globaltimer_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > WAIT_LIMIT_NS) return false;
    }
  }
  return true;
}

// ODD: p is odd; SOLO: one CTA
template <int MAXT, bool ODD, bool SOLO>
__global__ void __launch_bounds__(MAXT, 1) jacobi_persist_kernel(const PersistArgs a) {
  constexpr int NR = MAXT > 512 ? 2 : UR;  // row pairs in flight: what the registers hold
  extern __shared__ __align__(16) float sm[];
  const int p = a.p, pe = p + (p & 1), np = pe / 2, ring = pe - 1;
  const int G = int(gridDim.x), g = int(blockIdx.x), NT = int(blockDim.x), tid = int(threadIdx.x);
  const int ks = g * a.ppc, ke = min(ks + a.ppc, np), cnt = ke - ks;
  const int v0 = g * a.vc, vn = max(0, min(a.vc, p - v0)), vp = (a.vc + 3) / 4;
  constexpr bool solo = SOLO;
  const bool lone = !SOLO && ring_lone(np, a.ppc);
  // shared memory: V^T columns [plane][row][4], angles [2 rounds][pair] (c, s, t), solo: the
  // published angles by x, rows [2 rounds][local row][pe], the diagonal of A
  float4* V = reinterpret_cast<float4*>(sm);
  float4* pars = V + vp * pe;
  float4* sN = pars + 2 * np;
  float* rows = reinterpret_cast<float*>(sN + pe);
  float* sD = rows + 4 * a.ppc * pe;
  __shared__ int s_abort;
  uint4* wR = a.words;                                              // [buffer][CTA][upper / lower][np]
  uint4* wN = wR + (solo ? 0 : size_t(4) * G * np);                 // [buffer][pe]
  auto box = [&](int buf, int cta, int which) { return wR + (size_t(buf * G + cta) * 2 + which) * np; };
  auto idx_at = [&](int t, int r) { return ring_index(t, r, ring); };
  auto came_from = [&](int t) { return ring_came_from(t, ring); };
  auto goes_to = [&](int t) { return ring_goes_to(t, ring); };
  // local row u < cnt: position ks + u; u >= cnt: position pe - ke + (u - cnt)
  auto pos_of = [&](int u) { return ring_row_position(u, ks, ke, pe); };
  auto row_at = [&](int t) { return t < np ? t - ks : cnt + t - (pe - ke); };
  // where local row u stands next; -1: at another CTA
  auto moves_to = [&](int u) {
    const int t = goes_to(pos_of(u));
    return ((t >= ks && t < ke) || (t >= pe - ke && t < pe - ks)) ? row_at(t) : -1;
  };

  for (int e = tid; e < 2 * cnt * pe; e += NT) {
    const int u = e / pe, c = e - u * pe, i = pos_of(u);
    rows[e] = (i < p && c < p) ? a.A[(long long)i * p + c] : 0.0f;
    rows[2 * a.ppc * pe + e] = 0.0f;  // column p of an odd p stays zero
  }
  for (int i = tid; i < p; i += NT) sD[i] = a.A[(long long)i * p + i];
  for (int e = tid; e < vp * pe; e += NT) {
    const int pl = e / pe, i = e - pl * pe, c = v0 + 4 * pl;
    V[e] = make_float4(c == i ? 1.0f : 0.0f, c + 1 == i ? 1.0f : 0.0f, c + 2 == i ? 1.0f : 0.0f,
                       c + 3 == i ? 1.0f : 0.0f);
  }
  if (tid == 0) s_abort = 0;
  __syncthreads();  // what this CTA reads of A is read: only now does it publish anything
  for (int u = tid; u < 2 * cnt; u += NT) {
    const int i = pos_of(u), j = ring - i;  // round 0: index = position
    if (i < j) {
      const float o = j < p ? rows[u * pe + j] : 0.0f;
      const float4 w = j < p ? pair_rotation(sD[i], sD[j], o) : make_float4(1.0f, 0.0f, 0.0f, 0.0f);
      if (solo) sN[i] = make_float4(w.x, w.z, o, 0.0f);
      else put_word(wN + i, w.x, w.z, o, tag_of(0));
    }
  }
  __syncthreads();

  const int side = ring_side_threads(a.ppc, np), workers = NT - side;
  const int copy = 2 * a.ppc * pe;  // floats between the two copies of the rows
  const bool can_up = g < G - 1, can_low = g > 0;
  if (tid >= workers) {
    // ---- the next round's elements and angles: row u's partner is at position ty, that one's at ring - ty ----
    const int u = tid - workers;
    const bool holds = u < 2 * cnt;
    const int hu = holds ? (u < cnt ? u : 2 * cnt - 1 - u) : 0;
    const int tx = holds ? pos_of(u) : 0, ty = holds ? came_from(ring - goes_to(tx)) : 0, kc = min(ty, ring - ty);
    const bool watches = lone && u == 2 * a.ppc;  // waits for the lone CTA's word
    int r = 0;
    for (int q = 0; q < a.rounds; ++q) {
      const int buf = q & 1;
      const int x = idx_at(tx, r), y = idx_at(ty, r), z = idx_at(ring - ty, r);
      const bool up = idx_at(ks + hu, r) < idx_at(ring - ks - hu, r), low = y < z;
      const float* ri = rows + buf * copy + (up ? hu : 2 * cnt - 1 - hu) * pe;
      const float* rj = rows + buf * copy + (up ? 2 * cnt - 1 - hu : hu) * pe;
      const int c0 = low ? y : z, c1 = low ? z : y;
      const bool is_i = (u < cnt) == up;
      if (watches) {
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (!await_word(w, wN + buf * pe + ring_lone_index(np, r, ring), tag_of(q))) s_abort = 1;
      }
      __syncthreads();
      if (s_abort) break;
      const bool publishes = q + 1 < a.rounds && holds && ring_publishes(x, y, tx, np, lone);
      const bool real = y > x && (!ODD || y < p);
      if (publishes && !real && !solo) put_word(wN + (buf ^ 1) * pe + x, 1.0f, 0.0f, 0.0f, tag_of(q + 1));
      if (publishes && real) {  // otherwise the partner's owner does it
        float b00 = ri[c0], b01 = ri[c1], b10 = rj[c0], b11 = rj[c1];
        rotate_block(pars[buf * np + ks + hu], pars[buf * np + kc], ks + hu == kc, b00, b01, b10, b11);
        const float o = is_i ? (low ? b00 : b01) : (low ? b10 : b11);
        const float4 w = pair_rotation(sD[x], sD[y], o);
        if (solo) sN[x] = make_float4(w.x, w.z, o, 0.0f);
        else put_word(wN + (buf ^ 1) * pe + x, w.x, w.z, o, tag_of(q + 1));
      }
      if (++r == ring) r = 0;
      if (solo) __syncthreads();
    }
  } else {
    // ---- column pair k2 and, NR at a time, the row pairs grp, grp + groups, ... of an order that
    // takes the two with a row to send first ----
    const int lanes = (np + 31) / 32 * 32;
    int groups = workers / lanes, grp = tid / lanes, k2 = tid - grp * lanes;
    asm volatile("" : "+r"(groups), "+r"(grp), "+r"(k2));  // opaque: not to be divided again in every round
    const bool active = k2 < np;
    auto turn = [&](int n) { return n == 0 ? 0 : (n == 1 ? cnt - 1 : n - 1); };
    // what stays the same in every round, for the first NR row pairs: where the rows stand and go
    // (floats; -1: sent away), and the rounds [first, first + len) in which the lower position
    // holds the smaller index
    const bool once = cnt <= NR * groups;
    int st_u[NR], st_ou[NR], st_ol[NR], st_du[NR], st_dl[NR], st_f[NR], st_len[NR];
    auto set_turn = [&](int z, int n) {
      const int u = turn(n), t = ks + u;
      st_u[z] = u;
      st_ou[z] = u * pe;
      st_ol[z] = (2 * cnt - 1 - u) * pe;
      const int du = moves_to(u), dl = moves_to(2 * cnt - 1 - u);
      st_du[z] = du < 0 ? -1 : du * pe;
      st_dl[z] = dl < 0 ? -1 : dl * pe;
      st_f[z] = t + 1;
      st_len[z] = t == 0 ? 0 : ring - 2 * t;
    };
#pragma unroll
    for (int z = 0; z < NR; ++z) set_turn(z, min(grp + z * groups, cnt - 1));
    uint4* in_up = box(0, g, 0) + k2;
    uint4* in_low = box(0, g, 1) + k2;
    uint4* out_up = can_low ? box(0, g - 1, 0) + k2 : nullptr;   // the row at position ks
    uint4* out_low = can_up ? box(0, g + 1, 1) + k2 : nullptr;   // at pe - ke
    const size_t flip = size_t(2) * G * np;                       // words between the two buffers
    // the rows in transit: group 0 takes the upper one, and the lower one if it is the only group
    const bool takes_up = can_up && active && grp == 0, takes_low = can_low && active && grp == (groups > 1 ? 1 : 0);
    const uint4 none = make_uint4(0u, 0u, 0u, 0u);
    uint4 wn = none, wu = none, wl = none;  // looks at the next round's angle and row words
    bool ok = true;
    int x2 = k2, y2 = active ? ring - k2 : 0;  // the pair's indices: they move up by one each round
    int xp = 0, yp = 0;
    int r = 0;
    for (int q = 0; q < a.rounds; ++q) {
      const unsigned tag = tag_of(q), next = tag_of(q + 1);
      const int buf = q & 1;
      const bool more = q + 1 < a.rounds;
      float4* par = pars + buf * np;
      float* cur = rows + buf * copy;
      float* nxt = rows + (buf ^ 1) * copy;
      const int i2 = min(x2, y2), j2 = max(x2, y2);
      const bool has_j2 = !ODD || j2 < p;
      // 1. every pair's angle, and the whole diagonal after this round; the rows that moved here
      // (the ends of the upper run, from CTA g + 1, and of the lower one, from g - 1)
      float4 r2 = make_float4(1.0f, 0.0f, 0.0f, 0.0f);
      if (grp == 0 && active) {
        if (!solo) ok = await_word(wn, wN + buf * pe + i2, tag) && ok;  // the padding index's pair too
        if (has_j2) {
          float o;
          if (solo) {
            const float4 v = sN[i2];
            r2.x = v.x;
            r2.z = v.y;
            o = v.z;
          } else {
            r2.x = __uint_as_float(wn.x);
            r2.z = __uint_as_float(wn.y);
            o = __uint_as_float(wn.z);
          }
          r2.y = r2.z * r2.x;
          sD[i2] = fmaf(-r2.z, o, sD[i2]);  // the pair's own block in rotate_block
          sD[j2] = fmaf(r2.z, o, sD[j2]);
        }
        par[k2] = r2;
      }
      if (q > 0) {
        const int ip = min(xp, yp), jp = max(xp, yp);  // the columns of pair k2 in the round that sent them
        if (takes_up) {
          ok = await_word(wu, in_up + buf * flip, tag) && ok;
          cur[(cnt - 1) * pe + ip] = __uint_as_float(wu.x);
          if (!ODD || jp < p) cur[(cnt - 1) * pe + jp] = __uint_as_float(wu.y);
        }
        if (takes_low) {
          ok = await_word(wl, in_low + buf * flip, tag) && ok;
          cur[(2 * cnt - 1) * pe + ip] = __uint_as_float(wl.x);
          if (!ODD || jp < p) cur[(2 * cnt - 1) * pe + jp] = __uint_as_float(wl.y);
        }
      }
      if (!ok) s_abort = 1;
      __syncthreads();
      if (s_abort) break;
      // 2. this CTA's rows
      if (grp != 0 && active) r2 = par[k2];
      if (active) {
        for (int n0 = grp; n0 < cnt; n0 += NR * groups) {
          if (!once) {
#pragma unroll
            for (int z = 0; z < NR; ++z) set_turn(z, min(n0 + z * groups, cnt - 1));
          }
          float b[NR][4];
          float4 r1[NR];
#pragma unroll
          for (int z = 0; z < NR; ++z) {
            if (n0 + z * groups < cnt) {
              const bool up = unsigned(r - st_f[z]) >= unsigned(st_len[z]);  // the upper position holds i
              const float* ri = cur + (up ? st_ou[z] : st_ol[z]);
              const float* rj = cur + (up ? st_ol[z] : st_ou[z]);
              r1[z] = par[ks + st_u[z]];
              b[z][0] = ri[i2];
              b[z][1] = ri[j2];
              b[z][2] = rj[i2];
              b[z][3] = rj[j2];
            }
          }
#pragma unroll
          for (int z = 0; z < NR; ++z) {
            if (n0 + z * groups < cnt) {
              const int u = st_u[z];
              const bool up = unsigned(r - st_f[z]) >= unsigned(st_len[z]);
              rotate_block(r1[z], r2, ks + u == k2 && has_j2, b[z][0], b[z][1], b[z][2], b[z][3]);
              if (ODD && max(idx_at(ks + u, r), idx_at(ring - ks - u, r)) == p) b[z][2] = b[z][3] = 0.0f;  // no such row
              const float u0 = up ? b[z][0] : b[z][2], u1 = up ? b[z][1] : b[z][3];  // the upper row's values
              const float l0 = up ? b[z][2] : b[z][0], l1 = up ? b[z][3] : b[z][1];
              if (more) {
                if (st_du[z] >= 0) {
                  nxt[st_du[z] + i2] = u0;
                  if (has_j2) nxt[st_du[z] + j2] = u1;
                } else {
                  put_word(out_up + (buf ^ 1) * flip, u0, u1, 0.0f, next);
                }
                if (st_dl[z] >= 0) {
                  nxt[st_dl[z] + i2] = l0;
                  if (has_j2) nxt[st_dl[z] + j2] = l1;
                } else {
                  put_word(out_low + (buf ^ 1) * flip, l0, l1, 0.0f, next);
                }
              } else {  // the last round's rows stay where they are
                nxt[st_ou[z] + i2] = u0;
                if (has_j2) nxt[st_ou[z] + j2] = u1;
                nxt[st_ol[z] + i2] = l0;
                if (has_j2) nxt[st_ol[z] + j2] = l1;
              }
            }
          }
        }
        // 3. this CTA's columns of V^T
        if (has_j2) {
#pragma unroll 2
          for (int pl = grp; pl < vp; pl += groups) {
            float4 u = V[pl * pe + i2], v = V[pl * pe + j2];
            rotate_rows(r2.x, r2.y, u.x, v.x);
            rotate_rows(r2.x, r2.y, u.y, v.y);
            rotate_rows(r2.x, r2.y, u.z, v.z);
            rotate_rows(r2.x, r2.y, u.w, v.w);
            V[pl * pe + i2] = u;
            V[pl * pe + j2] = v;
          }
        }
        // 4. the pair's indices in the next round, and a first look at its words
        xp = x2;
        yp = y2;
        if (x2 != 0) x2 = x2 == ring ? 1 : x2 + 1;  // position 0 keeps index 0
        y2 = y2 == ring ? 1 : y2 + 1;
        if (!solo && more) {
          if (grp == 0) wn = get_word(wN + (buf ^ 1) * pe + min(x2, y2));
          if (takes_up) wu = get_word(in_up + (buf ^ 1) * flip);
          if (takes_low) wl = get_word(in_low + (buf ^ 1) * flip);
        }
      }
      if (++r == ring) r = 0;
      if (solo) __syncthreads();  // the next angles are in shared memory
    }
  }

  // every CTA has read its last words before the memory that holds them is written
  __syncthreads();
  if (!solo) {
    if (tid == 0) {
      __threadfence();
      atomicAdd(a.done, 1u);
      const unsigned long long t0 = globaltimer_ns();
      while (*reinterpret_cast<volatile unsigned*>(a.done) < unsigned(G))
        if (globaltimer_ns() - t0 > WAIT_LIMIT_NS) {
          s_abort = 1;
          break;
        }
    }
    __syncthreads();
  }
  if (s_abort) {
    if (tid == 0) {
      record_status(a.status, DEV_TIMEOUT);
      *a.failed = 1u;  // A and V^T are not a result: the outputs become NaN
    }
    return;
  }
  const int rl = (a.rounds - 1) % ring;  // rows stand where the last round had them
  const float* last = rows + (a.rounds & 1) * copy;
  for (int e = tid; e < 2 * cnt * p; e += NT) {
    const int u = e / p, c = e - u * p, i = idx_at(pos_of(u), rl);
    if (i < p) a.A[(long long)i * p + c] = last[u * pe + c];
  }
  for (int e = tid; e < p * vn; e += NT) {
    const int i = e / vn, c = e - i * vn;
    a.Vt[(long long)i * p + v0 + c] = reinterpret_cast<const float*>(V + (c >> 2) * pe + i)[c & 3];
  }
}

// sqrt(off-diagonal sum of squares / total sum of squares) of A: CTA b sums the rows b, b + grid,
// ... into part[b] (off-diagonal, total); the finish adds the parts in order
__global__ void __launch_bounds__(256) off_norm_kernel(const float* __restrict__ A, int p, double2* __restrict__ part) {
  double off = 0.0, all = 0.0;
  for (int i = blockIdx.x; i < p; i += gridDim.x)
    for (int c = threadIdx.x; c < p; c += 256) {
      const double v = A[(long long)i * p + c], v2 = v * v;
      all += v2;
      if (c != i) off += v2;
    }
  __shared__ double s_off[256], s_all[256];
  s_off[threadIdx.x] = off;
  s_all[threadIdx.x] = all;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      s_off[threadIdx.x] += s_off[threadIdx.x + h];
      s_all[threadIdx.x] += s_all[threadIdx.x + h];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = make_double2(s_off[0], s_all[0]);
}

__global__ void __launch_bounds__(32) off_norm_finish_kernel(const double2* __restrict__ part, int n,
                                                             const unsigned* __restrict__ failed,
                                                             float* __restrict__ out) {
  double off = 0.0, all = 0.0;
  for (int e = threadIdx.x; e < n; e += 32) {
    off += part[e].x;
    all += part[e].y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    off += __shfl_xor_sync(0xffffffffu, off, o);
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  if (threadIdx.x == 0) *out = *failed ? NAN : all > 0.0 ? float(sqrt(off / all)) : 0.0f;
}

// block i: the rank of eigenvalue A_ii among all (decreasing, smaller index first on ties);
// if below k, row rank of the output is row i of V^T with the sign of its largest entry. All NaN if
// the rounds gave up.
__global__ void __launch_bounds__(256) select_kernel(const float* __restrict__ A, const float* __restrict__ Vt, int p,
                                                     int k, const unsigned* __restrict__ failed,
                                                     float* __restrict__ comps, float* __restrict__ eig) {
  const int i = blockIdx.x;
  if (*failed) {
    if (i >= k) return;
    for (int c = threadIdx.x; c < p; c += 256) comps[(long long)i * p + c] = NAN;
    if (threadIdx.x == 0) eig[i] = NAN;
    return;
  }
  const float li = A[(long long)i * p + i];
  __shared__ int s_rank[256];
  __shared__ float s_best[256];
  __shared__ int s_bi[256];
  int cnt = 0;
  for (int j = threadIdx.x; j < p; j += 256) {
    const float lj = A[(long long)j * p + j];
    if (lj > li || (lj == li && j < i)) ++cnt;
  }
  s_rank[threadIdx.x] = cnt;
  float best = -1.0f;
  int bi = p;
  for (int c = threadIdx.x; c < p; c += 256) {
    const float v = fabsf(Vt[(long long)i * p + c]);
    if (v > best) {
      best = v;
      bi = c;
    }
  }
  s_best[threadIdx.x] = best;
  s_bi[threadIdx.x] = bi;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      s_rank[threadIdx.x] += s_rank[threadIdx.x + h];
      const float ob = s_best[threadIdx.x + h];
      const int oi = s_bi[threadIdx.x + h];
      if (ob > s_best[threadIdx.x] || (ob == s_best[threadIdx.x] && oi < s_bi[threadIdx.x])) {
        s_best[threadIdx.x] = ob;
        s_bi[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  const int rank = s_rank[0];
  if (rank >= k) return;
  const float sign = Vt[(long long)i * p + s_bi[0]] < 0.0f ? -1.0f : 1.0f;
  for (int c = threadIdx.x; c < p; c += 256) comps[(long long)rank * p + c] = sign * Vt[(long long)i * p + c];
  if (threadIdx.x == 0) eig[rank] = li;
}

// out[r][q] = sum_c ((x_rc - mean_c) / scale_c) comps[q][c]; 32 x 32 tiles (rows x components)
__global__ void __launch_bounds__(256) transform_kernel(const float* __restrict__ x, int m, int p,
                                                        const float* __restrict__ mean, const float* __restrict__ scale,
                                                        const float* __restrict__ comps, int k, float* __restrict__ out) {
  __shared__ float zs[T32][T32 + 1], cs_[T32][T32 + 1];
  const int r0 = blockIdx.y * T32, q0 = blockIdx.x * T32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  for (int c0 = 0; c0 < p; c0 += T32) {
    for (int e = threadIdx.x; e < T32 * T32; e += 256) {
      const int a = e / T32, b = e % T32;
      const int r = r0 + a, c = c0 + b, q = q0 + a;
      zs[a][b] = (r < m && c < p) ? (x[(long long)r * p + c] - mean[c]) / scale[c] : 0.0f;
      cs_[a][b] = (q < k && c < p) ? comps[(long long)q * p + c] : 0.0f;
    }
    __syncthreads();
#pragma unroll 8
    for (int b = 0; b < T32; ++b) {
      const float w = cs_[tx][b];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = fmaf(zs[ty * 4 + u][b], w, acc[u]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = r0 + ty * 4 + u, q = q0 + tx;
    if (r < m && q < k) out[(long long)r * k + q] = acc[u];
  }
}

__global__ void __launch_bounds__(256) minmax_fit_kernel(const float* __restrict__ y, int m, int k,
                                                         float* __restrict__ lo, float* __restrict__ hi) {
  const int c = blockIdx.x * 32 + (threadIdx.x & 31), rg = threadIdx.x >> 5;
  float mn = INFINITY, mx = -INFINITY;
  if (c < k)
    for (int r = rg; r < m; r += 8) {
      const float v = y[(long long)r * k + c];
      mn = fminf(mn, v);
      mx = fmaxf(mx, v);
    }
  __shared__ float smn[8][32], smx[8][32];
  smn[rg][threadIdx.x & 31] = mn;
  smx[rg][threadIdx.x & 31] = mx;
  __syncthreads();
  if (rg == 0 && c < k) {
    for (int g = 1; g < 8; ++g) {
      mn = fminf(mn, smn[g][threadIdx.x]);
      mx = fmaxf(mx, smx[g][threadIdx.x]);
    }
    lo[c] = mn;
    hi[c] = mx;
  }
}

__global__ void minmax_apply_kernel(float* __restrict__ y, long long n, int k, const float* __restrict__ lo,
                                    const float* __restrict__ hi, float range_max) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int c = int(e % k);
    const float span = hi[c] - lo[c];
    float v = span > 0.0f ? (y[e] - lo[c]) / span * range_max : 0.0f;
    y[e] = fminf(fmaxf(v, 0.0f), range_max);
  }
}

struct Workspace {
  float* A;
  float* Vt;
  int2* ij;
  float4* cs;
  unsigned* done;    // CTAs finished in the current Jacobi round
  unsigned* failed;  // a wait of the one-launch form ran out
};

inline size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

inline size_t workspace_bytes(int p) {
  const size_t pe = size_t(p + (p & 1));
  return 2 * round256(size_t(p) * p * sizeof(float)) + round256(pe / 2 * sizeof(int2)) +
         round256(pe / 2 * sizeof(float4)) + 256;
}

inline Workspace carve(void* ws, int p) {
  uint8_t* b = static_cast<uint8_t*>(ws);
  const size_t pe = size_t(p + (p & 1));
  Workspace w;
  w.A = reinterpret_cast<float*>(b);
  b += round256(size_t(p) * p * sizeof(float));
  w.Vt = reinterpret_cast<float*>(b);
  b += round256(size_t(p) * p * sizeof(float));
  w.ij = reinterpret_cast<int2*>(b);
  b += round256(pe / 2 * sizeof(int2));
  w.cs = reinterpret_cast<float4*>(b);
  b += round256(pe / 2 * sizeof(float4));
  w.done = reinterpret_cast<unsigned*>(b);
  w.failed = w.done + 1;
  return w;
}

inline PersistPlan plan_of(const dk_ctx* ctx, int p) {
  const size_t mat_bytes = round256(size_t(p) * p * sizeof(float));
  return persist_plan(p, ctx->sm_count, 2 * mat_bytes, mat_bytes);
}

// the fit on a carved workspace (shared by the entry points); plan: plan_of's, or one of no CTAs for a
// launch per round
dk_status fit(dk_ctx* ctx, const float* x, int m, int p, int k, int sweeps, const Workspace& w,
              const PersistPlan& plan, float* mean, float* scale, float* comps, float* eig, float* off_norm,
              cudaStream_t st) {
  const size_t cov_bytes = size_t(p) * p * sizeof(float), mat_bytes = round256(cov_bytes);
  if (plan.ctas > 1) {
    // no word after the covariance (A's padding and V^T's part), which a former call may have used,
    // has a tag yet; cleared from a 256-byte boundary, before the covariance is written
    const size_t from = cov_bytes & ~size_t(255);
    if (cudaMemsetAsync(reinterpret_cast<uint8_t*>(w.A) + from, 0, 2 * mat_bytes - from, st) != cudaSuccess)
      return DK_ERR_CUDA;
  }
  col_stats_kernel<<<(p + 7) / 8, 64, 0, st>>>(x, m, p, mean, scale);
  const int nt = (p + T32 - 1) / T32;
  cov_kernel<<<nt * (nt + 1) / 2, 256, 0, st>>>(x, m, p, mean, scale, w.A);
  const int pe = p + (p & 1), np = pe / 2, rounds = sweeps * (pe - 1);
  if (cudaMemsetAsync(w.done, 0, 2 * sizeof(unsigned), st) != cudaSuccess) return DK_ERR_CUDA;  // and failed
  bool persistent = false;
  if (plan.ctas > 0) {
    uint8_t* box = reinterpret_cast<uint8_t*>(w.Vt) + mat_bytes - plan.box_bytes;
    using Kernel = void (*)(PersistArgs);
    const bool small = plan.threads <= 512;  // one CTA: always
    const Kernel odd = plan.ctas == 1 ? jacobi_persist_kernel<512, true, true>
                       : small        ? jacobi_persist_kernel<512, true, false>
                                      : jacobi_persist_kernel<1024, true, false>;
    const Kernel even = plan.ctas == 1 ? jacobi_persist_kernel<512, false, true>
                        : small        ? jacobi_persist_kernel<512, false, false>
                                       : jacobi_persist_kernel<1024, false, false>;
    const void* kern = reinterpret_cast<const void*>(p & 1 ? odd : even);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(plan.smem)) != cudaSuccess)
      return DK_ERR_CUDA;
    PersistArgs a{w.A,  w.Vt, reinterpret_cast<uint4*>(box), w.done, w.failed, ctx->status, p, plan.ppc,
                  plan.vc, rounds};
    void* args[] = {&a};
    persistent = cudaLaunchCooperativeKernel(kern, dim3(plan.ctas), dim3(plan.threads), args, plan.smem, st) ==
                 cudaSuccess;
    if (!persistent) cudaGetLastError();  // a device that cannot hold all CTAs at once
  }
  if (!persistent) {
    // beyond what shared memory holds: one launch per round
    const int fill_blocks = int(((long long)p * p + 255) / 256 < 4096 ? ((long long)p * p + 255) / 256 : 4096);
    eye_kernel<<<fill_blocks, 256, 0, st>>>(w.Vt, p);
    jacobi_params_kernel<<<(np + 255) / 256, 256, 0, st>>>(w.A, p, pe, 0, w.ij, w.cs);
    for (int q = 0; q < rounds; ++q) {
      const int r_next = q + 1 < rounds ? (q + 1) % (pe - 1) : -1;
      jacobi_rotate_kernel<<<np, 256, 0, st>>>(w.A, w.Vt, p, np, w.ij, w.cs, w.done, pe, r_next);
    }
  }
  if (off_norm) {
    // the rotation table is done with: it holds the partial sums, one 16-byte entry per CTA
    double2* part = reinterpret_cast<double2*>(w.cs);
    off_norm_kernel<<<np, 256, 0, st>>>(w.A, p, part);
    off_norm_finish_kernel<<<1, 32, 0, st>>>(part, np, w.failed, off_norm);
  }
  select_kernel<<<p, 256, 0, st>>>(w.A, w.Vt, p, k, w.failed, comps, eig);
  return launch_status();
}

}  // namespace pca
}  // namespace dk

using namespace dk;

DK_API size_t dk_pca_workspace_bytes(int p) { return p < 2 || p > DK_PCA_MAX_FEATURES ? 0 : pca::workspace_bytes(p); }

DK_API dk_status dk_pca_fit(dk_ctx* ctx, const float* x, int m, int p, int k, int sweeps, void* workspace,
                            size_t workspace_bytes, float* mean, float* scale, float* components,
                            float* eigenvalues, float* off_norm, void* stream) {
  if (!ctx || !x || !workspace || !mean || !scale || !components || !eigenvalues) return DK_ERR_ARG;
  if (m < 2 || p < 2 || k < 1 || k > p || sweeps < 1 || sweeps > 100) return DK_ERR_ARG;
  if (p > DK_PCA_MAX_FEATURES) return DK_ERR_UNSUPPORTED;
  if (workspace_bytes < pca::workspace_bytes(p) || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return DK_ERR_WORKSPACE;
  return pca::fit(ctx, x, m, p, k, sweeps, pca::carve(workspace, p), pca::plan_of(ctx, p), mean, scale, components,
                  eigenvalues, off_norm, static_cast<cudaStream_t>(stream));
}

DK_API dk_status dk_pca_transform(dk_ctx* ctx, const float* x, int m, int p, const float* mean, const float* scale,
                                  const float* components, int k, int fit_range, float range_max, float* lo,
                                  float* hi, float* out, void* stream) {
  if (!ctx || !x || !mean || !scale || !components || !lo || !hi || !out) return DK_ERR_ARG;
  if (m < 1 || p < 1 || k < 1 || k > p || !(range_max > 0.0f)) return DK_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  pca::transform_kernel<<<dim3((k + pca::T32 - 1) / pca::T32, (m + pca::T32 - 1) / pca::T32), 256, 0, st>>>(
      x, m, p, mean, scale, components, k, out);
  if (fit_range) pca::minmax_fit_kernel<<<(k + 31) / 32, 256, 0, st>>>(out, m, k, lo, hi);
  const long long n = (long long)m * k;
  const int blocks = int((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192);
  pca::minmax_apply_kernel<<<blocks, 256, 0, st>>>(out, n, k, lo, hi, range_max);
  return launch_status();
}

// ---------------------------------------------------------------------------------------
// dk_pca_fit_noalloc: the same fit with its working memory in a fixed device array.
//
// For callers that cannot hand this library device memory of their own: a host program
// whose device memory is owned and capped by another framework, a plug-in that receives
// only its input and output pointers, or a loop that must not stall on or fail in an
// allocation midway. The working memory for up to DK_PCA_NOALLOC_MAX_FEATURES features
// lives in the file-scope array below, which every GPU that loads the library holds until
// the process exits. Host code cannot pass the array's name to a kernel (on the host it
// names a stand-in, not device memory), so the first call on each device looks up the
// array's device address with that device current and keeps it for later calls.

namespace dk {
namespace pca {

constexpr size_t round256_c(size_t b) { return (b + 255) & ~size_t(255); }
constexpr size_t noalloc_bytes() {
  return 2 * round256_c(size_t(DK_PCA_NOALLOC_MAX_FEATURES) * DK_PCA_NOALLOC_MAX_FEATURES * sizeof(float)) +
         round256_c(DK_PCA_NOALLOC_MAX_FEATURES / 2 * sizeof(int2)) +
         round256_c(DK_PCA_NOALLOC_MAX_FEATURES / 2 * sizeof(float4)) + 256;
}

static __device__ __align__(256) unsigned char g_noalloc_scratch[noalloc_bytes()];

constexpr int MAX_DEVICES = 64;
static void* g_noalloc_ptr[MAX_DEVICES] = {};
static std::mutex g_noalloc_mu;

// device address of g_noalloc_scratch on `device`, looked up once with that device current
static dk_status noalloc_scratch(int device, void** out) {
  if (device < 0 || device >= MAX_DEVICES) return DK_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[device]) {
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) return DK_ERR_CUDA;
    if (cur != device && cudaSetDevice(device) != cudaSuccess) return DK_ERR_CUDA;
    void* ptr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (cur != device && cudaSetDevice(cur) != cudaSuccess) return DK_ERR_CUDA;
    if (e != cudaSuccess || !ptr) return DK_ERR_CUDA;
    g_noalloc_ptr[device] = ptr;
  }
  *out = g_noalloc_ptr[device];
  return DK_OK;
}

}  // namespace pca
}  // namespace dk

DK_API dk_status dk_pca_fit_noalloc(dk_ctx* ctx, const float* x, int m, int p, int k, int sweeps, float* mean,
                                    float* scale, float* components, float* eigenvalues, float* off_norm,
                                    void* stream) {
  if (!ctx || !x || !mean || !scale || !components || !eigenvalues) return DK_ERR_ARG;
  if (m < 2 || p < 2 || k < 1 || k > p || sweeps < 1 || sweeps > 100) return DK_ERR_ARG;
  if (p > DK_PCA_NOALLOC_MAX_FEATURES) return DK_ERR_UNSUPPORTED;
  void* scratch = nullptr;
  const dk_status s = pca::noalloc_scratch(ctx->device, &scratch);
  if (s != DK_OK) return s;
  // every part of the scratch that the fit reads is written earlier in the same call: the
  // covariance, the identity or the words of the one-launch form (whose place the fit clears), each
  // round's rotation table, the round counter, which the fit clears
  return pca::fit(ctx, x, m, p, k, sweeps, pca::carve(scratch, p), pca::plan_of(ctx, p), mean, scale, components,
                  eigenvalues, off_norm, static_cast<cudaStream_t>(stream));
}
