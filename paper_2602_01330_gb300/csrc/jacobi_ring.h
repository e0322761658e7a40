// The schedule of the one-launch Jacobi of pca.cu (jacobi_persist_kernel): which rows a CTA holds
// in which round, who publishes a word, and how the work is laid out. Plain functions, shared by
// the kernel and by host code that replays the schedule.
#pragma once

#include <stddef.h>

#ifdef __CUDACC__
#define DK_HD __host__ __device__ __forceinline__
#else
#define DK_HD inline
#endif

namespace dk {
namespace pca {

// Round-robin positions 0 .. ring are a ring with position 0 fixed; pair k holds the positions
// (k, ring - k). CTA g owns the pairs ks .. ke - 1, i.e. the rows at an upper run of positions
// ks .. ke - 1 and a lower run pe - ke .. pe - 1 - ks.
DK_HD int ring_index(int t, int r, int ring) {  // index at position t in round r, r < ring
  int x = t - 1 + r;
  if (x >= ring) x -= ring;
  return t == 0 ? 0 : 1 + x;
}
DK_HD int ring_came_from(int t, int ring) { return t == 0 ? 0 : (t == ring ? 1 : t + 1); }  // a round earlier
DK_HD int ring_goes_to(int t, int ring) { return t == 0 ? 0 : (t == 1 ? ring : t - 1); }
// position of local row u of a CTA with the pairs ks .. ke - 1
DK_HD int ring_row_position(int u, int ks, int ke, int pe) {
  const int cnt = ke - ks;
  return u < cnt ? ks + u : pe - ke + (u - cnt);
}

// Does the CTA that holds row x at position t publish a word for x's pair (x, y) of the next round?
// The row of the smaller index does: the pair's angle, or the identity when y is the padding index.
// With `lone`, the row that the last CTA moves from position np to np - 1 always does, the identity
// if it is the larger index.
//
// So every CTA publishes in every round, which is what makes two buffers of words enough (see
// jacobi_persist_kernel): both rows of some pair of the next round are the CTA's own. The upper
// run moves to the pairs ks - 1 .. ke - 2, the lower run to ks + 1 .. ke, so three or more pairs have
// ks + 1 in common; in the first CTA positions 0 and 1, in the last np and np + 1 meet (two pairs are
// enough). Only a last CTA of one pair has no such pair.
DK_HD bool ring_publishes(int x, int y, int t, int np, bool lone) { return y > x || (lone && t == np); }
DK_HD bool ring_lone(int np, int ppc) { return np > ppc && np % ppc == 1; }
// index whose word every CTA waits for, beside those of the pairs, where the last CTA is lone
DK_HD int ring_lone_index(int np, int r, int ring) { return ring_index(np - 1, r, ring); }

struct PersistPlan {
  int ctas, ppc, vc, threads;  // ppc: pairs per CTA; vc: columns of V^T per CTA; ctas = 0: no plan
  size_t smem, box_bytes;
};

constexpr int UR = 4;  // row pairs of a thread in flight

// Threads beside those of the rows: one for each of the CTA's 2 ppc rows and, with several CTAs,
// one that waits for the lone CTA's word.
DK_HD int ring_side_threads(int ppc, int np) { return (2 * ppc + (ppc < np ? 1 : 0) + 31) / 32 * 32; }

// Box memory (16-byte words): for several CTAs the rows in transit (2 buffers x CTAs x 2 rows x
// np column pairs), then the published angles (2 buffers x pe). It ends with V^T's part of the
// workspace, which is written only at the end, and reaches back into A's: the first row is
// sent in round 0 by a CTA that has everybody's angles, i.e. after every CTA has read its part
// of A. The fewest pairs per CTA that this and the SM count allow, but three at least (see
// ring_publishes): a CTA's work on its rows is what a round waits for.
inline PersistPlan persist_plan(int p, int sms, size_t box_cap, size_t angle_cap) {
  const int pe = p + (p & 1), np = pe / 2;
  const int lanes = (np + 31) / 32 * 32;  // one thread per column pair, groups of them over the rows
  constexpr size_t SMEM_CAP = 220 * 1024;
  auto make = [&](int ppc) {
    PersistPlan q;
    q.ppc = ppc;
    q.ctas = (np + ppc - 1) / ppc;
    q.vc = (p + q.ctas - 1) / q.ctas;
    // a thread per column pair, in groups over the row pairs when there are more than UR of
    // these, and warps of their own for the elements that the next round waits for
    const int side = ring_side_threads(ppc, np), room = (1024 - side) / lanes, want = (ppc + UR - 1) / UR;
    q.threads = lanes * (room < want ? room : want) + side;
    q.smem = size_t((q.vc + 3) / 4) * pe * 16 + size_t(2) * np * 16 + size_t(pe) * 16 + size_t(4) * ppc * pe * 4 +
             size_t(pe) * 4;
    q.box_bytes = size_t(32) * pe + (q.ctas > 1 ? size_t(32) * q.ctas * pe : 0);
    return q;
  };
  if (np <= 960 && size_t(32) * pe <= angle_cap) {
    const PersistPlan one = make(np);
    if (np < 32 && one.smem <= SMEM_CAP) return one;
    for (int ppc = 3; ppc < np; ++ppc) {
      const PersistPlan q = make(ppc);
      if (q.ctas > 1 && q.ctas <= sms && q.smem <= SMEM_CAP && q.box_bytes <= box_cap) return q;
    }
  }
  return PersistPlan{0, 0, 0, 0, 0, 0};
}

}  // namespace pca
}  // namespace dk
