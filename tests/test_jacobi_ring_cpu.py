"""The schedule of the one-launch Jacobi (csrc/jacobi_ring.h, shared with the kernel), replayed on
the host for every feature count that has a plan.

Two buffers of words are enough because every CTA publishes, in every round, at least one word
that every CTA waits for: whoever has all words of a round then knows that every CTA has read
those of the round before. So for each round: every CTA publishes, each index's word has one
writer, and the words that are waited for are among those that are published. Where the words lie
in the workspace: within V^T's part and the end of A's."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_01330_gb300", "csrc")

REPLAY = r"""
#include <stdio.h>
#include <stdlib.h>
#include <algorithm>
#include <vector>
#include "jacobi_ring.h"
using namespace dk::pca;
int main(int argc, char** argv) {
  const int sms = atoi(argv[1]), step = atoi(argv[2]);
  int plans = 0, lones = 0, last = 0, bad = 0;
  for (int p = 2; p <= 4096; p += step) {
    const size_t mat = (size_t(p) * p * 4 + 255) / 256 * 256;
    const PersistPlan plan = persist_plan(p, sms, 2 * mat, mat);
    if (plan.ctas == 0) continue;
    ++plans;
    last = p;
    const int pe = p + (p & 1), np = pe / 2, ring = pe - 1, G = plan.ctas;
    const bool lone = ring_lone(np, plan.ppc);
    lones += lone;
    if (plan.threads > 1024 || plan.box_bytes > 2 * mat || size_t(32) * pe > mat) bad |= 1;
    if ((G - 1) * plan.ppc >= np || G * plan.ppc < np || G > sms) bad |= 2;
    if (G == 1 && plan.threads > 512) bad |= 256;
    if (G == 1) continue;  // its words are in its own shared memory, behind barriers
    std::vector<int> writers(pe);
    for (int r = 0; r < ring && !(bad & 4); ++r) {  // published in round r for the next one
      const int rn = r + 1 == ring ? 0 : r + 1;
      std::fill(writers.begin(), writers.end(), 0);
      for (int g = 0; g < G; ++g) {
        const int ks = g * plan.ppc, ke = std::min(ks + plan.ppc, np);
        int awaited = 0;
        for (int u = 0; u < 2 * (ke - ks); ++u) {
          const int t = ring_row_position(u, ks, ke, pe), x = ring_index(t, r, ring);
          const int tn = ring_goes_to(t, ring), y = ring_index(ring - tn, rn, ring);
          if (ring_index(tn, rn, ring) != x || ring_index(ring_came_from(ring - tn, ring), r, ring) != y) bad |= 8;
          if (!ring_publishes(x, y, t, np, lone)) continue;
          ++writers[x];
          awaited += x < y || (lone && x == ring_lone_index(np, rn, ring));
        }
        if (awaited == 0) {  // nobody would know how far this CTA has come
          printf("p %d: CTA %d silent in round %d\n", p, g, r);
          bad |= 4;
          break;
        }
      }
      for (int k = 0; k < np; ++k)
        if (writers[std::min(ring_index(k, rn, ring), ring_index(ring - k, rn, ring))] != 1) bad |= 16;
      if (lone && writers[ring_lone_index(np, rn, ring)] != 1) bad |= 32;
      for (int x = 0; x < pe; ++x)
        if (writers[x] > 1) bad |= 64;
    }
    // the first round's words: by the rows of the upper runs, index = position
    if (lone && np - 1 != ring_lone_index(np, 0, ring)) bad |= 128;
  }
  printf("%d %d %d %d\n", bad, plans, lones, last);
  return 0;
}
"""


@pytest.mark.parametrize("sms,step", [(152, 1), (148, 7), (76, 7), (16, 11)])
def test_every_cta_publishes_in_every_round(tmp_path, sms, step):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "replay.cpp", str(tmp_path / "replay")
    src.write_text(REPLAY)
    subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe, str(sms), str(step)], check=True, capture_output=True, text=True).stdout
    bad, plans, lones, last = (int(v) for v in out.splitlines()[-1].split())
    assert bad == 0, out
    assert plans > 0 and lones > 0 and last >= 64  # several CTAs, a last one of one pair among them
    if sms == 152:
        assert last == 1372  # beyond, shared memory holds no plan: one launch per round
