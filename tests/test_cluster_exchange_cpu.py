"""Host-side check of the tile exchange inside a thread-block cluster (k_resident_cluster): a model of
its CTAs, with the sets of shared-memory tiles numbered by the library's own cluster_set (internal
header, compiled for the host with nvcc; no GPU).

A push reads its source and writes its destination at any time between its issue and its completion,
which only the destination sees.  The model runs the CTAs under random schedules, copies late and
piecewise, and checks that a CTA only ever uses the tiles of its own evaluation.  With one own tile
(written in place) the same model must find a mix of two evaluations."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "aqc_internal.h"
using namespace aqc;

constexpr int W = 3;  // words of a tile: copies and stores move one at a time
struct Tile { int v[W]; };
struct Copy { int src, dst, slot, e, at; };  // the own tile of `src` for evaluation e, words [0, at) done

static uint64_t st;
static unsigned rnd() { st = st * 6364136223846793005ull + 1442695040888963407ull; return (unsigned)(st >> 33); }

// own: number of own tiles (2: cluster_set, 1: in place)
static bool run(int ctas, int evals, int own, uint64_t seed) {
  st = seed;
  struct Cta {
    std::vector<Tile> tile[2];  // per set: the own one, then the partners'
    int e = 0, phase = 0, word = 0;
    std::vector<int> got;  // partners' tiles complete, by evaluation
  };
  std::vector<Cta> c(ctas);
  std::vector<Copy> fly;
  auto own_set = [&](int e) { return own == 2 ? cluster_set(e) : 0; };
  for (Cta& a : c) {
    for (auto& s : a.tile) s.assign(ctas, Tile{{-1, -1, -1}});
    a.got.assign(evals, 0);
    for (int i = 0; i < ctas; i++) a.tile[cluster_set(0)][i] = Tile{{0, 0, 0}};
    a.got[0] = ctas - 1;  // the first evaluation's tiles come from memory
  }
  for (long step = 0; step < 4000000; step++) {
    bool left = false;
    for (Cta& a : c) left = left || a.e < evals;
    if (!left) return true;
    const unsigned pick = rnd() % (unsigned)(ctas + 1);
    if (pick == (unsigned)ctas || rnd() % 8 == 0) {  // one word of a copy in flight
      if (fly.empty()) continue;
      const unsigned i = rnd() % (unsigned)fly.size();
      Copy& f = fly[i];
      c[f.dst].tile[cluster_set(f.e)][f.slot].v[f.at] = c[f.src].tile[own_set(f.e)][0].v[f.at];
      if (++f.at == W) {
        c[f.dst].got[f.e]++;
        fly.erase(fly.begin() + i);
      }
      continue;
    }
    Cta& a = c[pick];
    if (a.e >= evals) continue;
    switch (a.phase) {
      case 0:  // push, from the second evaluation on
        if (a.e > 0)
          for (int p = 1; p < ctas; p++) fly.push_back(Copy{(int)pick, (int)pick ^ p, p, a.e, 0});
        a.phase = 1;
        break;
      case 1:  // wait for the partners, then use every tile word by word (other CTAs and copies go on)
        if (a.got[a.e] < ctas - 1) break;
        a.phase = 2;
        a.word = 0;
        break;
      case 2: {
        const int t = a.word / W, w = a.word % W;
        if (a.tile[t ? cluster_set(a.e) : own_set(a.e)][t].v[w] != a.e) return false;
        if (++a.word == ctas * W) {
          a.phase = 3;
          a.word = 0;
        }
        break;
      }
      default:  // the own tile of the next evaluation
        a.tile[own_set(a.e + 1)][0].v[a.word] = a.e + 1;
        if (++a.word == W) {
          a.e++;
          a.phase = 0;
        }
    }
  }
  return false;  // a deadlock
}

int main() {
  int mixed = 0;
  for (int ctas = 2; ctas <= kResMaxCluster; ctas *= 2)
    for (uint64_t seed = 1; seed <= 40; seed++) {
      if (!run(ctas, 9, 2, seed)) { printf("a tile of another evaluation: %d CTAs, seed %d\n", ctas, (int)seed); return 1; }
      mixed += !run(ctas, 9, 1, seed);
    }
  if (!mixed) { printf("the model does not see an own tile overwritten under a copy\n"); return 1; }
  printf("ok\n");
  return 0;
}
"""


def test_pushed_tiles_are_not_overwritten_before_they_are_read(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "exchange.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "exchange"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_1311_3938_gb300", "csrc"), "-o", str(exe),
                    str(src)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
