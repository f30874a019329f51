"""The order in which the 4-bit conversion warps of the weights-as-rows kernel
wait for slots and stages (ColsConvert in csrc/internal.cuh), compiled for the
host from the same header and run against a model of the kernel's barriers.

Each of the sixteen warps executes the steps that ColsConvert gives it, beside
the weight producer and the MMA issuer; loads land in any order, MMAs complete
in order, and the next actor to move is drawn at random, with some actors and
some loads held back.  A barrier is its phase and its missing arrivals, and a
wait sees the phase's parity only, as on the device.  Checked: a slot that a
warp has waited for holds its load, and still does when the warp lets it go; a
stage waited for has been consumed; no barrier takes an arrival too many; every
MMA finds its halves converted; nothing waits forever."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_23805_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "internal.cuh"

struct Tile { bool codes; uint32_t kb; };
enum Kind { kSlot, kStage, kCodes, kRows, kNone, kPass };
struct Step { Kind k; uint32_t v, arg; };
struct Recorder {
  std::vector<Step> s;
  bool slot(uint32_t w) { s.push_back({kSlot, w, 0}); return true; }
  bool stage(uint32_t st) { s.push_back({kStage, st, 0}); return true; }
  void codes(uint32_t w, bool any) { s.push_back({kCodes, w, any}); }
  void rows(uint32_t w, uint32_t j) { s.push_back({kRows, w, j}); }
  void none() { s.push_back({kNone, 0, 0}); }
  void pass(uint32_t w) { s.push_back({kPass, w, 0}); }
};

struct Barrier {
  int expect = 1, pending = 1;
  long phase = 0;
  explicit Barrier(int n = 1) : expect(n), pending(n) {}
  bool arrive(int n) {
    pending -= n;
    if (pending < 0) return false;
    if (pending == 0) { pending = expect; ++phase; }
    return true;
  }
  bool passed(uint32_t parity) const { return (phase & 1) != (long)parity; }
};

struct Rng {
  uint64_t s;
  uint32_t operator()(uint32_t n) {
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    return (uint32_t)((s >> 33) % n);
  }
};

// 0, or what went wrong
static int run(const std::vector<Tile>& tiles, uint32_t ring_s, uint32_t ring_w, uint64_t seed) {
  Rng rnd{seed * 2654435761u + 12345};
  std::vector<Step> prog[16];
  for (int w = 0; w < 16; ++w) {
    msi::ColsConvert c(w >> 2);
    Recorder r;
    for (const Tile& t : tiles) c.tile(t.codes, t.kb, r);
    prog[w] = r.s;
  }
  uint32_t n_slots = 0, n_st = 0;
  for (const Tile& t : tiles) {
    n_slots += t.codes ? (t.kb + 3) / 4 : t.kb;
    n_st += (t.kb + 3) / 4;
  }
  std::vector<Barrier> wfull(ring_w), wempty(ring_w, Barrier(16)), sempty(ring_s), afull(4, Barrier(4));
  std::vector<long> content(ring_w, -1);
  std::vector<char> landed(n_slots, 0), consumed(n_st, 0);
  std::vector<uint32_t> flying;                    // armed slots whose load has not landed
  std::vector<int> converted(4, 0);                // half stages each set's warps have finished, by set
  uint32_t pw = 0, issued = 0, done = 0, half = 0; // producer; MMA: stages issued and completed
  size_t pc[16] = {};
  const auto log2 = [](uint32_t n) { uint32_t l = 0; while ((1u << l) < n) ++l; return l; };
  const uint32_t wl = log2(ring_w), sl = log2(ring_s);
  // actors: 16 warps, producer, MMA issue, MMA completion, landing; some slow
  int slow[20];
  for (int& v : slow) v = rnd(4) == 0 ? 1 + (int)rnd(60) : 0;
  const uint32_t slow_slot = rnd(3) ? rnd(n_slots) : n_slots;
  int idle = 0;
  while (true) {
    bool all = pw == n_slots && done == n_st && flying.empty();
    for (int w = 0; w < 16 && all; ++w) all = pc[w] == prog[w].size();
    if (all) return 0;
    if (++idle > 20000) return 1;                  // nothing moves
    const bool held = idle < 10000;                // the slow ones are held back
    const uint32_t a = rnd(20);
    if (held && slow[a] && rnd(slow[a] + 1) != 0) continue;
    if (a < 16) {
      if (pc[a] == prog[a].size()) continue;
      const Step& s = prog[a][pc[a]];
      const int set = a >> 2;
      const uint32_t wi = s.v & (ring_w - 1);
      if (s.k == kSlot) {
        if (!wfull[wi].passed((s.v >> wl) & 1u)) continue;
        if (content[wi] != (long)s.v || !landed[s.v]) return 2;
      } else if (s.k == kStage) {
        if (s.v >= 2) {
          const uint32_t p = s.v - 2;
          if (!sempty[p & (ring_s - 1)].passed((p >> sl) & 1u)) continue;
          if (!consumed[p]) return 3;
        }
      } else if (s.k == kNone) {
        if (!afull[set].arrive(1)) return 4;
      } else {
        if (content[wi] != (long)s.v || !landed[s.v]) return 5;
        if (s.k == kCodes && !wempty[wi].arrive(2)) return 6;
        if (s.k == kPass && !wempty[wi].arrive(1)) return 6;
        if ((s.k == kCodes || (s.k == kRows && s.arg)) && !afull[set].arrive(1)) return 4;
      }
      ++pc[a];
    } else if (a == 16) {
      if (pw == n_slots || !wempty[pw & (ring_w - 1)].passed(((pw >> wl) & 1u) ^ 1u)) continue;
      content[pw & (ring_w - 1)] = pw;
      flying.push_back(pw++);
    } else if (a == 17) {
      if (issued == n_st) continue;
      const uint32_t h = 2 * issued + half;        // half stage: set h & 3, its (h >> 2)-th
      if (!afull[h & 3].passed((h >> 2) & 1u)) continue;
      if (afull[h & 3].phase != (long)(h >> 2) + 1) return 7;
      half ^= 1;
      if (half == 0) ++issued;
    } else if (a == 18) {
      if (done == issued) continue;
      consumed[done] = 1;
      if (!sempty[done & (ring_s - 1)].arrive(1)) return 8;
      ++done;
    } else {
      if (flying.empty()) continue;
      const size_t i = rnd((uint32_t)flying.size());
      const uint32_t w = flying[i];
      if (held && w == slow_slot && rnd(400) != 0) continue;
      flying.erase(flying.begin() + i);
      landed[w] = 1;
      if (!wfull[w & (ring_w - 1)].arrive(1)) return 9;
    }
    idle = 0;
  }
}

int main() {
  // K blocks of up and down tiles: (H / 64, I / 64)
  const uint32_t shapes[][2] = {{4, 2}, {4, 10}, {12, 2}, {20, 10}, {32, 8}, {8, 4}};
  int bad = 0;
  for (const auto& s : shapes) {
    const uint32_t u = s[0], d = s[1];
    // a CTA's sequences: shared up tiles, codes, shared down tiles, codes
    const std::vector<Tile> seqs[] = {
        {{true, u}, {true, u}, {false, d}, {true, d}, {true, d}},
        {{false, u}, {true, u}, {false, d}, {true, d}, {false, d}, {true, d}},
        {{true, u}, {false, d}, {false, d}, {true, d}, {true, d}, {true, d}},
        {{false, u}, {false, u}, {true, u}, {true, u}, {true, u}, {false, d}, {true, d}, {true, d}},
        {{true, u}, {true, d}, {false, d}, {true, d}, {false, d}, {true, d}, {true, d}}};
    for (const auto& q : seqs)
      for (uint32_t rs : {2u, 4u})
        for (uint32_t rw : {4u, 8u})
          for (uint64_t seed = 0; seed < 60; ++seed) {
            const int r = run(q, rs, rw, seed);
            if (r != 0) {
              if (bad < 10) printf("FAIL kb %u %u sequence of %zu rings %u %u seed %d: code %d\n", u, d, q.size(), rs, rw, (int)seed, r);
              ++bad;
            }
          }
  }
  printf("%d %s\n", bad, bad == 0 ? "ok" : "failures");
  return bad == 0 ? 0 : 1;
}
'''


def test_conversion_waits_name_one_phase(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "convert.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "convert"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout
