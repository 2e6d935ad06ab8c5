"""Which units of a matrix every warp of the cluster kernel multiplies (cluster_plan in csrc/cluster_pass.cuh), against the shares of the
whole-pass kernel's CTAs (stage_shares in csrc/pass_kernel.cuh): host code, built with nvcc and run on the CPU."""
import os
import subprocess

import pytest

from paper_2602_05499_b200 import build

CHECK = r"""
#include "%s/cluster_pass.cuh"
#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>
using namespace sdfp;
#define REQUIRE(x) do { if (!(x)) { printf("line %%d: %%s (kind %%d rank %%d)\n", __LINE__, #x, kind, rank); return 1; } } while (0)
int main(int argc, char** argv) {
  const int d = atoi(argv[1]), f = atoi(argv[2]), vocab = atoi(argv[3]), slots = atoi(argv[4]), rows = atoi(argv[5]), grid = 148;
  int kind = -1, rank = -1;
  if (argc > 6) {  // does a layout exist, shared memory left aside?
    const ClPlan p = cluster_plan(d, f, vocab, atoi(argv[6]), grid, slots);
    return cluster_layout(d, f, d / 64, 64, 2, rows, 96, atoi(argv[6]), slots, p, 1 << 29).total > 0 ? 2 : 3;
  }
  const ClPlan whole = cluster_plan(d, f, vocab, 2, grid, 1 << 14);
  const int places = std::max(slots, whole.most_cuts);
  const ClPlan plan = cluster_plan(d, f, vocab, 2, grid, places);
  for (kind = 0; kind < CL_KINDS; ++kind) {
    const int n_pairs = cl_pairs_of(kind, d, f, vocab), KT = (kind == CL_DOWN ? f : d) / 16, NT = n_pairs / 8, groups = (NT + 7) / 8;
    std::vector<StageShare> shares(grid);
    stage_shares(shares.data(), groups, KT, grid);
    std::map<std::pair<int, int>, std::pair<int, int>> unit;  // (group, k-tile) -> (piece, class), as the CTAs of the whole-pass kernel take them
    std::vector<int> pieces(groups, 0);
    for (const StageShare& s : shares)
      for (int u = 0; u < s.n; ++u) {
        const int g = (s.ub + u) / KT, kt = (s.ub + u) %% KT;
        if (u == 0 || kt == 0) pieces[g]++;
        unit[{g, kt}] = {pieces[g] - 1, u %% kClasses};
      }
    int covered = 0;
    for (rank = 0; rank < kClCtas; ++rank) {
      const unsigned char* at = plan.bytes.data() + (size_t)rank * plan.stride;
      const ClMine& m = reinterpret_cast<const ClMine*>(at)[kind];
      const ClRound* rounds = reinterpret_cast<const ClRound*>(at + plan.rounds_at) + m.round0;
      const ClEntry* entries = reinterpret_cast<const ClEntry*>(at + plan.entries_at) + m.entry0;
      REQUIRE(m.p0 == covered && m.p0 == cl_first_pair(n_pairs, rank, 2));
      covered += m.np;
      int quads = 0, used[kClasses] = {};
      for (int r = 0; r < m.n_rounds; ++r) {
        const ClRound& rd = rounds[r];
        REQUIRE(rd.quad0 == quads);
        quads += rd.n_quads;
        for (int i = 0; i < rows * rd.n_quads; ++i) REQUIRE((int)((unsigned)i * rd.magic >> 20) == i / rd.n_quads);
        const int end = (m.p0 + 4 * quads - 1) / 8 + 1;
        REQUIRE((m.p0 + 4 * rd.quad0) / 8 == rd.tile0 && (end - rd.tile0) * rd.np <= places);
        std::set<std::pair<int, int>> done;  // (place, class)
        for (int cls = 0; cls < kClasses; ++cls) {
          std::vector<int> kts;
          for (bool last = false; !last;) {
            REQUIRE(used[cls] < m.n_entries);
            const ClEntry& e = entries[cls * m.n_entries + used[cls]++];
            last = e.last != 0;
            REQUIRE(e.n_tiles >= 1 && e.n_tiles <= m.tile_width && e.np == rd.np && (!last || (e.last == 2) == (r + 1 == m.n_rounds)));
            if (e.kt >= 0) {
              kts.push_back(e.kt);
              for (int t = 0; t < e.n_tiles; ++t) {  // the weights read are the tile's, and its unit is this class's
                const int w = e.w + t * 32 + (t >= e.wrap ? (KT - 1) * 256 : 0), first = e.w / 256 / KT * 8 + e.w %% 256 / 32, tile = w / 256 / KT * 8 + w %% 256 / 32;
                REQUIRE(w / 256 %% KT == e.kt && tile == first + t && tile < NT && (unit[{tile / 8, e.kt}].second == cls));
              }
            }
            if (e.slot >= 0) {
              const int tile = rd.tile0 + e.slot / e.np, piece = e.slot %% e.np;
              std::vector<int> want;
              for (int kt = 0; kt < KT; ++kt)
                if (unit[{tile / 8, kt}] == std::make_pair(piece, cls)) want.push_back(kt);
              REQUIRE(want == kts);  // in order, nothing left out
              for (int t = 0; t < e.n_tiles; ++t) REQUIRE(e.slot + t * e.np < places && done.insert({e.slot + t * e.np, cls}).second);
              kts.clear();
            }
          }
          REQUIRE(kts.empty());
        }
        REQUIRE((int)done.size() == (end - rd.tile0) * rd.np * kClasses);
        for (int t = rd.tile0; t < end; ++t) REQUIRE(pieces[t / 8] == rd.np);
      }
      REQUIRE(4 * quads == m.np);
    }
    REQUIRE(covered == n_pairs);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "check.cu", d / "check"
    src.write_text(CHECK % build.CSRC)
    cmd = [os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-o", str(exe), str(src)]
    done = subprocess.run(cmd, capture_output=True, text=True)
    assert done.returncode == 0, done.stdout + done.stderr
    return str(exe)


@pytest.mark.parametrize("d,f,vocab,slots,rows", [
    (128, 64, 16, 8, 16),        # half a tile per CTA, CTAs and classes without a unit
    (256, 688, 2048, 8, 5),      # three pieces, groups that end inside a CTA's share
    (512, 1376, 32000, 11, 9),   # the lm-head cut evenly: pieces that begin at any class, many rounds
    (512, 1376, 4096, 3, 2),     # less room than a stage's sums: rounds in the layers too
    (768, 2064, 4096, 51, 2),
    (1088, 80, 272, 1, 16),      # ... a tile at a time
    (640, 8192, 1008, 24, 1),    # long contractions, many pieces
])
def test_plan_is_the_whole_pass_kernels(checker, d, f, vocab, slots, rows):
    done = subprocess.run([checker] + [str(x) for x in (d, f, vocab, slots, rows)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


@pytest.mark.parametrize("d,f,vocab,slots,rows,bytes_per,held", [
    (256, 688, 2048, 8, 5, 2, True), (256, 688, 2048, 8, 5, 4, True),
    (2048, 4096, 2048, 64, 2, 2, True),
    (2112, 4096, 2048, 64, 2, 2, False),       # more columns than the first norm's sum is made of
    (256, 16384, 2048, 64, 16, 2, False),      # 1 MB of u: a stage's bytes do not fit the transaction count
    (256, 16320, 2048, 64, 15, 2, True),
    (128, 64, 65536, 8, 16, 4, True),          # (the lm-head's pairs are not divided by multiplication)
    (256, 688, 2048, 32768, 5, 2, False),      # a place's number does not fit
])
def test_layout_refuses_what_its_fields_do_not_hold(checker, d, f, vocab, slots, rows, bytes_per, held):
    done = subprocess.run([checker] + [str(x) for x in (d, f, vocab, slots, rows, bytes_per)], capture_output=True, text=True)
    assert done.returncode == (2 if held else 3)
