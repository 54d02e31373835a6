"""The symmetric forms' work split (csrc/cn_sym.h), compiled for the host and
enumerated: for one system and for an ensemble's table of rows, over tiles, sizes, CTA counts, stage sizes and bands, every unit
(row of tiles, block) on or above the diagonal belongs to exactly one CTA,
every CTA has one, no two segments share a slot, and the merge's view of
which CTAs hold a row agrees."""

import os
import shutil
import subprocess

import pytest

from conftest import ROOT

SOURCE = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "cn_sym.h"
using namespace cn;
#define CHECK(x) if (!(x)) { std::printf("%s: n %lld tile %lld cta %d\n", #x, (long long)n, (long long)tile, c); return 1; }
int main() {
  long launches = 0;
  for (int64_t tile : {64, 256, 512, 2048})
  for (int64_t n : {1LL, 31LL, 32LL, 33LL, 64LL, 65LL, 1000LL, 2047LL, 2048LL, 2049LL, 5000LL, 9999LL, 20000LL})
  for (int slots : {1, 2, 7, 304, 1216})
  for (int most : {1, 4, 8})
  for (int band : {0, 1, 3}) {
    SymGrid g{};
    g.n = n; g.n_tiles = (n + tile - 1) / tile; g.n_blocks = (n + 31) / 32; g.tile_blocks = tile / 32;
    const int w = band ? std::min<int>(band, g.n_tiles) : g.n_tiles;
    for (int r0 = 0; r0 < g.n_tiles; r0 += w) {
      int c = 0;
      g.row0 = r0; g.row1 = std::min(g.n_tiles, r0 + w);
      g.cost0 = g.row_start(r0); g.cost = g.row_start(g.row1) - g.cost0;
      g.grid = std::max<int64_t>(1, std::min<int64_t>(slots, g.cost / kSymCostPair));
      std::vector<std::vector<int>> own(g.row1 - r0, std::vector<int>(g.n_blocks, -1));
      std::vector<char> seg(g.grid + w, 0);
      for (c = 0; c < g.grid; ++c) {
        SymCursor cur;
        cur.seek(g, g.part(c));
        int units = 0, last = -1;
        while (cur.s < g.part(c + 1)) {
          const int64_t s0 = cur.s;
          int32_t I, b, nb;
          bool diag;
          cur.take(g, g.part(c + 1), most, &I, &b, &nb, &diag);
          CHECK(I >= r0 && I < g.row1 && nb >= 1 && nb <= most && b >= I * g.tile_blocks && b + nb <= g.n_blocks)
          for (int k = 0; k < nb; ++k, ++units) {
            CHECK(own[I - r0][b + k] == -1)
            own[I - r0][b + k] = c;
            CHECK(g.owner(s0 + (int64_t)k * (diag ? kSymCostDiag : kSymCostPair)) == c)
            CHECK((b + k < g.diag_end(I)) == diag)
          }
          if (I != last) {
            CHECK(c + I - r0 < (int)seg.size() && !seg[c + I - r0])
            seg[c + I - r0] = 1;
            last = I;
          }
        }
        CHECK(units > 0)
      }
      for (int I = r0; I < g.row1; ++I) {
        for (int b = 0; b < g.n_blocks; ++b) CHECK((own[I - r0][b] != -1) == (b >= I * g.tile_blocks))
        const int64_t s1 = g.row_start(I + 1) - (g.diag_end(I) < g.n_blocks ? kSymCostPair : kSymCostDiag);
        CHECK(g.owner(g.row_start(I)) == own[I - r0][I * g.tile_blocks] && g.owner(s1) == own[I - r0][g.n_blocks - 1])
        for (int64_t o = g.owner(g.row_start(I)); o <= g.owner(s1); ++o)
          CHECK(std::find(own[I - r0].begin(), own[I - r0].end(), (int)o) != own[I - r0].end())
      }
      ++launches;
    }
  }
  // ensembles: the rows of several clusters on one cost line
  for (int64_t tile : {64, 512, 2048})
  for (int set = 0; set < 4; ++set)
  for (int slots : {1, 5, 152, 1216})
  for (int most : {1, 2, 8}) {
    const std::vector<std::vector<int>> sizes = {{1}, {700, 1, 33, 64, 2048, 31}, {5000, 512, 511, 513}, {32, 32, 32, 32}};
    std::vector<SymRow> rows;
    int64_t cost = 0, n = 0;
    int c = 0;
    for (int m : sizes[set]) {
      const int nb = (m + 31) / 32, tb = tile / 32;
      for (int b = 0; b < nb; b += tb) {
        SymRow r{};
        r.cost = cost; r.p0 = n; r.n = m; r.n_blocks = nb; r.blk0 = b; r.diag_end = std::min(nb, b + tb);
        cost += r.length();
        rows.push_back(r);
      }
      n += m;
    }
    SymGrid g{};
    g.n = n; g.cost = cost; g.grid = std::max<int64_t>(1, std::min<int64_t>(slots, cost / kSymCostPair));
    std::vector<std::vector<int>> own;
    for (const SymRow& r : rows) own.push_back(std::vector<int>(r.n_blocks, -1));
    std::vector<char> seg(g.grid + rows.size(), 0);
    for (c = 0; c < g.grid; ++c) {
      SymCursor cur;
      sym_seek_rows(cur, rows.data(), rows.size(), g.part(c));
      int units = 0, last = -1;
      while (cur.s < g.part(c + 1)) {
        const int64_t s0 = cur.s;
        int32_t I, b, nb;
        bool diag;
        sym_take_rows(cur, rows.data(), rows.size(), g.part(c + 1), most, &I, &b, &nb, &diag);
        CHECK(I >= 0 && I < (int)rows.size() && nb >= 1 && nb <= most && b >= rows[I].blk0 && b + nb <= rows[I].n_blocks)
        for (int k = 0; k < nb; ++k, ++units) {
          CHECK(own[I][b + k] == -1 && (b + k < rows[I].diag_end) == diag)
          own[I][b + k] = c;
          CHECK(g.owner(s0 + (int64_t)k * (diag ? kSymCostDiag : kSymCostPair)) == c)
        }
        if (I != last) {
          CHECK(c + I < (int)seg.size() && !seg[c + I])
          seg[c + I] = 1;
          last = I;
        }
      }
      CHECK(units > 0)
    }
    for (size_t I = 0; I < rows.size(); ++I) {
      for (int b = 0; b < rows[I].n_blocks; ++b) CHECK((own[I][b] != -1) == (b >= rows[I].blk0))
      CHECK(g.owner(rows[I].cost) == own[I][rows[I].blk0] && g.owner(rows[I].last()) == own[I].back())
      for (int64_t o = g.owner(rows[I].cost); o <= g.owner(rows[I].last()); ++o)
        CHECK(std::find(own[I].begin(), own[I].end(), (int)o) != own[I].end())
    }
    ++launches;
  }
  std::printf("ok %ld\n", launches);
  return 0;
}
"""


def test_every_unit_has_one_owner(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "schedule.cpp", tmp_path / "schedule"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_astro_ph_0703100_gb300", "csrc"), "-I", os.path.join(cuda, "include"),
                    str(src), "-o", str(exe), "-L", os.path.join(cuda, "lib64"), "-lcudart_static", "-lpthread", "-ldl", "-lrt"],
                   check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.startswith("ok"), res.stdout
