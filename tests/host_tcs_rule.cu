// Host driver of tcs_wins (csrc/contract_tcs.cu): random tile lists against the rule
// restated tile by tile, and its time on a list of many tiles per column window.
// Prints the number of lists, of disagreements and of lists where the rule holds, then
// the ratio of its time to the restatement's.
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <random>
#include <vector>

#include "contract_tcs.cu"

using namespace bsi;

namespace {

// Column entries: runs of one ring triple, w3 channels padded to a multiple of 8.
int add_list(std::vector<ColEntry> &cols, int runs, int w3, int nu0, bool swap_first) {
  const int off = (int)cols.size();
  for (int r = 0; r < runs; ++r)
    for (int q = 0; q < (w3 + 7) / 8 * 8; ++q)
      cols.push_back(ColEntry{q < w3 ? 7 * r + nu0 + q : -1, r, nu0 + q, swap_first && r == 0});
  return off;
}

bool rule(const std::vector<TcTile> &tiles, const std::vector<TcGroup> &groups,
          const std::vector<ColEntry> &cols, bool fixed_order) {
  double cs = 0, cl = 0;
  for (const TcTile &t : tiles) {
    const TcGroup &G = groups[t.group];
    if (!G.dsum || G.out_full) return false;
    const int pa = std::min(32, G.nu1_hi - t.nu1_0), pb = std::min(16, G.nu2_hi - t.nu2_0);
    if (fixed_order && pa > 16) return false;
    const int npa = pa > 16 ? 32 : 16, dmax = t.diag ? t.nu2_0 - t.nu1_0 : 32;
    const int nst = std::max(0, std::min(G.Kpad - t.kseg * G.kseg_len, G.kseg_len)) / 32;
    const int halves = (0 < pa && -(pb - 1) <= dmax) + (16 < pa && 16 - (pb - 1) <= dmax);
    cl += 2.0 * (1700.0 * nst + 12000.0);
    for (int c0 = t.col0; c0 < std::min(t.ncol, t.col0 + 256); c0 += 128) {
      const int n = std::min(128, t.ncol - c0);
      long long red = 0;
      for (int g = 0; g < n;) {  // a segment: one ring triple
        const ColEntry f = cols[t.col_off + c0 + g];
        int e = g, last = g;
        for (; e < n; ++e) {
          const ColEntry c = cols[t.col_off + c0 + e];
          if (c.field < 0) continue;
          if (c.trip != f.trip || c.swapped != f.swapped) break;
          last = e;
        }
        if (fixed_order && g / 32 != last / 32) return false;
        red += (long long)(npa + 15) * (16 + cols[t.col_off + c0 + last].nu3 - f.nu3);
        g = e;
      }
      if (red > 12544) return false;
      const int w = (n + 15) / 16 * 16;
      cs += halves * (nst * std::max(8.5 * w, G.kexp ? 1050.0 : 800.0) + 2500.0 + 60.0 * w) + 4000.0;
    }
  }
  return !tiles.empty() && cs < cl;
}

}  // namespace

int main() {
  std::mt19937 rng(1);
  auto pick = [&](int lo, int hi) { return lo + (int)(rng() % (unsigned)(hi - lo + 1)); };
  double dummy = 0;
  int kexp = 0, bad = 0, wins = 0;
  const int lists = 4000;
  for (int it = 0; it < lists; ++it) {
    std::vector<TcGroup> groups(pick(1, 3));
    const int nc = pick(1, 140);
    for (TcGroup &G : groups) {
      G = TcGroup{};
      G.nu1_hi = G.nu2_hi = nc;
      G.Kpad = 32 * pick(1, 300);
      G.kseg_len = 32 * pick(1, 300);
      G.dsum = &dummy;
      G.out_full = pick(0, 60) ? nullptr : &dummy;
      G.kexp = pick(0, 1) ? &kexp : nullptr;
    }
    std::vector<ColEntry> cols;
    std::vector<TcTile> tiles;
    for (int l = pick(1, 4); l > 0; --l) {
      const int g = pick(0, (int)groups.size() - 1), w3 = pick(1, nc), runs = pick(1, 12);
      const int off = add_list(cols, runs, w3, pick(0, nc - w3), pick(0, 1) != 0);
      const int n = (int)cols.size() - off, nk = pick(1, 3);
      for (int b = pick(1, 2); b > 0; --b)
        for (int c0 = 0; c0 < n; c0 += 256)
          for (int x = 0; x < nc; x += 32)
            for (int y = 0; y < nc; y += 16)
              for (int k = 0; k < nk; ++k)
                tiles.push_back(TcTile{g, b, 0, 0, x, y, off, n, c0, k, x > y, 0});
    }
    if (pick(0, 1)) std::shuffle(tiles.begin(), tiles.end(), rng);
    for (int fixed = 0; fixed < 2; ++fixed) {
      const bool want = rule(tiles, groups, cols, fixed != 0);
      bad += want != tcs_wins(tiles.data(), tiles.size(), groups.data(), cols.data(), fixed != 0);
      wins += want;
    }
  }
  // one list of 20 runs of 64 channels, 16 x 32 rectangles: 2560 tiles of 5 windows
  std::vector<TcGroup> groups(1);
  groups[0].nu1_hi = groups[0].nu2_hi = 512;
  groups[0].Kpad = groups[0].kseg_len = 4096;
  groups[0].dsum = &dummy;
  std::vector<ColEntry> cols;
  std::vector<TcTile> tiles;
  const int off = add_list(cols, 20, 64, 0, false), n = (int)cols.size() - off;
  for (int c0 = 0; c0 < n; c0 += 256)
    for (int x = 0; x < 512; x += 32)
      for (int y = 0; y < 512; y += 16) tiles.push_back(TcTile{0, 0, 0, 0, x, y, off, n, c0, 0, 0, 0});
  double best[2] = {1e9, 1e9};
  int sink = 0;
  for (int rep = 0; rep < 40; ++rep)
    for (int k = 0; k < 2; ++k) {
      const auto t0 = std::chrono::steady_clock::now();
      sink += k ? (int)rule(tiles, groups, cols, false)
                : (int)tcs_wins(tiles.data(), tiles.size(), groups.data(), cols.data(), false);
      best[k] = std::min(best[k], std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count());
    }
  std::printf("%d %d %d %.4f %d\n", 2 * lists, bad, wins, best[0] / best[1], sink);
  return 0;
}
