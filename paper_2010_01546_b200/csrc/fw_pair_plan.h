// Work lists of the CTA-pair kernels (fw_umma_pair.cu): tiles of a problem, their estimated times, and the widths of tiles and numbers of
// row slabs with which a launch ends earliest.  Plain C++, no device.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <map>
#include <mutex>
#include <vector>

namespace fw {

constexpr int GP_SR_F32 = 32;              // rows of X per stage, fp32 (48 KB stages, 4 in flight)
constexpr int GP_SR_BF16 = 64;             // bf16: the same 48 KB and 1024 tensor cycles per stage as fp32; with 32 rows
                                           // (512 cycles) the per-stage hand-offs left the tensor pipe idle a third of the time
constexpr int pair_sr(bool bf16) { return bf16 ? GP_SR_BF16 : GP_SR_F32; }
constexpr int GP_GCOLS = 128;              // columns per column group (chunks of 32 fp32 or 64 bf16 columns)
constexpr int GP_MAX_ITEMS = 2048;
constexpr int kMinPanel = 256;             // narrowest tile of a product

inline int pair_tiles_sym(int M16) {
  int t = 0;
  for (int c = 0; c < M16; c += 256) t += (M16 - c + 511) / 512;
  return t;
}
inline int pair_tiles_full(int M16, int panel) { return ((M16 + 255) / 256) * ((M16 + panel - 1) / panel); }

// Plans by what they were made for.  Host threads that work on different layers ask at the same time: every look is under the lock,
// and what is handed out is a copy.
template <class V>
class PlanMemo {
 public:
  bool find(const std::vector<int64_t>& key, V& v) {
    std::lock_guard<std::mutex> lock(mu_);
    const auto hit = plans_.find(key);
    if (hit == plans_.end()) return false;
    v = hit->second;
    return true;
  }
  void keep(const std::vector<int64_t>& key, const V& v) {
    std::lock_guard<std::mutex> lock(mu_);
    if (plans_.size() > 256) plans_.clear();
    plans_[key] = v;
  }

 private:
  std::mutex mu_;
  std::map<std::vector<int64_t>, V> plans_;
};

struct PairTile { int n0, n1, cols; bool skip; };   // cols: columns a CTA stages; skip: wholly below the diagonal of a symmetric product

inline void pair_tiles(int M, bool full, int panel, bool sym_out, std::vector<PairTile>& out) {
  const int M16 = (M + 15) / 16 * 16;
  out.clear();
  for (int I = 0; 256 * I < M16; ++I) {
    const int c_first = full ? 0 : 256 * I;
    for (int c = c_first, t = 0; c < M16; c += panel, ++t) {
      PairTile pt;
      const int pw = std::min(panel, M16 - c);
      pt.n0 = std::min(256, pw);
      pt.n1 = pw - pt.n0;
      const bool diag = !full && t == 0;
      // (a Gram tile counts whole groups: the row slabs chosen by this estimate fix how the sums are rounded)
      if (full) pt.cols = GP_GCOLS + pt.n0 / 2 + pt.n1 / 2;
      else pt.cols = GP_GCOLS * (1 + ((diag && pt.n0 == 256) ? 0 : 1) + (pt.n1 > 0 ? 1 : 0));
      pt.skip = full && sym_out && c + pt.n0 + pt.n1 <= 256 * I;
      out.push_back(pt);
    }
  }
}

// Estimated time of one tile over `rows` rows, microseconds: tensor time against staging time.  Staging rates
// are what a CTA sustains with every SM busy (measured: about 40 bytes per clock for bf16 tiles and 48 for fp32
// tiles, which then run at the TF32 tensor rate).
inline double pair_tile_us(const PairTile& t, bool bf16, int fix, double rows) {
  const double clk_us = 1800.0;                                   // SM clocks per microsecond under load
  const double tensor = (t.n0 + t.n1) / 512.0 * (bf16 ? 16.0 : 32.0);
  const double load = t.cols * (bf16 ? 2.0 / 40.0 : 4.0 / 48.0) * (1.0 + 0.2 * (fix & 1) + 0.4 * (fix >> 1));
  const double fixed = 4.0 + 128.0 * (t.n0 + t.n1) * 4.0 / 80e3;  // prologue, pipeline fill, epilogue stores
  return fixed + rows * std::max(tensor, load) / clk_us;
}

struct PairSpec {
  int M; int64_t rows; bool bf16, full, colsums, sym_out = false; int split_cap; int panel = 512, fix = 0, round_out = 0;
  std::vector<PairTile> tiles;
  int splits; int64_t per;     // chosen: splits, stages per split
};

// When the longest-first list schedule of the items over the resident CTA pairs ends.
inline double pair_makespan(std::vector<double>& items, int slots) {
  std::sort(items.begin(), items.end(), [](double a, double b) { return a > b; });
  std::vector<double> slot(slots, 0.0);
  for (double c : items) *std::min_element(slot.begin(), slot.end()) += c;
  return *std::max_element(slot.begin(), slot.end());
}

// Columns of the products' tiles: 512 moves the fewest bytes per output, but one layer of M = 2304 is 45 such tiles on 74
// pairs of SMs, or 72 of 320 columns that take three quarters of the time.  The search takes the host 1 ms for 16 layers of M = 1024 to 2500 and is made
// once per list of problems: every re-sync asks for two, one a product.
inline int pair_choose_panel(const std::vector<PairSpec>& P, int slots) {
  static PlanMemo<int> memo;
  std::vector<int64_t> key(1, slots);
  for (const PairSpec& p : P) { key.push_back(p.M); key.push_back(p.sym_out * 4 + p.fix); }
  int panel = 512;
  if (memo.find(key, panel)) return panel;
  double best = 0;
  std::vector<PairTile> tiles;
  std::vector<double> items;
  for (int w = 512; w >= kMinPanel; w -= 64) {
    items.clear();
    for (const PairSpec& p : P) {
      pair_tiles(p.M, true, w, p.sym_out, tiles);
      for (const PairTile& t : tiles)
        if (!t.skip) items.push_back(pair_tile_us(t, false, p.fix, (double)p.M));
    }
    if (items.size() > (size_t)GP_MAX_ITEMS) break;
    const double end = pair_makespan(items, slots);
    if (w == 512 || end < best) { best = end; panel = w; }
  }
  memo.keep(key, panel);
  return panel;
}

// Chooses the split count of every problem so that the longest-first list schedule of all (tile, split) items
// over the resident CTA pairs ends earliest, counting what each further split costs the reduction that follows.  forced, debug:
// tuning aids.
inline void pair_choose_splits(std::vector<PairSpec>& P, int slots, int forced, bool debug) {
  struct Choice { std::vector<int> splits; double us; };
  Choice best{std::vector<int>(P.size(), 1), 1e300};
  std::vector<double> items;
  // the search costs the host a fraction of a millisecond: its result is kept per list of problems
  static PlanMemo<Choice> memo;
  std::vector<int64_t> key;
  key.push_back(slots);
  for (const PairSpec& p : P) {
    key.push_back(p.M); key.push_back(p.rows); key.push_back(p.split_cap); key.push_back(p.panel);
    key.push_back((p.bf16 ? 1 : 0) | (p.full ? 2 : 0) | (p.fix << 5) | (p.sym_out ? 8 : 0) | (p.colsums ? 16 : 0));
  }
  const bool known = memo.find(key, best);
  for (int step = 0; !known && step < 64; ++step) {
    const double tau = 6.0 * std::pow(1.12, step);                // target item time, 6 us .. 7.5 ms
    double extra = 0;
    size_t count = 0;
    items.clear();
    std::vector<int> sp(P.size());
    for (size_t l = 0; l < P.size(); ++l) {
      PairSpec& p = P[l];
      double longest = 0;
      for (const PairTile& t : p.tiles)
        if (!t.skip) longest = std::max(longest, pair_tile_us(t, p.bf16, p.fix, (double)p.rows));
      const int SRh = pair_sr(p.bf16);
      const int64_t nsr = (p.rows + SRh - 1) / SRh;
      int64_t s = (int64_t)(longest / tau + 0.5);
      s = std::max<int64_t>(1, std::min<int64_t>(s, std::min<int64_t>(p.split_cap, nsr)));
      const int64_t per = (nsr + s - 1) / s;
      s = (nsr + per - 1) / per;
      sp[l] = (int)s;
      for (const PairTile& t : p.tiles) {
        if (t.skip) continue;
        for (int64_t k = 0; k < s; ++k) {
          const double r = (double)std::min<int64_t>(per * SRh, p.rows - k * per * SRh);
          items.push_back(pair_tile_us(t, p.bf16, p.fix, r));
        }
        count += (size_t)s;
      }
      // the reduction reads every partial once (upper triangle), at about 4 TB/s
      if (!p.full) extra += (double)(s - 1) * 0.55 * 4.0 * p.M * (double)p.M / 4e6;
    }
    if (count > (size_t)GP_MAX_ITEMS) continue;
    const double span = pair_makespan(items, slots) + extra;
    if (span < best.us) best = Choice{sp, span};
  }
  if (!known) memo.keep(key, best);
  for (size_t l = 0; l < P.size(); ++l) {
    PairSpec& p = P[l];
    const int64_t nsr = (p.rows + pair_sr(p.bf16) - 1) / pair_sr(p.bf16);
    int64_t s = best.splits[l];
    if (forced > 0) s = std::max<int64_t>(1, std::min<int64_t>(forced, std::min<int64_t>(p.split_cap, nsr)));
    if (debug) fprintf(stderr, "[fw] pair: M=%d rows=%lld tiles=%zu splits=%lld (cap %d) est %.1f us\n", p.M, (long long)p.rows, p.tiles.size(), (long long)s, p.split_cap, best.us);
    const int64_t per = (nsr + s - 1) / s;
    p.splits = (int)((nsr + per - 1) / per);
    p.per = per;
  }
}

}  // namespace fw
