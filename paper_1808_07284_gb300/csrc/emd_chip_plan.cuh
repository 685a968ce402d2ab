// Layout of the on-chip solve (emd_chip.cuh, emd_chip_w.cuh): its sizes, the buffers of its exchanges
// and how a batch is dealt to the SMs.  Host code without CUDA, so that a plan can be looked at
// where there is no GPU.
#pragma once

#include <algorithm>
#include <cstddef>
#include <utility>
#include <vector>

#ifdef __CUDACC__
#define EMD_HOST_DEVICE __host__ __device__
#else
#define EMD_HOST_DEVICE
#endif

namespace emd {

inline size_t align256(size_t x) { return (x + 255u) & ~static_cast<size_t>(255u); }
inline int ntp_of(int nt) { return (nt + 31) / 32 * 32; }  // pitch of a plane's rows

constexpr int kChipWorkers = 15;   // worker warps of a CTA (and a decider warp)
constexpr int kTallWorkers = 11;   // worker warps of a tall CTA: 168 registers a thread
constexpr int kChipMaxRows = 128;  // staged rows of a CTA at most (shared memory)
constexpr int kWMaxRows = 385;     // staged rows of a tall CTA at most
constexpr int kChipTJ = 120;       // owned time samples of a strip
constexpr int kChipMaxCtas = 160;  // CTAs of a launch at most (its jobs are a kernel argument)

enum ChipForm { kChipTile = 0, kChipMarch = 1, kChipMarchTall = 2 };

// One CTA's part of a gather.
struct ChipJob {
  int gather, seg, strip, segs, strips, i0, h;
  int group, rows;  // CTAs of the gather, staged rows of its tallest CTA
};

// Exchange buffers of a gather, in the workspace of its planes: packets of the cells that other CTAs
// hold as halo, two rows of every segment ([parity][seg][which][ntp]) and two samples of every
// strip ([parity][strip][side][nr]).
EMD_HOST_DEVICE inline size_t chip_row_packets(int segs, int ntp) {
  return segs > 1 ? static_cast<size_t>(2) * segs * 2 * ntp : 0;
}
EMD_HOST_DEVICE inline size_t chip_exchange_bytes(int segs, int strips, int nr, int ntp) {
  return 16 * (chip_row_packets(segs, ntp) + static_cast<size_t>(2) * strips * 2 * nr);
}

// The exchange buffers (packets: ux, ut of the last-but-one owned row; ux of the second one; ut of the
// second owned sample and ut, ux of the last-but-one) are followed, for tall CTAs, by [cta][rows][5]
// [128] streamed values.
constexpr int kTallRow = 5 * 128;
EMD_HOST_DEVICE inline size_t chip_w_tall_floats(int rows) { return static_cast<size_t>(rows) * kTallRow; }

// How the on-chip solve (emd_chip.cuh) lays a batch out: waves of gathers that are on chip side
// by side, one cooperative launch per wave.
struct ChipPlan {
  std::vector<std::vector<ChipJob>> waves;
  std::vector<int> form;  // a wave's kernel: ChipForm
  double cost = 0.0;      // estimated time of one pass over every gather, us
};

// Estimated us per pass of a wave whose tallest CTA stages n rows: the pass boundary and the rows.
// Measured: 2.8 us at 16 rows and 5.4 at 70 in the tile pass's form; 8.25 at 123 in the marching
// pass's; 16.7 at 217 and 23.2 at 327 in tall CTAs.  With the isotropic cost, whose square root and division
// take issue slots: 3.3 at 14 rows, 7.4 at 70; 11.8 at 92, 14.6 at 123; 22.5 at 150, 32.9 at 253, 44.8 at 327 and
// 58.3 at 383, where the streamed rows no longer stay in L2.
inline double chip_pass_us(int n, bool march, bool iso) {
  if (iso) {
    if (n > kChipMaxRows) return 4.5 + 0.12 * n + 0.13 * std::max(0, n - 327);
    return march ? 2.4 + 0.099 * n : 2.2 + 0.076 * n;
  }
  if (n > kChipMaxRows) return 3.9 + 0.059 * n;
  return march ? 2.4 + 0.048 * n : 2.0 + 0.049 * n;
}

// Estimated us per pass of the streaming solves (tile and marching pass) over `cells` cells:
// about 10 us of decision chain and 5.9 us per million cells, from L2 or from HBM alike; with the
// isotropic cost 23.5 us at 1.4 million cells, 38 at 3.2, 54 at 5.2, 172 at 20.7 and 256 at 30.7.
inline double stream_pass_us(double cells, bool iso) { return iso ? 12.0 + 7.8e-6 * cells : 10.0 + 5.9e-6 * cells; }

inline int chip_strips(int nt) { return (nt + kChipTJ - 1) / kChipTJ; }

// Staged rows of a gather's CTAs at the fewest rows that `cap` CTAs allow (0: it needs more CTAs
// however tall they are).
inline int chip_min_rows(int nt, int nr, int cap) {
  const int segs = cap / chip_strips(nt);
  return segs < 1 ? 0 : (nr + segs - 1) / segs + 3;
}

// Whether a gather's state fits on `cap` SMs, and in its planes what the on-chip solve keeps there:
// the exchange buffers and, for tall CTAs, their streamed values.
inline bool chip_fits(int nt, int nr, int cap, bool march) {
  const int strips = chip_strips(nt), ntp = ntp_of(nt), rows = chip_min_rows(nt, nr, cap);
  if (rows == 0 || rows > (march ? kWMaxRows : kChipMaxRows)) return false;
  const size_t planes = 9 * align256(sizeof(float) * static_cast<size_t>(nr) * ntp);
  const int lowest = kChipWorkers - 3;  // receivers of the lowest CTAs (chip_plan)
  size_t need = chip_exchange_bytes((nr + lowest - 1) / lowest, strips, nr, ntp);
  if (march && nr > kChipMaxRows - 3) {
    const int tall = (nr + kChipMaxRows - 3) / (kChipMaxRows - 2);  // segments of tall CTAs at most
    need = std::max(need, chip_exchange_bytes(tall, strips, nr, ntp) +
                              4 * static_cast<size_t>(tall) * strips * chip_w_tall_floats((nr + tall - 1) / tall + 3));
  }
  return need <= planes;
}

// The plan whose estimated pass is shortest, over the height of the CTAs (taller ones put more
// gathers beside each other, lower ones spread a gather over more SMs); no waves when a gather
// does not fit.
inline ChipPlan chip_plan(int B, const int *nt, const int *nr, int cap, bool march, bool iso) {
  // staged rows of the tallest CTA: whole rows per worker warp, up to what the layout holds
  std::vector<int> heights;
  for (int n = kChipWorkers; n < kChipMaxRows; n += kChipWorkers) heights.push_back(n);
  heights.push_back(kChipMaxRows);
  if (march)
    for (int n = kChipMaxRows / kTallWorkers * kTallWorkers + kTallWorkers; n <= kWMaxRows;
         n += kTallWorkers)
      heights.push_back(n);
  auto is_tall = [](int n) { return n > kChipMaxRows; };
  std::vector<ChipJob> g(B);
  std::vector<int> order(B), wave(B), start, used, rows;
  auto lay_out = [&](int height) -> double {  // estimated us per pass, or -1
    for (int b = 0; b < B; ++b) {
      ChipJob &J = g[b];
      J.gather = b;
      J.strips = chip_strips(nt[b]);
      const int nseg = (nr[b] + height - 4) / (height - 3);
      J.h = std::max(nr[b] > 1 ? 2 : 1, (nr[b] + nseg - 1) / nseg);
      J.segs = (nr[b] + J.h - 1) / J.h;
      if (static_cast<long long>(J.strips) * J.segs > cap) return -1.0;
      J.group = J.strips * J.segs;
      J.rows = J.h + 3;
    }
    start.assign(cap + 1, 0);  // the gathers in falling order of their CTAs (a counting sort)
    for (int b = 0; b < B; ++b) ++start[cap - g[b].group + 1];
    for (int i = 1; i <= cap; ++i) start[i] += start[i - 1];
    for (int b = 0; b < B; ++b) order[start[cap - g[b].group]++] = b;
    used.clear();
    rows.clear();
    // First fit, largest first; a wave's gathers share a layout.  Gathers of as many CTAs and the same
    // layout look on from the last one's wave, since no wave before it can take them: the waves are
    // walked once for each number of CTAs, not once for each gather (20,000 uneven gathers: 240 ms).
    size_t open = 0, from[2] = {0, 0};  // waves before `open` are full
    int group = -1;
    for (int b : order) {
      while (open < used.size() && used[open] + g[order.back()].group > cap) ++open;
      if (g[b].group != group) from[0] = from[1] = open;
      group = g[b].group;
      const bool tall = is_tall(g[b].rows);
      size_t w = std::max(open, from[tall]);
      while (w < used.size() && (used[w] + group > cap || is_tall(rows[w]) != tall)) ++w;
      if (w == used.size()) {
        used.push_back(0);
        rows.push_back(g[b].rows);
      }
      used[w] += group;
      rows[w] = std::max(rows[w], g[b].rows);
      from[tall] = w;
      wave[b] = static_cast<int>(w);
    }
    double cost = 0.0;
    for (int n : rows) cost += chip_pass_us(n, march, iso);
    return cost;
  };
  ChipPlan plan;
  int best = 0;
  for (const int height : heights) {
    const double cost = lay_out(height);
    if (cost < 0.0 || (best && cost >= plan.cost)) continue;
    best = height;
    plan.cost = cost;
  }
  if (!best) return plan;
  lay_out(best);
  std::vector<std::vector<int>> members(used.size());
  for (int b : order) members[wave[b]].push_back(b);
  for (size_t w = 0; w < members.size(); ++w) {
    plan.waves.emplace_back();
    plan.form.push_back(!march ? kChipTile : is_tall(rows[w]) ? kChipMarchTall : kChipMarch);
    for (int b : members[w])
      for (int seg = 0; seg < g[b].segs; ++seg)
        for (int strip = 0; strip < g[b].strips; ++strip) {
          ChipJob J = g[b];
          J.seg = seg;
          J.strip = strip;
          J.i0 = seg * g[b].h;
          J.h = std::min(g[b].h, nr[b] - J.i0);
          plan.waves.back().push_back(J);
        }
  }
  return plan;
}

// Copies of the elements `idx` of an array (empty for a null one).
template <class T>
std::vector<T> pick(const T *a, const std::vector<int> &idx) {
  std::vector<T> v;
  if (a)
    for (int b : idx) v.push_back(a[b]);
  return v;
}

// The gathers of a batch that are solved on chip (`on`, in order) and their plan.  Of three ways
// the one whose estimated pass is shortest: every gather that fits, only those whose own pass
// there is shorter than their share of a streamed pass, or none.
//
// *march: the form whose rounding the streaming solve of this batch has, the tile pass up to
// about 1.4 million cells (and for thin gathers), where the autotuner takes it, the marching pass
// above.  Measured crossing, single gathers: 400 x 3000 and 648 x 2000 take the tile pass, 400 x
// 3500 and 300 x 5000 the march.
inline ChipPlan choose_on_chip(int B, const int *nt, const int *nr, int cap, bool iso, bool whole_only,
                               std::vector<int> &on, bool *march) {
  double cells = 0.0;
  int receivers = 0;
  for (int b = 0; b < B; ++b) {
    cells += static_cast<double>(nt[b]) * nr[b];
    receivers = std::max(receivers, nr[b]);
  }
  *march = cells >= 1.4e6 && receivers > 8;
  ChipPlan plan;
  double best = stream_pass_us(cells, iso);
  on.clear();
  size_t tried = 0;
  for (const bool all : {true, false}) {
    std::vector<int> sub;
    double left = cells;
    for (int b = 0; b < B; ++b) {
      const double n = static_cast<double>(nt[b]) * nr[b];
      if (!chip_fits(nt[b], nr[b], cap, *march)) continue;
      const int rows = chip_min_rows(nt[b], nr[b], cap);
      if (!all && rows > kChipMaxRows &&
          chip_pass_us(rows, *march, iso) > stream_pass_us(n, iso) - stream_pass_us(0.0, iso))
        continue;
      sub.push_back(b);
      left -= n;
    }
    const int nb = static_cast<int>(sub.size());
    if (nb == 0 || sub.size() == tried || (whole_only && nb < B)) continue;
    tried = sub.size();
    ChipPlan q = chip_plan(nb, pick(nt, sub).data(), pick(nr, sub).data(), cap, *march, iso);
    const double cost = q.cost + (nb < B ? stream_pass_us(left, iso) : 0.0);
    if (q.waves.empty() || cost >= best) continue;
    best = cost;
    on = std::move(sub);
    plan = std::move(q);
  }
  return plan;
}

}  // namespace emd
