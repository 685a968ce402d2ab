// On-chip persistent solve: a gather whose whole state fits in the shared and tensor memory of
// the GPU is solved without touching DRAM or L2 except for halos, sums and the one read of its
// inputs and write of its outputs.  One launch does everything a solve needs: the balancing
// sums (k_prepare's), every PDHG iteration and the finalize pass.
//
// Layout.  A gather is cut into segments of h receivers by strips of 120 time samples, one CTA
// each (one CTA per SM).  A CTA holds its h x 120 cells and a halo of two receivers above, one
// below and four samples on each side: n = h + 3 rows of 128 samples, dealt in contiguous runs
// to fifteen worker warps (with the decider warp four per scheduler, so that a thread may hold
// 128 registers); lane l owns four consecutive samples, so every state value is private to one
// lane.  u^k (x, t) and phi live in tensor memory (12 words per lane and row, used as a
// lane-private store: it moves about 600 B per clock and SM, shared memory 128); div u, q =
// div(u^{k+1} - u^k) and the balanced f live in shared memory.  Time neighbours come by
// shuffles, receivers within a warp's run from registers, and the rows where two runs meet
// through small shared buffers.
//
// One iteration.  A warp walks its run upwards (falling receiver index).  At row r it completes
// phi^k of row r (p = div u + f and q of the last pass are stored, not recomputed), then
// u^{k+1}, div u^{k+1}, p, q and the linesearch sums of row r + 1.  The last row of a run needs
// u^{k+1} of the next run's first row and the first row needs phi and p, q of the last row
// above it, so these are taken after three barriers of the workers.  Every cell's arithmetic
// and rounding are those of the tile pass (emd_pass_tma.cuh), so both give the same iterates;
// emd_chip_w.cuh has the same solve with the arithmetic of the marching pass.
//
// Pass boundary.  No CTA waits for a broadcast or a memory barrier.  Every CTA's decider warp adds
// the CTA's sums to a few 64-bit words in L2 whose low byte counts the CTAs that have added
// (chip_fast_add, chip_fast_poll); once the counts are full, every CTA reads the same totals and takes the
// same decision.  The cells that neighbours hold as halo travel as 16-byte packets that carry the
// pass they belong to, and the workers fetch theirs while the decider decides.  (An exchange by
// FP64 sums, a release of a counter and its acquisition, which the first form had everywhere and
// passes with residual sums still take, costs about 5400 cycles from the last row to the next
// pass; now 3300.)
//
// Measured, us per pass, against the streaming solve: 64 x 256 2.8 (7.9: 5700 cycles, half of them the
// exchange's L2 round trip, half the workers' three barriers with one row between them), 321 x 401
// 2.9 (8.5), 400 x 3000 5.4 (16.7).
#pragma once

#include "emd_chip_plan.cuh"
#include "emd_pass_tma.cuh"

namespace emd {

constexpr int kChipTmemCols = 128;                      // tensor memory columns of a warp
constexpr int kChipRowCols = 12;                        // ... of one row: ux, ut, phi
static_assert((kChipMaxRows + kChipWorkers - 1) / kChipWorkers * kChipRowCols <= kChipTmemCols, "a run's rows");

constexpr int kChipSets = 3;                            // accumulator sets, used in turn
constexpr int kChipVals = 8;                            // sums of a pass
constexpr int kChipSpread = 8;                          // copies of each accumulator
constexpr int kChipWordSets = 2;                        // word sets of the fast exchange, used in turn
constexpr int kChipWordCopies = 4;                      // copies of the words of the fast exchange
constexpr int kChipWords = 16;                          // two words of each value

struct ChipJobs {
  ChipJob job[kChipMaxCtas];
};

// Dynamic shared memory of a CTA: the planes div u, q and f at a fixed stride (so that one row
// address serves the three of them), then four boundary rows per warp.
constexpr unsigned kChipRowBytes = 512;
constexpr unsigned kChipPlane = kChipMaxRows * kChipRowBytes;
constexpr unsigned kChipBound = kChipWorkers * kChipRowBytes;
constexpr size_t kChipSmem = 3 * kChipPlane + 4 * kChipBound + 128;

// ------------------------------------------------------------------ packed FP32 pairs
// Two IEEE operations per issue slot (the FMA lanes are the same: 127 against 113-117 lane
// operations per clock and SM; the saved issue slots go to loads, shuffles and selects).

using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void upk(f32x2 r, float &x, float &y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(r));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Four consecutive samples of one lane, as two pairs.
struct Q4 {
  f32x2 a, b;
};
__device__ __forceinline__ Q4 q4(float x, float y, float z, float w) { return {pk(x, y), pk(z, w)}; }
__device__ __forceinline__ Q4 q4s(float s) { return {pk(s, s), pk(s, s)}; }
__device__ __forceinline__ void un4(const Q4 &v, float (&o)[4]) {
  upk(v.a, o[0], o[1]);
  upk(v.b, o[2], o[3]);
}
__device__ __forceinline__ Q4 add4(const Q4 &x, const Q4 &y) { return {add2(x.a, y.a), add2(x.b, y.b)}; }
__device__ __forceinline__ Q4 sub4(const Q4 &x, const Q4 &y) { return {sub2(x.a, y.a), sub2(x.b, y.b)}; }
__device__ __forceinline__ Q4 mul4(const Q4 &x, const Q4 &y) { return {mul2(x.a, y.a), mul2(x.b, y.b)}; }
__device__ __forceinline__ Q4 fma4(const Q4 &x, const Q4 &y, const Q4 &z) {
  return {fma2(x.a, y.a, z.a), fma2(x.b, y.b, z.b)};
}
// Sixteen bytes of shared memory, by address in the shared window, at a constant offset.
template <unsigned OFF = 0>
__device__ __forceinline__ Q4 lds4(unsigned a) {
  Q4 v;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+%3];" : "=l"(v.a), "=l"(v.b) : "r"(a), "n"(OFF) : "memory");
  return v;
}
template <unsigned OFF = 0>
__device__ __forceinline__ void sts4(unsigned a, const Q4 &v) {
  asm volatile("st.shared.v2.b64 [%0+%1], {%2, %3};" ::"r"(a), "n"(OFF), "l"(v.a), "l"(v.b) : "memory");
}
__device__ __forceinline__ void sts1(unsigned a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ float lds1(unsigned a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
// Eight bytes of shared memory (a value written twice) as both pairs.
template <unsigned OFF = 0>
__device__ __forceinline__ Q4 lds_pair(unsigned a) {
  Q4 v;
  asm volatile("ld.shared.b64 %0, [%1+%2];" : "=l"(v.a) : "r"(a), "n"(OFF) : "memory");
  v.b = v.a;
  return v;
}

// x[j] - x[j - 1] over the lane's four samples; `left` is the last sample of the lane before.
__device__ __forceinline__ Q4 diff_left(const Q4 &v) {
  float x[4];
  un4(v, x);
  const float left = __shfl_up_sync(0xffffffffu, x[3], 1);
  return q4(x[0] - left, x[1] - x[0], x[2] - x[1], x[3] - x[2]);
}
// x[j + 1] - x[j].
__device__ __forceinline__ Q4 diff_right(const Q4 &v) {
  float x[4];
  un4(v, x);
  const float right = __shfl_down_sync(0xffffffffu, x[0], 1);
  return q4(x[1] - x[0], x[2] - x[1], x[3] - x[2], right - x[3]);
}

// shrink(v, al) inv = (v - clamp(v, -al, al)) inv: |v| <= al gives 0, else sign(v)(|v| - al).
__device__ __forceinline__ Q4 shrink4(const Q4 &v, float al, const Q4 &inv) {
  float x[4], t[4];
  un4(v, x);
#pragma unroll
  for (int q = 0; q < 4; ++q) t[q] = fminf(fmaxf(x[q], -al), al);
  return mul4(sub4(v, q4(t[0], t[1], t[2], t[3])), inv);
}

// div u of one row from the differences of its face fluxes.
__device__ __forceinline__ Q4 div4(const Q4 &dx_, const Q4 &dt_, const Q4 &rdx, const Q4 &rdt) {
  return fma4(dx_, rdx, mul4(dt_, rdt));
}

// ------------------------------------------------------------------ halo packets
// Two values of a cell and the pass they belong to, written and read as one 128-bit access, so a
// reader that sees the pass's tag has its values.

struct Packet {
  float x, y;
  int tag;
};
using PacketMem = uint4;
__device__ __forceinline__ void put_packet(PacketMem *p, float x, float y, int tag) {
  asm volatile(
      "{\n .reg .b64 lo, hi;\n .reg .b128 q;\n mov.b64 lo, {%1, %2};\n mov.b64 hi, {%3, %3};\n"
      " mov.b128 q, {lo, hi};\n st.relaxed.gpu.global.b128 [%0], q;\n}\n" ::"l"(p),
      "f"(x), "f"(y), "r"(tag)
      : "memory");
}
__device__ __forceinline__ Packet get_packet(const PacketMem *p) {
  Packet v;
  asm volatile(
      "{\n .reg .b32 again;\n .reg .b64 lo, hi;\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%3];\n"
      " mov.b128 {lo, hi}, q;\n mov.b64 {%0, %1}, lo;\n mov.b64 {%2, again}, hi;\n}\n"
      : "=f"(v.x), "=f"(v.y), "=r"(v.tag)
      : "l"(p)
      : "memory");
  return v;
}
// Repeats `ready` (a warp's attempt, true in every lane that has what it needs) until it is true in
// all lanes; false when the bound runs out.
template <class F>
__device__ __forceinline__ bool poll_warp(F ready) {
  if (__all_sync(0xffffffffu, ready())) return true;
  const unsigned long long t0 = global_ns();
  for (unsigned n = 0;; ++n) {
    if (__all_sync(0xffffffffu, ready())) return true;
    if ((n & 63u) == 63u && global_ns() - t0 > kSpinLimitNs) return false;
  }
}

// ------------------------------------------------------------------ tensor memory as a store

__device__ __forceinline__ void tmem_alloc_all(uint32_t *slot) {  // one warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n"
               "tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::"r"(smem_u32(slot))
               : "memory");
}
__device__ __forceinline__ void tmem_free_all(uint32_t base) {  // the same warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(base) : "memory");
}

// A row's tensor-memory state of one lane: ux, ut, phi.
struct RowState {
  Q4 ux, ut, ph;
};

__device__ __forceinline__ RowState tmem_load_row(uint32_t addr) {
  uint32_t r[12];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%12];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%13];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
        "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11])
      : "r"(addr), "r"(addr + 8)
      : "memory");
  auto g = [&](int i) { return q4(__uint_as_float(r[i]), __uint_as_float(r[i + 1]), __uint_as_float(r[i + 2]),
                                  __uint_as_float(r[i + 3])); };
  return {g(0), g(4), g(8)};
}

__device__ __forceinline__ void tmem_store_row(uint32_t addr, const RowState &s) {
  float x[4], t[4], p[4];
  un4(s.ux, x);
  un4(s.ut, t);
  un4(s.ph, p);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%2,%3,%4,%5,%6,%7,%8,%9};\n"
      "tcgen05.st.sync.aligned.32x32b.x4.b32 [%1], {%10,%11,%12,%13};\n" ::"r"(addr), "r"(addr + 8),
      "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(t[3]), "f"(p[0]),
      "f"(p[1]), "f"(p[2]), "f"(p[3])
      : "memory");
}

// This warp's earlier tensor-memory stores are complete (before it loads the rows again).
__device__ __forceinline__ void tmem_stores_done() {
  asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
}

// ------------------------------------------------------------------ barriers

// Barriers of a CTA of NW worker warps: the workers alone, or with the decider warp.
template <int NW = kChipWorkers>
__device__ __forceinline__ void bar_workers() {
  asm volatile("bar.sync 1, %0;\n" ::"n"(NW * 32) : "memory");
}
template <int ID, int NW = kChipWorkers>
__device__ __forceinline__ void bar_all() {
  asm volatile("bar.sync %0, %1;\n" ::"n"(ID), "n"((NW + 1) * 32) : "memory");
}
template <int ID, int NW = kChipWorkers>
__device__ __forceinline__ void bar_all_arrive() {
  asm volatile("bar.arrive %0, %1;\n" ::"n"(ID), "n"((NW + 1) * 32) : "memory");
}

// Totals of eight values over each group of eight lanes: lane l ends with the total of value l & 7
// over its group (FP32, pairwise).  Each step exchanges halves of the values, so seven shuffles do.
__device__ __forceinline__ float group_sum8(const float (&v)[8]) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  float a[4], b[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {  // lanes with bit 2 set keep values 4..7
    const bool hi = lane & 4;
    const float keep = hi ? v[i + 4] : v[i], send = hi ? v[i] : v[i + 4];
    a[i] = keep + __shfl_xor_sync(FULL, send, 4);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool hi = lane & 2;
    const float keep = hi ? a[i + 2] : a[i], send = hi ? a[i] : a[i + 2];
    b[i] = keep + __shfl_xor_sync(FULL, send, 2);
  }
  const bool hi = lane & 1;
  const float keep = hi ? b[1] : b[0], send = hi ? b[0] : b[1];
  return keep + __shfl_xor_sync(FULL, send, 1);
}

// Warp totals of eight values: lane l ends with the total of value l & 7 (all 32 lanes summed, FP32).
__device__ __forceinline__ float warp_sum8(const float (&v)[8]) {
  float s = group_sum8(v);
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  return s;
}

// The same with the last two additions, whose rounding counts most, in a pair of floats.
__device__ __forceinline__ float warp_sum8_pair(const float (&v)[8], float &low) {
  constexpr unsigned FULL = 0xffffffffu;
  float s = group_sum8(v), t, e;
  two_sum(s, __shfl_xor_sync(FULL, s, 8), t, e);
  const float t16 = __shfl_xor_sync(FULL, t, 16), e16 = __shfl_xor_sync(FULL, e, 16);
  two_sum(t, t16, s, low);
  low += e + e16;
  return s;
}

// Sum of x over the lanes that share lane & 7 (the four groups of eight lanes), in every lane.
__device__ __forceinline__ double sum_groups(double x) {
  x += __shfl_xor_sync(0xffffffffu, x, 8);
  x += __shfl_xor_sync(0xffffffffu, x, 16);
  return x;
}

// The shared part of the kernel's CTA.
struct ChipShared {
  uint32_t tmem;
  int done, status, bad;
  float fmean;
  // each value four times, so that a 16-byte load gives a Q4: alpha, coef, theta,
  // 1 / (1 + eps alpha) of the pass, then 1/dx, 1/dt
  alignas(16) float sc[6][4];
  float warm[6][4];                          // takes what the decision writes when it runs for nothing
  float part[16][kChipVals];                 // warp totals of a pass (zero for warps that are not there)
  float low[16][kChipVals];                  // tall CTAs: their low parts
  double dpart[16][4];                       // warp totals of the balancing sums
};

// Decider warp: the lanes with `adds` add x to value lane & 7 in a copy of accumulator set `set`,
// the CTA is counted, and once every CTA of the group is, `v` is the group's total of value
// lane & 7 in every lane.  Afterwards CTA 0 zeroes the set of the pass before, which every CTA
// has read by now and which is added to again two passes on.  False when the bounded wait ran
// out.  (Eight copies: two loads and three FP64 additions to read a total, each addition about
// 70 cycles of a chain that every CTA waits for.)
__device__ __forceinline__ bool chip_exchange(const Ctl &c, State *st, double *acc, int set, int cta,
                                              int group, unsigned step, bool adds, double x, double &v) {
  const int lane = threadIdx.x & 31;
  double *a = acc + set * (kChipSpread * kChipVals);
  if (adds) atomicAdd(a + (cta % kChipSpread) * kChipVals + (lane & 7), x);
  __syncwarp();
  if (lane == 0 && c.debug_fault != 2) red_release_add(&st->tiles_done, 1u);
  if (!__all_sync(0xffffffffu, wait_count(&st->tiles_done, step * static_cast<unsigned>(group)))) return false;
  static_assert(kChipSpread == 8 && kChipVals == 8, "two copies per lane");
  const double x0 = __ldcg(a + lane), x1 = __ldcg(a + 32 + lane);  // copies lane / 8 and 4 + lane / 8
  v = sum_groups(x0 + x1);
  if (cta == 0) {
    double *z = acc + ((set + kChipSets - 1) % kChipSets) * (kChipSpread * kChipVals);
    z[lane] = 0.0;
    z[32 + lane] = 0.0;
  }
  return true;
}

// The totals over a CTA's warps of their FP32 totals, to a pair (hi, lo) of floats that every lane
// holds for value lane & 7.  (Two-sums are 4-cycle operations; FP64 takes 64 cycles for each of
// the nine conversions and additions.)
// LOW: the warps' totals are pairs themselves, with these low parts.
template <bool LOW>
__device__ __forceinline__ void chip_block_pair(const float (&part)[16][kChipVals], const float (&low)[16][kChipVals],
                                                float &s, float &e) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
  float s0, e0, s1, e1;
  two_sum(part[g][q], part[g + 4][q], s0, e0);
  two_sum(part[g + 8][q], part[g + 12][q], s1, e1);
  two_sum(s0, s1, s, e);
  e += e0 + e1;
  if (LOW) e += (low[g][q] + low[g + 4][q]) + (low[g + 8][q] + low[g + 12][q]);
#pragma unroll
  for (int o = 8; o <= 16; o <<= 1) {
    const float so = __shfl_xor_sync(FULL, s, o), eo = __shfl_xor_sync(FULL, e, o);
    two_sum(s, so, s0, e0);
    s = s0;
    e = (e + eo) + e0;
  }
}
// hi in lanes 0..7 and lo in the others, so that lanes 0..15 add both.
__device__ __forceinline__ double chip_block_total(const ChipShared &sh) {
  float s, e;
  chip_block_pair<false>(sh.part, sh.low, s, e);
  return static_cast<double>((threadIdx.x & 31) < 8 ? s : e);
}

// The exchange of a pass's six linesearch sums.  A value x of a CTA (the pair s + e of lane & 7) is
// taken in fixed point, x = (A + B 2^-46) 2^-sa with integers |A| < 2^38 and |B| <= 2^46, and
// added as the two words 256 A + 1 and 256 B + 1: the low byte of a word counts the CTAs that have
// added to it, so one poll brings the totals and says whether they are complete, with no barrier
// between data and counter (1000 cycles) and no second read (700).  The integers add exactly in
// any order.  The words are never cleared: each CTA keeps the totals that it read last from a set,
// and a total is the difference (modulo 2^64).  Clearing them would need a fence before the next
// exchange (1000 cycles a pass); as it is, a set is added to again only after every CTA has added
// to the other one, which it does after its read of this one.  sa puts the last pass's total of the value's family (p: P_pp, P_qq; grad p: G_pp,
// G_qq) at 2^24, so a value keeps 24 bits down to 2^-46 of it and may grow 2^14 fold; a CTA whose
// value does not fit adds 2^47 for it, every CTA sees the total beyond 2^46 and all of them take
// the FP64 exchange for this pass.  v: the total in FP32; a, b: in fixed point.
struct FastTotal {
  long long a, b;
  float v;
  bool fits;
};
__device__ __forceinline__ void chip_fast_add(const Ctl &c, unsigned long long *words, int set, int cta, float s, float e,
                                              int sa) {
  const int lane = threadIdx.x & 31, q = lane & 7;
  unsigned long long *const w = words + set * (kChipWordCopies * kChipWords);
  const float scale = __int_as_float((127 + sa) << 23);
  const float hs = q < 6 ? s * scale : 0.0f, ls = q < 6 ? e * scale : 0.0f;
  const bool fits = fabsf(hs) < 0x1p38f;  // false for a NaN too
  const float a1 = rintf(hs), a2 = rintf(ls);
  const long long ia = fits ? __float2ll_rn(a1) + __float2ll_rn(a2) : 1ll << 47;
  const long long ib = fits ? __float2ll_rn((hs - a1) * 0x1p46f) + __float2ll_rn((ls - a2) * 0x1p46f) : 0;
  if (lane < 16 && c.debug_fault != 2)
    atomicAdd(w + (cta % kChipWordCopies) * kChipWords + 2 * q + (lane >> 3),
              (static_cast<unsigned long long>(lane < 8 ? ia : ib) << 8) + 1u);
}
// x0, y0: the totals last read from this set, replaced by those read now.
__device__ __forceinline__ bool chip_fast_poll(const unsigned long long *words, int set, int group, int sa,
                                               unsigned long long &x0, unsigned long long &y0, FastTotal &o) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, q = lane & 7;
  unsigned long long x = 0, y = 0;
  const unsigned long long *const src =
      words + set * (kChipWordCopies * kChipWords) + (lane >> 3) * kChipWords + 2 * q;
  const bool ok = poll_warp([&] {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];\n" : "=l"(x), "=l"(y) : "l"(src) : "memory");
#pragma unroll
    for (int d = 8; d <= 16; d <<= 1) {
      x += __shfl_xor_sync(FULL, x, d);
      y += __shfl_xor_sync(FULL, y, d);
    }
    return static_cast<int>((x - x0) & 255u) == group && static_cast<int>((y - y0) & 255u) == group;
  });
  o.a = static_cast<long long>(x - x0) >> 8;
  o.b = static_cast<long long>(y - y0) >> 8;
  x0 = x;
  y0 = y;
  o.v = fmaf(__ll2float_rn(o.b), 0x1p-46f, __ll2float_rn(o.a)) * __int_as_float((127 - sa) << 23);
  o.fits = __all_sync(FULL, llabs(o.a) < (1ll << 46));
  return ok;
}

// xi^lane, by the multiplications of decide_prep_lanes.
__device__ __forceinline__ double xi_power(double xi) {
  double xl = 1.0, base = xi;
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    if (((threadIdx.x & 31) >> b) & 1) xl *= base;
    base *= base;
  }
  return xl;
}

// FP32 copies of a decision's prepared coefficients, for the quick test below.
struct QuickPrep {
  float s2x, s2, cl;
  bool usable;
};
// What a decision needs besides the sums, while the pass runs: per lane the step sizes that trial
// would accept, and the quick test's coefficients from their FP32 copies.  (The FP64 test's own
// coefficients, decide_prep_lanes, only when that runs: with them, the FP64 of this preparation
// took 4600 cycles, longer than the pass of a small gather.)
__device__ __forceinline__ QuickPrep step_prep(const Ctl &c, DecidePrep &d, double xl) {
  d.s_lane = sqrt(1.0 + d.theta) * xl;
  d.alpha_l = d.alpha * d.s_lane;
  d.coef_l = c.delta * d.alpha_l;
  d.alpha_lf = static_cast<float>(d.alpha_l);
  d.coef_lf = static_cast<float>(d.coef_l);
  d.theta_lf = static_cast<float>(d.s_lane);
  d.inv_lf = 1.0f / (1.0f + static_cast<float>(c.eps * d.alpha_l));
  const float zeta = static_cast<float>(c.zeta);
  QuickPrep p;
  p.s2x = 2.0f * d.theta_lf;
  p.s2 = d.theta_lf * d.theta_lf;
  p.cl = d.coef_lf * d.alpha_lf / (zeta * zeta);
  p.usable = p.cl > 1e-25f && p.cl < 1e25f;
  return p;
}

// An FP64 total cut to FP32 by integer operations (a conversion would take the FP64 pipe): exact
// to 23 bits within 2^-60 .. 2^60, else 0 (an infinity for one that is not finite).
__device__ __forceinline__ float cut_f32(double v) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int ex = (hi >> 20) & 0x7ff;
  const float f = __int_as_float((hi & 0x80000000) | ((ex - 896) << 23) | ((hi & 0xfffff) << 3) |
                                 static_cast<int>(static_cast<unsigned>(lo) >> 29));
  return ex > 1023 - 60 && ex < 1023 + 60 ? f : ex == 0x7ff ? INFINITY : 0.0f;
}

// The linesearch decision from FP32 copies of the totals (f: value lane & 7), where those settle
// it: a trial counts as decided when the two sides of its test differ by more than 1e-5 of the
// magnitudes that enter them, ten times what rounding the totals to 24 bits and the few FP32
// operations can move them, so the FP64 test would decide alike.  Returns the trial (0-based),
// or -1 where FP64 has to look (near ties, zeros, values outside 2^-60 .. 2^60, non-finite
// sums, no passing trial among the first 32).  The FP64 test is five dependent operations of
// about 70 cycles for every CTA to wait for.
__device__ __forceinline__ int quick_decide(const Ctl &c, const QuickPrep &p, float f) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // values 6 and 7 (the residual's) only have to be finite
  const float mag_f = fabsf(f);
  if (!__all_sync(FULL, (lane & 7) < 6 ? mag_f > 0x1p-60f && mag_f < 0x1p60f : mag_f < INFINITY)) return -1;
  float a[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) a[q] = __shfl_sync(FULL, f, q);
  const float px = p.s2x * a[1], pd = fmaf(p.s2, a[2], a[0]);
  const float gx = p.s2x * a[4], gd = fmaf(p.s2, a[5], a[3]);
  const float lhs = p.cl * (gd + gx), rhs = pd + px;
  const float mag = p.cl * (gd + fabsf(gx)) + (pd + fabsf(px));
  const bool sure = p.usable && fabsf(lhs - rhs) > 1e-5f * mag;
  const unsigned known = __ballot_sync(FULL, sure);
  const unsigned pass = __ballot_sync(FULL, sure && lhs < rhs && lane < c.ls_max_trials);
  if (!pass) return -1;
  const unsigned below = (pass & (0u - pass)) - 1u;  // the trials before the first that passes
  return (known & below) == below ? __ffs(pass) - 1 : -1;
}

// The prox of four cells (prox_cell of emd_kernels.cuh, the same values).  With the isotropic cost most
// cells shrink to zero, and the square root and division of a zero or denormal norm leave the
// instructions' fast path (648 x 8000, hyperbolic: 60.8 us a pass, which streaming took 53.6 for; now 44.7).
// So a cell whose squared norm is surely below alpha^2 takes a norm of about alpha instead, and where all
// of a warp's cells are such the two are left out.
template <bool ISO>
__device__ __forceinline__ void chip_prox(const Q4 &ux, const Q4 &ut, const Q4 &gx, const Q4 &gt,
                                          float alpha, const Q4 &al, const Q4 &inv, Q4 &nx, Q4 &nt) {
  const Q4 vx = fma4(al, gx, ux), vt = fma4(al, gt, ut);
  if (ISO) {
    float x[4], t[4], n2[4];
    un4(vx, x);
    un4(vt, t);
    const float low = 0.9999995f * (alpha * alpha);  // below it sqrtf(n2) <= alpha
    bool any = false;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      n2[q] = __fmaf_rn(x[q], x[q], __fmul_rn(t[q], t[q]));
      any = any || !(n2[q] < low);
    }
    nx = mul4(q4s(0.0f), vx);  // zeros of the signs that the scaling by 0 gives
    nt = mul4(q4s(0.0f), vt);
    if (__any_sync(0xffffffffu, any)) {
      float a[4], b[4], iv, unused;
      upk(inv.a, iv, unused);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float n = sqrtf(n2[q] < low ? low : n2[q]);
        const float s = n > alpha ? (1.0f - alpha / n) * iv : 0.0f;
        a[q] = s * x[q];
        b[q] = s * t[q];
      }
      nx = q4(a[0], a[1], a[2], a[3]);
      nt = q4(b[0], b[1], b[2], b[3]);
    }
  } else {
    nx = shrink4(vx, alpha, inv);
    nt = shrink4(vt, alpha, inv);
  }
}

// What the warps of a CTA share: its part of the gather and its storage.
struct ChipCta {
  const Ctl &c;
  const ChipJob &J;
  const Shot &S;
  ChipShared &sh;
  State *st;
  int lane, warp, nr, nt, ntp;
  int n, cta;        // staged rows, index in the group
  int ra, rb;        // rows of this warp's run
  int gj0;           // time index of this lane's first sample
  uint32_t taddr;    // this warp's tensor memory
  unsigned smem;     // this lane's column of the first 512-byte row of shared memory
};

// The balancing sums over a lane's cells: f, f^2, |Pcal| + |Pobs| and Pcal - Pobs, each to about
// 48 bits in FP32 pairs (an FP64 instruction takes a scheduler 64 cycles).  Over a gather they are as near
// to the exact sums as k_prepare's FP64 ones, as long as FP32 holds them: see balance_in_range.
// (Squares in FP64 cost 12 us of a solve of 648 x 8000, and they or a third float for f 0.3 us of each of
// its passes by what they do to the kernel's registers.)
struct BalanceSums {
  Sum2 f, f2, ab;
  float de = 0.0f;  // rounding errors of the differences f = Pcal - Pobs
  __device__ __forceinline__ void add(float po, float pp) {
    float d, e;
    two_sum(pp, -po, d, e);
    de += e;
    f.add(d);
    const float dd = d * d;
    f2.add(dd);
    f2.lo += fmaf(d, d, -dd);
    two_sum(fabsf(pp), fabsf(po), d, e);
    ab.add(d);
    ab.lo += e;
  }
  __device__ __forceinline__ void store(const ChipCta &X) {
    const double t0 = warp_sum_d(f.value()), t1 = warp_sum_d(f2.value()), t2 = warp_sum_d(ab.value());
    const double t3 = warp_sum_d(f.value() + static_cast<double>(de));
    if (X.lane < 4) X.sh.dpart[X.warp][X.lane] = X.lane == 0 ? t0 : X.lane == 1 ? t1 : X.lane == 2 ? t2 : t3;
  }
};

// Whether FP32 held the balancing sums m of a gather of N cells.  It did not where one is not finite
// (squares of 1e18 and more; inputs that are not finite), nor where the sum of squares is so small
// that what its cells lose to the smallest step of a float, 2^-149 each, may reach 2^-53 of it (f of about 3e-15 and
// less).  A sum of zero stands: the passes' own sums of squares are zero too then, in any solve.
__device__ __forceinline__ bool balance_in_range(const double (&m)[4], double N) {
  return isfinite(m[0]) && isfinite(m[1]) && isfinite(m[2]) && isfinite(m[3]) && (m[1] == 0.0 || m[1] >= N * 0x1p-96);
}

// u of a warm start at (gi, gj), plane 0 (x) or 1 (t); the outer faces carry none.
__device__ __forceinline__ float chip_init_flux(const ChipCta &X, int plane, int gi, int gj) {
  const bool in = gi >= 0 && gi < X.nr && gj >= 0 && gj < X.nt && (plane ? gj > 0 : gi > 0);
  return in ? X.S.m_init[(static_cast<size_t>(plane) * X.nr + gi) * X.nt + gj] : 0.0f;
}

// An owned row of the solution to the caller's arrays, and its terms of the gap sums (up: phi of
// the row above, gtv: phi[j] - phi[j - 1]).
template <bool ISO>
__device__ __forceinline__ void chip_output_row(const ChipCta &X, bool vec, int gi, const Q4 &ux4, const Q4 &ut4,
                                                const Q4 &ph4, const Q4 &up, const Q4 &gtv, const Q4 &f4,
                                                Sum2 (&t)[4]) {
  const Shot &S = X.S;
  float ph[4], pu[4], gt[4], ux[4], ut[4], fb[4];
  un4(ph4, ph);
  un4(up, pu);
  un4(gtv, gt);
  un4(ux4, ux);
  un4(ut4, ut);
  un4(f4, fb);
  const size_t g = static_cast<size_t>(gi) * X.nt + X.gj0, m_t = static_cast<size_t>(X.nr) * X.nt;
  if (vec && X.gj0 < X.nt) {
    *reinterpret_cast<float4 *>(S.phi_out + g) = make_float4(ph[0], ph[1], ph[2], ph[3]);
    *reinterpret_cast<float4 *>(S.m_out + g) = make_float4(ux[0], ux[1], ux[2], ux[3]);
    *reinterpret_cast<float4 *>(S.m_out + m_t + g) = make_float4(ut[0], ut[1], ut[2], ut[3]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int gj = X.gj0 + q;
    if (gj >= X.nt) continue;
    if (!vec) {
      S.phi_out[g + q] = ph[q];
      S.m_out[g + q] = ux[q];
      S.m_out[m_t + g + q] = ut[q];
    }
    const float gx = gi > 0 ? (ph[q] - pu[q]) * S.rdx : 0.0f, gtt = gj > 0 ? gt[q] * S.rdt : 0.0f;
    gap_terms(t, ux[q], ut[q], ph[q], fb[q], gx, gtt, ISO);
  }
}
// Whether rows of the outputs can be written sixteen bytes at a time.
__device__ __forceinline__ bool chip_vec_out(const ChipCta &X) {
  return (X.nt & 3) == 0 &&
         ((reinterpret_cast<uintptr_t>(X.S.phi_out) | reinterpret_cast<uintptr_t>(X.S.m_out)) & 15u) == 0;
}
// This warp's gap sums for the decider: the high and the low parts as eight values.
__device__ __forceinline__ void chip_store_gap(const ChipCta &X, Sum2 (&t)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    t[q].warp_total();
    if (X.lane == 0) {
      X.sh.part[X.warp][q] = t[q].hi;
      X.sh.part[X.warp][4 + q] = t[q].lo;
    }
  }
}

// A lane's samples: whether f of each is needed (one halo sample more on the left than right), and
// 1/dt of the face left of each, 0 for outer faces and samples that nobody needs.
struct ChipLane {
  bool use[4];
  float rm[4];
  bool own;  // lanes 1..30 own their samples, 0 and 31 only feed their neighbours
};
__device__ __forceinline__ ChipLane chip_lane(const ChipCta &X) {
  ChipLane l;
  const int lane = X.lane;
  l.own = lane >= 1 && lane <= 30;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int gj = X.gj0 + q;
    l.use[q] = gj >= 0 && gj < X.nt && (lane > 0 || q >= 2) && (lane < 31 || q == 0);
    l.rm[q] = gj > 0 && gj < X.nt && (lane > 0 || q == 3) && (lane < 31 || q == 0) ? X.S.rdt : 0.0f;
  }
  return l;
}

// Takes the inputs of a run's rows in turn: row(r, Pobs, Pcal), samples that nobody needs as 0.  They
// are loaded three rows ahead (8000 x 648, 30 rows a warp: 18 us less for a solve; what else a solve takes
// beside its passes is the writes of the streamed values and of the outputs).
template <class F>
__device__ __forceinline__ void chip_input_rows(const ChipCta &X, const ChipLane &ln, F row) {
  struct In {
    float po[4], pp[4];
  } a{}, b{}, c{}, d{};
#pragma unroll 1
  for (int r = X.ra - 3; r < X.rb; ++r) {
    const int gi = X.J.i0 + 1 + r;
    const bool in = r + 3 < X.rb && gi >= 0 && gi < X.nr;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool use = in && ln.use[q];
      const size_t g = static_cast<size_t>(gi) * X.nt + X.gj0 + q;
      d.po[q] = use ? __ldg(X.S.p_obs + g) : 0.0f;
      d.pp[q] = use ? __ldg(X.S.p_pred + g) : 0.0f;
    }
    if (r >= X.ra) row(r, a.po, a.pp);
    a = b;
    b = c;
    c = d;
  }
}

// Warp totals of a pass's eight packed sums (the two lanes that only feed neighbours leave theirs
// out), for the decider.  LOW: in pairs, for the long runs of tall CTAs (with plain warp totals their
// reported residual was 1.5 times as far from 64 bits as the streaming solve's; now 0.8 times).
template <bool LOW = false>
__device__ __forceinline__ void chip_store_sums(const ChipCta &X, const f32x2 (&v)[8], bool own) {
  float t[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    float x, y;
    upk(v[q], x, y);
    t[q] = own ? x + y : 0.0f;
  }
  float low = 0.0f;
  const float tot = LOW ? warp_sum8_pair(t, low) : warp_sum8(t);
  if (X.lane < 8) X.sh.part[X.warp][X.lane] = tot;
  if (LOW && X.lane < 8) X.sh.low[X.warp][X.lane] = low;
}

// The decider warp: the balancing constants, every pass's decision and the gather's final state.
template <int NW>
__device__ __forceinline__ void chip_decider(const ChipCta &X) {
  const Ctl &c = X.c;
  const ChipJob &J = X.J;
  const Shot &S = X.S;
  ChipShared &sh = X.sh;
  State *const st = X.st;
  const int lane = X.lane, nr = X.nr, nt = X.nt, cta = X.cta;
  const float rdx = S.rdx, rdt = S.rdt;
  double *const acc = acc_of(c, J.gather);
  constexpr int kSlow = kChipSets * kChipSpread * kChipVals;  // doubles of the FP64 exchange, then the words
  static_assert(kSlow + kChipWordSets * kChipWordCopies * kChipWords <= kAccBufs * kSpread * kAcc, "a gather's accumulators");
  unsigned long long *const words = reinterpret_cast<unsigned long long *>(acc + kSlow);
  // the balancing sums: f, f^2, |Pcal| + |Pobs|, Pcal - Pobs
  bar_all<2, NW>();
  double v = 0.0;
  if ((lane & 7) < 4) {
    double p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = sh.dpart[(lane >> 3) + 4 * i][lane & 7];
    v = (p[0] + p[1]) + (p[2] + p[3]);
  }
  v = sum_groups(v);
  unsigned step = 1;
  int set = 0;
  bool ok = chip_exchange(c, st, acc, set, cta, J.group, step, lane < 8, v, v);
  DecidePrep pr;
  pr.k = 0;
  double m4[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) m4[q] = __shfl_sync(0xffffffffu, v, q);
  const double N = static_cast<double>(nr) * nt;
  const double fmean = c.balance ? m4[0] / N : 0.0;
  pr.fnorm = sqrt(fmax(m4[1] - 2.0 * fmean * m4[0] + N * fmean * fmean, 0.0));
  pr.alpha = c.alpha0 > 0.0 ? c.alpha0 : (c.linesearch ? 1.0 / sqrt(c.delta * S.lambda) : 1.0 / sqrt(S.lambda));
  pr.beta_fixed = 1.0 / (S.lambda * pr.alpha);
  pr.theta = 1.0;
  pr.coef = 0.0;  // pass 0: phi^0 is the initial potential
  // the values of the next pass, each written four times (lane 4 q + i: copy i of value q)
  auto publish_sc = [&](float (&dst)[6][4], float alpha, float coef, float theta, float inv) {
    const int q = lane >> 2;
    if (lane < 16) dst[q][lane & 3] = q == 0 ? alpha : q == 1 ? coef : q == 2 ? theta : inv;
  };
  publish_sc(sh.sc, static_cast<float>(pr.alpha), 0.0f, 1.0f, 1.0f / (1.0f + static_cast<float>(c.eps * pr.alpha)));
  if (lane >= 16 && lane < 24) sh.sc[lane >> 2][lane & 3] = lane < 20 ? rdx : rdt;
  // a gather whose sums left the range of FP32 is handed back: the streaming solve adds them in FP64
  const bool summed = balance_in_range(m4, N);
  bool done = !summed;
  int status = summed ? ST_OK : ST_NONFINITE;
  if (lane == 0) {
    sh.fmean = static_cast<float>(fmean);
    sh.done = done;
    sh.status = status;
    if (!ok) sh.bad = 1;
  }
  bar_all<4, NW>();
  int trials = 0;
  double r_feas = -1.0, r_step = -1.0;
  const bool quick = c.linesearch && c.debug_fault != 1;
  // fixed-point exponents of the two families for the next fast exchange
  int fset = 0, e_p = 0, e_g = 0;
  unsigned long long x0 = 0, y0 = 0, x1 = 0, y1 = 0;  // the totals last read from set fset, from the other
  bool scaled = false;
  const double xl = xi_power(c.xi);
  constexpr unsigned FULL = 0xffffffffu;
  while (ok && !done) {
    const QuickPrep qp = step_prep(c, pr, xl);  // overlaps the pass
    // passes with residual sums (and those without a scale yet) take the FP64 exchange
    const bool check = c.tol > 0.0 && (pr.k + 1) % c.check_every == 0;
    bool slow = !scaled || check || pr.k + 1 >= c.max_iter;
    bar_all<2, NW>();
    float hi, lo, f = 0.0f;
    chip_block_pair<NW == kTallWorkers>(sh.part, sh.low, hi, lo);
    FastTotal ft;
    const int sa = 24 - ((lane & 7) < 3 ? e_p : e_g);
    // The decision's instructions have left the instruction cache since the last pass (1300 cycles
    // against 300): they run once for nothing (into sh.warm) while the other CTAs' sums arrive.
    int w = -1;
    if (!slow) chip_fast_add(c, words, fset, cta, hi, lo, sa);
#pragma unroll 1
    for (int real = slow ? 2 : 0; real < 2; ++real) {
      if (real) {
        ok = chip_fast_poll(words, fset, J.group, sa, x0, y0, ft);
        f = ft.v;
      } else {
        f = hi;
      }
      w = quick ? quick_decide(c, qp, f) : -1;
      publish_sc(real ? sh.sc : sh.warm, __shfl_sync(FULL, pr.alpha_lf, w & 31), __shfl_sync(FULL, pr.coef_lf, w & 31),
                 __shfl_sync(FULL, pr.theta_lf, w & 31), __shfl_sync(FULL, pr.inv_lf, w & 31));
    }
    if (!slow) {
      fset ^= 1;
      const unsigned long long tx = x0, ty = y0;  // the other set's
      x0 = x1;
      y0 = y1;
      x1 = tx;
      y1 = ty;
      slow = !ft.fits;
    }
    if (ok && slow) {
      ++step;
      set = (set + 1) % kChipSets;
      ok = chip_exchange(c, st, acc, set, cta, J.group, step, lane < 16, static_cast<double>(lane < 8 ? hi : lo), v);
      f = cut_f32(v);
      w = quick && !check ? quick_decide(c, qp, f) : -1;
      if (w >= 0)
        publish_sc(sh.sc, __shfl_sync(FULL, pr.alpha_lf, w), __shfl_sync(FULL, pr.coef_lf, w),
                   __shfl_sync(FULL, pr.theta_lf, w), __shfl_sync(FULL, pr.inv_lf, w));
    }
    if (!ok) {
      if (lane == 0) sh.bad = 1;
      bar_all<4, NW>();
      break;
    }
    if (!slow && (w < 0 || c.trace))
      v = fma(static_cast<double>(ft.b), 0x1p-46, static_cast<double>(ft.a)) * __hiloint2double((1023 - sa) << 20, 0);
    if (w >= 0) {
      done = pr.k + 1 >= c.max_iter;
      if (lane == 0) sh.done = done;
      bar_all<4, NW>();
      trials += w + 1;
      if (c.trace && cta == 0) {
        Decision o;
        o.alpha = __shfl_sync(FULL, pr.alpha_l, w);
        o.theta = __shfl_sync(FULL, pr.s_lane, w);
        o.trials_now = w + 1;
        const double ppp = __shfl_sync(FULL, v, 0);
        if (lane == 0) write_trace(c, J.gather, pr.k, o, ppp, pr.fnorm);
      }
      pr.alpha = __shfl_sync(FULL, pr.alpha_l, w);
      pr.theta = __shfl_sync(FULL, pr.s_lane, w);
      pr.coef = __shfl_sync(FULL, pr.coef_l, w);
      ++pr.k;
    } else {
      double a_[9];
#pragma unroll
      for (int q = 0; q < 6; ++q) a_[q] = __shfl_sync(0xffffffffu, v, q);
      a_[6] = 0.0;
      a_[7] = __shfl_sync(0xffffffffu, v, 6);
      a_[8] = __shfl_sync(0xffffffffu, v, 7);
      decide_prep_lanes(c, pr);
      const Decision o = decide_core(c, pr, a_);
      trials += o.trials_now;
      done = o.done;
      status = o.status;
      if (o.status == ST_OK) publish_sc(sh.sc, o.alpha_f, o.coef_f, o.theta_f, o.inv_f);
      if (lane == 0) {
        sh.status = o.status;
        sh.done = o.done;
      }
      bar_all<4, NW>();
      if (cta == 0 && lane == 0) write_trace(c, J.gather, pr.k, o, a_[0], pr.fnorm);
      if (o.checked && cta == 0) residuals(pr, a_, r_feas, r_step);
      if (o.status == ST_OK) {
        pr.k = o.k_new;
        pr.alpha = o.alpha;
        pr.theta = o.theta;
        pr.coef = o.coef;
      }
    }
    if (sh.bad) ok = false;  // a worker's wait ran out
    {
      const float p2 = fmaxf(__shfl_sync(FULL, f, 0), __shfl_sync(FULL, f, 2));
      const float g2 = fmaxf(__shfl_sync(FULL, f, 3), __shfl_sync(FULL, f, 5));
      scaled = p2 > 0x1p-60f && p2 < 0x1p60f && g2 > 0x1p-60f && g2 < 0x1p60f;
      e_p = (__float_as_int(p2) >> 23) - 127;
      e_g = (__float_as_int(g2) >> 23) - 127;
    }
  }
  // the last pass's sums (or, when no pass ran, the balancing ones, which nobody reads)
  const double s_p2 = __shfl_sync(0xffffffffu, v, 0), s_u2 = __shfl_sync(0xffffffffu, v, 6),
               s_du2 = __shfl_sync(0xffffffffu, v, 7);
  double gap = 0.0;
  if (ok && status == ST_OK) {  // the finalize pass's sums
    bar_all<2, NW>();
    const double mine = chip_block_total(sh);
    ++step;
    set = (set + 1) % kChipSets;
    ok = chip_exchange(c, st, acc, set, cta, J.group, step, lane < 16, mine, gap);
  }
  if (!ok && lane == 0) atomicExch(c.error, 1);
  double g4[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    g4[q] = __shfl_sync(0xffffffffu, gap, q) + __shfl_sync(0xffffffffu, gap, 4 + q);
  if (ok && cta == 0 && lane == 0) {
    st->k = pr.k;
    st->trials = trials;
    st->status = status;
    st->alpha = pr.alpha;
    st->theta = pr.theta;
    st->coef = pr.coef;
    st->fmean = fmean;
    st->fnorm = pr.fnorm;
    st->mass_mu = S.area * 0.5 * (m4[2] + m4[3]);
    st->mass_nu = S.area * 0.5 * (m4[2] - m4[3]);
    st->imbalance = S.area * m4[3];
    st->r_feas = r_feas;
    st->r_step = r_step;
    st->s_p2 = s_p2;
    st->s_u2 = s_u2;
    st->s_du2 = s_du2;
    for (int q = 0; q < 4; ++q) st->gap_sums[q] = g4[q];
    st->done = 1;
    atomicAdd(c.n_done, 1);
  }
}

// A worker warp with the arithmetic of the tile pass.
template <bool ISO>
__device__ __forceinline__ void chip_worker(const ChipCta &X) {
  const Ctl &c = X.c;
  const ChipJob &J = X.J;
  const Shot &S = X.S;
  ChipShared &sh = X.sh;
  const int lane = X.lane, warp = X.warp, nr = X.nr, nt = X.nt, ntp = X.ntp, n = X.n, ra = X.ra, rb = X.rb;
  const int gj0 = X.gj0;
  const float rdx = S.rdx, rdt = S.rdt;
  // shared memory, this lane's column of every row: planes div u, q, f; then the boundary rows
  const unsigned plane = X.smem;
  const unsigned bound = plane + 3 * kChipPlane;  // + 0: phi^k of a run's last row
  constexpr unsigned kBUx = kChipBound;           // u^{k+1} (x) of a run's first row
  constexpr unsigned kBP = 2 * kChipBound, kBQ = 3 * kChipBound;  // p, q of a run's last row
  // exchange buffers
  PacketMem *const xrow = reinterpret_cast<PacketMem *>(S.f), *const xcol = xrow + chip_row_packets(J.segs, ntp);
  const size_t xrow_set = static_cast<size_t>(J.segs) * 2 * ntp, xcol_set = static_cast<size_t>(J.strips) * 2 * nr;
  const ChipLane ln = chip_lane(X);
  const bool own_lane = ln.own;
  const Q4 rdt_m = q4(ln.rm[0], ln.rm[1], ln.rm[2], ln.rm[3]);
  auto row_addr = [&](int r) { return plane + static_cast<unsigned>(r) * kChipRowBytes; };
  const unsigned brow = bound + static_cast<unsigned>(warp) * kChipRowBytes;  // this run's boundary row

  // div u and q of the strip's first and last-but-one sample go to the neighbouring strips, those of
  // the segment's first and last-but-one row to the neighbouring segments
  const bool edge_lane = lane == 1 || lane == 30;
  PacketMem *const xedge = xcol + (static_cast<size_t>(J.strip) * 2 + (lane == 30 ? 1 : 0)) * nr + J.i0 - 2;
  PacketMem *const xmine = xrow + static_cast<size_t>(J.seg) * 2 * ntp + gj0;
  auto put_row = [&](int which, int parity, const Q4 &d, const Q4 &q, int tag) {
    float d_[4], q_[4];
    un4(d, d_);
    un4(q, q_);
    PacketMem *const o = xmine + (parity ? xrow_set : 0) + which * ntp;
    if (own_lane && gj0 < ntp && J.segs > 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i) put_packet(o + i, d_[i], q_[i], tag);
    }
  };
  // this CTA's packets start without a tag
  for (int r = max(ra, 2); r < min(rb, J.h + 2); ++r) {
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      if (edge_lane) put_packet(xedge + (m ? xcol_set : 0) + r, 0.0f, 0.0f, 0);
      if (r == 2) put_row(0, m, q4s(0.0f), q4s(0.0f), 0);
      if (r == J.h) put_row(1, m, q4s(0.0f), q4s(0.0f), 0);
    }
  }
  // the halo sample that this lane fetches: even lanes sample -2, odd ones sample 120 of the
  // run's row lane / 2 (rows 0 and n - 1 come whole)
  const PacketMem *halo_src = nullptr;
  unsigned halo_dst = 0;
  {
    const int r = ra + (lane >> 1), side = lane & 1, gi = J.i0 - 2 + r, strip = J.strip + (side ? 1 : -1);
    if (r < rb && r > 0 && r < n - 1 && gi >= 0 && gi < nr && strip >= 0 && strip < J.strips) {
      halo_src = xcol + (static_cast<size_t>(strip) * 2 + (side ? 0 : 1)) * nr + gi;
      halo_dst = row_addr(r) - 16u * lane + (side ? 4 * 124 : 4 * 2);
    }
  }

  // ---- inputs, warm start and the balancing sums
  {
    BalanceSums sums;
    chip_input_rows(X, ln, [&](int r, const float (&po)[4], const float (&pp)[4]) {
      const int gi = J.i0 - 2 + r;
      const bool rin = gi >= 0 && gi < nr, rown = r >= 2 && r < J.h + 2;
      float f[4], ph[4], ux[4], ut[4], d[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int gj = gj0 + q;
        const bool in = rin && ln.use[q];
        const size_t g = static_cast<size_t>(gi) * nt + gj;
        f[q] = pp[q] - po[q];
        ph[q] = in && S.phi_init ? S.phi_init[g] : 0.0f;
        ux[q] = ut[q] = d[q] = 0.0f;
        if (in && S.m_init) {
          ux[q] = chip_init_flux(X, 0, gi, gj);
          ut[q] = chip_init_flux(X, 1, gi, gj);
          d[q] = fmaf(chip_init_flux(X, 0, gi + 1, gj) - ux[q], rdx, (chip_init_flux(X, 1, gi, gj + 1) - ut[q]) * rdt);
        }
        if (in && rown && own_lane) sums.add(po[q], pp[q]);
      }
      const unsigned a = row_addr(r);
      sts4(a, q4(d[0], d[1], d[2], d[3]));
      sts4<kChipPlane>(a, q4s(0.0f));
      sts4<2 * kChipPlane>(a, q4(f[0], f[1], f[2], f[3]));
      tmem_store_row(X.taddr + (r - ra) * kChipRowCols,
                     {q4(ux[0], ux[1], ux[2], ux[3]), q4(ut[0], ut[1], ut[2], ut[3]),
                      q4(ph[0], ph[1], ph[2], ph[3])});
    });
    tmem_stores_done();
    sums.store(X);
    bar_all<2>();
    bar_all<4>();
    const float fm = sh.fmean;
    for (int r = ra; r < rb; ++r) {  // the balanced f, zero outside the gather
      const int gi = J.i0 - 2 + r;
      const bool rin = gi >= 0 && gi < nr;
      float x[4];
      un4(lds4<2 * kChipPlane>(row_addr(r)), x);
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = rin && ln.use[q] ? x[q] - fm : 0.0f;
      sts4<2 * kChipPlane>(row_addr(r), q4(x[0], x[1], x[2], x[3]));
    }
  }

  // row r with phi^k completed from the last pass's div u and q (received ones at the halo)
  auto dual = [&](int r, const Q4 &cf, const Q4 &th) -> RowState {
    RowState s = tmem_load_row(X.taddr + (r - ra) * kChipRowCols);
    const unsigned a = row_addr(r);
    const Q4 p = add4(lds4(a), lds4<2 * kChipPlane>(a));
    s.ph = fma4(cf, fma4(th, lds4<kChipPlane>(a), p), s.ph);
    return s;
  };
  const unsigned sc_addr = smem_u32(&sh.sc[0][0]);

  int k = 0;
  while (!sh.bad) {
    if (sh.done) break;
    const float alpha = sh.sc[0][0];
    const Q4 al4 = lds_pair(sc_addr), cf = lds_pair<16>(sc_addr), th = lds_pair<32>(sc_addr);
    const Q4 inv4 = lds_pair<48>(sc_addr), rdx4 = lds_pair<64>(sc_addr), rdt4 = lds_pair<80>(sc_addr);
    const bool need_res = (c.tol > 0.0 && (k + 1) % c.check_every == 0) || k + 1 >= c.max_iter;
    f32x2 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 0ull;

    // u^{k+1} of a row from phi^k of it and of the row above
    // (PLAIN: an owned row away from the gather's first receiver, no residual sums)
    auto prox_row = [&](auto plain, int r, const RowState &s, const Q4 &ph_up, Q4 &nx, Q4 &nv) {
      constexpr bool PLAIN = decltype(plain)::value;
      const int gi = J.i0 - 2 + r;
      const Q4 rx = PLAIN || (gi > 0 && gi < nr) ? rdx4 : q4s(0.0f);
      const Q4 gx = mul4(sub4(s.ph, ph_up), rx), gt = mul4(diff_left(s.ph), rdt_m);
      chip_prox<ISO>(s.ux, s.ut, gx, gt, alpha, al4, inv4, nx, nv);
      if (!PLAIN && need_res && r >= 2 && r < J.h + 2) {
        const Q4 dx_ = sub4(nx, s.ux), dt_ = sub4(nv, s.ut);
        v[6] = fma2(nx.a, nx.a, fma2(nv.a, nv.a, v[6]));
        v[6] = fma2(nx.b, nx.b, fma2(nv.b, nv.b, v[6]));
        v[7] = fma2(dx_.a, dx_.a, fma2(dt_.a, dt_.a, v[7]));
        v[7] = fma2(dx_.b, dx_.b, fma2(dt_.b, dt_.b, v[7]));
      }
    };
    PacketMem *const xe = xedge + (k & 1 ? xcol_set : 0);
    const int tag = k + 1;
    // p, q of a row, its sums that need no other row, and the halo cells others hold
    // (PLAIN: an owned row that no other segment holds as halo)
    auto flux_row = [&](auto plain, int r, const Q4 &ux, const Q4 &ut, const Q4 &ux_dn, Q4 &p, Q4 &q) {
      constexpr bool PLAIN = decltype(plain)::value;
      const unsigned a = row_addr(r);
      const Q4 dn = div4(sub4(ux_dn, ux), diff_right(ut), rdx4, rdt4);
      p = add4(dn, lds4<2 * kChipPlane>(a));
      q = sub4(dn, lds4(a));
      sts4(a, dn);
      sts4<kChipPlane>(a, q);
      if (PLAIN || (r >= 2 && r < J.h + 2)) {
        const Q4 gp = mul4(diff_left(p), rdt_m), gq = mul4(diff_left(q), rdt_m);
        v[0] = fma2(p.b, p.b, fma2(p.a, p.a, v[0]));
        v[1] = fma2(p.b, q.b, fma2(p.a, q.a, v[1]));
        v[2] = fma2(q.b, q.b, fma2(q.a, q.a, v[2]));
        v[3] = fma2(gp.b, gp.b, fma2(gp.a, gp.a, v[3]));
        v[4] = fma2(gp.b, gq.b, fma2(gp.a, gq.a, v[4]));
        v[5] = fma2(gq.b, gq.b, fma2(gq.a, gq.a, v[5]));
        const f32x2 de = lane == 30 ? dn.b : dn.a, qe = lane == 30 ? q.b : q.a;
        float d0, q0, unused;
        upk(de, d0, unused);
        upk(qe, q0, unused);
        if (edge_lane) put_packet(xe + r, d0, q0, tag);
        if (!PLAIN && r == 2) put_row(0, k & 1, dn, q, tag);
        if (!PLAIN && r == J.h) put_row(1, k & 1, dn, q, tag);
      }
    };
    // receiver-direction gradient sums of row r from p, q of it and of the row above
    auto grad_row = [&](auto plain, int r, const Q4 &p, const Q4 &q, const Q4 &pu, const Q4 &qu) {
      if (!decltype(plain)::value && !(r >= 2 && r < J.h + 2 && J.i0 - 2 + r > 0)) return;
      const Q4 gp = mul4(sub4(p, pu), rdx4), gq = mul4(sub4(q, qu), rdx4);
      v[3] = fma2(gp.b, gp.b, fma2(gp.a, gp.a, v[3]));
      v[4] = fma2(gp.b, gq.b, fma2(gp.a, gq.a, v[4]));
      v[5] = fma2(gq.b, gq.b, fma2(gq.a, gq.a, v[5]));
    };

    // ---- the run, upwards: row r's phi^k, then row r + 1's flux and sums.  The rows go two
    // per trip, so what one row hands to the next changes registers instead of being copied.
    struct Carry {
      RowState cur;          // the row below with phi^k completed (u still u^k)
      Q4 ux_dn, p_dn, q_dn;  // of the row below that: u^{k+1} (x), p, q
    };
    auto step = [&](auto plain, int r, const Carry &in, Carry &out) {
      out.cur = dual(r, cf, th);
      Q4 nx, nv;
      prox_row(plain, r + 1, in.cur, out.cur.ph, nx, nv);
      tmem_store_row(X.taddr + (r + 1 - ra) * kChipRowCols, {nx, nv, in.cur.ph});
      out.ux_dn = nx;
      flux_row(plain, r + 1, nx, nv, in.ux_dn, out.p_dn, out.q_dn);
      if (r + 2 < rb - 1) grad_row(plain, r + 2, in.p_dn, in.q_dn, out.p_dn, out.q_dn);
    };
    const BoolConst<true> plain{};
    const BoolConst<false> any{};
    Carry x, y;
    x.p_dn = x.q_dn = x.ux_dn = q4s(0.0f);
    if (ra < rb) {
      const RowState s = dual(rb - 1, cf, th);
      sts4(brow, s.ph);
      x.cur = s;
      if (ra < rb - 1) {  // the last row's flux waits for the next run's first row
        x.cur = dual(rb - 2, cf, th);
        Q4 nx, nv;
        prox_row(any, rb - 1, s, x.cur.ph, nx, nv);
        tmem_store_row(X.taddr + (rb - 1 - ra) * kChipRowCols, {nx, nv, s.ph});
        x.ux_dn = nx;
      }
      int r = rb - 3;
#pragma unroll 1
      while (r >= ra) {
        if (!need_res && r + 1 < J.h && r >= 3 && r > ra) {  // rows r + 1 and r are plain
          step(plain, r, x, y);
          step(plain, r - 1, y, x);
          r -= 2;
        } else {
          step(any, r, x, y);
          x = y;
          --r;
        }
      }
    }
    // ---- the first row of the run: phi^k of the row above comes from the run before
    bar_workers();
    Q4 p_a = q4s(0.0f), q_a = q4s(0.0f);  // p, q of row ra
    if (ra < rb) {
      if (ra > 0) {
        Q4 nx, nv;
        prox_row(any, ra, x.cur, lds4(brow - kChipRowBytes), nx, nv);
        sts4<kBUx>(brow, nx);
        tmem_store_row(X.taddr, {nx, nv, x.cur.ph});
        if (ra < rb - 1) {
          flux_row(any, ra, nx, nv, x.ux_dn, p_a, q_a);
          if (ra + 1 < rb - 1) grad_row(any, ra + 1, x.p_dn, x.q_dn, p_a, q_a);
        }
      } else {
        tmem_store_row(X.taddr, x.cur);  // row 0 carries phi^k only
      }
    }
    tmem_stores_done();
    bar_workers();
    // ---- the last row of the run: u^{k+1} of the row below comes from the next run
    const int L = rb - 1;
    if (ra < rb && L >= 1 && L < n - 1) {
      const RowState s = tmem_load_row(X.taddr + (L - ra) * kChipRowCols);
      Q4 p, q;
      flux_row(any, L, s.ux, s.ut, lds4<kBUx + kChipRowBytes>(brow), p, q);
      sts4<kBP>(brow, p);
      sts4<kBQ>(brow, q);
      if (L == ra) {
        p_a = p;
        q_a = q;
      } else if (L - 1 >= 1) {  // the row above in this run: p = div u + f, q as stored
        const unsigned a = row_addr(L - 1);
        grad_row(any, L, p, q, add4(lds4(a), lds4<2 * kChipPlane>(a)), lds4<kChipPlane>(a));
      }
    }
    bar_workers();
    if (ra < rb && ra >= 2 && ra < n - 1)
      grad_row(any, ra, p_a, q_a, lds4<kBP - kChipRowBytes>(brow), lds4<kBQ - kChipRowBytes>(brow));

    chip_store_sums(X, v, own_lane);
    bar_all_arrive<2>();
    // ---- halo values of the pass: received div u and q
    bool got = true;
    if (ra < rb) {
      Packet e;
      got = poll_warp([&] {
        if (halo_src) e = get_packet(halo_src + (k & 1 ? xcol_set : 0));
        return !halo_src || e.tag == tag;
      });
      if (halo_src) {
        sts1(halo_dst, e.x);
        sts1(halo_dst + kChipPlane, e.y);
      }
      for (int w = 0; w < 2; ++w) {
        const int r = w ? n - 1 : 0, gi = J.i0 - 2 + r, seg = J.seg + (w ? 1 : -1);
        if (r < ra || r >= rb || seg < 0 || seg >= J.segs || gi < 0 || gi >= nr) continue;
        const PacketMem *const o = xrow + (k & 1 ? xrow_set : 0) + (static_cast<size_t>(seg) * 2 + (w ? 0 : 1)) * ntp + gj0;
        float d_[4] = {0.f, 0.f, 0.f, 0.f}, q_[4] = {0.f, 0.f, 0.f, 0.f};
        got = poll_warp([&] {
          bool all = true;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (!ln.use[i]) continue;
            const Packet x = get_packet(o + i);
            d_[i] = x.x;
            q_[i] = x.y;
            all = all && x.tag == tag;
          }
          return all;
        }) && got;
        sts4(row_addr(r), q4(d_[0], d_[1], d_[2], d_[3]));
        sts4<kChipPlane>(row_addr(r), q4(q_[0], q_[1], q_[2], q_[3]));
      }
    }
    if (!got && lane == 0) sh.bad = 1;
    bar_all<4>();  // the decision
    ++k;
  }

  // ---- finalize: phi^K, the outputs and the duality gap's sums
  if (!sh.bad && sh.status == ST_OK) {
    const Q4 cf = lds_pair<16>(sc_addr), th = lds_pair<32>(sc_addr);
    Sum2 t[4];
    for (int r = ra; r < rb; ++r) {
      const RowState s = dual(r, cf, th);
      tmem_store_row(X.taddr + (r - ra) * kChipRowCols, s);
      if (r == rb - 1) sts4(brow, s.ph);
    }
    tmem_stores_done();
    bar_workers();
    const bool vec = chip_vec_out(X);
    Q4 up = ra < rb && ra > 0 ? lds4(brow - kChipRowBytes) : q4s(0.0f);
    for (int r = ra; r < rb; ++r) {
      const RowState s = tmem_load_row(X.taddr + (r - ra) * kChipRowCols);
      const Q4 gtv = diff_left(s.ph);
      if (r >= 2 && r < J.h + 2 && own_lane)
        chip_output_row<ISO>(X, vec, J.i0 - 2 + r, s.ux, s.ut, s.ph, up, gtv, lds4<2 * kChipPlane>(row_addr(r)), t);
      up = s.ph;
    }
    chip_store_gap(X, t);
    bar_all_arrive<2>();
  }
}

}  // namespace emd
