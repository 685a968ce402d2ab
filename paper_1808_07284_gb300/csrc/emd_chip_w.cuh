// The on-chip solve of emd_chip.cuh with the arithmetic of the marching pass (emd_march.cuh): the
// dual step is taken from the extrapolated flux w = u^k + theta (u^k - u^{k-1}), so u^{k-1} is kept
// in place of div u and q.  Gathers and batches that would stream through the marching pass are
// solved in this form, those that would take the tile pass in the other one, so the rounding of
// a size's iterates does not depend on where its state lives.
//
// Storage.  u^m lies in slot m & 1 of a row: pass k reads u^k and u^{k-1} and writes u^{k+1} over
// the latter.  Tensor memory holds the flux of a run's first eight (tall: ten) rows, 16 columns each;
// shared memory gives every warp row slots for phi, the flux of further rows (four slots a row)
// and f.  CTAs of up to 128 rows keep everything there.
//
// Tall CTAs (up to 385 rows, for gathers of up to about 6 million cells) have eleven worker warps
// with more registers: phi stays in shared memory, and the flux of the rows past those ten and f stream from a buffer of the CTA's own
// in global memory, which stays in L2: about 21 B per cell and pass on 8000 x 648, and none from
// DRAM.  A row's streamed values are loaded one row ahead, into registers.
//
// Halo.  phi^k of the halo rows -2 and h and samples -2 and 120 needs u of one row or sample more:
// both components of row -2, the x flux of row h + 1 and the t flux of samples -2 and 121 come
// from the neighbours after every pass; the rest of the halo's flux is computed here (with the
// isotropic cost, whose shrinkage needs both components, ux of sample -2 comes too).
//
// Measured, us per pass, against the streaming solve: 480 x 4000 8.2 (20.4): a row of a warp takes
// 240 cycles of its scheduler, about 200 of them on the FMA pipe, and the pass boundary 3500 of
// 17000 cycles.  648 x 8000, tall, 22.8 (43.7): 350 cycles a row, three warps a scheduler and the streamed
// values' L2 latency.
#pragma once

#include "emd_chip.cuh"

namespace emd {

constexpr int kWRowCols = 16;      // tensor memory columns of a row: two slots of ux, ut

// The storage of a CTA of NW worker warps.
template <int NW>
struct WLayout {
  static constexpr int kSmemRows = static_cast<int>((kChipSmem - 128) / kChipRowBytes);
  static constexpr int kTmemCols = 512 / ((NW + 3) / 4) / kWRowCols * kWRowCols;  // of a warp
  static constexpr int kTmemRows = kTmemCols / kWRowCols;     // rows of a run whose flux lies there
  static constexpr int kSlots = (kSmemRows - 3 * NW - 2 * (NW + 1)) / NW;  // row slots of a warp
  static constexpr int kMaxRows = NW * kSlots;                // staged rows of a CTA at most
  // boundary rows: phi^k of every run's last row, p, q of it, u (x) of every run's first row in
  // two slots (and of the row below the last run)
  static constexpr unsigned kBound = kMaxRows * kChipRowBytes;
  static constexpr unsigned kBP = NW * kChipRowBytes, kBQ = 2 * kBP, kBUx = 3 * kBP;
  static constexpr unsigned kBUxSlot = (NW + 1) * kChipRowBytes;
};
static_assert(kWMaxRows == WLayout<kTallWorkers>::kMaxRows, "staged rows of a tall CTA at most");
static_assert(2 * ((kChipMaxRows + kChipWorkers - 1) / kChipWorkers) + 4 <= WLayout<kChipWorkers>::kSlots &&
                  (kChipMaxRows + kChipWorkers - 1) / kChipWorkers <= WLayout<kChipWorkers>::kTmemRows + 1,
              "a run of 9 rows has no streamed values");

__device__ __forceinline__ Q4 ldg4(const float *p) {
  const float4 t = __ldcg(reinterpret_cast<const float4 *>(p));
  return q4(t.x, t.y, t.z, t.w);
}
__device__ __forceinline__ void stg4(float *p, const Q4 &v) {
  float o[4];
  un4(v, o);
  __stcg(reinterpret_cast<float4 *>(p), make_float4(o[0], o[1], o[2], o[3]));
}

// A row's flux slot in tensor memory: ux, ut.
__device__ __forceinline__ void tmem_load_flux(uint32_t addr, Q4 &ux, Q4 &ut) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(addr)
      : "memory");
  ux = q4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
  ut = q4(__uint_as_float(r[4]), __uint_as_float(r[5]), __uint_as_float(r[6]), __uint_as_float(r[7]));
}
// Both slots, with one wait.
__device__ __forceinline__ void tmem_load_flux2(uint32_t a0, uint32_t a1, Q4 &x0, Q4 &t0, Q4 &x1, Q4 &t1) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
        "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15])
      : "r"(a0), "r"(a1)
      : "memory");
  auto g = [&](int i) { return q4(__uint_as_float(r[i]), __uint_as_float(r[i + 1]), __uint_as_float(r[i + 2]),
                                  __uint_as_float(r[i + 3])); };
  x0 = g(0);
  t0 = g(4);
  x1 = g(8);
  t1 = g(12);
}
__device__ __forceinline__ void tmem_store_flux(uint32_t addr, const Q4 &ux, const Q4 &ut) {
  float x[4], t[4];
  un4(ux, x);
  un4(ut, t);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(addr), "f"(x[0]),
               "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(t[3])
               : "memory");
}

// Four words of tensor memory per lane.
__device__ __forceinline__ Q4 tmem_load_quad(uint32_t addr) {
  uint32_t r[4];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
      : "r"(addr)
      : "memory");
  return q4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
}
__device__ __forceinline__ void tmem_store_quad(uint32_t addr, const Q4 &v) {
  float x[4];
  un4(v, x);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(addr), "f"(x[0]), "f"(x[1]),
               "f"(x[2]), "f"(x[3])
               : "memory");
}

// A worker warp with the arithmetic of the marching pass.
template <bool ISO, bool TALL, int NW>
__device__ __forceinline__ void chip_worker_w(const ChipCta &X) {
  using LY = WLayout<NW>;
  constexpr int kWSlots = LY::kSlots, kWTmemRows = LY::kTmemRows;
  constexpr unsigned kWBound = LY::kBound, kWBP = LY::kBP, kWBQ = LY::kBQ, kWBUx = LY::kBUx, kWBUxSlot = LY::kBUxSlot;
  const Ctl &c = X.c;
  const ChipJob &J = X.J;
  const Shot &S = X.S;
  ChipShared &sh = X.sh;
  const int lane = X.lane, warp = X.warp, nr = X.nr, ntp = X.ntp, n = X.n, ra = X.ra, rb = X.rb;
  const int gj0 = X.gj0, run = rb - ra;
  constexpr int kRounds = (kWSlots + 15) / 16;  // two edge samples of 16 rows are fetched in a round
  const ChipLane ln = chip_lane(X);
  const bool own_lane = ln.own;
  const Q4 rdt_m = q4(ln.rm[0], ln.rm[1], ln.rm[2], ln.rm[3]);

  // ---- where the rows of this run live
  const unsigned slots = X.smem + static_cast<unsigned>(warp) * (kWSlots * kChipRowBytes);
  const unsigned a_ph = slots;               // phi of row ra
  int nf = 1 << 30;                          // rows of the run from nf on have their f streamed
  unsigned a_u = 0, a_f;                     // flux, f of row ra (if those were in slots)
  float *tall = nullptr;                     // streamed values ux0, ut0, ux1, ut1, f: row r at + kTallRow r
  if (TALL) {
    nf = min(run, kWSlots - run);
    a_f = slots + static_cast<unsigned>(run) * kChipRowBytes;
    tall = S.f + chip_exchange_bytes(J.segs, J.strips, nr, ntp) / 4 + X.cta * chip_w_tall_floats(J.rows) + 4 * lane;
  } else {
    constexpr unsigned kRun = (kChipMaxRows + kChipWorkers - 1) / kChipWorkers;
    a_f = slots + kRun * kChipRowBytes;
    a_u = slots + (2 * kRun - 4 * kWTmemRows) * kChipRowBytes;
  }
  auto u_slot = [&](int i, int m) { return a_u + static_cast<unsigned>(4 * i + 2 * m) * kChipRowBytes; };
  auto load_flux = [&](int r, int m, Q4 &ux, Q4 &ut) {
    const int i = r - ra;
    if (i < kWTmemRows) {
      tmem_load_flux(X.taddr + i * kWRowCols + 8 * m, ux, ut);
    } else if (!TALL) {
      ux = lds4(u_slot(i, m));
      ut = lds4<kChipRowBytes>(u_slot(i, m));
    } else {
      ux = ldg4(tall + r * kTallRow + 256 * m);
      ut = ldg4(tall + r * kTallRow + 256 * m + 128);
    }
  };
  auto store_flux = [&](int r, int m, const Q4 &ux, const Q4 &ut) {
    const int i = r - ra;
    if (i < kWTmemRows) {
      tmem_store_flux(X.taddr + i * kWRowCols + 8 * m, ux, ut);
    } else if (!TALL) {
      sts4(u_slot(i, m), ux);
      sts4<kChipRowBytes>(u_slot(i, m), ut);
    } else {
      stg4(tall + r * kTallRow + 256 * m, ux);
      stg4(tall + r * kTallRow + 256 * m + 128, ut);
    }
  };
  auto phi_addr = [&](int r) { return a_ph + static_cast<unsigned>(r - ra) * kChipRowBytes; };
  auto load_f = [&](int r) {
    return !TALL || r - ra < nf ? lds4(a_f + static_cast<unsigned>(r - ra) * kChipRowBytes)
                                : ldg4(tall + r * kTallRow + 512);
  };
  auto store_f = [&](int r, const Q4 &v) {
    if (!TALL || r - ra < nf)
      sts4(a_f + static_cast<unsigned>(r - ra) * kChipRowBytes, v);
    else
      stg4(tall + r * kTallRow + 512, v);
  };
  const unsigned brow = X.smem + kWBound + static_cast<unsigned>(warp) * kChipRowBytes;  // this run's boundary row
  auto bux = [&](int m) { return brow + kWBUx + static_cast<unsigned>(m) * kWBUxSlot; };
  // exchange buffers
  PacketMem *const xrow = reinterpret_cast<PacketMem *>(S.f), *const xcol = xrow + chip_row_packets(J.segs, ntp);
  const size_t xrow_set = static_cast<size_t>(J.segs) * 2 * ntp, xcol_set = static_cast<size_t>(J.strips) * 2 * nr;
  const bool edge_lane = lane == 1 || lane == 30;
  PacketMem *const xedge = xcol + (static_cast<size_t>(J.strip) * 2 + (lane == 30 ? 1 : 0)) * nr + J.i0 - 2;
  PacketMem *const xmine = xrow + static_cast<size_t>(J.seg) * 2 * ntp + gj0;
  auto put_row = [&](int which, int parity, const Q4 &ux, const Q4 &ut, int tag) {
    float x[4], t[4];
    un4(ux, x);
    un4(ut, t);
    PacketMem *const o = xmine + (parity ? xrow_set : 0) + which * ntp;
    if (own_lane && gj0 < ntp && J.segs > 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i) put_packet(o + i, x[i], t[i], tag);
    }
  };
  // this CTA's packets start without a tag
  for (int r = max(ra, 2); r < min(rb, J.h + 2); ++r) {
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      if (edge_lane) put_packet(xedge + (m ? xcol_set : 0) + r, 0.0f, 0.0f, 0);
      if (r == J.h) put_row(0, m, q4s(0.0f), q4s(0.0f), 0);
      if (r == 3) put_row(1, m, q4s(0.0f), q4s(0.0f), 0);
    }
  }

  // ---- inputs, warm start and the balancing sums
  {
    BalanceSums sums;
    chip_input_rows(X, ln, [&](int r, const float (&po)[4], const float (&pp)[4]) {
      const int gi = J.i0 - 2 + r;
      const bool rin = gi >= 0 && gi < nr, rown = r >= 2 && r < J.h + 2;
      float f[4], ph[4], ux[4], ut[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int gj = gj0 + q;
        const bool in = rin && ln.use[q];
        const size_t g = static_cast<size_t>(gi) * X.nt + gj;
        f[q] = pp[q] - po[q];
        ph[q] = in && S.phi_init ? S.phi_init[g] : 0.0f;
        ux[q] = in && S.m_init ? chip_init_flux(X, 0, gi, gj) : 0.0f;
        ut[q] = (in || (lane == 31 && q == 1)) && S.m_init ? chip_init_flux(X, 1, gi, gj) : 0.0f;
        if (in && rown && own_lane) sums.add(po[q], pp[q]);
      }
      const Q4 ux4 = q4(ux[0], ux[1], ux[2], ux[3]), ut4 = q4(ut[0], ut[1], ut[2], ut[3]);
#pragma unroll
      for (int m = 0; m < 2; ++m) {  // u^{-1} := u^0
        store_flux(r, m, ux4, ut4);
        if (r == ra) sts4(bux(m), ux4);
      }
      sts4(phi_addr(r), q4(ph[0], ph[1], ph[2], ph[3]));
      store_f(r, q4(f[0], f[1], f[2], f[3]));
    });
    if (run > 0 && rb == n) {  // the row below the last one: its x flux
      float ux[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        ux[q] = ln.use[q] && S.m_init ? chip_init_flux(X, 0, J.i0 - 2 + n, gj0 + q) : 0.0f;
#pragma unroll
      for (int m = 0; m < 2; ++m) sts4(bux(m) + kChipRowBytes, q4(ux[0], ux[1], ux[2], ux[3]));
    }
    tmem_stores_done();
    sums.store(X);
    bar_all<2, NW>();
    bar_all<4, NW>();
    const float fm = sh.fmean;
    for (int r = ra; r < rb; ++r) {  // the balanced f, zero outside the gather
      const int gi = J.i0 - 2 + r;
      const bool rin = gi >= 0 && gi < nr;
      float x[4];
      un4(load_f(r), x);
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = rin && ln.use[q] ? x[q] - fm : 0.0f;
      store_f(r, q4(x[0], x[1], x[2], x[3]));
    }
  }

  const unsigned sc_addr = smem_u32(&sh.sc[0][0]);

  struct Row {
    Q4 bx, bt, ph, f, wx;  // u^k, the completed phi^k, f (tall), w (x)
  };
  struct Pre {
    Q4 bx, bt, ax, at, f;  // u^k, u^{k-1}, f of a row
  };

  int k = 0;
  while (!sh.bad) {
    if (sh.done) break;
    const int mb = k & 1, mn = mb ^ 1;  // slots of u^k; of u^{k-1}, then u^{k+1}
    const float alpha = sh.sc[0][0];
    const Q4 al4 = lds_pair(sc_addr), cf = lds_pair<16>(sc_addr), th = lds_pair<32>(sc_addr);
    const Q4 inv4 = lds_pair<48>(sc_addr), rdx4 = lds_pair<64>(sc_addr), rdt4 = lds_pair<80>(sc_addr);
    Q4 cfx;
    cfx.a = cfx.b = mul2(cf.a, rdx4.a);
    const bool need_res = (c.tol > 0.0 && (k + 1) % c.check_every == 0) || k + 1 >= c.max_iter;
    f32x2 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 0ull;
    PacketMem *const xe = xedge + (mb ? xcol_set : 0);
    const int tag = k + 1;
    const uint32_t tb = X.taddr + 8 * mb, tn = X.taddr + 8 * mn;

    auto fetch = [&](int r, Pre &p) {
      const int i = r - ra;
      if (i < kWTmemRows) {
        tmem_load_flux2(tb + i * kWRowCols, tn + i * kWRowCols, p.bx, p.bt, p.ax, p.at);
      } else {
        load_flux(r, mb, p.bx, p.bt);
        load_flux(r, mn, p.ax, p.at);
      }
      p.f = load_f(r);
    };
    // phi^k of row r: phi^{k-1} + c (f + div w); wx_dn: w (x) of the row below
    auto dual = [&](unsigned a_phi, const Pre &p, const Q4 &wx_dn, Row &o) {
      const Q4 wt = fma4(th, sub4(p.bt, p.at), p.bt);
      o.wx = fma4(th, sub4(p.bx, p.ax), p.bx);
      const Q4 x = fma4(cf, fma4(diff_right(wt), rdt4, p.f), lds4(a_phi));
      o.ph = fma4(cfx, sub4(wx_dn, o.wx), x);
      o.bx = p.bx;
      o.bt = p.bt;
      if (TALL) o.f = p.f;
    };
    // u^{k+1} of a row from phi^k of it and of the row above
    auto prox = [&](const Row &s, const Q4 &ph_up, const Q4 &rx, Q4 &nx, Q4 &nv) {
      const Q4 gx = mul4(sub4(s.ph, ph_up), rx), gt = mul4(diff_left(s.ph), rdt_m);
      chip_prox<ISO>(s.bx, s.bt, gx, gt, alpha, al4, inv4, nx, nv);
    };
    // the samples of an owned row that the neighbouring strips hold as halo; e: the row's place
    auto give_edge = [&](PacketMem *e, const Q4 &nx, const Q4 &nv) {
      float t[4], x[4];
      un4(nv, t);
      un4(nx, x);
      if (edge_lane) put_packet(e, lane == 30 ? t[2] : t[1], x[2], tag);
    };
    // any row: the flux, stored and handed to the CTAs that hold it as halo
    auto prox_row = [&](int r, const Row &s, const Q4 &ph_up, Q4 &nx, Q4 &nv) {
      const int gi = J.i0 - 2 + r;
      prox(s, ph_up, gi > 0 && gi < nr ? rdx4 : q4s(0.0f), nx, nv);
      store_flux(r, mn, nx, nv);
      sts4(phi_addr(r), s.ph);
      if (r >= 2 && r < J.h + 2) {
        give_edge(xe + r, nx, nv);
        if (r == J.h) put_row(0, mb, nx, nv, tag);
        if (r == 3) put_row(1, mb, nx, nv, tag);
      }
    };
    // p, q of a row and its sums that need no other row; ddx: its step (x)
    auto flux_row = [&](auto plain, int r, const Q4 &nx, const Q4 &nv, const Q4 &bx, const Q4 &bt, const Q4 &f,
                        const Q4 &nx_dn, const Q4 &ddx_dn, Q4 &p, Q4 &q, Q4 &ddx) {
      constexpr bool PLAIN = decltype(plain)::value;
      ddx = sub4(nx, bx);
      const Q4 ddt = sub4(nv, bt);
      p = fma4(rdx4, sub4(nx_dn, nx), fma4(diff_right(nv), rdt4, f));
      q = fma4(rdx4, sub4(ddx_dn, ddx), mul4(diff_right(ddt), rdt4));
      if (PLAIN || (r >= 2 && r < J.h + 2)) {
        const Q4 gp = mul4(diff_left(p), rdt_m), gq = mul4(diff_left(q), rdt_m);
        v[0] = fma2(p.b, p.b, fma2(p.a, p.a, v[0]));
        v[1] = fma2(p.b, q.b, fma2(p.a, q.a, v[1]));
        v[2] = fma2(q.b, q.b, fma2(q.a, q.a, v[2]));
        v[3] = fma2(gp.b, gp.b, fma2(gp.a, gp.a, v[3]));
        v[4] = fma2(gp.b, gq.b, fma2(gp.a, gq.a, v[4]));
        v[5] = fma2(gq.b, gq.b, fma2(gq.a, gq.a, v[5]));
        if (!PLAIN && need_res) {
          v[6] = fma2(nx.a, nx.a, fma2(nv.a, nv.a, v[6]));
          v[6] = fma2(nx.b, nx.b, fma2(nv.b, nv.b, v[6]));
          v[7] = fma2(ddx.a, ddx.a, fma2(ddt.a, ddt.a, v[7]));
          v[7] = fma2(ddx.b, ddx.b, fma2(ddt.b, ddt.b, v[7]));
        }
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

    // ---- the run, upwards: row r's phi^k, then row r + 1's flux and sums, two rows per trip
    const BoolConst<true> plain{};
    const BoolConst<false> any{};
    struct Carry {
      Row cur;                       // the row below
      Q4 nx_dn, ddx_dn, p_dn, q_dn;  // of the row below that: u^{k+1} (x), its step, p, q
      Pre pre;                       // the next row
    };
    auto step = [&](int r, const Carry &in, Carry &out) {  // any rows
      Pre p;
      if (TALL) {
        if (r > ra) fetch(r - 1, out.pre);
      } else {
        fetch(r, p);
      }
      dual(phi_addr(r), TALL ? in.pre : p, in.cur.wx, out.cur);
      Q4 nv;
      prox_row(r + 1, in.cur, out.cur.ph, out.nx_dn, nv);
      flux_row(any, r + 1, out.nx_dn, nv, in.cur.bx, in.cur.bt, TALL ? in.cur.f : load_f(r + 1), in.nx_dn, in.ddx_dn,
               out.p_dn, out.q_dn, out.ddx_dn);
      if (r + 2 < rb - 1) {
        grad_row(any, r + 2, in.p_dn, in.q_dn, out.p_dn, out.q_dn);
      } else {  // p, q of the row above the run's last one, for that row's turn
        sts4<kWBP>(brow, out.p_dn);
        sts4<kWBQ>(brow, out.q_dn);
      }
    };
    // Plain rows: r + 1 owned, not the gather's first receiver, held by no other segment, no residual
    // sums.  The addresses of row r run along, i = r - ra.  STREAM: the values of rows r - 1 to r + 1
    // stream; else each is looked for where it lies.
    struct At {
      unsigned ph, f;
      uint32_t tb, tn;
      PacketMem *xe;
      const float *gb, *gf;  // streamed u^k, f
      float *gn;             // streamed u^{k-1}, then u^{k+1}
      int i;
    };
    auto plain_step = [&](auto stream, const At &a, int off, const Carry &in, Carry &out) {
      constexpr bool STREAM = decltype(stream)::value;
      const int o = -off, i = a.i - off;  // row r - off
      Pre p;
      if (TALL) {  // the row above, where it lies
        if (!STREAM && i <= kWTmemRows) {
          tmem_load_flux2(a.tb + (o - 1) * kWRowCols, a.tn + (o - 1) * kWRowCols, out.pre.bx, out.pre.bt, out.pre.ax,
                          out.pre.at);
        } else {
          out.pre.bx = ldg4(a.gb + (o - 1) * kTallRow);
          out.pre.bt = ldg4(a.gb + (o - 1) * kTallRow + 128);
          out.pre.ax = ldg4(a.gn + (o - 1) * kTallRow);
          out.pre.at = ldg4(a.gn + (o - 1) * kTallRow + 128);
        }
        out.pre.f = !STREAM && i <= nf ? lds4(a.f + (o - 1) * static_cast<int>(kChipRowBytes)) : ldg4(a.gf + (o - 1) * kTallRow);
      } else {
        tmem_load_flux2(a.tb + o * kWRowCols, a.tn + o * kWRowCols, p.bx, p.bt, p.ax, p.at);
        p.f = lds4(a.f + o * static_cast<int>(kChipRowBytes));
      }
      const unsigned ph = a.ph + o * static_cast<int>(kChipRowBytes);
      dual(ph, TALL ? in.pre : p, in.cur.wx, out.cur);
      Q4 nv;
      prox(in.cur, out.cur.ph, rdx4, out.nx_dn, nv);
      if (!TALL || (!STREAM && i + 1 < kWTmemRows)) {
        tmem_store_flux(a.tn + (o + 1) * kWRowCols, out.nx_dn, nv);
      } else {
        stg4(a.gn + (o + 1) * kTallRow, out.nx_dn);
        stg4(a.gn + (o + 1) * kTallRow + 128, nv);
      }
      sts4<kChipRowBytes>(ph, in.cur.ph);
      give_edge(a.xe + o + 1, out.nx_dn, nv);
      flux_row(plain, 0, out.nx_dn, nv, in.cur.bx, in.cur.bt,
               TALL ? in.cur.f : lds4<kChipRowBytes>(a.f + o * static_cast<int>(kChipRowBytes)), in.nx_dn, in.ddx_dn,
               out.p_dn, out.q_dn, out.ddx_dn);
      if (ISO || i + 2 < run - 1) {
        grad_row(plain, 0, in.p_dn, in.q_dn, out.p_dn, out.q_dn);
      } else {
        sts4<kWBP>(brow, out.p_dn);
        sts4<kWBQ>(brow, out.q_dn);
      }
    };
    Carry x, y;
    x.p_dn = x.q_dn = x.nx_dn = x.ddx_dn = q4s(0.0f);
    if (run > 0) {
      Pre p;
      fetch(rb - 1, p);
      const Q4 b_dn = lds4(bux(mb) + kChipRowBytes), a_dn = lds4(bux(mn) + kChipRowBytes);
      Row s;
      dual(phi_addr(rb - 1), p, fma4(th, sub4(b_dn, a_dn), b_dn), s);
      sts4(brow, s.ph);
      x.cur = s;
      if (run > 1) {  // the last row's p, q wait for the next run's first row
        fetch(rb - 2, p);
        if (TALL && run > 2) fetch(rb - 3, x.pre);
        dual(phi_addr(rb - 2), p, s.wx, x.cur);
        Q4 nv;
        prox_row(rb - 1, s, x.cur.ph, x.nx_dn, nv);
        x.ddx_dn = sub4(x.nx_dn, s.bx);
      }
      // rows [lo, hi] are plain as the upper row of a step; they go two per trip
      const int lo = max(3, ra + (TALL ? 1 : 0)), hi = need_res ? -1 : ISO ? min(J.h - 2, rb - 4) : J.h - 2;
      int r = rb - 3;
#pragma unroll 1
      while (r >= ra) {
        if (r > hi || r <= lo) {
          step(r, x, y);
          x = y;
          --r;
          continue;
        }
        const int off = r * kTallRow;
        At a{phi_addr(r), a_f + static_cast<unsigned>(r - ra) * kChipRowBytes, tb + (r - ra) * kWRowCols,
             tn + (r - ra) * kWRowCols, xe + r, tall + off + 256 * mb, tall + off + 512, tall + off + 256 * mn, r - ra};
        auto stretch = [&](auto stream, int end) {
#pragma unroll 1
          for (; r > end; r -= 2) {
            plain_step(stream, a, 0, x, y);
            plain_step(stream, a, 1, y, x);
            a.ph -= 2 * kChipRowBytes;
            a.f -= 2 * kChipRowBytes;
            a.tb -= 2 * kWRowCols;
            a.tn -= 2 * kWRowCols;
            a.xe -= 2;
            a.gb -= 2 * kTallRow;
            a.gf -= 2 * kTallRow;
            a.gn -= 2 * kTallRow;
            a.i -= 2;
          }
        };
        if (TALL) stretch(BoolConst<TALL>{}, max(lo, ra + 1 + max(kWTmemRows, nf)));
        stretch(BoolConst<false>{}, lo);
      }
    }
    // ---- the first row of the run: phi^k of the row above comes from the run before
    bar_workers<NW>();
    Q4 p_a = q4s(0.0f), q_a = q4s(0.0f);  // p, q of row ra
    if (run > 0) {
      if (ra > 0) {
        Q4 nx, nv;
        prox_row(ra, x.cur, lds4(brow - kChipRowBytes), nx, nv);
        sts4(bux(mn), nx);
        if (run > 1) {
          Q4 ddx;
          flux_row(any, ra, nx, nv, x.cur.bx, x.cur.bt, TALL ? x.cur.f : load_f(ra), x.nx_dn, x.ddx_dn, p_a, q_a, ddx);
          if (run > 2) grad_row(any, ra + 1, x.p_dn, x.q_dn, p_a, q_a);
        }
      } else {
        sts4(phi_addr(0), x.cur.ph);  // row 0 carries phi^k only
      }
    }
    tmem_stores_done();
    bar_workers<NW>();
    // ---- the last row of the run: u^{k+1} of the row below comes from the next run
    const int L = rb - 1;
    if (run > 0 && L >= 1 && L < n - 1) {
      Q4 nx, nv, bx, bt, p, q, ddx;
      load_flux(L, mn, nx, nv);
      load_flux(L, mb, bx, bt);
      const Q4 nx_dn = lds4(bux(mn) + kChipRowBytes);
      flux_row(any, L, nx, nv, bx, bt, load_f(L), nx_dn, sub4(nx_dn, lds4(bux(mb) + kChipRowBytes)), p, q, ddx);
      if (run == 2)
        grad_row(any, L, p, q, p_a, q_a);
      else if (run > 2)
        grad_row(any, L, p, q, lds4<kWBP>(brow), lds4<kWBQ>(brow));
      if (run == 1) {
        p_a = p;
        q_a = q;
      }
      sts4<kWBP>(brow, p);
      sts4<kWBQ>(brow, q);
    }
    bar_workers<NW>();
    if (run > 0 && ra >= 2 && ra < n - 1)
      grad_row(any, ra, p_a, q_a, lds4<kWBP - kChipRowBytes>(brow), lds4<kWBQ - kChipRowBytes>(brow));

    chip_store_sums<TALL>(X, v, own_lane);
    bar_all_arrive<2, NW>();
    // ---- halo flux of the pass
    bool got = true;
    if (run > 0) {
      // rows -2 and h + 1
      auto halo_row = [&](int seg, int which, Q4 &ux, Q4 &ut) {
        const PacketMem *const o = xrow + (mb ? xrow_set : 0) + (static_cast<size_t>(seg) * 2 + which) * ntp + gj0;
        float x[4] = {0.f, 0.f, 0.f, 0.f}, t[4] = {0.f, 0.f, 0.f, 0.f};
        got = poll_warp([&] {
          bool all = true;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (!ln.use[i]) continue;
            const Packet p = get_packet(o + i);
            x[i] = p.x;
            t[i] = p.y;
            all = all && p.tag == tag;
          }
          return all;
        }) && got;
        ux = q4(x[0], x[1], x[2], x[3]);
        ut = q4(t[0], t[1], t[2], t[3]);
      };
      Q4 hx, ht;
      if (ra == 0 && J.seg > 0) {
        halo_row(J.seg - 1, 0, hx, ht);
        store_flux(0, mn, hx, ht);
      }
      if (rb == n && J.seg + 1 < J.segs && J.i0 - 2 + n < nr) {
        halo_row(J.seg + 1, 1, hx, ht);
        sts4(bux(mn) + kChipRowBytes, hx);
      }
      tmem_stores_done();
      // Lane l fetches side l & 1 of the run's rows ra + l / 2 (+ 16, ...): the t flux of samples -2
      // and 121 (and, with the isotropic cost, the x flux of sample -2), and puts it in its row: an
      // element of the row where that is in shared or global memory; rows in tensor memory are
      // rewritten by the warp.
      const int e_side = lane & 1, e_strip = J.strip + (e_side ? 1 : -1);
      const bool e_any = e_strip >= 0 && e_strip < J.strips;
      const PacketMem *const e_src = xcol + (mb ? xcol_set : 0) + (static_cast<size_t>(e_strip) * 2 + (e_side ? 0 : 1)) * nr;
      float et[kRounds], ex[kRounds];
      got = poll_warp([&] {
        bool all = true;
#pragma unroll
        for (int w = 0; w < kRounds; ++w) {
          const int r = ra + (lane >> 1) + 16 * w, gi = J.i0 - 2 + r;
          et[w] = ex[w] = 0.0f;
          if (!(r < rb && e_any && gi >= 0 && gi < nr)) continue;
          const Packet p = get_packet(e_src + gi);
          et[w] = p.x;
          ex[w] = p.y;
          all = all && p.tag == tag;
        }
        return all;
      }) && got;
      auto edges = [&](int comp, const float (&e)[kRounds]) {
        const bool mine = comp == 1 || !e_side;
#pragma unroll
        for (int w = 0; w < kRounds; ++w) {
          const int r = ra + (lane >> 1) + 16 * w, i = r - ra;
          if (r >= rb || i < kWTmemRows || !mine) continue;
          const unsigned o = e_side ? 125u : 2u;  // the sample's place in the row
          if (!TALL)
            sts1(u_slot(i, mn) - 16u * lane + comp * kChipRowBytes + 4u * o, e[w]);
          else
            __stcg(tall - 4 * lane + r * kTallRow + (2 * mn + comp) * 128 + o, e[w]);
        }
        // (lane 0 holds row ra: its x flux also lies in the boundary row)
        if (comp == 0 && lane == 0) sts1(bux(mn) + 8u, e[0]);
        Q4 u[kWTmemRows];
        const uint32_t a = tn + 4 * comp;
#pragma unroll
        for (int i = 0; i < kWTmemRows; ++i)
          if (i < run) u[i] = tmem_load_quad(a + i * kWRowCols);
#pragma unroll
        for (int i = 0; i < kWTmemRows; ++i) {
          const float e0 = __shfl_sync(0xffffffffu, e[0], 2 * i), e1 = __shfl_sync(0xffffffffu, e[0], 2 * i + 1);
          if (i >= run) continue;
          float t[4];
          un4(u[i], t);
          tmem_store_quad(a + i * kWRowCols, q4(t[0], lane == 31 && comp ? e1 : t[1], lane == 0 ? e0 : t[2], t[3]));
        }
      };
      edges(1, et);
      if (ISO) edges(0, ex);
      tmem_stores_done();
    }
    if (!got && lane == 0) sh.bad = 1;
    bar_all<4, NW>();  // the decision
    ++k;
  }

  // ---- finalize: phi^K (from div u^K and div u^{K-1}, as the finalize pass forms it), the outputs
  // and the duality gap's sums
  if (!sh.bad && sh.status == ST_OK) {
    const int mb = k & 1, ma = mb ^ 1;
    const Q4 cf = lds_pair<16>(sc_addr), th = lds_pair<32>(sc_addr);
    const Q4 rdx4 = lds_pair<64>(sc_addr), rdt4 = lds_pair<80>(sc_addr);
    Sum2 t[4];
    if (run > 0) {
      Q4 b_dn = lds4(bux(mb) + kChipRowBytes), a_dn = lds4(bux(ma) + kChipRowBytes);
      Q4 bx, bt, ax, at, f, bx1, bt1, ax1, at1, f1;  // of this row and of the next
      auto load = [&](int r) {
        load_flux(r, mb, bx1, bt1);
        load_flux(r, ma, ax1, at1);
        f1 = load_f(r);
      };
      load(rb - 1);
#pragma unroll 1
      for (int r = rb - 1; r >= ra; --r) {
        bx = bx1;
        bt = bt1;
        ax = ax1;
        at = at1;
        f = f1;
        if (r > ra) load(r - 1);
        const Q4 db = div4(sub4(b_dn, bx), diff_right(bt), rdx4, rdt4);
        const Q4 da = div4(sub4(a_dn, ax), diff_right(at), rdx4, rdt4);
        const Q4 ph = fma4(cf, fma4(th, sub4(db, da), add4(db, f)), lds4(phi_addr(r)));
        sts4(phi_addr(r), ph);
        if (r == rb - 1) sts4(brow, ph);
        b_dn = bx;
        a_dn = ax;
      }
    }
    bar_workers<NW>();
    const bool vec = chip_vec_out(X);
    Q4 up = run > 0 && ra > 0 ? lds4(brow - kChipRowBytes) : q4s(0.0f);
    Q4 ux, ut, f, ux1, ut1, f1;
    if (run > 0) {
      load_flux(ra, mb, ux1, ut1);
      f1 = load_f(ra);
    }
#pragma unroll 1
    for (int r = ra; r < rb; ++r) {
      ux = ux1;
      ut = ut1;
      f = f1;
      if (r + 1 < rb) {
        load_flux(r + 1, mb, ux1, ut1);
        f1 = load_f(r + 1);
      }
      const Q4 ph = lds4(phi_addr(r)), gtv = diff_left(ph);
      if (r >= 2 && r < J.h + 2 && own_lane)
        chip_output_row<ISO>(X, vec, J.i0 - 2 + r, ux, ut, ph, up, gtv, f, t);
      up = ph;
    }
    chip_store_gap(X, t);
    bar_all_arrive<2, NW>();
  }
}

__host__ __device__ constexpr int chip_workers(int form) { return form == kChipMarchTall ? kTallWorkers : kChipWorkers; }

template <bool ISO, int FORM>
__global__ void __launch_bounds__((chip_workers(FORM) + 1) * 32, 1) k_solve_chip(const Ctl c, const __grid_constant__ ChipJobs jobs) {
  constexpr int NW = chip_workers(FORM), kCols = FORM == kChipTile ? kChipTmemCols : WLayout<NW>::kTmemCols;
  extern __shared__ float4 dyn4[];
  __shared__ ChipShared sh;
  const ChipJob &J = jobs.job[blockIdx.x];
  const Shot &S = c.shots[J.gather];
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  const int n = J.h + 3;

  if (warp == 0) tmem_alloc_all(&sh.tmem);
  if (threadIdx.x == 0) {
    sh.done = 0;
    sh.status = ST_OK;
    sh.bad = 0;
  }
  if (threadIdx.x < 16 * kChipVals) (&sh.part[0][0])[threadIdx.x] = (&sh.low[0][0])[threadIdx.x] = 0.0f;  // of warps that are not there
  if (threadIdx.x < 16 * 4) (&sh.dpart[0][0])[threadIdx.x] = 0.0;
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");

  // a worker's run: rows [ra, rb).  The leftover rows go to the warps after the first one, whose
  // halo rows take the general row code; empty runs are at the end
  const int base = n / NW, rem = n % NW, lead = base > 0 ? 1 : 0;
  auto first_row = [&](int w) { return w * base + min(max(w - lead, 0), rem); };
  const int ra = first_row(warp), rb = first_row(warp + 1);
  const ChipCta X{c, J, S, sh, c.states + J.gather, lane, warp, S.nr, S.nt, S.ntp, n,
                  J.seg * J.strips + J.strip, ra, rb, J.strip * kChipTJ - 4 + 4 * lane,
                  sh.tmem + (static_cast<uint32_t>(warp & 3) << 21) + (warp >> 2) * kCols,
                  ((smem_u32(dyn4) + 127u) & ~127u) + 16u * lane};
  if (warp == NW)
    chip_decider<NW>(X);
  else if constexpr (FORM == kChipTile)
    chip_worker<ISO>(X);
  else
    chip_worker_w<ISO, FORM == kChipMarchTall, NW>(X);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) tmem_free_all(sh.tmem);
}

}  // namespace emd
