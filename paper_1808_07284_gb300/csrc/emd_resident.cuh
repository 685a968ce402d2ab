// Shared-memory-resident solve for small gathers: one CTA holds a whole gather in shared memory for
// the entire solve, so a PDHG iteration is four short phases between barriers, a warp sum and the
// linesearch decision -- no global memory traffic, atomics or cross-CTA waits.  In a batch every
// gather gets its own CTA and the gathers run independently (the paper solves one EMD per shot).
//
// Such a pass is a chain of latencies, so every step is short: a thread owns whole quads of four
// consecutive samples (rows padded to a multiple of four), div u and q of the last pass are kept
// instead of formed again, the totals of the warps are added in float pairs, and a decision
// settles in FP32 wherever that is certain (quick_decide).  FP64, 64 cycles an instruction, is
// left to the decider warp, which prepares the next decision's step sizes beside the pass.
//
// Shared planes, one float4 per quad: ux, ut (u^k, then u^{k+1}), phi, div u, q, p, f.  Every
// cell's arithmetic and rounding are those of the tile pass.  Measured: 1 x 1024 1.4 us per pass (5.3 with
// six barriers, scalar cells and FP64 totals and decisions), 20 x 200 3.4, 64 x 112 4.9.
#pragma once

#include "emd_chip.cuh"

namespace emd {

constexpr int kResWarps = 15;            // cell-work warps at most (and the decider warp)
constexpr int kResPlanes = 7;
constexpr int kResidentMaxCells = 7168;  // cells of a gather at most, and with its rows padded:
constexpr int kResidentMaxPadded = 8128;

inline int resident_quads(int nt, int nr) { return nr * ((nt + 3) / 4); }
inline size_t resident_smem_bytes(int quads) { return static_cast<size_t>(quads) * kResPlanes * 16; }

struct ResShared {
  alignas(16) float sc[4];     // alpha, coef, theta, 1 / (1 + eps alpha)
  // Warp totals of a pass (zero for warps that are not there), in pairs of floats: a small gather has
  // few warps to average their rounding (with plain totals the reported residual of 1 x 1024 was 8.2e-9
  // from 64 bits, in FP64 above the warp 5.7e-9; now 4.9e-9, for 0.01 of 1.44 us a pass).
  float part[16][kChipVals], low[16][kChipVals];
  int done, status;
};

__global__ void __launch_bounds__((kResWarps + 1) * 32, 1) k_solve_resident(Ctl c) {
  const int g = blockIdx.x;
  const Shot &S = c.shots[g];
  State *st = c.states + g;
  extern __shared__ float4 dyn4[];
  __shared__ ResShared sh;
  const int nr = S.nr, nt = S.nt, ntp = S.ntp, quads_row = (nt + 3) / 4, quads = nr * quads_row;
  const float rdx = S.rdx, rdt = S.rdt;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int workers = blockDim.x / 32 - 1, NT = workers * 32;
  float4 *const UX = dyn4, *const UT = UX + quads, *const PH = UT + quads, *const DV = PH + quads;
  float4 *const QQ = DV + quads, *const PP = QQ + quads, *const FF = PP + quads;
  auto bar = [&](int id, int threads) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); };

  // ---- load the gather: balanced f, u^0, phi^{-1} (the warm start) from the prepared planes
  const float fmean = st->fmean_f;
  for (int e = tid; e < quads; e += blockDim.x) {
    const int i = e / quads_row, j = 4 * (e - i * quads_row), o = i * ntp + j;
    float f[4], ux[4], ut[4], ph[4], d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool in = j + q < nt;
      f[q] = in ? S.f[o + q] - fmean : 0.0f;
      ux[q] = in ? S.ux[0][o + q] : 0.0f;
      ut[q] = in ? S.ut[0][o + q] : 0.0f;
      ph[q] = in ? S.ph[1][o + q] : 0.0f;
      const float xl = i > 0 ? ux[q] : 0.0f, xr = in && i + 1 < nr ? S.ux[0][o + ntp + q] : 0.0f;
      const float tl = j + q > 0 ? ut[q] : 0.0f, tr = j + q + 1 < nt ? S.ut[0][o + q + 1] : 0.0f;
      d[q] = in ? fmaf(xr - xl, rdx, (tr - tl) * rdt) : 0.0f;
    }
    FF[e] = make_float4(f[0], f[1], f[2], f[3]);
    UX[e] = make_float4(ux[0], ux[1], ux[2], ux[3]);
    UT[e] = make_float4(ut[0], ut[1], ut[2], ut[3]);
    PH[e] = make_float4(ph[0], ph[1], ph[2], ph[3]);
    DV[e] = make_float4(d[0], d[1], d[2], d[3]);
    QQ[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (int q = tid; q < 16 * kChipVals; q += blockDim.x) (&sh.part[0][0])[q] = (&sh.low[0][0])[q] = 0.0f;
  if (tid == 0) {
    sh.sc[0] = st->alpha_f;
    sh.sc[1] = st->coef_f;
    sh.sc[2] = st->theta_f;
    sh.sc[3] = st->inv_f;
    sh.done = 0;
    sh.status = ST_OK;
  }
  __syncthreads();

  if (warp == workers) {
    // ================================================================ decider warp
    constexpr unsigned FULL = 0xffffffffu;
    DecidePrep pr;
    pr.k = 0;
    pr.alpha = st->alpha;
    pr.theta = st->theta;
    pr.coef = st->coef;
    pr.beta_fixed = st->beta_fixed;
    pr.fnorm = st->fnorm;
    const double xl = xi_power(c.xi);  // the same in every pass
    const bool quick = c.linesearch && c.debug_fault != 1;
    int trials = 0, status = ST_OK;
    bool done = false;
    double r_feas = -1.0, r_step = -1.0, v = 0.0;
    while (!done) {
      const QuickPrep qp = step_prep(c, pr, xl);  // beside the pass
      const bool check = c.tol > 0.0 && (pr.k + 1) % c.check_every == 0;
      bar(2, NT + 32);
      float hi, lo;
      chip_block_pair<true>(sh.part, sh.low, hi, lo);
      const int w = quick && !check ? quick_decide(c, qp, hi) : -1;
      if (w >= 0) {
        const float a = __shfl_sync(FULL, pr.alpha_lf, w), cf = __shfl_sync(FULL, pr.coef_lf, w);
        const float th = __shfl_sync(FULL, pr.theta_lf, w), iv = __shfl_sync(FULL, pr.inv_lf, w);
        done = pr.k + 1 >= c.max_iter;
        if (lane == 0) {
          *reinterpret_cast<float4 *>(sh.sc) = make_float4(a, cf, th, iv);
          sh.done = done;
        }
        bar(4, NT + 32);
        trials += w + 1;
        pr.alpha = __shfl_sync(FULL, pr.alpha_l, w);
        pr.theta = __shfl_sync(FULL, pr.s_lane, w);
        pr.coef = __shfl_sync(FULL, pr.coef_l, w);
        if (c.trace) {
          Decision o;
          o.alpha = pr.alpha;
          o.theta = pr.theta;
          o.trials_now = w + 1;
          const double ppp = __shfl_sync(FULL, static_cast<double>(hi) + static_cast<double>(lo), 0);
          if (lane == 0) write_trace(c, g, pr.k, o, ppp, pr.fnorm);
        }
        if (done) v = static_cast<double>(hi) + static_cast<double>(lo);
        ++pr.k;
      } else {
        v = static_cast<double>(hi) + static_cast<double>(lo);
        double a_[9];
#pragma unroll
        for (int q = 0; q < 6; ++q) a_[q] = __shfl_sync(FULL, v, q);
        a_[6] = 0.0;
        a_[7] = __shfl_sync(FULL, v, 6);
        a_[8] = __shfl_sync(FULL, v, 7);
        decide_prep_lanes(c, pr);
        const Decision o = decide_core(c, pr, a_);
        trials += o.trials_now;
        done = o.done;
        status = o.status;
        if (lane == 0) {
          if (o.status == ST_OK) *reinterpret_cast<float4 *>(sh.sc) = make_float4(o.alpha_f, o.coef_f, o.theta_f, o.inv_f);
          sh.status = o.status;
          sh.done = o.done;
        }
        bar(4, NT + 32);
        if (lane == 0) write_trace(c, g, pr.k, o, a_[0], pr.fnorm);
        if (o.checked) residuals(pr, a_, r_feas, r_step);
        if (o.status == ST_OK) {
          pr.k = o.k_new;
          pr.alpha = o.alpha;
          pr.theta = o.theta;
          pr.coef = o.coef;
        }
      }
    }
    const double s_p2 = __shfl_sync(FULL, v, 0), s_u2 = __shfl_sync(FULL, v, 6), s_du2 = __shfl_sync(FULL, v, 7);
    if (lane == 0) {
      st->k = pr.k;
      st->trials = trials;
      st->status = status;
      st->alpha = pr.alpha;
      st->theta = pr.theta;
      st->coef = pr.coef;
      publish(st, c.eps);
      st->coef_f = 0.0f;  // phi^K is complete: the finalize pass adds nothing to it
      st->r_feas = r_feas;
      st->r_step = r_step;
      st->s_p2 = s_p2;
      st->s_u2 = s_u2;
      st->s_du2 = s_du2;
      st->done = 1;
      atomicAdd(c.n_done, 1);
    }
    return;
  }

  // ================================================================== cell-work warps
  int k = 0;
  float coef, theta;
  while (true) {
    const float4 sc = *reinterpret_cast<const float4 *>(sh.sc);
    const float alpha = sc.x, inv = sc.w;
    coef = sc.y;
    theta = sc.z;
    if (sh.done) break;
    const bool need_res = (c.tol > 0.0 && (k + 1) % c.check_every == 0) || k + 1 >= c.max_iter;
    // ---- phi^k = phi^{k-1} + c_k (p_{k-1} + theta_k q_{k-1})
    auto dual = [&](int e) {
      const float4 d = DV[e], f = FF[e], q = QQ[e];
      float4 ph = PH[e];
      ph.x = fmaf(coef, fmaf(theta, q.x, d.x + f.x), ph.x);
      ph.y = fmaf(coef, fmaf(theta, q.y, d.y + f.y), ph.y);
      ph.z = fmaf(coef, fmaf(theta, q.z, d.z + f.z), ph.z);
      ph.w = fmaf(coef, fmaf(theta, q.w, d.w + f.w), ph.w);
      PH[e] = ph;
    };
    for (int e = tid; e < quads; e += NT) dual(e);
    bar(1, NT);
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // ---- u^{k+1} = shrink(u^k + alpha grad phi^k, alpha) / (1 + eps alpha)
    for (int e = tid; e < quads; e += NT) {
      const int i = e / quads_row, j = 4 * (e - i * quads_row);
      const float4 p4 = PH[e], u4 = i > 0 ? PH[e - quads_row] : p4, x4 = UX[e], t4 = UT[e];
      const float left = j > 0 ? reinterpret_cast<const float *>(PH)[4 * e - 1] : 0.0f;
      const float ph[5] = {left, p4.x, p4.y, p4.z, p4.w}, up[4] = {u4.x, u4.y, u4.z, u4.w};
      const float bx[4] = {x4.x, x4.y, x4.z, x4.w}, bt[4] = {t4.x, t4.y, t4.z, t4.w};
      float nx[4], nv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float gx = (ph[q + 1] - up[q]) * rdx;  // 0 at receiver 0
        const float gt = j + q > 0 && j + q < nt ? (ph[q + 1] - ph[q]) * rdt : 0.0f;
        prox_cell(fmaf(alpha, gx, bx[q]), fmaf(alpha, gt, bt[q]), alpha, inv, c.iso, nx[q], nv[q]);
      }
      UX[e] = make_float4(nx[0], nx[1], nx[2], nx[3]);
      UT[e] = make_float4(nv[0], nv[1], nv[2], nv[3]);
      if (need_res) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float dx_ = nx[q] - bx[q], dt_ = nv[q] - bt[q];
          v[6] += nx[q] * nx[q] + nv[q] * nv[q];
          v[7] += dx_ * dx_ + dt_ * dt_;
        }
      }
    }
    bar(1, NT);
    // ---- div u^{k+1}, p = div u^{k+1} + f, q = div(u^{k+1} - u^k)
    for (int e = tid; e < quads; e += NT) {
      const int i = e / quads_row, j = 4 * (e - i * quads_row);
      const float4 x4 = UX[e], t4 = UT[e], f4 = FF[e], d4 = DV[e];
      const float4 n4 = i + 1 < nr ? UX[e + quads_row] : make_float4(0.f, 0.f, 0.f, 0.f);
      const float right = j + 4 < nt ? reinterpret_cast<const float *>(UT)[4 * e + 4] : 0.0f;
      const float t[5] = {t4.x, t4.y, t4.z, t4.w, right}, x[4] = {x4.x, x4.y, x4.z, x4.w}, n[4] = {n4.x, n4.y, n4.z, n4.w};
      const float f[4] = {f4.x, f4.y, f4.z, f4.w}, d[4] = {d4.x, d4.y, d4.z, d4.w};
      float dn[4], p[4], qq[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        dn[q] = fmaf(n[q] - x[q], rdx, (t[q + 1] - t[q]) * rdt);
        p[q] = dn[q] + f[q];
        qq[q] = dn[q] - d[q];
      }
      DV[e] = make_float4(dn[0], dn[1], dn[2], dn[3]);
      PP[e] = make_float4(p[0], p[1], p[2], p[3]);
      QQ[e] = make_float4(qq[0], qq[1], qq[2], qq[3]);
    }
    bar(1, NT);
    // ---- the sums
    for (int e = tid; e < quads; e += NT) {
      const int i = e / quads_row, j = 4 * (e - i * quads_row);
      const float4 p4 = PP[e], q4_ = QQ[e], pu4 = i > 0 ? PP[e - quads_row] : p4, qu4 = i > 0 ? QQ[e - quads_row] : q4_;
      const float pl = j > 0 ? reinterpret_cast<const float *>(PP)[4 * e - 1] : 0.0f;
      const float ql = j > 0 ? reinterpret_cast<const float *>(QQ)[4 * e - 1] : 0.0f;
      const float p[5] = {pl, p4.x, p4.y, p4.z, p4.w}, qv[5] = {ql, q4_.x, q4_.y, q4_.z, q4_.w};
      const float pu[4] = {pu4.x, pu4.y, pu4.z, pu4.w}, qu[4] = {qu4.x, qu4.y, qu4.z, qu4.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float m = j + q > 0 && j + q < nt ? rdt : 0.0f;
        const float gpx = (p[q + 1] - pu[q]) * rdx, gpt = (p[q + 1] - p[q]) * m;
        const float gqx = (qv[q + 1] - qu[q]) * rdx, gqt = (qv[q + 1] - qv[q]) * m;
        v[0] = fmaf(p[q + 1], p[q + 1], v[0]);
        v[1] = fmaf(p[q + 1], qv[q + 1], v[1]);
        v[2] = fmaf(qv[q + 1], qv[q + 1], v[2]);
        v[3] = fmaf(gpx, gpx, fmaf(gpt, gpt, v[3]));
        v[4] = fmaf(gpx, gqx, fmaf(gpt, gqt, v[4]));
        v[5] = fmaf(gqx, gqx, fmaf(gqt, gqt, v[5]));
      }
    }
    float low;
    const float tot = warp_sum8_pair(v, low);
    if (lane < 8) {
      sh.part[warp][lane] = tot;
      sh.low[warp][lane] = low;
    }
    asm volatile("bar.arrive 2, %0;\n" ::"r"(NT + 32) : "memory");
    bar(4, NT + 32);  // the decision
    ++k;
  }

  // ---- phi^K, and the solution into the planes that the finalize pass reads at k = K
  if (sh.status != ST_OK) return;
  const int kc = k % 3;
  for (int e = tid; e < quads; e += NT) {
    const int i = e / quads_row, j = 4 * (e - i * quads_row), o = i * ntp + j;  // 16-byte aligned rows
    const float4 d = DV[e], f = FF[e], q = QQ[e];
    float4 ph = PH[e];
    ph.x = fmaf(coef, fmaf(theta, q.x, d.x + f.x), ph.x);
    ph.y = fmaf(coef, fmaf(theta, q.y, d.y + f.y), ph.y);
    ph.z = fmaf(coef, fmaf(theta, q.z, d.z + f.z), ph.z);
    ph.w = fmaf(coef, fmaf(theta, q.w, d.w + f.w), ph.w);
    *reinterpret_cast<float4 *>(S.ux[kc] + o) = UX[e];
    *reinterpret_cast<float4 *>(S.ut[kc] + o) = UT[e];
    *reinterpret_cast<float4 *>(S.ph[(k + 1) & 1] + o) = ph;
  }
}

}  // namespace emd
