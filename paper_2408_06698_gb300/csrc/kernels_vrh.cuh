// a3 + a5 with the element's data in registers, the basis split over two lanes (FP32): volume
// term, facet lift and inverse mass.
//
// The structure of k_volume_r (a lane per (element, component a), the quadrature points
// walked in the same order by every lane, broadcast basis rows, the other components taken
// by shuffles, f_a = w_q (div^W u_a + W . grad^ u_a) tested against phi_i, register pairs, the
// products that vanish by degree left out), with each (element, component) pair on two
// lanes: half h owns the basis indices i = 2 t + h (coefficients c_i, test accumulators r_i,
// with a separate wind its coefficients) and the modal gradient entries G_c[j], j = 2 t + h <
// dim P^{k-1} (and those of div^ W).  Per point a lane forms its half's partial sums, and one
// shuffle each with the other half completes them; both halves then hold the same f_a and
// accumulate their own r_i.  The tables are staged with their basis columns permuted so that
// each half reads one contiguous block of a row (half h at column offset h HP).  Half the
// registers per lane of k_volume_r: a register kernel at k = 5, where a whole basis does not
// fit in one lane.  Separate wind and VJP as in k_volume_r.
//
// Bound: FMA register reads and the shuffles.  Measured (CUDA events, per launch): 18^3 x 6,
// k = 5, w = u 437 -> 351 us (scalar FMAs, dense Dm and TrM products before); 13^3 x 6, k = 5,
// separate wind 633 -> 192 us (a warp per element before).
#pragma once
#include "f32x2.cuh"
#include "kernels.cuh"
#include "kernels_vr.cuh"

namespace hopu {

template <int D, int K, int MODE = kVolSame>
struct VolRH {
  using S = Shape<D, K>;
  static constexpr int NB = S::nb, NB1 = cnbasis(D, K - 1), NF = S::nf, NL = S::nloc, NQ = S::nq, GT = S::gt;
  static constexpr int LPE = 2 * D;               // lanes per element: (component, half)
  static constexpr int ELW = 32 / LPE;            // elements per warp
  static constexpr int NH = (NB + 1) / 2;         // basis indices of half 0 (half 1: NB - NH)
  static constexpr int NH1 = (NB1 + 1) / 2;       // modal-gradient indices of half 0
  static constexpr int NP = (NH + 1) / 2, NP1 = (NH1 + 1) / 2;  // pairs of a half
  static constexpr int HP = r4i(NH);              // one half's block of a permuted row
  static constexpr int RW = 2 * HP;               // permuted row width
  static constexpr int NBQ = (RW / 4) % 2 == 0 ? RW + 4 : RW;  // Bt row stride: an odd multiple of 16 bytes
  static constexpr int NG = (D + 1) * NF * D;
  static constexpr int O_WQ = NQ * NBQ;           // Bt [NQ][NBQ], permuted columns
  static constexpr int O_DM = r4i(O_WQ + NQ);     // Dm [D][NB1][RW], permuted columns
  static constexpr int O_TRM = O_DM + D * NB1 * RW;   // TrM [(D+1) NF][RW], permuted columns
  static constexpr int O_W = O_TRM + (D + 1) * NF * RW;
  static constexpr int PER_WARP = r4i(ELW * NL);  // the warp's element records: in (u, w), and out
  static constexpr int GW = r4i(ELW * NG);        // the warp's facet moments
  static constexpr int NBUF = MODE == kVolSame ? 2 : 3;
  static constexpr int NGAM = MODE == kVolAdjSame ? 2 : 1;
  // tables above 64 KB: one CTA of 8 warps (6 with two sets of moments) per SM; else CTAs of 4
  // warps, as many as fit
  static constexpr int WARPS = O_W * 4 > 64 * 1024 ? (NGAM == 2 ? 6 : 8) : 4;
  static constexpr int O_G = O_W + WARPS * NBUF * PER_WARP;
  static constexpr size_t SMEM = size_t(O_G + WARPS * NGAM * GW) * 4;
  static constexpr int REGS = (MODE == kVolWind ? 3 * NH + NH1 : 2 * NH) + D * NH1;  // a lane's vectors
  static constexpr int MINB = WARPS > 4 ? 1 : (REGS <= 60 ? 4 : 3);
  static constexpr bool OK = REGS <= 160 && SMEM <= 220 * 1024 && NB >= 2;
};

// Arguments as k_volume_r.
template <int D, int K, int MODE>
__global__ void __launch_bounds__(32 * VolRH<D, K, MODE>::WARPS, VolRH<D, K, MODE>::MINB)
    k_volume_rh(DevMesh m, DevTabs tb, const float* __restrict__ in1, const float* __restrict__ in2,
                const float* __restrict__ gam, const float* __restrict__ gam2, float* out, Combine cmb) {
  using C = VolRH<D, K, MODE>;
  constexpr bool WIND = MODE == kVolWind, ADJ = MODE >= kVolAdjU;
  constexpr bool ROW = WIND || MODE == kVolAdjU;   // the wind enters through its reference components
  constexpr int NB = C::NB, NB1 = C::NB1, NF = C::NF, NL = C::NL, NQ = C::NQ, GT = C::GT;
  constexpr int NBQ = C::NBQ, HP = C::HP, RW = C::RW, NG = C::NG, ELW = C::ELW, LPE = C::LPE;
  constexpr int NH = C::NH, NH1 = C::NH1, NP = C::NP, NP1 = C::NP1;
  extern __shared__ __align__(16) float sm[];
  pdl_trigger();
  {  // tables with permuted basis columns (zero padding)
    const float* Btg = static_cast<const float*>(tb.Bt);
    const float* Wqg = static_cast<const float*>(tb.Wq);
    const float* Dmg = static_cast<const float*>(tb.Dm);
    const float* TrMg = static_cast<const float*>(tb.TrM);
    constexpr int NBQG = row_stride<float>(NB);  // Bt rows in global memory
    for (int t = threadIdx.x; t < NQ * NBQ; t += blockDim.x) {
      const int q = t / NBQ, p = t - q * NBQ, h = p / HP, i = 2 * (p - h * HP) + h;
      sm[t] = (p < RW && i < NB) ? Btg[q * NBQG + i] : 0.0f;
    }
    for (int t = threadIdx.x; t < NQ; t += blockDim.x) sm[C::O_WQ + t] = Wqg[t];
    for (int t = threadIdx.x; t < D * NB1 * RW; t += blockDim.x) {
      const int row = t / RW, p = t - row * RW, h = p / HP, i = 2 * (p - h * HP) + h;
      sm[C::O_DM + t] = i < NB ? Dmg[row * NB + i] : 0.0f;
    }
    for (int t = threadIdx.x; t < (D + 1) * NF * RW; t += blockDim.x) {
      const int row = t / RW, p = t - row * RW, h = p / HP, i = 2 * (p - h * HP) + h;
      sm[C::O_TRM + t] = i < NB ? TrMg[row * NB + i] : 0.0f;
    }
  }
  const float* sBt = sm;
  const float* sWq = sm + C::O_WQ;
  const float* sDm = sm + C::O_DM;
  const float* sTrM = sm + C::O_TRM;
  pdl_wait();
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool lane_on = lane < LPE * ELW;
  const int el = lane_on ? lane / LPE : 0;
  const int rr = lane_on ? lane - el * LPE : 0;
  const int a = rr >> 1, h = rr & 1;
  const int a1 = (a + 1) % D, a2 = (a + 2) % D;
  const int nh = h ? NB - NH : NH;          // this half's basis indices
  const int pt = lane ^ 1;                  // the other half of this (element, component)
  // the other components' lanes of the same half (idle lanes talk to themselves)
  const int p1 = lane_on ? el * LPE + a1 * 2 + h : lane;
  const int p2 = lane_on ? el * LPE + a2 * 2 + h : lane;
  float* sIn = sm + C::O_W + warp * C::NBUF * C::PER_WARP;
  float* sY = sIn + C::PER_WARP;
  float* sIn2 = sY + (MODE == kVolSame ? 0 : C::PER_WARP);
  float* sG = sm + C::O_G + warp * C::NGAM * C::GW;
  const int64_t ngroups = (m.E + ELW - 1) / ELW, gstep = (int64_t)gridDim.x * C::WARPS;
  auto count = [&](int64_t g) { return (m.E - g * ELW < ELW) ? (int)(m.E - g * ELW) : ELW; };
  auto request = [&](int64_t g) {
    warp_copy_records<NL, ELW>(sIn, in1, g * ELW, count(g), lane);
    if (MODE != kVolSame) warp_copy_records<NL, ELW>(sIn2, in2, g * ELW, count(g), lane);
  };
  auto halves = [&](float v) { return v + __shfl_sync(kFull, v, pt); };
  int64_t grp = (int64_t)warp * gridDim.x + blockIdx.x;
  if (grp < ngroups) request(grp);
  cp_commit();
  for (; grp < ngroups; grp += gstep) {
    const int64_t e0 = grp * ELW;
    const int ne = count(grp);
    const bool act = lane_on && el < ne;
    const int64_t e = act ? e0 + el : e0;  // inactive lanes read the group's first element
    const float* gp = m.geoF + e * GT;
    // M = |det J| J^-1: its columns a, a + 1, a + 2 (w = u), column a (kVolAdjW) or row a in M0
    constexpr bool COLS = MODE == kVolSame || MODE == kVolAdjSame;
    float M0[D], M1[COLS ? D : 1], M2[COLS ? D : 1];
#pragma unroll
    for (int cc = 0; cc < D; ++cc) {
      M0[cc] = __ldg(gp + 2 * D * D + (ROW ? a * D + cc : cc * D + a));
      if constexpr (COLS) {
        M1[cc] = __ldg(gp + 2 * D * D + cc * D + a1);
        M2[cc] = D == 3 ? __ldg(gp + 2 * D * D + cc * D + a2) : 0.0f;
      }
    }
    const float invabs = __ldg(gp + 3 * D * D);
    // this half's coefficients, entries 2 t + h (zero beyond the half): c those whose gradient is
    // taken, ev those evaluated at the points (as in k_volume_r)
    f2 c[NP], ev[MODE == kVolSame ? 1 : NP];
    cp_wait<0>();
    __syncwarp();
    {
      const int oe = (act ? el : 0) * NL + h, o = oe + a * NB;
      const float* sC = ADJ ? sIn2 : sIn;
      const float sc = ADJ ? invabs : 1.0f;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const bool in0 = 2 * j < nh, in1_ = 2 * j + 1 < nh;
        c[j] = f2_pack(in0 ? sC[o + 4 * j] : 0.0f, in1_ ? sC[o + 4 * j + 2] : 0.0f);
        if constexpr (ADJ) c[j] = f2_mul(c[j], f2_dup(sc));
        if constexpr (ROW) {
          float v[2] = {0.0f, 0.0f};
          const float* wp = (WIND ? sIn2 : sIn) + oe + 4 * j;
#pragma unroll
          for (int b = 0; b < D; ++b) {
            if (in0) v[0] = fmaf(M0[b], wp[b * NB], v[0]);
            if (in1_) v[1] = fmaf(M0[b], wp[b * NB + 2], v[1]);
          }
          ev[j] = f2_pack(v[0], v[1]);
        } else if constexpr (ADJ) {
          ev[j] = f2_pack(in0 ? sIn[o + 4 * j] : 0.0f, in1_ ? sIn[o + 4 * j + 2] : 0.0f);
        }
      }
    }
    __syncwarp();
    // this group's facet moments and the next group's coefficients arrive during the points
    warp_copy_records<NG, ELW>(sG, gam, e0, ne, lane);
    if (MODE == kVolAdjSame) warp_copy_records<NG, ELW>(sG + C::GW, gam2, e0, ne, lane);
    if (grp + gstep < ngroups) request(grp + gstep);
    cp_commit();
    // this half's entry j = 2 t + h of the modal reference derivative sum_i Dm[cc][j][i] x_i, xo
    // the other half's coefficients (zero past dim P^{k-1})
    auto derivative = [&](const f2 (&x)[NP], const f2 (&xo)[NP], int cc, int t) -> float {
      const int j = 2 * t + h;
      const bool in = j < NB1;
      const int i0 = cnbasis(D, mode_degree(D, 2 * t));  // no terms below: the lower of the two halves' rows
      const float* drow = sDm + (cc * NB1 + (in ? j : 0)) * RW;
      const float* mine = drow + h * HP;
      const float* other = drow + (1 - h) * HP;
      f2 s0 = f2_zero(), s1 = f2_zero();
#pragma unroll
      for (int t4 = 0; t4 < NH; t4 += 4)
        if (2 * t4 + 8 > i0) {
          f2 d[2], o[2];
          lds_f2(mine + t4, d[0], d[1]);
          lds_f2(other + t4, o[0], o[1]);
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const int jj = t4 / 2 + w;
            if (jj < NP && 4 * jj + 4 > i0) {
              s0 = f2_fma(d[w], x[jj < NP ? jj : 0], s0);
              s1 = f2_fma(o[w], xo[jj < NP ? jj : 0], s1);
            }
          }
        }
      return in ? f2_sum(f2_add(s0, s1)) : 0.0f;
    };
    auto swap = [&](const f2 (&x)[NP], f2 (&xo)[NP]) {
#pragma unroll
      for (int j = 0; j < NP; ++j)
        xo[j] = f2_pack(__shfl_sync(kFull, f2_x(x[j]), pt), __shfl_sync(kFull, f2_y(x[j]), pt));
    };
    // separate wind: this half's modal coefficients of div^ W = sum_a d^_a W_a, a term per lane
    f2 dw[WIND ? NP1 : 1];
    if constexpr (WIND) {
      f2 xo[NP];
      swap(ev, xo);
      float pd[2 * NP1];
#pragma unroll
      for (int t = 0; t < 2 * NP1; ++t) pd[t] = t < NH1 ? derivative(ev, xo, a, t) : 0.0f;
      __syncwarp();  // keeps the products of the two derivatives apart (registers)
#pragma unroll
      for (int t = 0; t < NH1; ++t) {
        const float v = pd[t];
        pd[t] += __shfl_sync(kFull, v, p1);
        if (D == 3) pd[t] += __shfl_sync(kFull, v, p2);
      }
#pragma unroll
      for (int j = 0; j < NP1; ++j) dw[j] = f2_pack(pd[2 * j], pd[2 * j + 1]);
      __syncwarp();
    }
    // modal reference gradients of u_a
    f2 G[D][NP1];
    {
      f2 xo[NP];
      swap(c, xo);
#pragma unroll
      for (int cc = 0; cc < D; ++cc)
#pragma unroll
        for (int j = 0; j < NP1; ++j)
          G[cc][j] = f2_pack(derivative(c, xo, cc, 2 * j), 2 * j + 1 < NH1 ? derivative(c, xo, cc, 2 * j + 1) : 0.0f);
    }
    f2 r[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) r[j] = f2_zero();
    // two points per pass (an odd last point is paired with itself at weight 0)
    constexpr int QB = vol_point_block(MODE, NQ);  // points whose test sums run together
    float* yp = sY + ((act ? el : 0) * D + a) * NB + h;  // this lane's output entries
#pragma unroll 1
    for (int q0 = 0; q0 < NQ; q0 += QB) {
      const int qe = q0 + QB < NQ ? q0 + QB : NQ;
#pragma unroll 1
      for (int q = q0; q < qe; q += 2) {
        const bool two = q + 1 < NQ;
        const int qs[2] = {q, two ? q + 1 : q};
        f2 us[2], gs[2][D], ws[2], ds[2], ff[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          us[x] = ws[x] = ds[x] = f2_zero();
#pragma unroll
          for (int cc = 0; cc < D; ++cc) gs[x][cc] = f2_zero();
        }
#pragma unroll
        for (int t4 = 0; t4 < NH; t4 += 4)
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            f2 p[2];
            lds_f2(sBt + qs[x] * NBQ + h * HP + t4, p[0], p[1]);
#pragma unroll
            for (int w = 0; w < 2; ++w) {
              const int j = t4 / 2 + w, jc = j < NP ? j : 0, j1 = j < NP1 ? j : 0;
              if (!ADJ && j < NP) us[x] = f2_fma(p[w], c[jc], us[x]);
              if constexpr (MODE != kVolSame) {
                if (j < NP) ws[x] = f2_fma(p[w], ev[jc], ws[x]);
              }
              if constexpr (WIND) {
                if (j < NP1) ds[x] = f2_fma(p[w], dw[j1], ds[x]);
              }
              if (j < NP1) {
#pragma unroll
                for (int cc = 0; cc < D; ++cc) gs[x][cc] = f2_fma(p[w], G[cc][j1], gs[x][cc]);
              }
            }
          }
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const float u = ADJ ? 0.0f : halves(f2_sum(us[x]));
          float gd[D];
#pragma unroll
          for (int cc = 0; cc < D; ++cc) gd[cc] = halves(f2_sum(gs[x][cc]));
          const float wa = MODE == kVolSame ? u : halves(f2_sum(ws[x]));
          float f = 0.0f;
          if constexpr (ROW) {  // (div^ W) u_a + W . grad^ u_a, or - W . grad^ z_a
            if (WIND) f = halves(f2_sum(ds[x])) * u;
#pragma unroll
            for (int cc = 0; cc < D; ++cc) f = fmaf(__shfl_sync(kFull, wa, el * LPE + 2 * cc), gd[cc], f);
          }
          if constexpr (MODE == kVolSame) {
            float pd = 0.0f;
#pragma unroll
            for (int cc = 0; cc < D; ++cc) pd = fmaf(M0[cc], gd[cc], pd);
            float dv = pd + __shfl_sync(kFull, pd, p1);
            if (D == 3) dv += __shfl_sync(kFull, pd, p2);
            f = dv * u;
          }
          if constexpr (COLS) {  // W = M u with the other components' u
            const float u1 = __shfl_sync(kFull, wa, p1);
            const float u2 = D == 3 ? __shfl_sync(kFull, wa, p2) : 0.0f;
#pragma unroll
            for (int cc = 0; cc < D; ++cc) {
              float W = fmaf(M1[cc], u1, M0[cc] * wa);
              if (D == 3) W = fmaf(M2[cc], u2, W);
              f = fmaf(W, gd[cc], f);
            }
          }
          if constexpr (MODE == kVolAdjW || MODE == kVolAdjSame) {  // sum_c M[c][a] sum_b u_b d^_c z_b
#pragma unroll
            for (int cc = 0; cc < D; ++cc) {
              const float v = wa * gd[cc];
              float ug = v + __shfl_sync(kFull, v, p1);
              if (D == 3) ug += __shfl_sync(kFull, v, p2);
              f = fmaf(M0[cc], ug, f);
            }
          }
          if (ADJ) f = -f;
          ff[x] = f2_dup(f * (x == 0 || two ? sWq[qs[x]] : 0.0f));
        }
#pragma unroll
        for (int t4 = 0; t4 < NH; t4 += 4) {
          f2 ta[2], tc[2];
          lds_f2(sBt + qs[0] * NBQ + h * HP + t4, ta[0], ta[1]);
          lds_f2(sBt + qs[1] * NBQ + h * HP + t4, tc[0], tc[1]);
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const int j = t4 / 2 + w;
            if (j < NP) r[j < NP ? j : 0] = f2_fma(tc[w], ff[1], f2_fma(ta[w], ff[0], r[j < NP ? j : 0]));
          }
        }
      }
      if (QB < NQ && qe < NQ) {
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          if (act && 2 * j < nh) yp[4 * j] = f2_x(r[j]) + (q0 ? yp[4 * j] : 0.0f);
          if (act && 2 * j + 1 < nh) yp[4 * j + 2] = f2_y(r[j]) + (q0 ? yp[4 * j + 2] : 0.0f);
          r[j] = f2_zero();
        }
      }
    }
    // facet lift of component a, this half: r_t += sum_fm TrM[fm][2 t + h] gam[e][fm][a]
    cp_wait<0>();
    __syncwarp();
    {
      const float* gl = sG + (act ? el : 0) * NG + a;
#pragma unroll 1
      for (int f = 0; f <= D; ++f) {
#pragma unroll
        for (int mm = 0; mm < NF; ++mm) {
          const f2 gv = f2_dup(MODE == kVolAdjSame ? gl[(f * NF + mm) * D] + gl[C::GW + (f * NF + mm) * D]
                                                 : gl[(f * NF + mm) * D]);
          const int i0 = cnbasis(D, mode_degree(D - 1, mm) - 1);  // lower degrees have no such trace
          const float* trow = sTrM + (f * NF + mm) * RW + h * HP;
#pragma unroll
          for (int t4 = 0; t4 < NH; t4 += 4)
            if (2 * t4 + 8 > i0) {
              f2 t[2];
              lds_f2(trow + t4, t[0], t[1]);
#pragma unroll
              for (int w = 0; w < 2; ++w) {
                const int j = t4 / 2 + w;
                if (j < NP && 4 * j + 4 > i0) r[j < NP ? j : 0] = f2_fma(t[w], gv, r[j < NP ? j : 0]);
              }
            }
        }
      }
    }
    if constexpr (QB < NQ) {
      if (act) {
#pragma unroll
        for (int j = 0; j < NP; ++j)
          r[j] = f2_add(r[j], f2_pack(2 * j < nh ? yp[4 * j] : 0.0f, 2 * j + 1 < nh ? yp[4 * j + 2] : 0.0f));
      }
    }
    // inverse mass, then coalesced stores of the warp's element records
    if (act) {
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        if (2 * j < nh) yp[4 * j] = f2_x(r[j]) * (ADJ ? 1.0f : invabs);
        if (2 * j + 1 < nh) yp[4 * j + 2] = f2_y(r[j]) * (ADJ ? 1.0f : invabs);
      }
    }
    __syncwarp();
    for (int t = lane; t < ne * NL; t += 32) {
      const int64_t idx = e0 * NL + t;
      out[idx] = combine_at<float>(cmb, sY[t], idx);
    }
    __syncwarp();
  }
}

}  // namespace hopu
