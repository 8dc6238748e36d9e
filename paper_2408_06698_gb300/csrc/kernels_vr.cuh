// a3 + a5 with the element's data in registers (FP32): volume term, facet lift and inverse mass;
// w = u first, a separate wind and the VJP below.
//
// A warp takes ELW = 32 / D elements and a lane owns one (element, component a) pair: the
// coefficients c of u_a, its modal reference gradients G_c = Dm_c c (c < D, dim P^{k-1}
// entries each) and the accumulators r of its test integrals stay in registers for the whole
// element, as pairs of neighbouring basis indices (f32x2.cuh).  The quadrature points are
// walked in the same order by every lane, so the basis row phi(x_q) is one broadcast
// shared-memory load for the whole warp; per point a lane forms
//   u_a = sum_i phi_i c_i,   d^_c u_a = sum_j phi_j G_c[j],
// takes the other components' u from its element's lanes (two shuffles) for W = M u
// (M = |det J| J^-1), sums its share sum_c M[c][a] d^_c u_a of div^ W over them, and adds
// f_a = w_q (div^W u_a + W . grad^ u_a) phi_i to r_i (the element-wise integration by parts of
// the conservative form, as the other volume kernels).  The facet lift
// sum_fm TrM[fm][i] gam[e][fm][a] and 1/|det J| follow; the outputs leave through a per-warp
// staging buffer with coalesced stores.  Differentiation lowers the degree and a trace does
// not raise it: Dm[c][j][i] = 0 for deg phi_j >= deg phi_i and TrM[m][i] = 0 for
// deg psi_m > deg phi_i, and both products run over the rest only.  The group's records
// arrive by cp.async, requested one group ahead (short ones are loaded directly, DIRECT below).
//
// GTAB: the reference gradients at the points come from staged tables of d phi_i / d xhat_c
// instead of the modal gradients G held in registers (d n_{b,k-1} fewer registers, more
// resident warps, d n_b instead of d n_{b,k-1} FMAs per point); 6-warp CTAs amortise the
// tables.  The autotuner picks between the two.
//
// FUSE: the element part of the back-projection R E^-1 (a7) follows in the same kernel:
// chat = det J J^-1 y (lane b mixes the element's components from the staging buffer and
// keeps component b in registers), ell = D chat (every lane forms its component's share of
// each row, D staged per CTA, the shares summed by shuffles); interior rows are combined
// into the V_h output, facet rows go to lf with the sign sigma.
//
// Separate wind (kVolWind): lane a holds the modal coefficients of the reference component
// W_a = sum_b M[a][b] w_b and those of div^ W = sum_a d^_a W_a (summed over the element's lanes
// once), evaluates both at the points with the same basis row and takes the other W by
// shuffles; one point per pass where the registers end (k = 4).
//
// VJP (kVolAdj*): the volume parts of the cotangents of u and w (kernels_adj.cuh) have the same
// shape, the gradient taken of z = ybar / |det J| and the facet moments those of the adjoint
// facet kernel; each cotangent is one run of the point loop, with w = u one for their sum.  A
// single loop for both cotangents would hold two accumulator sets beside G, which ends the
// registers at k = 3; the warp-per-element kernel that did so kept its 2 x 64 sums in local
// memory (16^3 x 6, k = 3: 1272 us against 61 us for the two launches; k = 4: 4045 against 178).
//
// Bound: the FMA units' register reads (three distinct 64-bit operands per paired FMA: a copy
// of the inner loop alone ran at 210 cycles per point and warp at k = 4, against 139 of FMA
// issue, whether the rows came once or twice from shared memory).  Measured (CUDA events, per
// launch): 32^3 x 6, k = 4, w = u 629 -> 528 us (scalar FMAs, dense Dm and TrM products and
// strided coefficient loads before), separate wind 1815 -> 761 us (a warp per element before;
// the basis split over two lanes 1054 us); 24^3 x 6, k = 3, w = u 90 -> 84 us; 16^3 x 6, k = 3,
// separate wind 57 -> 37 us.
#pragma once
#include "f32x2.cuh"
#include "kernels.cuh"

namespace hopu {

// What the point loop of the register volume kernels evaluates and tests.
enum VolMode {
  kVolSame = 0,     // y: w = u
  kVolWind = 1,     // y: separate wind
  kVolAdjU = 2,     // VJP, cotangent of u: f = -W . grad^ z
  kVolAdjW = 3,     // VJP, cotangent of w: f = -sum_c M[c][a] sum_b u_b d^_c z_b
  kVolAdjSame = 4   // VJP with w = u: the sum of both
};

// Separate wind and VJP, many points: the test sums run in blocks of points whose partial sums
// meet in the output staging buffer.  One running sum over 100 points rounded the operator 6 %
// more than a warp per element, whose points are summed pairwise; one over 46 points rounded
// the wind's cotangent 20 % more (at k = 3 the blocks cost 5 us of 61).
__host__ __device__ constexpr int vol_point_block(int mode, int nq) {
  const int lim = mode == kVolWind ? 64 : (mode == kVolAdjSame ? 100 : 16);
  return (mode != kVolSame && nq > lim) ? (nq / 8 + 1) * 2 : nq;
}

template <int D, int K, bool GTAB = false, int MODE = kVolSame>
struct VolR {
  using S = Shape<D, K>;
  static constexpr int NB = S::nb, NB1 = cnbasis(D, K - 1), NF = S::nf, NL = S::nloc, NQ = S::nq, GT = S::gt;
  static constexpr int NP = (NB + 1) / 2, NP1 = (NB1 + 1) / 2;  // pairs of basis indices
  static constexpr int ELW = 32 / D;                 // elements per warp
  static constexpr int WARPS = GTAB ? 6 : 4;
  static constexpr int NBQ = row_stride<float>(NB);  // Bt rows (point-major, as in global memory)
  static constexpr int NB4 = r4i(NB);                // Dm / TrM rows padded for 16-byte loads
  static constexpr int NG = (D + 1) * NF * D;
  static constexpr int O_DBT = NQ * NBQ;             // GTAB: [D][NQ][NBQ] reference gradients
  static constexpr int O_WQ = O_DBT + (GTAB ? D * NQ * NBQ : 0);
  static constexpr int O_DM = r4i(O_WQ + NQ);
  static constexpr int O_TRM = O_DM + (GTAB ? 0 : D * NB1 * NB4);
  static constexpr int O_W = O_TRM + (D + 1) * NF * NB4;
  static constexpr int PER_WARP = r4i(ELW * NL);     // the warp's element records: in, and out
  static constexpr int GW = r4i(ELW * NG);           // the warp's facet moments
  // few coefficients and no other component's: a lane loads its own instead of taking them from the
  // buffer (2D, k = 2, 160^2, w = u, with the rounded geometry: 12.0 -> 10.2 us)
  static constexpr bool DIRECT = (D == 2 || K == 1) && MODE != kVolWind && MODE != kVolAdjU;
  static constexpr int NBUF = DIRECT ? 1 : MODE == kVolSame ? 2 : 3;  // records: in (none, one or two fields), out
  static constexpr int NGAM = MODE == kVolAdjSame ? 2 : 1;
  static constexpr int O_G = O_W + WARPS * NBUF * PER_WARP;
  static constexpr size_t SMEM = size_t(O_G + WARPS * NGAM * GW) * 4;
  static constexpr int NLR = row_stride<float>(NL);  // rows of the row-major D in global memory
  static constexpr int NDP = D * NB4;                // fused back-projection: D [NL][D blocks of NB4]
  static constexpr int O_D = O_G + WARPS * GW;
  static constexpr size_t SMEM_FUSE = size_t(O_D + NL * NDP) * 4;
  static constexpr int REGS = (MODE == kVolWind ? 3 * NB + NB1 : 2 * NB) + (GTAB ? 0 : D * NB1);  // c, r, G of a lane (and w, div w)
  static constexpr int XP = REGS <= 140 ? 2 : 1;  // quadrature points per pass
  static constexpr int MINB = GTAB ? 2 : (REGS <= 90 ? 3 : 2);  // resident CTAs asked of the register allocator
  static constexpr bool OK = REGS <= 190 && SMEM <= 200 * 1024;
  static constexpr bool FUSE_OK = OK && SMEM_FUSE <= 200 * 1024;
};

// A warp copies the records of ne consecutive elements (NV values each) starting at element e0.
template <int NV, int GROUP>
__device__ __forceinline__ void warp_copy_records(float* dst, const float* src, int64_t e0, int ne, int lane) {
  constexpr int CH = gcd_pow2(GROUP * NV * 4);  // a whole group starts on a multiple of its size
  const char* s = reinterpret_cast<const char*>(src + e0 * NV);
  char* d = reinterpret_cast<char*>(dst);
  if (ne == GROUP) {
    for (int t = lane; t < GROUP * NV * 4 / CH; t += 32) cp_async<CH>(d + t * CH, s + t * CH);
  } else {
    for (int t = lane; t < ne * NV; t += 32) cp_async<4>(d + 4 * t, s + 4 * t);
  }
}

// in1: the field evaluated at the points (u; the wind for kVolAdjU); in2: the wind (kVolWind) or
// the cotangent ybar (VJP); gam2: the wind's moments (kVolAdjSame).
template <int D, int K, bool FUSE, bool GTAB, int MODE>
__global__ void __launch_bounds__(32 * VolR<D, K, GTAB, MODE>::WARPS, VolR<D, K, GTAB, MODE>::MINB)
    k_volume_r(DevMesh m, DevTabs tb, const float* __restrict__ in1, const float* __restrict__ in2,
               const float* __restrict__ gam, const float* __restrict__ gam2, float* out, Combine cmb,
               float* __restrict__ lf) {
  using C = VolR<D, K, GTAB, MODE>;
  constexpr bool WIND = MODE == kVolWind, ADJ = MODE >= kVolAdjU;
  constexpr bool ROW = WIND || MODE == kVolAdjU;   // the wind enters through its reference components
  using S = Shape<D, K>;
  constexpr int NB = C::NB, NB1 = C::NB1, NF = C::NF, NL = C::NL, NQ = C::NQ, GT = C::GT;
  constexpr int NBQ = C::NBQ, NB4 = C::NB4, NG = C::NG, ELW = C::ELW, NP = C::NP, NP1 = C::NP1;
  extern __shared__ __align__(16) float sm[];
  pdl_trigger();
  {
    const float* Btg = static_cast<const float*>(tb.Bt);
    const float* Wqg = static_cast<const float*>(tb.Wq);
    const float* Dmg = static_cast<const float*>(tb.Dm);
    const float* TrMg = static_cast<const float*>(tb.TrM);
    for (int t = threadIdx.x; t < NQ * NBQ; t += blockDim.x) sm[t] = Btg[t];
    if (GTAB) {
      const float* dBtg = static_cast<const float*>(tb.dBt);
      for (int t = threadIdx.x; t < D * NQ * NBQ; t += blockDim.x) sm[C::O_DBT + t] = dBtg[t];
    }
    for (int t = threadIdx.x; t < NQ; t += blockDim.x) sm[C::O_WQ + t] = Wqg[t];
    for (int t = threadIdx.x; t < (GTAB ? 0 : D * NB1 * NB4); t += blockDim.x) {
      const int row = t / NB4, i = t - row * NB4;
      sm[C::O_DM + t] = i < NB ? Dmg[row * NB + i] : 0.0f;
    }
    for (int t = threadIdx.x; t < (D + 1) * NF * NB4; t += blockDim.x) {
      const int row = t / NB4, i = t - row * NB4;
      sm[C::O_TRM + t] = i < NB ? TrMg[row * NB + i] : 0.0f;
    }
    if (FUSE) {  // row rr, component block b: D[rr][b*nb + i] at rr*NDP + b*NB4 + i (16-byte rows)
      const float* Dg = static_cast<const float*>(tb.Drow);
      for (int t = threadIdx.x; t < NL * C::NDP; t += blockDim.x) {
        const int rr = t / C::NDP, col = t - rr * C::NDP, b = col / NB4, i = col - b * NB4;
        sm[C::O_D + t] = i < NB ? Dg[rr * C::NLR + b * NB + i] : 0.0f;
      }
    }
  }
  const float* sBt = sm;
  const float* sWq = sm + C::O_WQ;
  const float* sDm = sm + C::O_DM;
  const float* sTrM = sm + C::O_TRM;
  pdl_wait();
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool lane_on = lane < D * ELW;
  const int el = lane_on ? lane / D : 0;
  const int a = lane_on ? lane - el * D : 0;
  const int a1 = (a + 1) % D, a2 = (a + 2) % D;
  // the other lanes of the element (idle lanes talk to themselves)
  const int p1 = lane_on ? el * D + a1 : lane;
  const int p2 = lane_on ? el * D + a2 : lane;
  float* sIn = sm + C::O_W + warp * C::NBUF * C::PER_WARP;
  float* sY = sIn + (C::DIRECT ? 0 : C::PER_WARP);
  float* sIn2 = sY + (MODE == kVolSame ? 0 : C::PER_WARP);
  float* sG = sm + C::O_G + warp * C::NGAM * C::GW;
  const int64_t ngroups = (m.E + ELW - 1) / ELW, gstep = (int64_t)gridDim.x * C::WARPS;
  auto count = [&](int64_t g) { return (m.E - g * ELW < ELW) ? (int)(m.E - g * ELW) : ELW; };
  int64_t grp = (int64_t)warp * gridDim.x + blockIdx.x;
  auto request = [&](int64_t g) {
    if (C::DIRECT) return;
    warp_copy_records<NL, ELW>(sIn, in1, g * ELW, count(g), lane);
    if (MODE != kVolSame) warp_copy_records<NL, ELW>(sIn2, in2, g * ELW, count(g), lane);
  };
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
    // c: the coefficients whose gradient is taken (u; z = ybar / |det J| in the VJP);
    // ev: those evaluated at the points (c itself when w = u; the modal W_a = sum_b M[a][b] w_b,
    // the wind's reference component a; u in the wind's cotangent)
    f2 c[NP], ev[MODE == kVolSame ? 1 : NP];
    if constexpr (C::DIRECT) {
      const float* pc = (ADJ ? in2 : in1) + e * NL + a * NB;
      const float* pe = in1 + e * NL + a * NB;
      const float sc = ADJ ? invabs : 1.0f;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const bool pair = 2 * j + 1 < NB;
        c[j] = f2_pack(__ldg(pc + 2 * j), pair ? __ldg(pc + 2 * j + 1) : 0.0f);
        if constexpr (ADJ) {
          c[j] = f2_mul(c[j], f2_dup(sc));
          ev[j] = f2_pack(__ldg(pe + 2 * j), pair ? __ldg(pe + 2 * j + 1) : 0.0f);
        }
      }
    } else {
      cp_wait<0>();
      __syncwarp();
      const int oe = (act ? el : 0) * NL, o = oe + a * NB;
      const float* sC = ADJ ? sIn2 : sIn;
      const float sc = ADJ ? invabs : 1.0f;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const bool pair = 2 * j + 1 < NB;
        c[j] = f2_pack(sC[o + 2 * j], pair ? sC[o + 2 * j + 1] : 0.0f);
        if constexpr (ADJ) c[j] = f2_mul(c[j], f2_dup(sc));
        if constexpr (ROW) {
          const float* sWn = WIND ? sIn2 : sIn;
          float v[2] = {0.0f, 0.0f};
#pragma unroll
          for (int w = 0; w < 2; ++w)
            if (2 * j + w < NB) {
#pragma unroll
              for (int b = 0; b < D; ++b) v[w] = fmaf(M0[b], sWn[oe + b * NB + 2 * j + w], v[w]);
            }
          ev[j] = f2_pack(v[0], v[1]);
        } else if constexpr (ADJ) {
          ev[j] = f2_pack(sIn[o + 2 * j], pair ? sIn[o + 2 * j + 1] : 0.0f);
        }
      }
    }
    __syncwarp();
    // this group's facet moments and the next group's coefficients arrive during the points
    warp_copy_records<NG, ELW>(sG, gam, e0, ne, lane);
    if (MODE == kVolAdjSame) warp_copy_records<NG, ELW>(sG + C::GW, gam2, e0, ne, lane);
    if (grp + gstep < ngroups) request(grp + gstep);
    cp_commit();
    // entry `row` of the modal reference derivative Dm_cc of the coefficients x
    auto derivative = [&](const f2 (&x)[NP], int cc, int row) -> float {
      const int i0 = cnbasis(D, mode_degree(D, row));  // the first index of higher degree
      const float* drow = sDm + (cc * NB1 + row) * NB4;
      f2 s = f2_zero();
#pragma unroll
      for (int i = 0; i < NB; i += 4)
        if (i + 4 > i0) {
          f2 t[2];
          lds_f2(drow + i, t[0], t[1]);
#pragma unroll
          for (int w = 0; w < 2; ++w)
            if (i + 2 * w + 2 > i0 && i + 2 * w < NB) s = f2_fma(t[w], x[i / 2 + w < NP ? i / 2 + w : 0], s);
        }
      return f2_sum(s);
    };
    // separate wind: modal coefficients of div^ W = sum_a d^_a W_a, a term from each lane
    f2 dw[WIND ? NP1 : 1];
    if constexpr (WIND) {
      float pd[NB1];
#pragma unroll
      for (int j = 0; j < NB1; ++j) pd[j] = derivative(ev, a, j);
      __syncwarp();  // keeps the products of the two derivatives apart (registers)
#pragma unroll
      for (int j = 0; j < NB1; ++j) {
        const float v = pd[j];
        pd[j] += __shfl_sync(kFull, v, p1);
        if (D == 3) pd[j] += __shfl_sync(kFull, v, p2);
      }
#pragma unroll
      for (int j = 0; j < NP1; ++j) dw[j] = f2_pack(pd[2 * j], 2 * j + 1 < NB1 ? pd[2 * j + 1 < NB1 ? 2 * j + 1 : 0] : 0.0f);
      __syncwarp();
    }
    // modal reference gradients of u_a (not with GTAB)
    constexpr int NG1 = GTAB ? 1 : NP1;
    f2 G[D][NG1];
    if constexpr (!GTAB) {
#pragma unroll
      for (int cc = 0; cc < D; ++cc)
#pragma unroll
        for (int j = 0; j < NP1; ++j)
          G[cc][j] = f2_pack(derivative(c, cc, 2 * j), 2 * j + 1 < NB1 ? derivative(c, cc, 2 * j + 1) : 0.0f);
    }
    f2 r[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) r[j] = f2_zero();
    // two points per pass where the registers allow it: the loads and shuffles of one overlap
    // the arithmetic of the other (an odd last point is paired with itself at weight 0)
    constexpr int XP = C::XP;
    constexpr int QB = vol_point_block(MODE, NQ);  // points whose test sums run together
    float* yp = sY + ((act ? el : 0) * D + a) * NB;  // this lane's output entries
#pragma unroll 1
    for (int q0 = 0; q0 < NQ; q0 += QB) {
      const int qe = q0 + QB < NQ ? q0 + QB : NQ;
#pragma unroll 1
      for (int q = q0; q < qe; q += XP) {
        const bool two = q + 1 < NQ;
        const int qs[2] = {q, two ? q + 1 : q};
        float u[XP], gd[XP][D], wa[XP], dvs[XP];
        {
          f2 us[XP], gs[XP][D], ws[XP], ds[XP];
#pragma unroll
          for (int x = 0; x < XP; ++x) {
            us[x] = ws[x] = ds[x] = f2_zero();
#pragma unroll
            for (int cc = 0; cc < D; ++cc) gs[x][cc] = f2_zero();
          }
#pragma unroll
          for (int i = 0; i < NB; i += 4)
#pragma unroll
            for (int x = 0; x < XP; ++x) {
              f2 t[2];
              lds_f2(sBt + qs[x] * NBQ + i, t[0], t[1]);
#pragma unroll
              for (int w = 0; w < 2; ++w) {
                const int j = i / 2 + w;
                if (!ADJ && j < NP) us[x] = f2_fma(t[w], c[j < NP ? j : 0], us[x]);
                if constexpr (MODE != kVolSame) {
                  if (j < NP) ws[x] = f2_fma(t[w], ev[j < NP ? j : 0], ws[x]);
                }
                if constexpr (WIND) {
                  if (j < NP1) ds[x] = f2_fma(t[w], dw[j < NP1 ? j : 0], ds[x]);
                }
                if constexpr (!GTAB) {
                  if (j < NP1) {
#pragma unroll
                    for (int cc = 0; cc < D; ++cc) gs[x][cc] = f2_fma(t[w], G[cc][j < NG1 ? j : 0], gs[x][cc]);
                  }
                }
              }
            }
          if constexpr (GTAB) {  // d^_c u_a = sum_i (d phi_i / d xhat_c)(x_q) c_i
#pragma unroll
            for (int cc = 0; cc < D; ++cc)
#pragma unroll
              for (int i = 0; i < NB; i += 4)
#pragma unroll
                for (int x = 0; x < XP; ++x) {
                  f2 t[2];
                  lds_f2(sm + C::O_DBT + (cc * NQ + qs[x]) * NBQ + i, t[0], t[1]);
#pragma unroll
                  for (int w = 0; w < 2; ++w)
                    if (i / 2 + w < NP) gs[x][cc] = f2_fma(t[w], c[i / 2 + w < NP ? i / 2 + w : 0], gs[x][cc]);
                }
          }
#pragma unroll
          for (int x = 0; x < XP; ++x) {
            u[x] = f2_sum(us[x]);
            wa[x] = MODE == kVolSame ? u[x] : f2_sum(ws[x]);
            dvs[x] = f2_sum(ds[x]);
#pragma unroll
            for (int cc = 0; cc < D; ++cc) gd[x][cc] = f2_sum(gs[x][cc]);
          }
        }
        f2 ff[XP];
#pragma unroll
        for (int x = 0; x < XP; ++x) {
          float f = 0.0f;
          if constexpr (ROW) {  // (div^ W) u_a + W . grad^ u_a, or - W . grad^ z_a
            if (WIND) f = dvs[x] * u[x];
#pragma unroll
            for (int cc = 0; cc < D; ++cc) f = fmaf(__shfl_sync(kFull, wa[x], el * D + cc), gd[x][cc], f);
          }
          if constexpr (MODE == kVolSame) {
            // div^ W = sum_b sum_c M[c][b] d^_c u_b
            float pd = 0.0f;
#pragma unroll
            for (int cc = 0; cc < D; ++cc) pd = fmaf(M0[cc], gd[x][cc], pd);
            float dv = pd + __shfl_sync(kFull, pd, p1);
            if (D == 3) dv += __shfl_sync(kFull, pd, p2);
            f = dv * u[x];
          }
          if constexpr (COLS) {  // W = M u with the other components' u
            const float u1 = __shfl_sync(kFull, wa[x], p1);
            const float u2 = D == 3 ? __shfl_sync(kFull, wa[x], p2) : 0.0f;
#pragma unroll
            for (int cc = 0; cc < D; ++cc) {
              float W = fmaf(M1[cc], u1, M0[cc] * wa[x]);
              if (D == 3) W = fmaf(M2[cc], u2, W);
              f = fmaf(W, gd[x][cc], f);
            }
          }
          if constexpr (MODE == kVolAdjW || MODE == kVolAdjSame) {  // sum_c M[c][a] sum_b u_b d^_c z_b
#pragma unroll
            for (int cc = 0; cc < D; ++cc) {
              const float v = wa[x] * gd[x][cc];
              float ug = v + __shfl_sync(kFull, v, p1);
              if (D == 3) ug += __shfl_sync(kFull, v, p2);
              f = fmaf(M0[cc], ug, f);
            }
          }
          if (ADJ) f = -f;
          ff[x] = f2_dup(f * (x == 0 || two ? sWq[qs[x]] : 0.0f));
        }
#pragma unroll
        for (int i = 0; i < NB; i += 4) {
          f2 t[XP][2];
#pragma unroll
          for (int x = 0; x < XP; ++x) lds_f2(sBt + qs[x] * NBQ + i, t[x][0], t[x][1]);
#pragma unroll
          for (int x = 0; x < XP; ++x)
#pragma unroll
            for (int w = 0; w < 2; ++w) {
              const int j = i / 2 + w;
              if (j < NP) r[j < NP ? j : 0] = f2_fma(t[x][w], ff[x], r[j < NP ? j : 0]);
            }
        }
      }
      if (QB < NQ && qe < NQ) {
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          if (act) {
            yp[2 * j] = f2_x(r[j]) + (q0 ? yp[2 * j] : 0.0f);
            if (2 * j + 1 < NB) yp[2 * j + 1] = f2_y(r[j]) + (q0 ? yp[2 * j + 1] : 0.0f);
          }
          r[j] = f2_zero();
        }
      }
    }
    // facet lift of component a: r_i += sum_fm TrM[fm][i] gam[e][fm][a]
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
          const float* trow = sTrM + (f * NF + mm) * NB4;
#pragma unroll
          for (int i = 0; i < NB; i += 4)
            if (i + 4 > i0) {
              f2 t[2];
              lds_f2(trow + i, t[0], t[1]);
#pragma unroll
              for (int w = 0; w < 2; ++w) {
                const int j = i / 2 + w;
                if (j < NP && 2 * j + 2 > i0) r[j < NP ? j : 0] = f2_fma(t[w], gv, r[j < NP ? j : 0]);
              }
            }
        }
      }
    }
    if constexpr (QB < NQ) {
      if (act) {
#pragma unroll
        for (int j = 0; j < NP; ++j) r[j] = f2_add(r[j], f2_pack(yp[2 * j], 2 * j + 1 < NB ? yp[2 * j + 1] : 0.0f));
      }
    }
    // inverse mass, then coalesced stores of the warp's element records
    if (act) {
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        yp[2 * j] = f2_x(r[j]) * (ADJ ? 1.0f : invabs);
        if (2 * j + 1 < NB) yp[2 * j + 1] = f2_y(r[j]) * (ADJ ? 1.0f : invabs);
      }
    }
    __syncwarp();
    if constexpr (!FUSE) {
      for (int t = lane; t < ne * NL; t += 32) {
        const int64_t idx = e0 * NL + t;
        out[idx] = combine_at<float>(cmb, sY[t], idx);
      }
    } else {
      // chat[b][i] = sum_c Pi[b][c] y[c][i], Pi = det J J^-1 (lane b of the element), kept in
      // registers; row rr of ell = D chat is the sum over the element's lanes of
      // sum_i D[rr][b*nb + i] chat[b][i], reduced by shuffles and written by lane rr / nb
      float Pi[D];
#pragma unroll
      for (int cc = 0; cc < D; ++cc) Pi[cc] = __ldg(gp + D * D + a * D + cc);
      const float* ye = sY + (act ? el : 0) * NL;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        float v[2] = {0.0f, 0.0f};
#pragma unroll
        for (int w = 0; w < 2; ++w)
          if (2 * j + w < NB) {
#pragma unroll
            for (int cc = 0; cc < D; ++cc) v[w] = fmaf(Pi[cc], ye[cc * NB + 2 * j + w], v[w]);
          }
        r[j] = f2_pack(v[0], v[1]);
      }
      const float* sD = sm + C::O_D + a * NB4;
      const int* codes = m.efc + e * (D + 1);
#pragma unroll 1
      for (int rr = 0; rr < NL; ++rr) {
        const float* drow = sD + rr * C::NDP;
        f2 s = f2_zero();
#pragma unroll
        for (int i = 0; i < NB; i += 4) {
          f2 t[2];
          lds_f2(drow + i, t[0], t[1]);
#pragma unroll
          for (int w = 0; w < 2; ++w)
            if (i / 2 + w < NP) s = f2_fma(t[w], r[i / 2 + w < NP ? i / 2 + w : 0], s);
        }
        const float part = f2_sum(s);
        float v = part + __shfl_sync(kFull, part, p1);
        if (D == 3) v += __shfl_sync(kFull, part, p2);
        if (act && rr / NB == a) {
          if (rr < (D + 1) * NF) {
            lf[e * (D + 1) * NF + rr] = (__ldg(codes + rr / NF) & 2) ? -v : v;
          } else {
            const int64_t idx = m.NF * NF + e * S::nint + (rr - (D + 1) * NF);
            out[idx] = combine_at<float>(cmb, v, idx);
          }
        }
      }
    }
    __syncwarp();
  }
}

}  // namespace hopu
