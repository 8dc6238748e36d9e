// a4 with the facet's data in registers (FP32): the facet flux moments of the HOPU form.
//
// A warp takes FPW = 32 / D facets and a lane owns one (facet, component a) pair.  Per facet
// mode m (the orthonormal facet basis psi_m) the lane forms its component of both sides'
// modal traces tau^X_m = sum_i TrM_{f_X}[m][i] c^X_a[i] from the coefficients it holds in
// registers (the degree <= 1 terms compensated, as in k_facet), the jump J_m = tau^A - tau^B
// and the averaged wind <w>_m; the facet's lanes sum J_m . n and <w>_m . n by shuffles, which
// gives (I - Pi^l) J in modal form (modes below dim P^l(F) keep only (J_m . n) n).  The facet
// quadrature points are then walked in the same order by every lane, with w.n, J and
// (I - Pi^l) J at the point, h = w_q/2 |w.n| (I - Pi^l) J and -w_q/2 (w.n) J accumulated into
// the moments alpha_m and beta_m in registers; beta's low modes keep their normal part
// ((I - Pi^l) h), both are scaled by a_F and written element-major as in k_facet
// (alpha + beta for side A, alpha - beta for side B).  Boundary facets (fb == fa) write side A
// only; inlet facets take side B's trace of u from the given data and keep the wind's own
// trace.
//
// The points of the collapsed rule are a grid (t_i, t_j) on which psi_m = A_p(t_i) B_m(t_j):
// a row j first contracts the modes over their second index (g_p = sum B_m c_m), each of its
// points then takes K + 1 products instead of dim P^K(F), and the test runs the same way back.
// At k = 4 (49 points, 15 modes) that is 22 FMAs per point and field instead of 45.  Fields
// that share a table value run as register pairs (f32x2.cuh): (J, (I - Pi^l) J) at the points,
// (alpha, beta) in the test, neighbouring basis indices in the traces.  A basis function of
// degree n has a trace of degree <= n, so TrM[m][i] = 0 where deg psi_m > deg phi_i: those
// products are left out, and only the modes of degree <= 1 have degree <= 1 terms to
// compensate.  Where a record is long (STAGE) the records of a group's two sides arrive in shared memory by
// 16-byte cp.async (one buffer per warp: the next group's records are requested as soon as
// the current ones are in registers, and land during its points); loaded straight from
// global memory, a lane's 35 consecutive values at k = 4 cost about 30 cache lines per
// warp-wide load.  A separate wind's records go through the same buffer between the two.
//
// Bound: FP32 FMA and issue (two scheduler-resident warps short of hiding the shuffles).
// Measured (CUDA events, per launch): 32^3 x 6, k = 4, w = u 443 -> 288 us (dense points and
// scalar FMAs before; 390 us with pairs and staged records alone), separate wind 1235 -> 435 us
// (a warp per facet before); 13^3 x 6, k = 5, separate wind 207 -> 64 us; 16^3 x 6, k = 3,
// separate wind 42 -> 29 us.  Three resident CTAs at k <= 4 although k = 4 then spills about
// ten registers outside the point loop.
#pragma once
#include "f32x2.cuh"
#include "kernels.cuh"

namespace hopu {

template <int D, int K>
struct FacR {
  using S = Shape<D, K>;
  static constexpr int NB = S::nb, NF = S::nf, NL = S::nloc, NQF = S::nqf;
  static constexpr int FPW = 32 / D;     // facets per warp
  static constexpr int WARPS = 4;
  static constexpr int NB4 = r4i(NB), NBP = (NB + 1) / 2;  // basis indices: padded row, pairs
  static constexpr int O_TRM = 0;                                // [(D+1) NF][NB4]
  static constexpr int O_LOW = O_TRM + (D + 1) * NF * NB4;       // [D+1][D+1][4]  TrM[f][m < 4][i <= D], mode-minor
  static constexpr int MF = S::mf;                               // facet points per direction
  static constexpr int AST = r4i(2 * (K + 1)), BST = D == 3 ? r4i(2 * NF) : 0;
  static constexpr int O_A = O_LOW + (D + 1) * (D + 1) * 4;      // [MF][AST]  A_p(t_i), each value twice
  static constexpr int O_B = O_A + MF * AST;                     // [MF][BST]  B_m(t_j), each value twice (3D)
  static constexpr int O_WF = O_B + MF * BST;                    // [NQF]      w_q / 2, i fastest
  static constexpr int O_GEO = O_WF + r4i(NQF);                  // per warp: FPW (n, a_F)
  static constexpr int GEO = r4i(FPW * (D + 1));
  static constexpr int O_REC = O_GEO + WARPS * GEO;              // per warp: 2 FPW coefficient records
  // a record starts at its element's offset modulo 16 bytes; strides keep scalar reads of
  // neighbouring lanes in different banks
  static constexpr int CH = (NL % 4 == 0 ? NL : r4i(NL + 3)) / 4;  // 16-byte chunks of a record
  static constexpr int RST = 4 * (CH % 2 ? CH : CH + 1);
  // 2D and k = 1: a lane's 3 to 15 coefficients of a side lie in one or two cache lines, and it loads
  // them itself; through the buffer the SSP-RK3 substep of a 160^2 k = 1 square took 58.9 us (53.7), of
  // 8^2 k = 4 43.9 (41.8), and a separate wind waited for its turn of the buffer (32 triangles, k = 4:
  // 6.0 against 4.7 us an apply)
  static constexpr bool STAGE = D == 3 && K > 1;
  static constexpr size_t SMEM = size_t(O_REC + (STAGE ? WARPS * 2 * FPW * RST : 0)) * 4;
  static constexpr int REGS = 2 * NB + 3 * NF;                   // coefficients and the modal vectors
  // 3D k = 2: at three CTAs an apply with w = u of 12^3 x 6 (2074 groups, 1824 warps) took two rounds and
  // 16.2 us, at four (12 bytes spilled) 12.1; 20^3 37.1 -> 36.2 us
  static constexpr int MINB = REGS <= 40 ? 4 : REGS <= 120 ? 3 : 2;
};

// Both sides' records of a group's facets into the warp's buffer: record r < FPW is side A of
// facet r, record FPW + r its side B (pa, pb: this lane's facet's elements * 4 + f).  A record is
// copied by CH lanes, RPI records per step, as the 16-byte chunks that hold it.
template <int D, int K>
__device__ __forceinline__ void facet_request(const float* src, float* sRec, int pa, int pb, int lane) {
  using C = FacR<D, K>;
  if (!C::STAGE) {
    cp_commit();  // the geometry
    return;
  }
  constexpr int NL = C::NL, FPW = C::FPW, CH = C::CH, RST = C::RST;
  constexpr int RPI = CH <= 16 ? (CH <= 8 ? 4 : 2) : 1, LPR = 32 / RPI;
  const int cr = lane / LPR, cc0 = lane - cr * LPR;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int ids = (side ? pb : pa) >> 2;
#pragma unroll 5
    for (int r0 = 0; r0 < FPW; r0 += RPI) {
      const int r = r0 + cr;
      const int64_t start = (int64_t)__shfl_sync(kFull, ids, r * D & 31) * NL;
      const int shift = NL % 4 ? int(start & 3) : 0;
      float* dst = sRec + (side * FPW + r) * RST;
#pragma unroll
      for (int c = cc0; c < ((CH + LPR - 1) / LPR) * LPR; c += LPR) {
        const int left = shift + NL - 4 * c;  // floats up to the record's end
        if (r < FPW && left > 0) {
          if (NL % 4) cp_async_part(dst + 4 * c, src + (start - shift) + 4 * c, left < 4 ? 4 * left : 16);
          else cp_async<16>(dst + 4 * c, src + start + 4 * c);
        }
      }
    }
  }
  cp_commit();
}

// Component a of facet fl's record of one side, as pairs of neighbouring basis indices: from the
// buffer, or (unless STAGE) from element e of src.
template <int D, int K>
__device__ __forceinline__ void facet_take(const float* src, const float* sRec, int side, int fl, int a, int64_t e,
                                           f2 (&c)[FacR<D, K>::NBP]) {
  using C = FacR<D, K>;
  constexpr int NB = C::NB, NL = C::NL;
  if constexpr (!C::STAGE) {
    const float* p = src + e * NL + a * NB;
#pragma unroll
    for (int j = 0; j < C::NBP; ++j) c[j] = f2_pack(__ldg(p + 2 * j), 2 * j + 1 < NB ? __ldg(p + 2 * j + 1) : 0.0f);
    return;
  }
  const float* p = sRec + (side * C::FPW + fl) * C::RST + a * NB;
  if constexpr (NL % 4 == 0 && NB % 4 == 0) {
#pragma unroll
    for (int j = 0; j < C::NBP; j += 2) lds_f2(p + 2 * j, c[j], c[j + 1]);
  } else {
    if (NL % 4) p += (e * NL) & 3;
#pragma unroll
    for (int j = 0; j < C::NBP; ++j) c[j] = f2_pack(p[2 * j], 2 * j + 1 < NB ? p[2 * j + 1] : 0.0f);
  }
}

// Plain part of mode mm's trace (row: TrM[f][mm]) from the basis indices that have one: those of
// the mode's degree on, and, unless all are wanted, past the compensated ones (i <= D) for the
// modes of degree <= 1.
template <int D, int K>
__device__ __forceinline__ float facet_plain_trace(int mm, const float* row, const f2 (&c)[FacR<D, K>::NBP], bool all) {
  constexpr int NB = FacR<D, K>::NB, NBP = FacR<D, K>::NBP;
  const int n = mode_degree(D - 1, mm);
  const int i0 = (n <= 1 && !all) ? D + 1 : cnbasis(D, n - 1);
  f2 s = f2_zero();
  float odd = 0.0f;
#pragma unroll
  for (int i = 0; i < NB; i += 4)
    if (i + 4 > i0) {
      f2 t[2];
      lds_f2(row + i, t[0], t[1]);
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int j = i + 2 * w;
        if (j >= NB || j + 2 <= i0) continue;
        const f2 cj = c[j / 2 < NBP ? j / 2 : 0];
        if (j < i0) odd = f2_y(t[w]) * f2_y(cj);
        else s = f2_fma(t[w], cj, s);
      }
    }
  return (i0 & 1) ? f2_sum(s) + odd : f2_sum(s);
}

// Tables of a facet kernel: trace matrices, the point factors A and B (each value twice), w_q / 2.
template <int D, int K>
__device__ __forceinline__ void facet_stage_tables(const DevTabs& tb, float* sm) {
  using C = FacR<D, K>;
  constexpr int NB = C::NB, NF = C::NF, NB4 = C::NB4, MF = C::MF, AST = C::AST, BST = C::BST;
  const float* TrMg = static_cast<const float*>(tb.TrM);
  const float* FAg = static_cast<const float*>(tb.FacA);  // [MF][K+1]
  const float* FBg = static_cast<const float*>(tb.FacB);  // [MF][NF]
  const float* Wfg = static_cast<const float*>(tb.Wf);
  for (int t = threadIdx.x; t < (D + 1) * NF * NB4; t += blockDim.x) {
    const int row = t / NB4, i = t - row * NB4;
    sm[C::O_TRM + t] = i < NB ? TrMg[row * NB + i] : 0.0f;
  }
  for (int t = threadIdx.x; t < (D + 1) * (D + 1) * 4; t += blockDim.x) {
    const int mm = t & 3, i = (t >> 2) % (D + 1), f = (t >> 2) / (D + 1);
    sm[C::O_LOW + t] = mm < NF ? TrMg[(f * NF + mm) * NB + i] : 0.0f;
  }
  for (int t = threadIdx.x; t < MF * AST; t += blockDim.x) {
    const int i = t / AST, p = (t - i * AST) >> 1;
    sm[C::O_A + t] = p <= K ? FAg[i * (K + 1) + p] : 0.0f;
  }
  if constexpr (D == 3) {
    for (int t = threadIdx.x; t < MF * BST; t += blockDim.x) {
      const int j = t / BST, mm = (t - j * BST) >> 1;
      sm[C::O_B + t] = mm < NF ? FBg[j * NF + mm] : 0.0f;
    }
  }
  for (int t = threadIdx.x; t < C::NQF; t += blockDim.x)
    sm[C::O_WF + t] = 0.5f * Wfg[D == 3 ? (t % MF) * MF + t / MF : t];  // rule order: q = i MF + j
}

template <int D, int K, bool WSEP>
__global__ void __launch_bounds__(32 * FacR<D, K>::WARPS, FacR<D, K>::MINB)
    k_facet_r(DevMesh m, DevTabs tb, const float* __restrict__ uL, const float* __restrict__ wL, int lconst,
              const int8_t* __restrict__ facet_l, float* __restrict__ gam, double* __restrict__ diss) {
  using C = FacR<D, K>;
  constexpr int NF = C::NF, NB4 = C::NB4, FPW = C::FPW, NBP = C::NBP, RST = C::RST;
  constexpr int MF = C::MF, AST = C::AST, BST = C::BST;
  extern __shared__ __align__(16) float sm[];
  pdl_trigger();
  facet_stage_tables<D, K>(tb, sm);
  const float* sTrM = sm + C::O_TRM;
  const float* sLow = sm + C::O_LOW;
  const float* sA = sm + C::O_A;
  const float* sB = sm + C::O_B;
  const float* sWf = sm + C::O_WF;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* sRec = sm + C::O_REC + warp * 2 * FPW * RST;
  float* sGeo = sm + C::O_GEO + warp * C::GEO;
  const bool lane_on = lane < D * FPW;
  const int fl = lane_on ? lane / D : 0;
  const int a = lane_on ? lane - fl * D : 0;
  const int p1 = lane_on ? fl * D + (a + 1) % D : lane;
  const int p2 = lane_on ? fl * D + (a + 2) % D : lane;
  auto lanes_sum = [&](float v) {
    float s = v + __shfl_sync(kFull, v, p1);
    if (D == 3) s += __shfl_sync(kFull, v, p2);
    return s;
  };
  const int64_t ngroups = (m.NF + FPW - 1) / FPW, gstep = (int64_t)gridDim.x * C::WARPS;
  auto request = [&](const float* src, int pa, int pb) { facet_request<D, K>(src, sRec, pa, pb, lane); };
  auto take = [&](const float* src, int side, int64_t e, f2 (&c)[NBP]) { facet_take<D, K>(src, sRec, side, fl, a, e, c); };
  auto plain = [&](int mm, const float* row, const f2 (&c)[NBP], bool all) {
    return facet_plain_trace<D, K>(mm, row, c, all);
  };
  int64_t grp = (int64_t)warp * gridDim.x + blockIdx.x;
  int npa = 0, npb = 0;  // the next group's elements of this lane's facet
  auto sides = [&](int64_t g) {
    if (g >= ngroups) return;
    const int64_t F = g * FPW + ((lane_on && g * FPW + fl < m.NF) ? fl : 0);
    npa = m.fa[F];
    npb = m.fb[F];
  };
  // (n, a_F) of a group's facets
  auto request_geo = [&](int64_t g) {
    const int64_t i0 = g * FPW * (D + 1), end = m.NF * (D + 1);
    for (int t = lane; t < FPW * (D + 1); t += 32)
      if (i0 + t < end) cp_async<4>(sGeo + t, m.fgeoF + i0 + t);
  };
  sides(grp);
  if (grp < ngroups) request_geo(grp);  // mesh data: before the wait for the previous kernel
  pdl_wait();
  __syncthreads();
  if (grp < ngroups) request(uL, npa, npb);
  for (; grp < ngroups; grp += gstep) {
    const int64_t F0 = grp * FPW;
    const bool act = lane_on && F0 + fl < m.NF;
    const int64_t F = act ? F0 + fl : F0;  // inactive lanes compute the group's first facet
    const int pa = npa, pb = npb;
    const int64_t eA = pa >> 2, eB = pb >> 2;
    const int fA = pa & 3, fB = pb & 3;
    sides(grp + gstep);
    const int l = facet_l ? int(facet_l[F]) : lconst;
    const int nl = (l < 0) ? 0 : cnbasis(D - 1, l);
    const int inl = m.inlet ? m.inlet[F] : -1;
    const float* ext = inl >= 0 ? static_cast<const float*>(m.inlet_modes) + (int64_t)inl * NF * D : nullptr;
    const float* trA = sTrM + fA * NF * NB4;
    const float* trB = sTrM + fB * NF * NB4;
    // modal traces of component a: jump J and averaged wind Wv
    float n[D], aF, na;  // na: this lane's component of n
    float J[NF], Wv[NF];
    {
      f2 cA[NBP], cB[NBP];
      cp_wait<0>();
      __syncwarp();
      take(uL, 0, eA, cA);
      take(uL, 1, eB, cB);
      {
        const float* fg = sGeo + (act ? fl : 0) * (D + 1);
#pragma unroll
        for (int cc = 0; cc < D; ++cc) n[cc] = fg[cc];
        aF = fg[D];
        na = (a == 0) ? n[0] : (a == 1 ? n[1] : n[D - 1]);
      }
      __syncwarp();
      if (grp + gstep < ngroups) request_geo(grp + gstep);
      if (WSEP) request(wL, pa, pb);
      else if (grp + gstep < ngroups) request(uL, npa, npb);
      // the degree <= 1 terms of the modes of degree <= 1, compensated; modes 0, 1 and 2, 3
      // paired (mode 3, and mode 2 in 2D, have none)
      f2 sA[2], kA[2], sB[2], kB[2];
#pragma unroll
      for (int i = 0; i <= D; ++i) {
        f2 ta[2], tbv[2];
        lds_f2(sLow + (fA * (D + 1) + i) * 4, ta[0], ta[1]);
        lds_f2(sLow + (fB * (D + 1) + i) * 4, tbv[0], tbv[1]);
        const float xa = (i & 1) ? f2_y(cA[i / 2]) : f2_x(cA[i / 2]);
        const float xb = (i & 1) ? f2_y(cB[i / 2]) : f2_x(cB[i / 2]);
        const f2 xa2 = f2_dup(xa), nxa2 = f2_dup(-xa), xb2 = f2_dup(xb), nxb2 = f2_dup(-xb);
#pragma unroll
        for (int h = 0; h < D - 1; ++h) {
          if (i == 0) {
            dot2_first_f2(sA[h], kA[h], ta[h], xa2, nxa2);
            dot2_first_f2(sB[h], kB[h], tbv[h], xb2, nxb2);
          } else {
            dot2_step_f2(sA[h], kA[h], ta[h], xa2, nxa2);
            dot2_step_f2(sB[h], kB[h], tbv[h], xb2, nxb2);
          }
        }
      }
#pragma unroll
      for (int mm = 0; mm < NF; ++mm) {
        float ta_, tb_;
        const float pl = plain(mm, trA + mm * NB4, cA, false);
        const float pr = plain(mm, trB + mm * NB4, cB, false);
        if (mm < D) {  // degree <= 1: main sums and corrections
          const int h = mm / 2;
          const float sa = (mm & 1) ? f2_y(sA[h]) : f2_x(sA[h]);
          const float ca = __fadd_rn((mm & 1) ? f2_y(kA[h]) : f2_x(kA[h]), pl);
          float sb = (mm & 1) ? f2_y(sB[h]) : f2_x(sB[h]);
          float cb = __fadd_rn((mm & 1) ? f2_y(kB[h]) : f2_x(kB[h]), pr);
          if (ext) {
            sb = ext[mm * D + a];
            cb = 0.0f;
          }
          ta_ = __fadd_rn(sa, ca);
          tb_ = __fadd_rn(sb, cb);
          J[mm] = __fadd_rn(__fsub_rn(sa, sb), __fsub_rn(ca, cb));
        } else {
          ta_ = pl;
          tb_ = ext ? ext[mm * D + a] : pr;
          J[mm] = ta_ - tb_;
        }
        Wv[mm] = ext ? ta_ : 0.5f * (ta_ + tb_);  // an inlet keeps the wind's own trace
      }
    }
    if (WSEP) {  // the wind's traces from its own coefficients
      f2 wA[NBP], wB[NBP];
      if (C::STAGE) {
        cp_wait<0>();
        __syncwarp();
      }
      take(wL, 0, eA, wA);
      take(wL, 1, eB, wB);
      if (C::STAGE) __syncwarp();
      if (grp + gstep < ngroups) request(uL, npa, npb);
#pragma unroll
      for (int mm = 0; mm < NF; ++mm) {
        const float s0 = plain(mm, trA + mm * NB4, wA, true);
        const float s1 = plain(mm, trB + mm * NB4, wB, true);
        Wv[mm] = ext ? s0 : 0.5f * (s0 + s1);
      }
    }
    // normal components over the facet's lanes: wvn_m = <w>_m . n, and (I - Pi^l) J in modal
    // form (modes below nl keep only (J_m . n) n), paired with J
    f2 JP[NF];
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const float jn = lanes_sum(J[mm] * na);
      Wv[mm] = lanes_sum(Wv[mm] * na);  // now <w>_m . n
      JP[mm] = f2_pack(J[mm], mm < nl ? jn * na : J[mm]);
    }
    // facet quadrature points (t_i, t_j): pairs (alpha, beta) of the moments; alpha central,
    // beta the upwind part
    f2 ab[NF];
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) ab[mm] = f2_zero();
    float dsum = 0.0f;
#pragma unroll 1
    for (int j = 0; j < (D == 3 ? MF : 1); ++j) {
      f2 g[K + 1], hs[K + 1];
      float gw[K + 1];
#pragma unroll
      for (int p = 0; p <= K; ++p) {
        g[p] = hs[p] = f2_zero();
        gw[p] = 0.0f;
      }
      const float* bj = sB + j * BST;
      if constexpr (D == 3) {
#pragma unroll
        for (int mm = 0; mm < NF; mm += 2) {
          f2 b[2];
          lds_f2(bj + 2 * mm, b[0], b[1]);
#pragma unroll
          for (int w = 0; w < 2; ++w)
            if (mm + w < NF) {
              const int n1 = mode_degree(2, mm + w), p = mm + w - n1 * (n1 + 1) / 2;
              g[p] = f2_fma(b[w], JP[mm + w], g[p]);
              gw[p] = fmaf(f2_x(b[w]), Wv[mm + w], gw[p]);
            }
        }
      } else {
#pragma unroll
        for (int p = 0; p <= K; ++p) {
          g[p] = JP[p];
          gw[p] = Wv[p];
        }
      }
#pragma unroll
      for (int i = 0; i < MF; ++i) {
        f2 A[K + 2], v = f2_zero();
        float wn = 0.0f;
#pragma unroll
        for (int p = 0; p <= K; p += 2) lds_f2(sA + i * AST + 2 * p, A[p], A[p + 1]);
#pragma unroll
        for (int p = 0; p <= K; ++p) {
          v = f2_fma(A[p], g[p], v);              // (J, (I - Pi^l) J) at the point
          wn = fmaf(f2_x(A[p]), gw[p], wn);
        }
        const float hw = sWf[j * MF + i] * wn;    // w_q/2 w.n
        const f2 t = f2_mul(v, f2_pack(-hw, fabsf(hw)));
        dsum = fmaf(f2_y(t), f2_y(v), dsum);
#pragma unroll
        for (int p = 0; p <= K; ++p) hs[p] = f2_fma(A[p], t, hs[p]);
      }
      if constexpr (D == 3) {
#pragma unroll
        for (int mm = 0; mm < NF; mm += 2) {
          f2 b[2];
          lds_f2(bj + 2 * mm, b[0], b[1]);
#pragma unroll
          for (int w = 0; w < 2; ++w)
            if (mm + w < NF) {
              const int n1 = mode_degree(2, mm + w), p = mm + w - n1 * (n1 + 1) / 2;
              ab[mm + w] = f2_fma(b[w], hs[p], ab[mm + w]);
            }
        }
      } else {
#pragma unroll
        for (int p = 0; p <= K; ++p) ab[p] = hs[p];
      }
    }
    // (I - Pi^l) h: the low modes of beta keep their normal part; scale by a_F; write
    float* gA = gam + (eA * (D + 1) + fA) * NF * D + a;
    float* gB = gam + (eB * (D + 1) + fB) * NF * D + a;
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const float am = f2_x(ab[mm]);
      float bm = f2_y(ab[mm]);
      const float bn = lanes_sum(bm * na);
      if (mm < nl) bm = bn * na;
      if (act) gA[mm * D] = aF * (am + bm);
      if (act && pb != pa) gB[mm * D] = aF * (am - bm);
    }
    if (diss) {
      const float tot = lanes_sum(dsum);
      if (act && a == 0) diss[F] = double(aF) * double(tot);
    }
  }
  cp_wait<0>();
}

}  // namespace hopu
