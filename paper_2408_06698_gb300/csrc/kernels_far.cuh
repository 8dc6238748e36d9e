// The facet part of the adjoint (VJP) of the apply, FP32, with the facet's data in registers: the
// layout of k_facet_r (staged records, degree-structured traces, sum-factorised points, register
// pairs) applied to the transposed form of k_facet_adj (same moments, same points).
//
// A lane owns one (facet, component a) pair.  From the coefficients of both sides it forms the
// modal traces of u_a and of z_a = ybar_a / |det J| (each side with its own inverse mass), and of
// w_a with a separate wind: the jumps [[u]]_m, [[z]]_m, the averages <u>_m and <w>_m; the facet's
// lanes sum the normal parts by shuffles, giving <w>.n, (I - Pi^l)[[u]] and (I - Pi^l)[[z]] in
// modal form.  At the facet points: w.n, the pairs ([[z]], (I - Pi)[[z]]) and (<u>, (I - Pi)[[u]]),
// s = 1/2 <u>.[[z]] + 1/4 sign(w.n) (I - Pi)[[u]].(I - Pi)[[z]] (summed over the lanes), and the
// moments
//   alpha_m += w_q psi_m 1/2 (w.n) [[z]]_a,  beta_m += w_q psi_m 1/2 |w.n| (I - Pi)[[z]]_a,
//   gamma_m += w_q psi_m s
// in registers; beta's low modes keep their normal part; alpha +- beta (sides A / B) go to the
// ubar moments, gamma n_a to the wbar moments, scaled by a_F, element-major.
//
// Bound: FP32 FMA and shuffles.  Measured (CUDA events, per launch): separate wind 16^3 x 6 k = 3
// 84 -> 44 us, 16^3 k = 4 261 -> 104 us, 10^3 k = 5 138 -> 49 us (a warp per facet before); w = u
// 12^3 k = 3 27 -> 25 us (dense points, scalar FMAs and strided loads before), 10^3 k = 5 131 ->
// 41 us.  At k = 5 about a hundred registers spill outside the point loop.
#pragma once
#include "kernels.cuh"
#include "kernels_fr.cuh"

namespace hopu {

template <int D, int K, bool WSEP>
__global__ void __launch_bounds__(32 * FacR<D, K>::WARPS, K <= 3 ? 3 : 2)
    k_facet_adj_r(DevMesh m, DevTabs tb, const float* __restrict__ uL, const float* __restrict__ wL,
                  const float* __restrict__ ybar, int lconst, const int8_t* __restrict__ facet_l,
                  float* __restrict__ gamU, float* __restrict__ gamW) {
  using C = FacR<D, K>;
  constexpr int NF = C::NF, NB4 = C::NB4, FPW = C::FPW, NBP = C::NBP, RST = C::RST;
  constexpr int MF = C::MF, AST = C::AST, BST = C::BST, GT = Shape<D, K>::gt;
  extern __shared__ __align__(16) float sm[];
  pdl_trigger();
  facet_stage_tables<D, K>(tb, sm);
  const float* sTrM = sm + C::O_TRM;
  const float* sA = sm + C::O_A;
  const float* sB = sm + C::O_B;
  const float* sWf = sm + C::O_WF;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* sRec = sm + C::O_REC + warp * 2 * FPW * RST;
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
  int64_t grp = (int64_t)warp * gridDim.x + blockIdx.x;
  int npa = 0, npb = 0;  // the next group's elements of this lane's facet
  auto sides = [&](int64_t g) {
    if (g >= ngroups) return;
    const int64_t F = g * FPW + ((lane_on && g * FPW + fl < m.NF) ? fl : 0);
    npa = m.fa[F];
    npb = m.fb[F];
  };
  sides(grp);
  pdl_wait();
  __syncthreads();
  if (grp < ngroups) facet_request<D, K>(uL, sRec, npa, npb, lane);
  for (; grp < ngroups; grp += gstep) {
    const int64_t F0 = grp * FPW;
    const bool act = lane_on && F0 + fl < m.NF;
    const int64_t F = act ? F0 + fl : F0;  // inactive lanes compute the group's first facet
    const int pa = npa, pb = npb;
    const int64_t eA = pa >> 2, eB = pb >> 2;
    const int fA = pa & 3, fB = pb & 3;
    sides(grp + gstep);
    const double* fg = m.fgeo + F * (D + 1);
    float n[D];
#pragma unroll
    for (int cc = 0; cc < D; ++cc) n[cc] = float(fg[cc]);
    const float aF = float(fg[D]);
    const float na = (a == 0) ? n[0] : (a == 1 ? n[1] : n[D - 1]);  // this lane's component of n
    const int l = facet_l ? int(facet_l[F]) : lconst;
    const int nl = (l < 0) ? 0 : cnbasis(D - 1, l);
    const float iA = float(m.geoT[eA * GT + 3 * D * D]), iB = float(m.geoT[eB * GT + 3 * D * D]);
    const float* trA = sTrM + fA * NF * NB4;
    const float* trB = sTrM + fB * NF * NB4;
    // both sides' coefficients of the field in the buffer; the next field's are requested
    f2 cA[NBP], cB[NBP];
    auto next = [&](const float* src, int ra, int rb, bool more) {
      cp_wait<0>();
      __syncwarp();
      facet_take<D, K>(sRec, 0, fl, a, eA, cA);
      facet_take<D, K>(sRec, 1, fl, a, eB, cB);
      __syncwarp();
      if (more) facet_request<D, K>(src, sRec, ra, rb, lane);
    };
    f2 UP[NF], ZP[NF];  // (<u>, (I - Pi^l)[[u]]) and ([[z]], (I - Pi^l)[[z]]), modal
    float Wn[NF];
    next(ybar, pa, pb, true);
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const float tA = facet_plain_trace<D, K>(mm, trA + mm * NB4, cA, true);
      const float tB = facet_plain_trace<D, K>(mm, trB + mm * NB4, cB, true);
      const float ju = tA - tB, av = 0.5f * (tA + tB);
      const float jn = lanes_sum(ju * na);
      UP[mm] = f2_pack(av, mm < nl ? jn * na : ju);
      if (!WSEP) Wn[mm] = lanes_sum(av * na);
    }
    if (WSEP) next(wL, pa, pb, true);
    else next(uL, npa, npb, grp + gstep < ngroups);
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const float jz = iA * facet_plain_trace<D, K>(mm, trA + mm * NB4, cA, true) -
                       iB * facet_plain_trace<D, K>(mm, trB + mm * NB4, cB, true);
      const float jn = lanes_sum(jz * na);
      ZP[mm] = f2_pack(jz, mm < nl ? jn * na : jz);
    }
    if (WSEP) {
      next(uL, npa, npb, grp + gstep < ngroups);
#pragma unroll
      for (int mm = 0; mm < NF; ++mm) {
        const float tA = facet_plain_trace<D, K>(mm, trA + mm * NB4, cA, true);
        const float tB = facet_plain_trace<D, K>(mm, trB + mm * NB4, cB, true);
        Wn[mm] = lanes_sum((0.5f * (tA + tB)) * na);
      }
    }
    f2 ab[NF];
    float gs[NF];
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      ab[mm] = f2_zero();
      gs[mm] = 0.0f;
    }
#pragma unroll 1
    for (int j = 0; j < (D == 3 ? MF : 1); ++j) {
      f2 gu[K + 1], gz[K + 1], hs[K + 1];
      float gw[K + 1], hg[K + 1];
#pragma unroll
      for (int p = 0; p <= K; ++p) {
        gu[p] = gz[p] = hs[p] = f2_zero();
        gw[p] = hg[p] = 0.0f;
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
              gu[p] = f2_fma(b[w], UP[mm + w], gu[p]);
              gz[p] = f2_fma(b[w], ZP[mm + w], gz[p]);
              gw[p] = fmaf(f2_x(b[w]), Wn[mm + w], gw[p]);
            }
        }
      } else {
#pragma unroll
        for (int p = 0; p <= K; ++p) {
          gu[p] = UP[p];
          gz[p] = ZP[p];
          gw[p] = Wn[p];
        }
      }
#pragma unroll
      for (int i = 0; i < MF; ++i) {
        f2 A[K + 2], vu = f2_zero(), vz = f2_zero();
        float wn = 0.0f;
#pragma unroll
        for (int p = 0; p <= K; p += 2) lds_f2(sA + i * AST + 2 * p, A[p], A[p + 1]);
#pragma unroll
        for (int p = 0; p <= K; ++p) {
          vu = f2_fma(A[p], gu[p], vu);
          vz = f2_fma(A[p], gz[p], vz);
          wn = fmaf(f2_x(A[p]), gw[p], wn);
        }
        const float hq = sWf[j * MF + i];         // w_q / 2
        const float sg = (wn > 0.0f) ? 0.5f : ((wn < 0.0f) ? -0.5f : 0.0f);
        const f2 pr = f2_mul(vu, vz);             // <u>_a [[z]]_a, (I - Pi)[[u]]_a (I - Pi)[[z]]_a
        const float s = hq * lanes_sum(fmaf(sg, f2_y(pr), f2_x(pr)));
        const float hw = hq * wn;
        const f2 t = f2_mul(vz, f2_pack(hw, fabsf(hw)));
#pragma unroll
        for (int p = 0; p <= K; ++p) {
          hs[p] = f2_fma(A[p], t, hs[p]);
          hg[p] = fmaf(f2_x(A[p]), s, hg[p]);
        }
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
              gs[mm + w] = fmaf(f2_x(b[w]), hg[p], gs[mm + w]);
            }
        }
      } else {
#pragma unroll
        for (int p = 0; p <= K; ++p) {
          ab[p] = hs[p];
          gs[p] = hg[p];
        }
      }
    }
    // (I - Pi^l) beta: the low modes keep their normal part; scale by a_F; write
    const int64_t sa = (eA * (D + 1) + fA) * NF * D + a, sb = (eB * (D + 1) + fB) * NF * D + a;
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const float am = f2_x(ab[mm]);
      float bm = f2_y(ab[mm]);
      const float bn = lanes_sum(bm * na);
      if (mm < nl) bm = bn * na;
      const float gm = aF * (gs[mm] * na);
      if (act) {
        gamU[sa + mm * D] = aF * (am + bm);
        gamW[sa + mm * D] = gm;
        if (pb != pa) {
          gamU[sb + mm * D] = aF * (am - bm);
          gamW[sb + mm * D] = gm;
        }
      }
    }
  }
  cp_wait<0>();
}

}  // namespace hopu
