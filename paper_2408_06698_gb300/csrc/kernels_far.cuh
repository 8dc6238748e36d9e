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
// sign(w.n) jumps at w.n = 0, and a point where |w.n| is no larger than its rounding error takes the
// sign of that error: another order of the sums flips it, and one flipped point moves wbar by 1e-6 to
// 1e-4 of its norm (16^3 x 6, k = 3: 4.1e-5 seen, two of a hundred random winds changed by more than
// 2e-6).  So w.n has one order here and in k_facet_adj: a separate wind's traces by ascending basis
// index, the normal component by ascending component, and, where the factorised value lies within the
// rounding errors of the two ways to sum it, the sum over the modes themselves.  All lanes of a facet
// then take one sign.  (w = u: the traces are those of u, in pairs.)
//
// Bound: FP32 FMA and shuffles.  Measured (CUDA events, per launch): separate wind 16^3 x 6 k = 3
// 84 -> 44 us, 16^3 k = 4 261 -> 113 us, 10^3 k = 5 138 -> 54 us (a warp per facet before; 44, 100
// and 49 us with the wind's traces in pairs, which other signs came with); w = u
// 12^3 k = 3 27 -> 25 us (dense points, scalar FMAs and strided loads before), 10^3 k = 5 131 ->
// 41 us.  At k = 5 about twenty registers spill outside the point loop.
#pragma once
#include "kernels.cuh"
#include "kernels_fr.cuh"

namespace hopu {

// A mode's trace as dot_ss sums it: every basis index, in order.  The entries of TrM that vanish by
// degree are 1e-15 of quadrature rounding, and they count: 3 c, the trace of a degree 3 function's
// coefficient alone, lies half-way between two FP32 values for every fourth c.
template <int D, int K>
__device__ __forceinline__ float facet_chain_trace(const float* row, const f2 (&c)[FacR<D, K>::NBP]) {
  constexpr int NB = FacR<D, K>::NB;
  float s = 0.0f;
#pragma unroll
  for (int i = 0; i < NB; i += 4) {
    f2 t[2];
    lds_f2(row + i, t[0], t[1]);
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int j = i + 2 * w;
      if (j < NB) s = fmaf(f2_x(t[w]), f2_x(c[j / 2]), s);
      if (j + 1 < NB) s = fmaf(f2_y(t[w]), f2_y(c[j / 2]), s);
    }
  }
  return s;
}

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
  // v . n of a vector held by the facet's lanes, by ascending component: the same bits in every lane
  auto normal = [&](float v, const float (&n)[D]) {
    float s = 0.0f;
#pragma unroll
    for (int cc = 0; cc < D; ++cc) s = fmaf(__shfl_sync(kFull, v, fl * D + cc), n[cc], s);
    return s;
  };
  auto half_sign = [](float v) { return (v > 0.0f) ? 0.5f : ((v < 0.0f) ? -0.5f : 0.0f); };
  const float* Psi = static_cast<const float*>(tb.Psi);  // [NF][NQF], rule order q = i MF + j
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
    const float* fg = m.fgeoF + F * (D + 1);
    float n[D];
#pragma unroll
    for (int cc = 0; cc < D; ++cc) n[cc] = __ldg(fg + cc);
    const float aF = __ldg(fg + D);
    const float na = (a == 0) ? n[0] : (a == 1 ? n[1] : n[D - 1]);  // this lane's component of n
    const int l = facet_l ? int(facet_l[F]) : lconst;
    const int nl = (l < 0) ? 0 : cnbasis(D - 1, l);
    const float iA = __ldg(m.geoF + eA * GT + 3 * D * D), iB = __ldg(m.geoF + eB * GT + 3 * D * D);
    const float* trA = sTrM + fA * NF * NB4;
    const float* trB = sTrM + fB * NF * NB4;
    // both sides' coefficients of the field in the buffer; the next field's are requested
    f2 cA[NBP], cB[NBP];
    auto next = [&](const float* cur, const float* src, int ra, int rb, bool more) {
      if (C::STAGE) {
        cp_wait<0>();
        __syncwarp();
      }
      facet_take<D, K>(cur, sRec, 0, fl, a, eA, cA);
      facet_take<D, K>(cur, sRec, 1, fl, a, eB, cB);
      if (C::STAGE) {
        __syncwarp();
        if (more) facet_request<D, K>(src, sRec, ra, rb, lane);
      }
    };
    f2 UP[NF], ZP[NF];  // (<u>, (I - Pi^l)[[u]]) and ([[z]], (I - Pi^l)[[z]]), modal
    float Wn[NF];
    next(uL, ybar, pa, pb, true);
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const float tA = facet_plain_trace<D, K>(mm, trA + mm * NB4, cA, true);
      const float tB = facet_plain_trace<D, K>(mm, trB + mm * NB4, cB, true);
      const float ju = tA - tB, av = 0.5f * (tA + tB);
      const float jn = lanes_sum(ju * na);
      UP[mm] = f2_pack(av, mm < nl ? jn * na : ju);
      if (!WSEP) Wn[mm] = normal(av, n);
    }
    if (WSEP) next(ybar, wL, pa, pb, true);
    else next(ybar, uL, npa, npb, grp + gstep < ngroups);
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const float jz = iA * facet_plain_trace<D, K>(mm, trA + mm * NB4, cA, true) -
                       iB * facet_plain_trace<D, K>(mm, trB + mm * NB4, cB, true);
      const float jn = lanes_sum(jz * na);
      ZP[mm] = f2_pack(jz, mm < nl ? jn * na : jz);
    }
    if (WSEP) {
      next(wL, uL, npa, npb, grp + gstep < ngroups);
#pragma unroll
      for (int mm = 0; mm < NF; ++mm) {
        const float tA = facet_chain_trace<D, K>(trA + mm * NB4, cA), tB = facet_chain_trace<D, K>(trB + mm * NB4, cB);
        Wn[mm] = normal(0.5f * (tA + tB), n);
      }
    }
    // the factorised w.n and the sum over the modes differ by at most (NF + 2 K + 6) roundings of
    // sum_m |psi_m| |(w.n)_m|, and |psi_m| < 2 (K + 1) at the facet points
    float near0 = 0.0f;
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) near0 += fabsf(Wn[mm]);
    near0 *= (NF + 2 * K + 6) * 2 * (K + 1) * 0x1p-24f;
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
      float least = INFINITY;  // of |w.n| at the row's points
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
        least = fminf(least, fabsf(wn));
        const float sg = half_sign(wn);
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
      // a point whose sign the sum over the modes decides: about one in ten thousand, so the row is
      // walked again for it (a branch per point parts the arithmetic of neighbouring points:
      // 122 us for 113 at k = 4)
      // (2D: the factorised sum is the sum over the modes)
      if (D == 3 && __any_sync(kFull, least <= near0)) {
#pragma unroll 1
        for (int i = 0; i < MF; ++i) {
          f2 A[K + 2];
          float wn = 0.0f, wm = 0.0f, vu = 0.0f, vz = 0.0f;
#pragma unroll
          for (int p = 0; p <= K; p += 2) lds_f2(sA + i * AST + 2 * p, A[p], A[p + 1]);
#pragma unroll
          for (int p = 0; p <= K; ++p) {
            vu = fmaf(f2_x(A[p]), f2_y(gu[p]), vu);
            vz = fmaf(f2_x(A[p]), f2_y(gz[p]), vz);
            wn = fmaf(f2_x(A[p]), gw[p], wn);
          }
          const float* psi = Psi + i * MF + j;
#pragma unroll
          for (int mm = 0; mm < NF; ++mm) wm = fmaf(__ldg(psi + mm * C::NQF), Wn[mm], wm);
          const float d = fabsf(wn) <= near0 ? half_sign(wm) - half_sign(wn) : 0.0f;
          const float s = sWf[j * MF + i] * lanes_sum(d * (vu * vz));
#pragma unroll
          for (int p = 0; p <= K; ++p) hg[p] = fmaf(f2_x(A[p]), s, hg[p]);
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
