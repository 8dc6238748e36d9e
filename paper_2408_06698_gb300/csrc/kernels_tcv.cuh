// a3 + a5 on the tensor cores (HOPU_FP32_TC, 3D k = 3, 4, STAGE wind w = u): volume term, facet
// lift and inverse mass, with the elements along the MMA rows.
//
// A tile is 40 elements: the 128 MMA rows (and TMEM lanes) are (element, component) pairs, 30 per
// lane quarter.  Per tile
//   A   c_a[i] of every row, split into three BF16 parts (24 bits), to TMEM (packed pairs);
//   D1  = A B1^T: u_a and its three reference derivatives at the quadrature points (B1 rows: phi_i
//         and d phi_i / d xhat_c at the points), in two halves of the points, each with its own
//         completion, so that the second half's products run under the first half's points;
//   F   thread (row, point group) reads its points' columns, forms the gradient s_b = sum_c M[c][b]
//         d^_c u_a (M = |det J| J^-1), takes the other components' u and s by shuffles and
//         f = w_q ((sum_b s_b of component b) u_a + sum_b u_b s_b), the integrand of k_volume_r,
//         split into three BF16 parts over D1's columns;
//   G   the row's facet moments gam[fm], split likewise;
//   D2  = F B2^T + G B3^T: the tested volume term (B2 rows: phi_i over the points) and the facet
//         lift (B3 rows: TrM over the facet modes), one column block per part of B (a product
//         with all of them is one MMA of three times the width: at N = 48 an MMA costs about the
//         same 80 cycles as at 144);
//   y   = D2 / |det J| from registers through shared memory to coalesced stores, while the next
//         tile's D1 runs.
// The coefficient records and the facet moments of a tile arrive by one bulk copy each, requested
// while the previous tile computes.
//
// Accuracy: a product of two FP32 values is the six products of their BF16 parts of order up to
// 2^-16 (hh, hm, mh, mm, hl, lh), every one exact and accumulated in FP32, the small ones first or
// apart; what is dropped is 2^-24 of the product, below FP32 rounding, where 3xTF32 leaves 2^-21.
//
// Bound: the phases of a tile run one after another (one tile's D1 and A fill the TMEM at k = 4):
// products 5.2 k, points 4.4 k, the rest 3.6 k of 13.2 k cycles.  12 worker warps (3 groups) of 128
// registers; 16 of them beside the MMA warp would leave 96 and spill.  A warp of its own issues the
// MMAs: an issuing worker blocked 3 k cycles per tile on the tensor pipe's queue, and with it every
// barrier; its products are unrolled, with descriptors by increments (in a loop that built each
// descriptor an MMA took its 80 cycles to issue).  Measured (CUDA events, per launch): 32^3 x 6, k = 4
// 528 us (k_volume_r) -> 211 us, on the way 366 (one completion for all of D1, the lift on the CUDA
// cores, bound by its shared-memory loads), 330 (the lift as a product, halves) and 239 (MMAs issued
// from a loop); 16^3 x 6, k = 3 34 -> 26 us.  Error of the operator
// against 64 bits, 32^3, k = 4: 3.6e-7 against 3.7e-7 with k_volume_r on Taylor-Green, 4.5e-7 against
// 4.8e-7 on random coefficients.
#pragma once
#include "f32x2.cuh"
#include "kernels.cuh"
#include "kernels_tc.cuh"
#include "tc.cuh"

namespace hopu {

template <int D, int K>
struct VolTe {
  using S = Shape<D, K>;
  static constexpr int NB = S::nb, NF = S::nf, NL = S::nloc, NQ = S::nq;
  static constexpr int EPQ = 32 / D, TM = 4 * EPQ;          // elements per lane quarter and per tile
  static constexpr int GRP = vol_te_groups(NB), WT = 128 * GRP, THREADS = WT + 32;  // workers; + the MMA warp
  static constexpr int NQP = vol_te_nqp(NQ);                // points, padded to chunks of 4
  static constexpr int P0 = vol_te_p0(NQ), P1 = NQP - P0;   // points of the two halves
  static constexpr int KP = vol_te_kp(NB);                  // K of A
  static constexpr int KF = vol_te_kf(NQ);                  // K of F
  static constexpr int KG = vol_te_kg((D + 1) * NF);        // K of G
  static constexpr int N1 = 4 * NQP, NS = vol_te_ns(NB);    // N of D1; columns of a block of D2
  static constexpr int NC0 = P0 / 4, NC1 = P1 / 4, NCZ = (KF - NQP) / 4;  // chunks: halves, zero padding
  static constexpr int FC = KF / 2, GC = KG / 2;            // TMEM columns of one part of F and G
  // TMEM columns: D1 [0, N1); F [0, 3 FC), G [GO, GO + 3 GC) and D2 [DO, AO) in its place; A [AO, TEND).
  // Blocks of D2: F hh | order 2^-8 | order 2^-16 | 8 unused | G hh
  static constexpr uint32_t GO = 3 * FC, DO = GO + 3 * GC, DG = DO + 3 * NS + 8;
  // EARLY: A lies behind D2 and the next tile's is written while D2 runs; at k = 3 that would take
  // more than half of the TMEM and the second CTA with it, so A waits until D2 has been read
  static constexpr bool EARLY = K == 4;
  static constexpr uint32_t AO = EARLY && DG + NS > (uint32_t)N1 ? DG + NS : (uint32_t)N1;
  static constexpr uint32_t TEND = AO + 3 * KP / 2 > DG + NS ? AO + 3 * KP / 2 : DG + NS;
  static constexpr uint32_t TCOLS = TEND <= 128 ? 128 : TEND <= 256 ? 256 : 512;
  static constexpr size_t B1 = size_t(N1) * KP * 2;         // bytes of one part
  static constexpr size_t B2 = size_t(3 * NS + 8) * KF * 2, B3 = size_t(4 * NS + 8) * KG * 2;  // stacked parts
  static constexpr size_t TAB = 3 * B1 + B2 + B3;
  static constexpr int NG = (D + 1) * NF * D, NFM = (D + 1) * NF;
  static constexpr int IPG = ((NB + GRP - 1) / GRP + 1) / 2 * 2;   // basis indices of a group
  static constexpr size_t IN_BYTES = size_t(TM) * NL * 4, G_BYTES = size_t(TM) * NG * 4;
  static constexpr size_t O_IN = TAB;
  static constexpr size_t O_G = O_IN + IN_BYTES;
  static constexpr size_t O_OUT = O_G + G_BYTES;
  static constexpr size_t O_WQ = O_OUT + IN_BYTES;
  static constexpr size_t O_BAR = O_WQ + size_t(KF) * 4;
  static constexpr size_t SMEM = O_BAR + 80;
  static constexpr bool OK = D == 3 && (K == 3 || K == 4) && SMEM <= 227 * 1024 && TEND <= 512 && 4 * P0 <= 256 &&
                             P0 % 4 == 0 && P1 % 4 == 0 && 3 * FC <= 4 * P0 && (3 * NS + 8) % 16 == 0 &&
                             TAB % 16 == 0 && IN_BYTES % 16 == 0 && G_BYTES % 16 == 0 && KP / 16 <= GRP &&
                             DG + (GRP - 1) * IPG + 16 <= TCOLS;
};

// x as three BF16 parts, two values per register (low half first): p0 + p1 + p2 = x to 24 bits
__device__ __forceinline__ void split_bf16x3(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
  auto pack = [](float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
  };
  auto rest = [](f2 v, uint32_t p) { return f2_sub(v, f2_pack(__uint_as_float(p << 16), __uint_as_float(p & 0xffff0000u))); };
  f2 v = f2_pack(x, y);
  p0 = pack(x, y);
  v = rest(v, p0);
  p1 = pack(f2_x(v), f2_y(v));
  v = rest(v, p1);
  p2 = pack(f2_x(v), f2_y(v));
}

template <int D, int K>
__global__ void __launch_bounds__(VolTe<D, K>::THREADS, K == 3 ? 2 : 1)
    k_volume_te(DevMesh m, const unsigned char* __restrict__ tab, const float* __restrict__ Wqg,
                const float* __restrict__ uL, const float* __restrict__ gam, float* out, Combine cmb) {
  using C = VolTe<D, K>;
  constexpr int NB = C::NB, NL = C::NL, P0 = C::P0, P1 = C::P1, KP = C::KP, KF = C::KF, KG = C::KG, NT = C::WT;
  constexpr int TM = C::TM, EPQ = C::EPQ, GRP = C::GRP, FC = C::FC, GC = C::GC, NG = C::NG, NS = C::NS, IPG = C::IPG;
  constexpr int GT = Shape<D, K>::gt, NFM = C::NFM;
  constexpr uint32_t SB1 = (KP / 8) * 128, SB2 = (KF / 8) * 128, SB3 = (KG / 8) * 128;  // stride byte offsets
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sIn = reinterpret_cast<float*>(smem_raw + C::O_IN);        // [TM][NL]  u of a tile
  float* sG = reinterpret_cast<float*>(smem_raw + C::O_G);          // [TM][NG]  facet moments of a tile
  float* sOut = reinterpret_cast<float*>(smem_raw + C::O_OUT);      // [TM][NL]  y of a tile
  float* sWq = reinterpret_cast<float*>(smem_raw + C::O_WQ);        // [KF], zero past the points
  // mbarriers: 0 tables, 1 and 2 the halves of D1, 3 D2, 4 u, 5 moments; 6 A and 7 F, G ready for
  // the MMA warp
  uint64_t* mb = reinterpret_cast<uint64_t*>(smem_raw + C::O_BAR);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mb + 8);
  volatile uint32_t* stop = tslot + 1;  // the workers gave up
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q4 = warp & 3, grp = warp >> 2;                         // lane quarter, group
  const bool lane_on = lane < D * EPQ;
  const int le = lane_on ? lane / D : 0, a = lane_on ? lane - le * D : 0;
  const int el = q4 * EPQ + le;                                     // the row's element of the tile
  const int a1 = (a + 1) % D, a2 = (a + 2) % D;
  const int p1 = lane_on ? le * D + a1 : lane, p2 = lane_on ? le * D + a2 : lane;
  if (warp == 0) {
    tc::tmem_alloc(tslot, C::TCOLS);
    pdl_trigger();  // behind the allocation, see pdl_trigger
  }
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) tc::mbar_init(mb + i, 1);
    *stop = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int t = tid; t < KF; t += C::THREADS) sWq[t] = t < C::NQ ? Wqg[t] : 0.0f;
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (tid == 0) {  // the constant B operands (written at context creation)
    tc::mbar_expect_tx(mb, (uint32_t)C::TAB);
    tc::bulk_g2s(smem_raw, tab, (uint32_t)C::TAB, mb);
  }
  const uint32_t tbase = *tslot;
  const uint32_t tquad = tbase + ((uint32_t)(q4 * 32) << 16);
  const uint32_t sb1 = tc::smem_u32(smem_raw), sb2 = sb1 + (uint32_t)(3 * C::B1), sb3 = sb2 + (uint32_t)C::B2;
  const int64_t ntiles = (m.E + TM - 1) / TM;
  bool ok = __syncthreads_and(tc::mbar_wait(mb, 0)) != 0;
  if (warp == NT / 32) {
    // the MMA warp: issuing blocks while the tensor pipe's queue is full, and no worker waits for it
    if (lane == 0 && ok) {
      const uint32_t limit = tc::mma_warp_limit(m.tc_wait_limit);
      uint32_t ph = 0;
      pdl_wait();
#pragma unroll 1
      for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ph ^= 1u) {
        if (!tc::mbar_wait(mb + 6, ph, limit) || *stop) break;
        tc::fence_after_sync();
        constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};  // small products first
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t b = sb1 + (h ? (4 * P0 / 8) * SB1 : 0);
#pragma unroll
          for (int x = 0; x < 6; ++x)
#pragma unroll
            for (int ks = 0; ks < KP / 16; ++ks)
              tc::mma_f16_ts(tbase + (h ? 4 * P0 : 0), tbase + C::AO + PA[x] * (KP / 2) + 8 * ks,
                             tc::sdesc(b + PB[x] * (uint32_t)C::B1, 128, SB1) + 16 * ks,
                             tc::idesc_bf16(128, h ? 4 * P1 : 4 * P0), x > 0 || ks > 0);
          tc::commit(mb + 1 + h);
        }
        if (!tc::mbar_wait(mb + 7, ph, limit) || *stop) break;
        tc::fence_after_sync();
        // Part x of G and F against parts 0 .. 2 - x of B3 and B2, stacked along N, so that a block
        // of D2 takes the products of one order and no small product is rounded into a large sum.
        // B3's rows are parts 0, 1, 2, 8 zero rows, part 0: its hh block lies behind the others
        // (the workers zeroed F's hh block, which the first product does not set).
        constexpr int NN[3] = {3 * NS + 8, 2 * NS, NS + 8};
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const uint32_t id = tc::idesc_bf16(128, NN[x]);
#pragma unroll
          for (int ks = 0; ks < KG / 16; ++ks)
            tc::mma_f16_ts(tbase + C::DO + (x == 0 ? 1 : x) * NS, tbase + C::GO + x * GC + 8 * ks,
                           tc::sdesc(sb3 + (x == 0 ? (NS / 8) * SB3 : 0), 128, SB3) + 16 * ks, id, x > 0 || ks > 0);
#pragma unroll
          for (int ks = 0; ks < KF / 16; ++ks)
            tc::mma_f16_ts(tbase + C::DO + x * NS, tbase + x * FC + 8 * ks, tc::sdesc(sb2, 128, SB2) + 16 * ks, id, 1);
        }
        tc::commit(mb + 3);
      }
    }
  } else {
  // bit i: something completes on mbarrier i; phase bit i of the next completion to wait for
  uint32_t pend = 0, phase = 0;
  auto wsync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };  // the workers
  auto wait = [&](int i, uint32_t limit) -> bool {  // every worker; false: gave up
    if (!(pend & (1u << i))) return true;
    uint32_t r = tc::mbar_wait(mb + i, (phase >> i) & 1u, limit);
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.and.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(r), "n"(NT)
        : "memory");
    if (r) {
      pend &= ~(1u << i);
      phase ^= 1u << i;
    }
    return r != 0;
  };
  // one bulk copy for a full tile, plain loads for the ragged tail (the caller synchronises
  // before the buffer is read)
  auto fetch = [&](float* dst, const float* src, int nv, int64_t tile, int i) {
    const int64_t e0 = tile * TM;
    if (e0 + TM <= m.E) {
      if (tid == 0) {
        tc::mbar_expect_tx(mb + i, (uint32_t)(TM * nv * 4));
        tc::bulk_g2s(dst, src + e0 * nv, (uint32_t)(TM * nv * 4), mb + i);
      }
      pend |= 1u << i;
    } else {
      for (int64_t t = tid; t < (m.E - e0) * nv; t += NT) dst[t] = src[e0 * nv + t];
    }
  };
  // A of a tile: 16 coefficients of the row per thread of the first groups
  auto operand_a = [&](int64_t tile) {
    const bool act = lane_on && tile * TM + el < m.E;
    if (grp < KP / 16) {
      const float* c = sIn + ((act ? el : 0) * D + a) * NB;
      uint32_t v[3][8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int i = grp * 16 + 2 * t;
        split_bf16x3(act && i < NB ? c[i] : 0.0f, act && i + 1 < NB ? c[i + 1] : 0.0f, v[0][t], v[1][t], v[2][t]);
      }
#pragma unroll
      for (int x = 0; x < 3; ++x) tc::tmem_st_u32<8>(tquad + C::AO + (uint32_t)(x * (KP / 2) + grp * 8), v[x]);
      tc::tmem_st_wait();
    }
  };
  auto signal = [&](int i, uint32_t bits) {  // the workers' TMEM accesses so far, then mbarrier i
    tc::fence_before_sync();
    wsync();
    if (tid == 0) tc::mbar_arrive(mb + i);
    pend |= bits;
  };
  pdl_wait();
  int64_t tile = blockIdx.x;
  if (ok && tile < ntiles) {
    fetch(sIn, uL, NL, tile, 4);
    fetch(sG, gam, NG, tile, 5);
    wsync();
    ok = wait(4, 1u << 22);
    if (ok) {
      operand_a(tile);
      signal(6, 6u);
      if (tile + gridDim.x < ntiles) fetch(sIn, uL, NL, tile + gridDim.x, 4);  // sIn has been read
    }
  }
  for (; ok && tile < ntiles; tile += gridDim.x) {
    const int64_t e0 = tile * TM, nxt = tile + gridDim.x;
    const int nel = (m.E - e0 < TM) ? (int)(m.E - e0) : TM;
    const bool act = lane_on && el < nel;
    const float* gp = m.geoF + (act ? e0 + el : e0) * GT;
    f2 M0[D], M1[D], M2[D];  // columns a, a + 1, a + 2 of M = |det J| J^-1
#pragma unroll
    for (int cc = 0; cc < D; ++cc) {
      M0[cc] = f2_dup(__ldg(gp + 2 * D * D + cc * D + a));
      M1[cc] = f2_dup(__ldg(gp + 2 * D * D + cc * D + a1));
      M2[cc] = f2_dup(__ldg(gp + 2 * D * D + cc * D + a2));
    }
    const float invabs = __ldg(gp + 3 * D * D);
    auto shfl2 = [&](f2 v, int p) {
      return f2_pack(__shfl_sync(kFull, f2_x(v), p), __shfl_sync(kFull, f2_y(v), p));
    };
    // f at the four points of chunk c, whose columns are col + f * np (f = u and the derivatives),
    // as BF16 parts
    auto chunk = [&](int c, uint32_t col, int np, uint32_t (&F)[3][2]) {
      float v[4][4];
      const uint32_t ta = tquad + col;
      tc::ld4x4({ta, ta + np, ta + 2 * np, ta + 3 * np}, v);
      const float4 wq = *reinterpret_cast<const float4*>(sWq + 4 * c);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const f2 u = f2_pack(v[0][2 * h], v[0][2 * h + 1]);
        f2 s0 = f2_zero(), s1 = f2_zero(), s2 = f2_zero();
#pragma unroll
        for (int cc = 0; cc < D; ++cc) {
          const f2 g = f2_pack(v[cc + 1][2 * h], v[cc + 1][2 * h + 1]);
          s0 = f2_fma(M0[cc], g, s0);
          s1 = f2_fma(M1[cc], g, s1);
          s2 = f2_fma(M2[cc], g, s2);
        }
        const f2 dv = f2_add(f2_add(s0, shfl2(s0, p1)), shfl2(s0, p2));
        f2 f = f2_mul(dv, u);
        f = f2_fma(u, s0, f);
        f = f2_fma(shfl2(u, p1), s1, f);
        f = f2_fma(shfl2(u, p2), s2, f);
        f = f2_mul(f, h ? f2_pack(wq.z, wq.w) : f2_pack(wq.x, wq.y));
        split_bf16x3(f2_x(f), f2_y(f), F[0][h], F[1][h], F[2][h]);
      }
    };
    auto store_chunk = [&](int c, const uint32_t (&F)[3][2]) {
#pragma unroll
      for (int x = 0; x < 3; ++x) tc::tmem_st_u32<2>(tquad + (uint32_t)(x * FC + 2 * c), F[x]);
    };
    constexpr int J0 = (C::NC0 + GRP - 1) / GRP, J1 = (C::NC1 + GRP - 1) / GRP;
    ok = wait(1, m.tc_wait_limit);
    tc::fence_after_sync();
    if (!ok) break;
    {
      uint32_t F[J0][3][2];
#pragma unroll
      for (int j = 0; j < J0; ++j)
        if (j * GRP + grp < C::NC0) chunk(j * GRP + grp, 4 * (j * GRP + grp), P0, F[j]);
      tc::fence_before_sync();
      wsync();  // the first half of D1 has been read: F takes its place
      tc::fence_after_sync();
#pragma unroll
      for (int j = 0; j < J0; ++j)
        if (j * GRP + grp < C::NC0) store_chunk(j * GRP + grp, F[j]);
    }
    ok = wait(2, m.tc_wait_limit);
    tc::fence_after_sync();
    if (!ok) break;
#pragma unroll
    for (int j = 0; j < J1; ++j) {
      const int c = C::NC0 + j * GRP + grp;
      uint32_t F[3][2];
      if (j * GRP + grp < C::NC1) {
        chunk(c, 4 * P0 + 4 * (j * GRP + grp), P1, F);
        store_chunk(c, F);
      }
    }
    if (grp < C::NCZ) {
      const uint32_t Z[3][2] = {};
      store_chunk(C::NC0 + C::NC1 + grp, Z);
    }
    ok = wait(5, 1u << 22);
    if (!ok) break;
    {  // G, 16 moments of the row per group and step
      const float* gl = sG + (act ? el : 0) * NG + a;
      uint32_t v[(KG / 16 + GRP - 1) / GRP][3][8];
#pragma unroll
      for (int j = 0; j < (KG / 16 + GRP - 1) / GRP; ++j)
        if (j * GRP + grp < KG / 16) {
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            const int f = (j * GRP + grp) * 16 + 2 * t;
            split_bf16x3(act && f < NFM ? gl[f * D] : 0.0f, act && f + 1 < NFM ? gl[(f + 1) * D] : 0.0f, v[j][0][t],
                         v[j][1][t], v[j][2][t]);
          }
        }
      tc::fence_before_sync();
      wsync();  // the second half of D1 has been read: G takes its place
      tc::fence_after_sync();
#pragma unroll
      for (int j = 0; j < (KG / 16 + GRP - 1) / GRP; ++j)
        if (j * GRP + grp < KG / 16) {
#pragma unroll
          for (int x = 0; x < 3; ++x)
            tc::tmem_st_u32<8>(tquad + C::GO + (uint32_t)(x * GC + (j * GRP + grp) * 8), v[j][x]);
        }
    }
    {  // F's hh block of D2 starts from zero
      const uint32_t Z[4] = {};
#pragma unroll
      for (int j = 0; j < (NS / 4 + GRP - 1) / GRP; ++j)
        if (j * GRP + grp < NS / 4) tc::tmem_st_u32<4>(tquad + C::DO + 4 * (j * GRP + grp), Z);
    }
    tc::tmem_st_wait();
    signal(7, 8u);
    if (nxt < ntiles) {
      fetch(sG, gam, NG, nxt, 5);  // sG has been read
      if (C::EARLY) {
        ok = wait(4, 1u << 22);
        if (!ok) break;
        operand_a(nxt);
      }
    }
    ok = wait(3, m.tc_wait_limit);
    tc::fence_after_sync();
    if (!ok) break;
    float y[16];
    {
      float v[16];
      const uint32_t i0 = (uint32_t)(grp * IPG);
      float w[16];
      tc::ld16(tquad + C::DO + i0, y);
      tc::ld16(tquad + C::DG + i0, v);
      tc::ld16(tquad + C::DO + NS + i0, w);
#pragma unroll
      for (int j = 0; j < IPG; ++j) y[j] += v[j];
      tc::ld16(tquad + C::DO + 2 * NS + i0, v);
#pragma unroll
      for (int j = 0; j < IPG; ++j) y[j] = (y[j] + (w[j] + v[j])) * invabs;
    }
    if (nxt < ntiles) {
      if (!C::EARLY) {
        ok = wait(4, 1u << 22);
        if (!ok) break;
        tc::fence_before_sync();
        wsync();  // D2 has been read
        tc::fence_after_sync();
        operand_a(nxt);
      }
      signal(6, 6u);  // A is ready, D2 has been read
      if (nxt + gridDim.x < ntiles) fetch(sIn, uL, NL, nxt + gridDim.x, 4);
    }
    if (act) {
      float* yo = sOut + (el * D + a) * NB + grp * IPG;
#pragma unroll
      for (int j = 0; j < IPG; ++j)
        if (grp * IPG + j < NB) yo[j] = y[j];
    }
    wsync();
    for (int t = tid; t < nel * NL; t += NT) {
      const int64_t idx = e0 * NL + t;
      out[idx] = combine_at<float>(cmb, sOut[t], idx);
    }
  }
  if (!ok) {
    if (tid == 0) atomicOr(m.err, kErrTcTimeoutVol);
    // bounded (full limit): the copies in flight land and the MMAs drain before TMEM is freed
    for (int i = 1; i < 6; ++i)
      if (pend & (1u << i)) tc::mbar_wait(mb + i, (phase >> i) & 1u);
    wsync();
    if (tid == 0) {  // release the MMA warp
      *stop = 1u;
      __threadfence_block();
      tc::mbar_arrive(mb + 6);
      tc::mbar_arrive(mb + 7);
    }
  }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tbase, C::TCOLS);
  }
}

}  // namespace hopu
