// a1 (E: V_h -> L2) in HOPU_FP32_TC: Y = X Dinv^T per element by exact integer products on the
// tensor cores (tcgen05, kind::f16), then the contravariant Piola map.
//
// The reference change of basis is ill-conditioned on the high-degree modes: their coefficients
// are small differences of large functionals, which a plain FP32 or 3xTF32 product loses.  Here
// nothing is rounded before the sum is complete (the splitting of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication", with signed base-256 digits):
//   X      of an element, scaled by a power of two so that |X| < 128, is q0 + q1 2^-8 + q2 2^-16 +
//          q3 2^-24 with digits |q| <= 128, integers but for the last (more than 32 bits below the
//          element's largest value);
//   Dinv   by rows likewise, five digits (from 64 bits on the host);
//   D_l    = sum of q_i d_j^T over i + j = l, l < 5: products of integers that BF16 holds exactly;
//          a sum stays below 4 * KP * 2^14 < 2^24, so FP32 accumulation is exact in any order (from
//          l = 3 on, where q3 enters, to 2^-24 of D_l);
//   Y      = D_0 + 2^-8 D_1 + ... : the three small levels by Horner's rule, the first two joined by
//          TwoSum, one rounding.
// Two things are left out.  The larger is X's rounding: BF16 keeps 8 bits of the last digit, so a
// functional is held to 2^-32 of the element's largest, and one below 2^-8 of that to fewer than its 24
// bits; Y then errs by at most 2^-32 |X|max times the sum of |Dinv| over its row.  The products beyond
// the fifth level are 2^-37 of |X|max |Dinv|max each.
// The kernel before refined a 3xTF32 product with a compensated residual X - D Y over the nonzeros
// of D on the CUDA cores, which took half of its time.
//
// A tile is 128 elements (the MMA rows, one TMEM lane each); thread (lane quarter q, group g) owns
// element 32 q + lane.  Per tile
//   A   the digits of the group's quarter of X, packed pairs, to TMEM;
//   D   in parts of up to GP groups of 16 columns (3D: 5 basis indices x 3 components, so that a
//       thread has all components of its indices for the Piola map), all levels of a part beside
//       one another: digit i of X against the stacked digits 0 .. 4 - i of Dinv is one MMA of that
//       many blocks of columns, as an MMA of few columns costs as much as one of about 150;
//   uL  from registers through shared memory to coalesced stores, while the next part runs.  The next
//       tile's functionals are gathered meanwhile.
// A warp of its own issues the MMAs (issuing blocks while the tensor pipe's queue is full).
//
// Bound: the workers' phases, one after another (cycles per tile at k = 4, of 17 k: gather and copies
// 10 k before they were rid of their divisions, digits 1.9 k, reading D 0.6 k and the Piola map 1.2 k
// per part); the products (2.6 k per part) run under them.  16 warps beside the MMA warp leave 96
// registers.  Measured (CUDA events, per launch, 3 launches back to back and more): 32^3 x 6, k = 4
// 349 us (the refined kernel) -> 102 us, on the way 209 (a lane per element gathered: 32 lines per
// load), 150, 129 (MMAs issued without a loop); 16^3, k = 3 20 -> 11 us; 13^3, k = 5 166 us (k_v2l)
// -> 22 us.  Error of V_h -> L2 against 64 bits, 32^3, k = 4, largest / L2: Taylor-Green 7.64e-8 /
// 3.95e-8 with either, random 7.92e-8 / 4.54e-8 with either.  Five levels: with four the emulated
// error of a smooth field was 4e-8 of its largest coefficient, with five 1e-9.
#pragma once
#include "f32x2.cuh"
#include "kernels.cuh"
#include "kernels_tc.cuh"
#include "tc.cuh"

namespace hopu {

template <int D, int K>
struct V2lTcr {
  using S = Shape<D, K>;
  static constexpr int NL = S::nloc, NB = S::nb;
  static constexpr int XD = kV2lXDigits, LV = kV2lLevels;
  static constexpr int KP = v2l_tc_kp(NL);            // K
  static constexpr int CW = KP / 4, CP = CW / 2;      // functionals of a group, TMEM columns of a digit
  static constexpr int IPG = v2l_tc_ipg(D);           // basis indices of 16 columns
  static constexpr int NGR = v2l_tc_groups(D, NB), GP = v2l_tc_part(D, NB, NL);
  static constexpr int PARTS = (NGR + GP - 1) / GP;
  static constexpr int TM = 128, WT = 512, THREADS = WT + 32;
  static constexpr uint32_t DO = XD * KP / 2, TEND = DO + LV * 16 * GP;  // A [0, DO), levels behind
  static constexpr uint32_t TCOLS = TEND <= 32 ? 32 : TEND <= 64 ? 64 : TEND <= 128 ? 128 : TEND <= 256 ? 256 : 512;
  static constexpr size_t B_BYTES = size_t(LV) * 16 * NGR * KP * 2;
  static constexpr size_t N_BYTES = size_t(16) * NGR * 4;  // the scale of every column
  static constexpr int XST = NL | 1;                                  // row strides, odd: conflict-free
  __host__ __device__ static constexpr int w(int p) { return IPG * GP * (p + 1) < NB ? IPG * GP : NB - IPG * GP * p; }  // indices of a part
  __host__ __device__ static constexpr int ost(int p) { return (D * w(p)) | 1; }
  __host__ __device__ static constexpr uint32_t part_bytes(int p) {
    return uint32_t(LV) * 16 * (NGR - p * GP < GP ? NGR - p * GP : GP) * KP * 2;
  }
  // k = 5: the digits of Dinv do not fit beside X, and each part's arrive while the one before runs
  static constexpr bool STREAM = B_BYTES > 128 * 1024;
  static constexpr size_t O_N = STREAM ? 2 * size_t(part_bytes(0)) : B_BYTES;
  static constexpr size_t O_X = O_N + N_BYTES;
  static constexpr size_t O_ST = O_X + size_t(TM) * XST * 4;
  static constexpr size_t O_GEO = O_ST + size_t(TM) * ost(0) * 4;
  static constexpr size_t O_MAX = O_GEO + size_t(TM) * D * D * 4;
  static constexpr size_t O_CODE = O_MAX + size_t(4) * TM * 4;
  static constexpr size_t O_BAR = O_CODE + size_t(TM) * (D + 1) * 4;
  static constexpr size_t SMEM = O_BAR + 56;
  static constexpr bool OK = SMEM <= 227 * 1024 && GP > 0 && GP <= 4 && TEND <= 512 && CP % 2 == 0 && CW < 64 &&
                             4 * KP < 1024 && B_BYTES % 16 == 0 && N_BYTES % 16 == 0 && O_CODE % 16 == 0 && TM * (D + 1) <= WT;
};

template <int D, int K>
__global__ void __launch_bounds__(V2lTcr<D, K>::THREADS, 1)
    k_v2l_tcr(DevMesh m, const unsigned char* __restrict__ tab, const float* __restrict__ uV, float* __restrict__ uL) {
  using C = V2lTcr<D, K>;
  using S = Shape<D, K>;
  constexpr int NL = C::NL, KP = C::KP, NF = S::nf, NB = S::nb, NINT = S::nint, GT = S::gt;
  constexpr int XST = C::XST, TM = C::TM, NT = C::WT, DD = D * D, NFL = (D + 1) * NF, CW = C::CW, CP = C::CP;
  constexpr int XD = C::XD, LV = C::LV, GP = C::GP, NGR = C::NGR, PARTS = C::PARTS, IPG = C::IPG;
  constexpr uint32_t SBO = (KP / 8) * 128;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const float* sN = reinterpret_cast<const float*>(smem_raw + C::O_N);  // [16 NGR] scales of the columns
  float* sX = reinterpret_cast<float*>(smem_raw + C::O_X);                  // [TM][XST] X of the next tile, unsigned
  float* stage = reinterpret_cast<float*>(smem_raw + C::O_ST);              // [TM][ost] uL of a part
  float* sGeo = reinterpret_cast<float*>(smem_raw + C::O_GEO);              // [TM][D D] J / det J
  int* sCode = reinterpret_cast<int*>(smem_raw + C::O_CODE);                // [TM][D+1] facet codes of the next tile
  float* sMax = reinterpret_cast<float*>(smem_raw + C::O_MAX);              // [4][TM]   largest |X| of a group
  // mbarriers: 0 tables, 1 a part's MMAs, 2 the MMA warp may start the next part, 3 and 4 a part's digits
  uint64_t* mb = reinterpret_cast<uint64_t*>(smem_raw + C::O_BAR);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mb + 5);
  volatile uint32_t* stop = tslot + 1;  // the workers gave up
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, grp = warp >> 2;
  const int el = q * 32 + lane;  // this thread's element (TMEM lane)
  if (warp == 0) {
    tc::tmem_alloc(tslot, C::TCOLS);
    pdl_trigger();  // behind the allocation, see pdl_trigger
  }
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 5; ++i) tc::mbar_init(mb + i, 1);
    *stop = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (tid == 0) {  // the constant tables (written at context creation)
    tc::mbar_expect_tx(mb, (uint32_t)(C::N_BYTES + (C::STREAM ? 0 : C::B_BYTES)));
    tc::bulk_g2s(smem_raw + C::O_N, tab + C::B_BYTES, (uint32_t)C::N_BYTES, mb);
    if (!C::STREAM) tc::bulk_g2s(smem_raw, tab, (uint32_t)C::B_BYTES, mb);
  }
  const uint32_t tbase = *tslot;
  const uint32_t tquad = tbase + ((uint32_t)(q * 32) << 16);
  const int64_t ntiles = (m.E + TM - 1) / TM;
  bool ok = __syncthreads_and(tc::mbar_wait(mb, 0)) != 0;
  if (warp == NT / 32) {
    if (lane == 0 && ok) {
      const uint32_t sb = tc::smem_u32(smem_raw);
      const int64_t mine = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
      const uint32_t total = (uint32_t)(mine * PARTS);  // parts of this CTA; part c uses buffer c & 1
      const uint32_t limit = tc::mma_warp_limit(m.tc_wait_limit);
      uint32_t c = 0, loaded = 0, ph = 0;
      auto load = [&] {
        if (!C::STREAM || loaded >= total) return;
        const int p = (int)(loaded % PARTS);
        uint64_t* full = mb + 3 + (loaded & 1);
        tc::mbar_expect_tx(full, C::part_bytes(p));
        tc::bulk_g2s(smem_raw + (loaded & 1) * C::part_bytes(0), tab + (size_t)p * C::part_bytes(0), C::part_bytes(p), full);
        ++loaded;
      };
      load();
      load();
      bool go = true;
      pdl_wait();
#pragma unroll 1
      for (int64_t tile = blockIdx.x; go && tile < ntiles; tile += gridDim.x) {
#pragma unroll 1
        for (int p = 0; p < PARTS; ++p, ph ^= 1u) {
          go = tc::mbar_wait(mb + 2, ph, limit) && !*stop;
          if (!go) break;
          if (C::STREAM) {
            if (c > 0) load();  // part c - 1 is done: the workers have read its result
            go = tc::mbar_wait(mb + 3 + (c & 1), (c >> 1) & 1u, limit);
            if (!go) break;
            ++c;
          }
          tc::fence_after_sync();
          const uint32_t nh = 16u * (uint32_t)(NGR - p * GP < GP ? NGR - p * GP : GP);  // columns of a level
          const uint32_t b = sb + (uint32_t)(C::STREAM ? (c - 1) & 1 : p) * C::part_bytes(0);
          // one thread issues: descriptors by increments (16 per K step of 256 bytes), no loop
          const uint64_t bd = tc::sdesc(b, 128, SBO);
#pragma unroll
          for (int i = 0; i < XD; ++i) {
            // digits 0 .. LV - 1 - i of Dinv, at most 256 columns (GP = 4: four levels) per MMA
            constexpr int MX = 256 / (16 * GP);
            const uint32_t n0 = (LV - i < MX ? LV - i : MX) * nh, d = tbase + C::DO + i * nh;
            const uint32_t id0 = tc::idesc_bf16(128, (int)n0);
#pragma unroll
            for (int ks = 0; ks < KP / 16; ++ks) {
              const uint32_t a = tbase + (uint32_t)(i * (KP / 2) + 8 * ks);
              tc::mma_f16_ts(d, a, bd + 16 * ks, id0, i > 0 || ks > 0);
              if (LV - i > MX)
                tc::mma_f16_ts(d + n0, a, bd + 16 * ks + (MX * nh / 8) * (SBO / 16), tc::idesc_bf16(128, (int)((LV - i - MX) * nh)),
                               i > 0 || ks > 0);
            }
          }
          tc::commit(mb + 1);
        }
      }
      for (; C::STREAM && c < loaded; ++c) tc::mbar_wait(mb + 3 + (c & 1), (c >> 1) & 1u);  // gave up: copies land
    }
  } else {
    uint32_t phase = 0;
    bool pend = false;  // a part's MMAs are in flight
    auto wsync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };  // the workers
    auto wait = [&]() -> bool {  // every worker, for the part in flight; false: gave up
      uint32_t r = tc::mbar_wait(mb + 1, phase, m.tc_wait_limit);
      asm volatile(
          "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.and.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
          : "=r"(r)
          : "r"(r), "n"(NT)
          : "memory");
      if (r) {
        pend = false;
        phase ^= 1u;
      }
      return r != 0;
    };
    auto signal = [&] {  // the workers' TMEM accesses so far, then the MMA warp
      tc::fence_before_sync();
      wsync();
      if (tid == 0) tc::mbar_arrive(mb + 2);
      pend = true;
    };
    auto load_code = [&](int64_t tile) -> int {
      return tid < TM * (D + 1) && tile * TM + tid / (D + 1) < m.E ? __ldg(m.efc + tile * TM * (D + 1) + tid) : 0;
    };
    // the functionals of a tile (codes in sCode) without their signs: LW lanes take a facet's block, a
    // warp an element's interior block (a lane per element would touch 32 lines per load)
    auto gather = [&](int64_t tile) {
      constexpr int LW = NF <= 4 ? 4 : NF <= 8 ? 8 : NF <= 16 ? 16 : 32;
      static_assert(NF <= 32, "a block per LW lanes");
      const int64_t e0 = tile * TM;
      const int n = (m.E - e0 < TM) ? (int)(m.E - e0) : TM, j = tid % LW;
#pragma unroll 4
      for (int b = tid / LW; b < n * (D + 1); b += NT / LW) {
        const int r = b / (D + 1);
        if (j < NF) cp_async<4>(sX + r * XST + (b - r * (D + 1)) * NF + j, uV + (int64_t)(sCode[b] >> 2) * NF + j);
      }
      const float* in = uV + m.NF * NF + e0 * NINT;
#pragma unroll
      for (int i = lane; i < NINT; i += 32)
#pragma unroll 4
        for (int r = warp; r < n; r += NT / 32) cp_async<4>(sX + r * XST + NFL + i, in + r * NINT + i);
      cp_commit();
    };
    auto load_geo = [&](int64_t tile) {
      const int64_t e0 = tile * TM;
      const int n = (m.E - e0 < TM) ? (int)(m.E - e0) : TM;
      for (int t = tid; t < n * DD; t += NT) {
        const int r = t / DD;
        cp_async<4>(sGeo + t, m.geoF + (e0 + r) * GT + (t - r * DD));
      }
      cp_commit();
    };
    // digits of the gathered functionals to TMEM; returns the power of two that undoes their scale
    auto operand_a = [&]() -> float {
      float x[CW];
      uint64_t neg = 0;  // bit j: the orientation sign of functional grp CW + j
#pragma unroll
      for (int f = 0; f <= D; ++f) {
        const int lo = min(max(f * NF - grp * CW, 0), CW), hi = min(max((f + 1) * NF - grp * CW, 0), CW);
        neg |= sCode[el * (D + 1) + f] & 2 ? ((uint64_t)1 << hi) - ((uint64_t)1 << lo) : 0u;
      }
      float mx = 0.0f;
#pragma unroll
      for (int j = 0; j < CW; ++j) {
        const int s = grp * CW + j;
        x[j] = s < NL ? sX[el * XST + s] : 0.0f;
        x[j] = (neg >> j) & 1u ? -x[j] : x[j];
        mx = fmaxf(mx, fabsf(x[j]));
      }
      sMax[grp * TM + el] = mx;
      wsync();
#pragma unroll
      for (int g = 0; g < 4; ++g) mx = fmaxf(mx, sMax[g * TM + el]);
      // 2^(e - 127) <= mx < 2^(e - 126); from 2^-120 down the fourth digit alone shrinks
      uint32_t e = __float_as_uint(mx) >> 23;
      e = e < 7u ? 7u : e;
      const f2 inv = f2_dup(__uint_as_float((260u - e) << 23)), rnd = f2_dup(12582912.0f), base = f2_dup(256.0f);
#pragma unroll
      for (int c = 0; c < CP; c += 2) {
        uint32_t v[XD][2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          f2 r = f2_mul(f2_pack(x[2 * (c + t)], x[2 * (c + t) + 1]), inv);
#pragma unroll
          for (int i = 0; i < XD; ++i) {
            // the nearest integers; the last digit keeps the bits that BF16 has left
            const f2 d = i < XD - 1 ? f2_sub(f2_add(r, rnd), rnd) : r;
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(v[i][t]) : "f"(f2_y(d)), "f"(f2_x(d)));
            r = f2_mul(f2_sub(r, d), base);
          }
        }
#pragma unroll
        for (int i = 0; i < XD; ++i) tc::tmem_st_u32<2>(tquad + (uint32_t)(i * (KP / 2) + grp * CP + c), v[i]);
      }
      tc::tmem_st_wait();
      return __uint_as_float((e - 6u) << 23);
    };
    auto copy_out = [&](int64_t tile, int p) {  // p a constant
      const int W = C::w(p), n = (m.E - tile * TM < TM) ? (int)(m.E - tile * TM) : TM;
      float* o = uL + tile * TM * NL + p * GP * IPG;
#pragma unroll
      for (int s = lane; s < D * W; s += 32) {
        const int off = s / W * NB + s % W;
#pragma unroll 4
        for (int r = warp; r < n; r += NT / 32) o[r * NL + off] = stage[r * C::ost(p) + s];
      }
    };

    float back = 0.0f;
    pdl_wait();
    int64_t tile = blockIdx.x, prev = -1;
    if (ok && tile < ntiles) {
      const int c = load_code(tile);
      if (tid < TM * (D + 1)) sCode[tid] = c;
      wsync();
      gather(tile);
      cp_wait<0>();
      wsync();
      back = operand_a();
      signal();
    }
    for (; ok && tile < ntiles; tile += gridDim.x) {
      const int64_t nxt = tile + gridDim.x;
      load_geo(tile);
      const int code = nxt < ntiles ? load_code(nxt) : 0;
      if (prev >= 0) copy_out(prev, PARTS - 1);
      if (nxt < ntiles) {
        if (tid < TM * (D + 1)) sCode[tid] = code;
        wsync();
        gather(nxt);
      } else {
        cp_commit();
      }
#pragma unroll
      for (int p = 0; p < PARTS; ++p) {
        constexpr float r8 = 1.0f / 256.0f;
        const int ng = NGR - p * GP < GP ? NGR - p * GP : GP, nh = 16 * ng;
        if (p + 1 < PARTS) cp_wait<1>();  // the geometry
        else cp_wait<0>();                // and X of the next tile
        ok = wait();
        tc::fence_after_sync();
        if (!ok) break;
        float y[16];
        if (grp < ng) {
          const uint32_t col = tquad + C::DO + 16 * grp;
          float v[16], w[16];
          tc::ld16(col + (LV - 1) * nh, y);
#pragma unroll
          for (int l = LV - 2; l >= 2; --l) {
            tc::ld16(col + l * nh, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) y[j] = fmaf(y[j], r8, v[j]);
          }
          tc::ld16(col + nh, v);
          tc::ld16(col, w);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float a = __fmul_rn(w[j], 256.0f), s = __fadd_rn(a, v[j]), z = __fsub_rn(s, a);
            const float t = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(v[j], z));
            y[j] = __fadd_rn(s, fmaf(y[j], r8, t));
          }
        }
        if (p + 1 < PARTS) signal();  // D has been read
        if (grp < ng) {
          const int g = p * GP + grp;
#pragma unroll
          for (int t = 0; t < IPG; ++t) {
            const int i = g * IPG + t;
            if (i < NB) {
              float c[D];
#pragma unroll
              for (int b = 0; b < D; ++b) c[b] = y[t * D + b] * sN[16 * g + t * D + b] * back;
#pragma unroll
              for (int a = 0; a < D; ++a) {
                float acc = 0.0f;
#pragma unroll
                for (int b = 0; b < D; ++b) acc = fmaf(sGeo[el * DD + a * D + b], c[b], acc);
                stage[el * C::ost(p) + a * C::w(p) + i - p * GP * IPG] = acc;
              }
            }
          }
        }
        if (p + 1 < PARTS) {
          wsync();
          copy_out(tile, p);
        }
      }
      if (!ok) break;
      prev = tile;
      if (nxt < ntiles) {
        back = operand_a();
        signal();
      } else {
        wsync();
      }
    }
    if (ok) {
      if (prev >= 0) copy_out(prev, PARTS - 1);
    } else {
      if (tid == 0) atomicOr(m.err, kErrTcTimeoutV2l);
      // bounded (full limit): the copies and MMAs in flight drain before TMEM is freed
      cp_wait<0>();
      if (pend) tc::mbar_wait(mb + 1, phase);
      wsync();
      if (tid == 0) {  // release the MMA warp
        *stop = 1u;
        __threadfence_block();
        tc::mbar_arrive(mb + 2);
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
