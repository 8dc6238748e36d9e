// Launch wrappers of one kernel family (dimension D, order K, precision T).
#pragma once
#include <algorithm>
#include <type_traits>
#include <utility>

#include "kernels.cuh"
#include "kernels_adj.cuh"
#include "kernels_tc.cuh"
#include "kernels_tcr.cuh"
#include "kernels_tcv.cuh"
#include "kernels_adapt.cuh"
#include "kernels_vr.cuh"
#include "kernels_vrh.cuh"
#include "kernels_far.cuh"
#include "kernels_fr.cuh"

namespace hopu {

template <int D, int K, typename T>
class OpsImpl final : public Ops {
  using S = Shape<D, K>;
  static constexpr size_t kLimit = 200 * 1024;  // shared-memory budget per CTA
  static constexpr size_t sz = sizeof(T);
  static constexpr size_t r4(size_t n) { return ((n + 3) / 4) * 4; }

  using PW = ProjWCfg<D, K, T>;  // warp tiles of the projections
  // V_h -> L2 in FP32: the refined projection (its launch shape is set by configure())
  static constexpr bool kRef = std::is_same<T, float>::value;
  int ref_warps_ = 8, ref_staged_ = 0, csr_n_ = 0;
  size_t ref_smem_ = 0;

  // facet kernel: padded modal trace matrices, Psi, WPsi, Wf; per warp: coefficient
  // blocks, two [nqf][4] point buffers, modal jump / wind, moments (layout of k_facet)
  static constexpr size_t kNBQ = row_stride<T>(S::nb);
  static constexpr size_t kFacTab = r4(size_t(D + 1) * S::nf * r4(S::nb) + 2 * S::nf * S::nqf + S::nqf) * sz;
  static constexpr size_t facet_warp(bool wsep) {
    return (size_t(wsep ? 4 : 2) * D * r4(S::nb) + 2 * S::nqf * 4 + 2 * S::nf * 4 + 2 * S::nf * 4) * sz;
  }
  static constexpr bool kFacetTab = true;
  static constexpr size_t facet_smem(bool wsep) { return kFacTab + kWarps * facet_warp(wsep); }

  // volume kernel: Bt, Wq, Dm, TrM; per warp: coefficients, modal gradients, (W and its
  // divergence), signed facet moments (layout of k_volume)
  static constexpr int kNB1 = cnbasis(D, K - 1);
  static constexpr size_t kVolTab =  // Dm rows padded, Dm and TrM 16-byte aligned (layout of k_volume)
      r4(r4(r4(size_t(S::nq) * kNBQ + S::nq) + size_t(D) * kNB1 * r4(S::nb)) + size_t(D + 1) * S::nf * S::nb) * sz;
  static constexpr size_t volume_stage(bool wsep) {
    return r4(S::nloc) * (wsep ? 2 : 1) + r4(size_t(D + 1) * S::nf * D) + r4(S::gt * 8 / sz);  // FP64 geometry
  }
  static constexpr size_t volume_warp(bool wsep) {
    return (2 * volume_stage(wsep) + size_t(D) * r4(S::nb) + size_t(D) * D * r4(kNB1) +
            (wsep ? size_t(D) * r4(S::nb) + r4(kNB1) : 0)) * sz;
  }
  static constexpr bool kVolumeTab = kVolTab + kWarps * volume_warp(true) <= kLimit;
  static constexpr size_t volume_smem(bool wsep) { return (kVolumeTab ? kVolTab : 0) + kWarps * volume_warp(wsep); }
  using FC = FuseCfg<D, K, T>;
  static constexpr size_t kFuseTab = r4(size_t(FC::TAB)) * sz;
  static constexpr bool kFuse = kVolumeTab && FC::OK && kVolTab + kFuseTab + kWarps * volume_warp(false) <= kLimit;
  static constexpr size_t kFuseSmem = kVolTab + kFuseTab + kWarps * volume_warp(false);
  int g_fuse_ = 1;

  // adjoint kernels (layouts of k_facet_adj / k_volume_adj)
  static constexpr size_t facet_adj_warp(bool wsep) {
    return (size_t(wsep ? 6 : 4) * D * r4(S::nb) + 3 * S::nqf * 4 + 7 * S::nf * 4) * sz;
  }
  static constexpr size_t facet_adj_smem(bool wsep) { return kFacTab + kWarps * facet_adj_warp(wsep); }
  static constexpr size_t volume_adj_smem(bool wsep) {
    return kWarps * (2 * size_t(D) * r4(S::nb) + size_t(D) * D * r4(kNB1) + (wsep ? size_t(D) * r4(S::nb) : 0) +
                     2 * r4(size_t(D + 1) * S::nf * D)) * sz;
  }
  int g_fadj_ = 1, g_vadj_ = 1, g_eta_ = 1;
  static constexpr size_t eta_smem() {
    return (r4(size_t(D + 1) * S::nf * r4(S::nb) + S::nf * S::nqf + S::nqf) +
            kWarps * (2 * size_t(D) * r4(S::nb) + 2 * S::nf * 4)) * sz;
  }
  int nsm_ = 1;
  int tc_ = 0;  // FP32 only: 0 = FMA, 3 = 3xTF32 tensor cores, 1 = 1xTF32 tensor cores
  int g_v2l_tc_ = 1;
  static constexpr bool kTcV2l = std::is_same<T, float>::value && V2lTc<D, K>::OK;
  static constexpr bool kTcV2lR = std::is_same<T, float>::value && V2lTcr<D, K>::OK;
  int g_v2l_tcr_ = 1;
  static constexpr bool kTcVol = std::is_same<T, float>::value && VolTc<D, K>::OK;
  int g_vol_tc_ = 1;
  // tensor-core STAGE volume kernel with elements along the rows (3xBF16 parts: HOPU_FP32_TC only)
  static constexpr bool kTcVolE = std::is_same<T, float>::value && VolTe<D, K>::OK;
  int g_vol_te_ = 1;
  static constexpr bool kTcL2v = std::is_same<T, float>::value && L2vTc<D, K>::OK;
  int g_l2v_tc_ = 1;
  bool use_tc_l2v_ = false;  // autotuner choice of the element back-projection
  bool use_tc_v2l_ = true;  // autotuner choice of the projection (TF32 mode)
  int vvar_ = -1;           // STAGE volume variant (VolumeVariant), -1: unfused warp-per-element
  // register-resident FP32 volume kernel (STAGE wind) where the lane's registers suffice
  static constexpr bool kVolR = std::is_same<T, float>::value && VolR<D, K>::OK;
  static constexpr bool kVolRF = std::is_same<T, float>::value && VolR<D, K>::FUSE_OK;
  static constexpr bool kVolRT = std::is_same<T, float>::value && VolR<D, K, true>::OK;
  int g_volrt_ = 1;
  // register kernel with the basis split over two lanes; every FP32 order has one of the two
  static constexpr bool kVolRH = std::is_same<T, float>::value && VolRH<D, K>::OK;
  static_assert(!std::is_same<T, float>::value || kVolR || kVolRH, "a register volume kernel for every FP32 order");
  int g_volrh_ = 1;
  // separate wind in FP32: the register kernel, its half-basis form where a lane's registers run out
  static constexpr bool kVolRW = std::is_same<T, float>::value && VolR<D, K, false, kVolWind>::OK;
  static constexpr bool kVolRHW = std::is_same<T, float>::value && !kVolRW;
  int g_volw_ = 1;
  // volume part of the VJP in FP32: the register kernel of each cotangent (kVolAdjU, kVolAdjW,
  // kVolAdjSame), its half-basis form where a lane's registers run out
  static constexpr bool kVolAdjR = VolR<D, K, false, kVolAdjSame>::OK;
  int g_volar_[3] = {1, 1, 1};
  template <int MODE>
  using VolA = typename std::conditional<kVolAdjR, VolR<D, K, false, MODE>, VolRH<D, K, MODE>>::type;
  template <int MODE>
  cudaError_t setup_adj() {
    using R = VolA<MODE>;
    static_assert(R::OK, "a register kernel for every FP32 order");
    if constexpr (kVolAdjR) return setup(k_volume_r<D, K, false, false, MODE>, R::SMEM, 32 * R::WARPS, &g_volar_[MODE - kVolAdjU]);
    else return setup(k_volume_rh<D, K, MODE>, R::SMEM, 32 * R::WARPS, &g_volar_[MODE - kVolAdjU]);
  }
  template <int MODE>
  void launch_adj(const DevMesh& m, const LaunchTabs& t, const void* in1, const void* ybar, const void* gam,
                  const void* gam2, void* out, cudaStream_t st) {
    using R = VolA<MODE>;
    const int g = clamp_grid(g_volar_[MODE - kVolAdjU], (m.E + R::ELW - 1) / R::ELW, 1);
    if constexpr (kVolAdjR)
      launch(k_volume_r<D, K, false, false, MODE>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(in1),
             static_cast<const float*>(ybar), static_cast<const float*>(gam), static_cast<const float*>(gam2),
             static_cast<float*>(out), Combine(), static_cast<float*>(nullptr));
    else
      launch(k_volume_rh<D, K, MODE>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(in1),
             static_cast<const float*>(ybar), static_cast<const float*>(gam), static_cast<const float*>(gam2),
             static_cast<float*>(out), Combine());
  }
  // Separate wind on a small mesh (FP32): a warp per facet or element.  A register warp walks the points of
  // its 10 to 16 items one after another, which takes longer than the one pass of a warp per item; the
  // limits are items per SM.  us per call (graph of 20 calls), warp per item / register kernel:
  //   facet term, apply: 3D k = 4, 324 facets 17.1 / 22.1, 1500 27.3 / 28.1, 2592 33.0 / 31.8; k = 5, 324
  //     40.5 / 48.1, 768 (two CTAs on some SMs, each with its own tables) 53.0 / 44.1; 2D k = 3, 768
  //     4.3 / 5.0, 1728 6.7 / 5.6; k = 4, 768 5.8 / 5.9, 1728 7.5 / 7.1; other orders at most even;
  //   facet part of the VJP: 3D k = 2, 324 20.3 / 22.1, 1500 24.4 / 25.4, 6144 31.0 / 29.7; 2D k = 4, 48
  //     17.6 / 18.4, 1728 20.0 / 19.8; other orders at most 2 % apart at the smallest mesh;
  //   volume part of the VJP: 2D k = 4, 32 elements 18.4 / 26.9, 4608 29.5 / 31.6, 8192 37.4 / 34.5; k = 3, 4608
  //     20.2 / 22.3; k = 2, 512 11.9 / 14.1, 1152 13.1 / 14.2; 3D k = 2, 162 22.1 / 27.9, 4374 30.8 / 33.2, 6000
  //     35.7 / 35.2; k = 1, 384 13.7 / 14.7, 750 14.7 / 14.9; from 3D k = 3 on its sums spill (162 elements, 80 /
  //     45).  One cotangent alone takes the same kernel (the same bits) although the register kernel then runs
  //     once (2D k = 2, 2048 11.7 / 8.5): the lines of k = 1 and of 2D k = 2 lie lower for it.
  static constexpr int kFacSmall = D == 3 ? (K == 4 ? 12 : K == 5 ? 4 : 0) : (K >= 3 ? 8 : 0);
  static constexpr int kFacAdjSmall = (D == 3 && K == 2) || (D == 2 && K == 4) ? 10 : 0;
  static constexpr int kVolAdjSmall = K == 1 ? 4 : D == 2 ? (K == 2 ? 8 : 32) : K == 2 ? 32 : 0;
  bool small(int64_t items, int per_sm) const { return items <= (int64_t)per_sm * nsm_; }
  // the sizes these choices go by: this mesh's, or those of the mesh that it is a part of
  int64_t size_E_ = 0, size_F_ = 0;
  int64_t elems(const DevMesh& m) const { return size_E_ ? size_E_ : m.E; }
  int64_t facets(const DevMesh& m) const { return size_F_ ? size_F_ : m.NF; }
  int g_facar_[2] = {1, 1};  // facet part of the VJP in FP32: w = u, separate wind
  int g_volr_ = 1, g_volrf_ = 1;
  // facet term: register-resident kernel in FP32 (every order), a warp per facet in FP64 and on small
  // meshes
  static constexpr bool kFacR = std::is_same<T, float>::value;
  int g_facr_[2] = {1, 1};
  int g_v2l_ = 1, g_v2lpt_ = 1, g_fac_[2] = {1, 1}, g_vol_[2] = {1, 1}, g_elem_[2] = {1, 1}, g_fsum_ = 1;

  template <typename Kern>
  cudaError_t setup(Kern kern, size_t smem, int threads, int* grid, bool max_carveout = false) {
    cudaError_t err = cudaSuccess;
    if (smem > 48 * 1024) {
      err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (err != cudaSuccess) return err;
    }
    if (max_carveout) {  // the largest shared-memory carveout, so that it does not cut occupancy
      err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
      if (err != cudaSuccess) return err;
    }
    int occ = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    if (err != cudaSuccess) return err;
    if (max_carveout) {  // resident blocks by shared memory, threads and registers
      int dev = 0, sm_smem = 0, reserved = 0;
      cudaFuncAttributes fa{};
      if (cudaGetDevice(&dev) == cudaSuccess &&
          cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess &&
          cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) == cudaSuccess &&
          cudaFuncGetAttributes(&fa, kern) == cudaSuccess) {
        const int by_smem = sm_smem / (int)(smem + fa.sharedSizeBytes + reserved);
        const int by_threads = 2048 / threads;
        const int by_regs = fa.numRegs > 0 ? 65536 / (fa.numRegs * threads) : by_threads;
        occ = std::max(occ, std::min(by_smem, std::min(by_threads, by_regs)));
      }
    }
    *grid = nsm_ * std::max(occ, 1);
    return cudaSuccess;
  }

  // Every launch of the family carries the programmatic-stream-serialization attribute
  // (the kernels wait for their predecessor after their prologue, see pdl_wait).
  template <typename... KArgs, typename... Args>
  static void launch(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
  }

  static int clamp_grid(int g, int64_t items, int per_block) {
    const int64_t need = (items + per_block - 1) / per_block;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, need));
  }

 public:
  explicit OpsImpl(int tc = 0) : tc_(std::is_same<T, float>::value ? tc : 0) { vvar_ = default_volume_variant(); }
  // The V_h -> L2 change of basis on the tensor cores: one TF32 product in TF32 mode
  // (k_v2l_tc); in 3xTF32 mode the product of exact digits (k_v2l_tcr), which keeps the small
  // high-degree coefficients of smooth fields that a plain FP32 or 3xTF32 product loses.
  bool tensor_cores() const override { return (tc_ == 1 && kTcV2l) || (tc_ == 3 && kTcV2lR); }
  bool tensor_core_volume() const override { return tc_ != 0 && kTcVol; }
  bool tensor_core_volume_el() const override { return tc_ == 3 && kTcVolE; }
  void select(int v2l_tc, int volume_tc) override {
    use_tc_v2l_ = v2l_tc != 0 && tensor_cores();
    if (volume_tc != 0 && tensor_core_volume()) vvar_ = kVolTensor;
    else if (vvar_ == kVolTensor || vvar_ < 0) vvar_ = default_volume_variant();
  }
  void set_sizes(int64_t n_elems, int64_t n_facets) override {
    size_E_ = n_elems;
    size_F_ = n_facets;
  }
  int selected_v2l() const override { return (use_tc_v2l_ && tensor_cores()) ? 1 : 0; }
  int selected_volume() const override { return vvar_ == kVolTensor || vvar_ == kVolTensorEl ? 1 : 0; }
  bool volume_variant_ok(int v) const override {
    switch (v) {
      case kVolRegFused: return kVolRF;
      case kVolRegSplit: return kVolR;
      case kVolWarpFused: return kFuse;
      case kVolTensor: return tensor_core_volume();
      case kVolTensorEl: return tensor_core_volume_el();
      case kVolRegTab: return kVolRT;
      case kVolRegHalf: return kVolRH;
      default: return false;
    }
  }
  void select_volume_variant(int v) override {
    if (volume_variant_ok(v)) vvar_ = v;
  }
  int volume_variant() const override { return vvar_; }
  int default_volume_variant() const {
    return kVolR ? kVolRegSplit : (kVolRH ? kVolRegHalf : (kFuse ? kVolWarpFused : -1));
  }

  cudaError_t prepare() override {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    err = cudaDeviceGetAttribute(&nsm_, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    const int th = 32 * kWarps;
    if constexpr (!kRef) {
      if ((err = setup(k_v2l<D, K, T, false>, PW::SMEM, 32 * PW::WARPS, &g_v2l_)) != cudaSuccess) return err;
    }
    if ((err = setup(k_v2l<D, K, T, true>, PW::SMEM, 32 * PW::WARPS, &g_v2lpt_)) != cudaSuccess) return err;
    if constexpr (kTcVol) {
      if (tc_ && (err = setup(k_volume_tc<D, K>, VolTc<D, K>::SMEM, VolTc<D, K>::THREADS, &g_vol_tc_, true)) !=
                     cudaSuccess)
        return err;
    }
    if constexpr (kTcVolE) {
      if (tc_ == 3 && (err = setup(k_volume_te<D, K>, VolTe<D, K>::SMEM, VolTe<D, K>::THREADS, &g_vol_te_, true)) !=
                          cudaSuccess)
        return err;
    }
    if constexpr (kTcV2lR) {
      if (tc_ == 3 && (err = setup(k_v2l_tcr<D, K>, V2lTcr<D, K>::SMEM, V2lTcr<D, K>::THREADS, &g_v2l_tcr_, true)) !=
                          cudaSuccess)
        return err;
    }
    if constexpr (kTcV2l) {
      if (tc_ == 1) {
        err = setup(k_v2l_tc<D, K, false>, V2lTc<D, K>::SMEM, V2lTc<D, K>::THREADS, &g_v2l_tc_, true);
        if (err != cudaSuccess) return err;
      }
    }

    if constexpr (kTcL2v) {
      if (tc_) {
        err = tc_ == 3 ? setup(k_l2v_tc<D, K, true>, L2vTc<D, K>::SMEM, L2vTc<D, K>::THREADS, &g_l2v_tc_, true)
                       : setup(k_l2v_tc<D, K, false>, L2vTc<D, K>::SMEM, L2vTc<D, K>::THREADS, &g_l2v_tc_, true);
        if (err != cudaSuccess) return err;
      }
    }
    if ((err = setup(k_eta<D, K, T>, eta_smem(), th, &g_eta_)) != cudaSuccess) return err;
    if constexpr (std::is_same<T, float>::value) {
      using R = FacR<D, K>;
      if ((err = setup(k_facet_adj_r<D, K, false>, R::SMEM, 32 * R::WARPS, &g_facar_[0])) != cudaSuccess) return err;
      if ((err = setup(k_facet_adj_r<D, K, true>, R::SMEM, 32 * R::WARPS, &g_facar_[1])) != cudaSuccess) return err;
      if ((err = setup_adj<kVolAdjU>()) != cudaSuccess) return err;
      if ((err = setup_adj<kVolAdjW>()) != cudaSuccess) return err;
      if ((err = setup_adj<kVolAdjSame>()) != cudaSuccess) return err;
      if constexpr (kFacAdjSmall) {
        if ((err = setup(k_facet_adj<D, K, T, true>, facet_adj_smem(true), th, &g_fadj_)) != cudaSuccess) return err;
      }
      if constexpr (kVolAdjSmall) {
        if ((err = setup(k_volume_adj<D, K, T, true>, volume_adj_smem(true), th, &g_vadj_)) != cudaSuccess) return err;
      }
    } else {
      if ((err = setup(k_facet_adj<D, K, T, false>, facet_adj_smem(false), th, &g_fadj_)) != cudaSuccess) return err;
      if ((err = setup(k_facet_adj<D, K, T, true>, facet_adj_smem(true), th, &g_fadj_)) != cudaSuccess) return err;
      if ((err = setup(k_volume_adj<D, K, T, false>, volume_adj_smem(false), th, &g_vadj_)) != cudaSuccess) return err;
      if ((err = setup(k_volume_adj<D, K, T, true>, volume_adj_smem(true), th, &g_vadj_)) != cudaSuccess) return err;
    }
    if constexpr (kFacR) {
      using R = FacR<D, K>;
      if ((err = setup(k_facet_r<D, K, false>, R::SMEM, 32 * R::WARPS, &g_facr_[0])) != cudaSuccess) return err;
      if ((err = setup(k_facet_r<D, K, true>, R::SMEM, 32 * R::WARPS, &g_facr_[1])) != cudaSuccess) return err;
    }
    if constexpr (!kFacR) {
      if ((err = setup(k_facet<D, K, T, false, kFacetTab>, facet_smem(false), th, &g_fac_[0])) != cudaSuccess) return err;
    }
    if constexpr (!kFacR || kFacSmall) {
      if ((err = setup(k_facet<D, K, T, true, kFacetTab>, facet_smem(true), th, &g_fac_[1])) != cudaSuccess) return err;
    }
    if constexpr (!std::is_same<T, float>::value) {
      if ((err = setup(k_volume<D, K, T, false, kVolumeTab, false>, volume_smem(false), th, &g_vol_[0])) != cudaSuccess) return err;
    }
    if ((err = setup(k_volume<D, K, T, true, kVolumeTab, false>, volume_smem(true), th, &g_vol_[1])) != cudaSuccess) return err;
    if constexpr (kVolR) {
      if ((err = setup(k_volume_r<D, K, false, false, kVolSame>, VolR<D, K>::SMEM, 32 * VolR<D, K>::WARPS, &g_volr_)) != cudaSuccess)
        return err;
    }
    if constexpr (kVolRH) {
      if ((err = setup(k_volume_rh<D, K, kVolSame>, VolRH<D, K>::SMEM, 32 * VolRH<D, K>::WARPS, &g_volrh_)) != cudaSuccess)
        return err;
    }
    if constexpr (kVolRW) {
      using R = VolR<D, K, false, kVolWind>;
      if ((err = setup(k_volume_r<D, K, false, false, kVolWind>, R::SMEM, 32 * R::WARPS, &g_volw_)) != cudaSuccess) return err;
    }
    if constexpr (kVolRHW) {
      using R = VolRH<D, K, kVolWind>;
      if ((err = setup(k_volume_rh<D, K, kVolWind>, R::SMEM, 32 * R::WARPS, &g_volw_)) != cudaSuccess) return err;
    }
    if constexpr (kVolRT) {
      if ((err = setup(k_volume_r<D, K, false, true, kVolSame>, VolR<D, K, true>::SMEM, 32 * VolR<D, K, true>::WARPS,
                       &g_volrt_)) != cudaSuccess)
        return err;
    }
    if constexpr (kVolRF) {
      if ((err = setup(k_volume_r<D, K, true, false, kVolSame>, VolR<D, K>::SMEM_FUSE, 32 * VolR<D, K>::WARPS, &g_volrf_)) !=
          cudaSuccess)
        return err;
    }
    if constexpr (kFuse) {
      if ((err = setup(k_volume<D, K, T, false, true, true>, kFuseSmem, th, &g_fuse_)) != cudaSuccess) return err;
    }
    if ((err = setup(k_l2v_elem<D, K, T, false>, PW::SMEM, 32 * PW::WARPS, &g_elem_[0])) != cudaSuccess) return err;
    if ((err = setup(k_l2v_elem<D, K, T, true>, PW::SMEM, 32 * PW::WARPS, &g_elem_[1])) != cudaSuccess) return err;
    if ((err = setup(k_l2v_facet<D, K, T, false>, 0, 256, &g_fsum_)) != cudaSuccess) return err;
    return cudaSuccess;
  }

  // The refined FP32 projection stages the sparse rows of D and, when they fit, Dinv^T per
  // CTA; as many warps per CTA as fit in ~220 KB (16, 12, 8 or 4).
  cudaError_t configure(const LaunchTabs& t) override {
    if constexpr (kRef) {
      using R = ProjRCfg<D, K>;
      csr_n_ = t.csr_n;
      const size_t csr = size_t(csr_n_) * 16, tab = (R::TAB + 15) / 16 * 16;
      ref_staged_ = csr + tab + 8 * R::TILE <= 220 * 1024;
      const size_t fixed = csr + (ref_staged_ ? tab : 0);
      ref_warps_ = R::fit_warps(fixed);
      ref_smem_ = fixed + size_t(ref_warps_) * R::TILE;
      return setup(k_v2l<D, K, T, false>, ref_smem_, 32 * ref_warps_, &g_v2l_);
    }
    return cudaSuccess;
  }

  int v2l(const DevMesh& m, const LaunchTabs& t, const void* uV, void* uL, cudaStream_t st) override {
    if constexpr (kTcV2lR) {
      if (tc_ == 3 && use_tc_v2l_ && t.tcv2l) {
        const int g = clamp_grid(g_v2l_tcr_, m.E, V2lTcr<D, K>::TM);
        launch(k_v2l_tcr<D, K>, g, V2lTcr<D, K>::THREADS, V2lTcr<D, K>::SMEM, st, m,
               static_cast<const unsigned char*>(t.tcv2l), static_cast<const float*>(uV), static_cast<float*>(uL));
        return 1;
      }
    }
    if constexpr (kTcV2l) {
      if (tc_ == 1 && use_tc_v2l_) {
        const int g = clamp_grid(g_v2l_tc_, m.E, V2lTc<D, K>::TM);
        const int nlp = (S::nloc + 3) / 4 * 4;
        launch(k_v2l_tc<D, K, false>, g, V2lTc<D, K>::THREADS, V2lTc<D, K>::SMEM, st, m,
               static_cast<const float*>(t.Dinv), nlp, static_cast<const float*>(uV), static_cast<float*>(uL));
        return 1;
      }
    }
    if constexpr (kRef) {
      const int g = clamp_grid(g_v2l_, (m.E + PW::EW - 1) / PW::EW, 1);
      launch(k_v2l<D, K, T, false>, g, 32 * ref_warps_, ref_smem_, st, m, static_cast<const T*>(t.DinvT),
             static_cast<const float4*>(t.Dcsr), csr_n_, ref_staged_, static_cast<const T*>(uV),
             static_cast<T*>(uL));
    } else {
      const int g = clamp_grid(g_v2l_, (m.E + PW::EW - 1) / PW::EW, 1);
      launch(k_v2l<D, K, T, false>, g, 32 * PW::WARPS, PW::SMEM, st, m, static_cast<const T*>(t.DinvT),
             static_cast<const float4*>(nullptr), 0, 0, static_cast<const T*>(uV), static_cast<T*>(uL));
    }
    return 1;
  }

  int facet(const DevMesh& m, const LaunchTabs& t, const void* uL, const void* wL, int l,
            const int8_t* facet_l, void* gam, double* diss, cudaStream_t st) override {
    const bool wsep = (wL != nullptr && wL != uL);
    if constexpr (kFacR) {
      if constexpr (kFacSmall) {
        if (wsep && small(facets(m), kFacSmall)) {
          launch(k_facet<D, K, T, true, kFacetTab>, clamp_grid(g_fac_[1], m.NF, kWarps), 32 * kWarps, facet_smem(true), st,
              m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), l, facet_l, static_cast<T*>(gam), diss);
          return 1;
        }
      }
      using R = FacR<D, K>;
      const int g = clamp_grid(g_facr_[wsep ? 1 : 0], (m.NF + R::FPW - 1) / R::FPW, 1);
      if (wsep)
        launch(k_facet_r<D, K, true>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(wL), l, facet_l, static_cast<float*>(gam), diss);
      else
        launch(k_facet_r<D, K, false>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(uL), l, facet_l, static_cast<float*>(gam), diss);
    } else {
      const int g = clamp_grid(g_fac_[wsep ? 1 : 0], m.NF, kWarps);
      if (wsep)
        launch(k_facet<D, K, T, true, kFacetTab>, g, 32 * kWarps, facet_smem(true), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), l, facet_l, static_cast<T*>(gam), diss);
      else
        launch(k_facet<D, K, T, false, kFacetTab>, g, 32 * kWarps, facet_smem(false), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(uL), l, facet_l, static_cast<T*>(gam), diss);
    }
    return 1;
  }

  int volume(const DevMesh& m, const LaunchTabs& t, const void* uL, const void* wL, const void* gam,
             Combine c, void* out, cudaStream_t st) override {
    const bool wsep = (wL != nullptr && wL != uL);
    if constexpr (kTcVolE) {
      if (!wsep && vvar_ == kVolTensorEl && t.tcvole) {
        using R = VolTe<D, K>;
        launch(k_volume_te<D, K>, clamp_grid(g_vol_te_, m.E, R::TM), R::THREADS, R::SMEM, st, m,
               static_cast<const unsigned char*>(t.tcvole), static_cast<const float*>(t.Wq), static_cast<const float*>(uL), static_cast<const float*>(gam),
               static_cast<float*>(out), c);
        return 1;
      }
    }
    if constexpr (kVolRH) {
      if (!wsep && (vvar_ == kVolRegHalf || !kVolR)) {
        using R = VolRH<D, K>;
        const int g = clamp_grid(g_volrh_, (m.E + R::ELW - 1) / R::ELW, 1);
        launch(k_volume_rh<D, K, kVolSame>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(uL), static_cast<const float*>(gam), static_cast<const float*>(nullptr), static_cast<float*>(out), c);
        return 1;
      }
    }
    if constexpr (kVolRT) {
      if (!wsep && vvar_ == kVolRegTab) {
        using R = VolR<D, K, true>;
        const int g = clamp_grid(g_volrt_, (m.E + R::ELW - 1) / R::ELW, 1);
        launch(k_volume_r<D, K, false, true, kVolSame>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(uL), static_cast<const float*>(gam), static_cast<const float*>(nullptr), static_cast<float*>(out), c, static_cast<float*>(nullptr));
        return 1;
      }
    }
    if constexpr (kVolR) {
      if (!wsep) {
        using R = VolR<D, K>;
        const int g = clamp_grid(g_volr_, (m.E + R::ELW - 1) / R::ELW, 1);
        launch(k_volume_r<D, K, false, false, kVolSame>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(uL), static_cast<const float*>(gam), static_cast<const float*>(nullptr), static_cast<float*>(out), c, static_cast<float*>(nullptr));
        return 1;
      }
    }
    // Separate wind (and FP64).  FP32: the register kernels, except while the warp-per-element
    // kernel has a resident warp for every element: its one pass is then shorter than a register
    // warp's walk over 32 / D elements (FP32 k = 3, 162 elements: 10 against 16 us; 7986 elements:
    // 27 against 20 us; k = 4, 2058 elements: 37 against 39 us; 6000 elements: 70 against 53 us).
    const int g = clamp_grid(g_vol_[wsep ? 1 : 0], m.E, kWarps);
    if constexpr (kVolRW || kVolRHW) {
      if (elems(m) > (int64_t)g_vol_[1] * kWarps) {
        if constexpr (kVolRW) {
          using R = VolR<D, K, false, kVolWind>;
          launch(k_volume_r<D, K, false, false, kVolWind>, clamp_grid(g_volw_, (m.E + R::ELW - 1) / R::ELW, 1),
                 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL), static_cast<const float*>(wL),
                 static_cast<const float*>(gam), static_cast<const float*>(nullptr), static_cast<float*>(out), c, static_cast<float*>(nullptr));
        } else {
          using R = VolRH<D, K, kVolWind>;
          launch(k_volume_rh<D, K, kVolWind>, clamp_grid(g_volw_, (m.E + R::ELW - 1) / R::ELW, 1), 32 * R::WARPS, R::SMEM,
                 st, m, t, static_cast<const float*>(uL), static_cast<const float*>(wL),
                 static_cast<const float*>(gam), static_cast<const float*>(nullptr), static_cast<float*>(out), c);
        }
        return 1;
      }
      launch(k_volume<D, K, T, true, kVolumeTab, false>, g, 32 * kWarps, volume_smem(true), st,
          m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), static_cast<const T*>(gam),
          static_cast<T*>(out), c, nullptr);
    } else {
      if (wsep)
        launch(k_volume<D, K, T, true, kVolumeTab, false>, g, 32 * kWarps, volume_smem(true), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), static_cast<const T*>(gam),
            static_cast<T*>(out), c, nullptr);
      else
        launch(k_volume<D, K, T, false, kVolumeTab, false>, g, 32 * kWarps, volume_smem(false), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(uL), static_cast<const T*>(gam),
            static_cast<T*>(out), c, nullptr);
    }
    return 1;
  }

  bool has_fused() const override {
    return vvar_ == kVolRegFused || vvar_ == kVolWarpFused || vvar_ == kVolTensor;
  }

  int eta(const DevMesh& m, const LaunchTabs& t, const void* uL, int l, int8_t* facet_l, const EtaThresholds& th,
          double* eta_out, cudaStream_t st) override {
    const int g = clamp_grid(g_eta_, m.NF, kWarps);
    launch(k_eta<D, K, T>, g, 32 * kWarps, eta_smem(), st, m, t, static_cast<const T*>(uL), l, facet_l, th, eta_out);
    return 1;
  }

  int v2l_pt(const DevMesh& m, const LaunchTabs& t, const void* vV, void* yL, cudaStream_t st) override {
    const int g = clamp_grid(g_v2lpt_, (m.E + PW::EW - 1) / PW::EW, 1);
    launch(k_v2l<D, K, T, true>, g, 32 * PW::WARPS, PW::SMEM, st, m, static_cast<const T*>(t.Dn),
           static_cast<const float4*>(nullptr), 0, 0, static_cast<const T*>(vV), static_cast<T*>(yL));
    return 1;
  }

  int facet_adj(const DevMesh& m, const LaunchTabs& t, const void* uL, const void* wL, const void* ybar, int l,
                const int8_t* facet_l, void* gamU, void* gamW, cudaStream_t st) override {
    const bool wsep = (wL != nullptr && wL != uL);
    if constexpr (std::is_same<T, float>::value) {
      if constexpr (kFacAdjSmall) {
        if (wsep && small(facets(m), kFacAdjSmall)) {
          launch(k_facet_adj<D, K, T, true>, clamp_grid(g_fadj_, m.NF, kWarps), 32 * kWarps, facet_adj_smem(true), st,
              m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), static_cast<const T*>(ybar), l, facet_l,
              static_cast<T*>(gamU), static_cast<T*>(gamW));
          return 1;
        }
      }
      using R = FacR<D, K>;
      const int g = clamp_grid(g_facar_[wsep ? 1 : 0], (m.NF + R::FPW - 1) / R::FPW, 1);
      if (wsep)
        launch(k_facet_adj_r<D, K, true>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(wL), static_cast<const float*>(ybar), l, facet_l, static_cast<float*>(gamU),
               static_cast<float*>(gamW));
      else
        launch(k_facet_adj_r<D, K, false>, g, 32 * R::WARPS, R::SMEM, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(uL), static_cast<const float*>(ybar), l, facet_l, static_cast<float*>(gamU),
               static_cast<float*>(gamW));
    } else {
      const int g = clamp_grid(g_fadj_, m.NF, kWarps);
      if (wsep)
        launch(k_facet_adj<D, K, T, true>, g, 32 * kWarps, facet_adj_smem(true), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), static_cast<const T*>(ybar), l, facet_l,
            static_cast<T*>(gamU), static_cast<T*>(gamW));
      else
        launch(k_facet_adj<D, K, T, false>, g, 32 * kWarps, facet_adj_smem(false), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(uL), static_cast<const T*>(ybar), l, facet_l,
            static_cast<T*>(gamU), static_cast<T*>(gamW));
    }
    return 1;
  }

  int volume_adj(const DevMesh& m, const LaunchTabs& t, const void* uL, const void* wL, const void* ybar,
                 const void* gamU, const void* gamW, void* ubar, void* wbar, cudaStream_t st) override {
    const bool wsep = (wL != nullptr && wL != uL);
    if constexpr (std::is_same<T, float>::value) {
      if (!wsep) {
        launch_adj<kVolAdjSame>(m, t, uL, ybar, gamU, gamW, ubar, st);
        return 1;
      }
      if constexpr (kVolAdjSmall) {
        if (small(elems(m), kVolAdjSmall)) {
          launch(k_volume_adj<D, K, T, true>, clamp_grid(g_vadj_, m.E, kWarps), 32 * kWarps, volume_adj_smem(true), st,
              m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), static_cast<const T*>(ybar),
              static_cast<const T*>(gamU), static_cast<const T*>(gamW), static_cast<T*>(ubar), static_cast<T*>(wbar));
          return 1;
        }
      }
      if (ubar) launch_adj<kVolAdjU>(m, t, wL, ybar, gamU, nullptr, ubar, st);
      if (wbar) launch_adj<kVolAdjW>(m, t, uL, ybar, gamW, nullptr, wbar, st);
      return (ubar != nullptr) + (wbar != nullptr);
    } else {
      const int g = clamp_grid(g_vadj_, m.E, kWarps);
      if (wsep)
        launch(k_volume_adj<D, K, T, true>, g, 32 * kWarps, volume_adj_smem(true), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(wL), static_cast<const T*>(ybar),
            static_cast<const T*>(gamU), static_cast<const T*>(gamW), static_cast<T*>(ubar), static_cast<T*>(wbar));
      else
        launch(k_volume_adj<D, K, T, false>, g, 32 * kWarps, volume_adj_smem(false), st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(uL), static_cast<const T*>(ybar),
            static_cast<const T*>(gamU), static_cast<const T*>(gamW), static_cast<T*>(ubar), static_cast<T*>(nullptr));
      return 1;
    }
  }

  int volume_l2v(const DevMesh& m, const LaunchTabs& t, const void* uL, const void* gam, void* lf, Combine c,
                 void* outV, cudaStream_t st) override {
    if constexpr (kTcVol) {
      if (vvar_ == kVolTensor && tensor_core_volume() && t.tcvol) {
        const int g = clamp_grid(g_vol_tc_, m.E, VolTc<D, K>::EB);
        const int nlr = row_stride<float>(S::nloc);
        launch(k_volume_tc<D, K>, g, VolTc<D, K>::THREADS, VolTc<D, K>::SMEM, st,
            m, static_cast<const float*>(t.tcvol), static_cast<const float*>(t.Dm), static_cast<const float*>(t.Wq),
            static_cast<const float*>(t.TrM), static_cast<const float*>(t.Drow), nlr, static_cast<const float*>(uL),
            static_cast<const float*>(gam), static_cast<float*>(outV), c, static_cast<float*>(lf));
        return 1;
      }
    }
    if constexpr (kVolRF) {
      if (vvar_ == kVolRegFused) {
        using R = VolR<D, K>;
        const int g = clamp_grid(g_volrf_, (m.E + R::ELW - 1) / R::ELW, 1);
        launch(k_volume_r<D, K, true, false, kVolSame>, g, 32 * R::WARPS, R::SMEM_FUSE, st, m, t, static_cast<const float*>(uL),
               static_cast<const float*>(uL), static_cast<const float*>(gam), nullptr, static_cast<float*>(outV), c, static_cast<float*>(lf));
        return 1;
      }
    }
    if constexpr (kFuse) {
      if (vvar_ == kVolWarpFused) {
        const int g = clamp_grid(g_fuse_, m.E, kWarps);
        launch(k_volume<D, K, T, false, true, true>, g, 32 * kWarps, kFuseSmem, st,
            m, t, static_cast<const T*>(uL), static_cast<const T*>(uL), static_cast<const T*>(gam),
            static_cast<T*>(outV), c, static_cast<T*>(lf));
        return 1;
      }
    }
    return 0;
  }

  bool tensor_core_l2v() const override { return kTcL2v && tc_ != 0; }
  void select_l2v(int tc) override { use_tc_l2v_ = tc != 0 && tensor_core_l2v(); }
  int selected_l2v() const override { return use_tc_l2v_ && tensor_core_l2v() ? 1 : 0; }

  int l2v_elem(const DevMesh& m, const LaunchTabs& t, const void* yL, bool dual, void* lf, Combine c,
               void* outV, cudaStream_t st) override {
    if constexpr (kTcL2v) {
      if (!dual && use_tc_l2v_ && tc_ && t.tcl2v) {
        using LC = L2vTc<D, K>;
        const int g = clamp_grid(g_l2v_tc_, m.E, LC::TM);
        if (tc_ == 3)
          launch(k_l2v_tc<D, K, true>, g, LC::THREADS, LC::SMEM, st, m, static_cast<const float*>(t.tcl2v),
                 static_cast<const float*>(yL), static_cast<float*>(lf), static_cast<float*>(outV), c);
        else
          launch(k_l2v_tc<D, K, false>, g, LC::THREADS, LC::SMEM, st, m, static_cast<const float*>(t.tcl2v),
                 static_cast<const float*>(yL), static_cast<float*>(lf), static_cast<float*>(outV), c);
        return 1;
      }
    }
    const int g = clamp_grid(g_elem_[dual ? 1 : 0], (m.E + PW::EW - 1) / PW::EW, 1);
    if (dual)
      launch(k_l2v_elem<D, K, T, true>, g, 32 * PW::WARPS, PW::SMEM, st, 
          m, static_cast<const T*>(t.Dinv), static_cast<const T*>(yL), static_cast<T*>(lf), static_cast<T*>(outV), c);
    else
      launch(k_l2v_elem<D, K, T, false>, g, 32 * PW::WARPS, PW::SMEM, st, 
          m, static_cast<const T*>(t.DT), static_cast<const T*>(yL), static_cast<T*>(lf), static_cast<T*>(outV), c);
    return 1;
  }

  int l2v_facet(const DevMesh& m, const void* lf, bool dual, Combine c, void* outV, cudaStream_t st) override {
    const int gf = clamp_grid(g_fsum_, m.NF * S::nf, 256);
    if (dual)
      launch(k_l2v_facet<D, K, T, true>, gf, 256, 0, st, m, static_cast<const T*>(lf), static_cast<T*>(outV), c);
    else
      launch(k_l2v_facet<D, K, T, false>, gf, 256, 0, st, m, static_cast<const T*>(lf), static_cast<T*>(outV), c);
    return 1;
  }
};

}  // namespace hopu

#define HOPU_DEFINE_OPS(D, K)                                               \
  namespace hopu {                                                          \
  Ops* make_ops_##D##_##K(bool fp64, int tc) {                              \
    if (fp64) return new OpsImpl<D, K, double>();                           \
    return new OpsImpl<D, K, float>(tc);                                    \
  }                                                                         \
  }
