// Pairs of FP32 values in one 64-bit register and the packed arithmetic of sm_100+
// (add / mul / fma .rn.f32x2): one issue slot for two IEEE operations, each rounded as its
// scalar form.  The register kernels are bound by instruction issue, not by the FMA units
// (scalar FP32 FMAs were 78 % of their instructions), so packing their dot products and
// accumulations halves what they issue at the same results.
#pragma once
#include <cuda_runtime.h>

namespace hopu {

struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 f2_pack(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_pack(x, x); }
__device__ __forceinline__ float f2_x(f2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float f2_y(f2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }
__device__ __forceinline__ float f2_sum(f2 a) { return f2_x(a) + f2_y(a); }
__device__ __forceinline__ f2 f2_zero() { return f2{0ull}; }
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

// two pairs from a 16-byte aligned shared-memory address (not hoisted out of loops)
__device__ __forceinline__ void lds_f2(const float* p, f2& a, f2& b) {
  asm volatile("ld.shared.v2.b64 {%0,%1}, [%2];\n"
               : "=l"(a.v), "=l"(b.v)
               : "r"((unsigned)__cvta_generic_to_shared(p)));
}

// One step of the compensated dot product (dot2_step) on two independent sums: s + c gains
// a * x exactly up to the rounding of c.  nx = -x, so that p - a x comes from one FMA.
__device__ __forceinline__ void dot2_first_f2(f2& s, f2& c, f2 a, f2 x, f2 nx) {
  s = f2_mul(a, x);
  c = f2_sub(f2_zero(), f2_fma(a, nx, s));  // s - a x, negated: the product's rounding error
}
__device__ __forceinline__ void dot2_step_f2(f2& s, f2& c, f2 a, f2 x, f2 nx) {
  const f2 p = f2_mul(a, x);
  const f2 npe = f2_fma(a, nx, p);
  const f2 t = f2_add(s, p);
  const f2 z = f2_sub(t, s);
  const f2 se = f2_add(f2_sub(s, f2_sub(t, z)), f2_sub(p, z));
  s = t;
  c = f2_add(c, f2_sub(se, npe));
}

}  // namespace hopu
