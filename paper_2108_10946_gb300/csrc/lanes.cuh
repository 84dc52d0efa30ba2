// One DoF's values of SG consecutive shots (1, 2 or 4) as one register group: loads, stores, global
// accumulation without a result, and packed FP32x2 arithmetic.
#pragma once
#include "fwi_internal.h"

namespace fwi {

template <int SG>
struct alignas(4 * SG) Lanes {  // one DoF's values of SG consecutive shots
  float x[SG];
};
template <int SG>
__device__ __forceinline__ Lanes<SG> lanes_ld(const float* p) {
  return *reinterpret_cast<const Lanes<SG>*>(p);
}
template <int SG>
__device__ __forceinline__ Lanes<SG> lanes_ldcg(const float* p) {  // from L2, where atomics resolve
  Lanes<SG> r;
  if constexpr (SG == 4) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
    r.x[0] = v.x, r.x[1] = v.y, r.x[2] = v.z, r.x[3] = v.w;
  } else if constexpr (SG == 2) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    r.x[0] = v.x, r.x[1] = v.y;
  } else {
    r.x[0] = __ldcg(p);
  }
  return r;
}
template <int SG>
__device__ __forceinline__ void lanes_st(float* p, const Lanes<SG>& v) {
  *reinterpret_cast<Lanes<SG>*>(p) = v;
}
template <int SG>
__device__ __forceinline__ void lanes_add(float* p, const Lanes<SG>& v) {  // global, no result
  if constexpr (SG == 4) atomicAdd(reinterpret_cast<float4*>(p), make_float4(v.x[0], v.x[1], v.x[2], v.x[3]));
  else if constexpr (SG == 2) atomicAdd(reinterpret_cast<float2*>(p), make_float2(v.x[0], v.x[1]));
  else atomicAdd(p, v.x[0]);
}
// y += z on every shot
template <int SG>
__device__ __forceinline__ void lanes_acc(Lanes<SG>& y, const Lanes<SG>& z) {
  if constexpr (SG == 1) {
    y.x[0] += z.x[0];
  } else {
#pragma unroll
    for (int k = 0; k < SG; k += 2) {
      const float2 t = __fadd2_rn(make_float2(y.x[k], y.x[k + 1]), make_float2(z.x[k], z.x[k + 1]));
      y.x[k] = t.x;
      y.x[k + 1] = t.y;
    }
  }
}
template <int SG>
__device__ __forceinline__ Lanes<SG> lanes_fma(float a, const Lanes<SG>& x, const Lanes<SG>& y) {  // a x + y
  Lanes<SG> r;
  if constexpr (SG == 1) {
    r.x[0] = fmaf(a, x.x[0], y.x[0]);
  } else {
#pragma unroll
    for (int k = 0; k < SG; k += 2) {
      const float2 t = __ffma2_rn(make_float2(a, a), make_float2(x.x[k], x.x[k + 1]), make_float2(y.x[k], y.x[k + 1]));
      r.x[k] = t.x;
      r.x[k + 1] = t.y;
    }
  }
  return r;
}
template <int SG>
__device__ __forceinline__ Lanes<SG> lanes_mul(float a, const Lanes<SG>& x) {
  Lanes<SG> r;
#pragma unroll
  for (int k = 0; k < SG; ++k) r.x[k] = a * x.x[k];
  return r;
}

}  // namespace fwi
