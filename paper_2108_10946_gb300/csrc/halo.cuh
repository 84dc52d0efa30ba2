// Finish of the halo DoFs of the chunked layout: one thread per (DoF, SG shots). Their sums arrived
// from the chunks by atomics, so they are read from L2, and the accumulators cleared for the next
// step; then the increment update of chunk_sym.cuh's sym_finish, and in the damping layer the
// update of the auxiliaries.
//
// The kernel moves 110 bytes per DoF and four shots (2D layer: 310; 3D: 480) and is bound by how
// many of them are in flight: a layer DoF's place in the layer arrays follows from its number (the
// layer's halo DoFs are the last ones), so all of its reads go out at once, and the two kinds of DoF
// sit in different blocks.
#pragma once
#include "lanes.cuh"

namespace fwi {

// DoF dof, shots s0, s0 + 1, ...; u: the field, u_out: where it goes.
template <int D, int SG, int MODE>
__device__ __forceinline__ void halo_dof(const StepArgs& a, const float* u, float* u_out, int dof, int s0, bool layer) {
  const int S = a.S;
  const size_t ix = (size_t)dof * S + s0, rx = (size_t)(dof - a.h0) * S + s0;
  const Lanes<SG> uo = lanes_ld<SG>(u + ix), vo = lanes_ld<SG>(a.v + ix);
  const Lanes<SG> y = lanes_ldcg<SG>(a.r + rx);
  const float c1 = __ldg(a.cf + dof), c2 = __ldg(a.cf + (size_t)a.N + dof), c3 = __ldg(a.cf + 2 * (size_t)a.N + dof);
  Lanes<SG> zero, vn;
#pragma unroll
  for (int k = 0; k < SG; ++k) zero.x[k] = 0.f;
  if (!layer) {
    vn = lanes_fma<SG>(-c2, y, lanes_fma<SG>(-c3, uo, lanes_mul<SG>(c1, vo)));
  } else {
    const size_t pi = (size_t)(dof - a.p_halo);
    float* P = a.P + pi * D * S + s0;
    float* Pa = a.Pacc + pi * D * S + s0;
    Lanes<SG> p[D], q[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      p[d] = lanes_ld<SG>(P + (size_t)d * S);
      q[d] = lanes_ldcg<SG>(Pa + (size_t)d * S);
    }
    const float4* lc = reinterpret_cast<const float4*>(a.lcs) + pi * (D == 2 ? 2 : 3);
    const float4 A = __ldg(lc), B = D == 3 || MODE != 0 ? __ldg(lc + 1) : A;
    Lanes<SG> Yo = zero, yw = zero;
    float4 C = A;
    if constexpr (D == 3) {
      Yo = lanes_ld<SG>(a.Y + pi * S + s0);
      if (MODE != 0) {
        yw = lanes_ldcg<SG>(a.Yacc + pi * S + s0);
        C = __ldg(lc + 2);
      }
    }
    vn = lanes_fma<SG>(-c2, y, lanes_fma<SG>(-c3, uo, lanes_mul<SG>(c1, vo)));
    const float e1[3] = {A.x, A.y, A.z};
    const float e2[3] = {D == 2 ? (MODE == 0 ? A.z : B.x) : B.x, D == 2 ? (MODE == 0 ? A.w : B.y) : B.y, B.z};
#pragma unroll
    for (int d = 0; d < D; ++d) {
      lanes_st<SG>(P + (size_t)d * S, lanes_fma<SG>(-e2[d], q[d], lanes_mul<SG>(e1[d], p[d])));
      lanes_st<SG>(Pa + (size_t)d * S, zero);
    }
    if constexpr (D == 3) {
      if (MODE == 0) {
        vn = lanes_fma<SG>(-A.w, Yo, vn);
        lanes_st<SG>(a.Y + pi * S + s0, lanes_fma<SG>(a.dt, uo, Yo));
      } else {
        vn = lanes_fma<SG>(C.x, Yo, vn);
        lanes_st<SG>(a.Y + pi * S + s0, lanes_fma<SG>(B.w, yw, lanes_fma<SG>(-C.y, uo, Yo)));
        lanes_st<SG>(a.Yacc + pi * S + s0, zero);
      }
    }
  }
  Lanes<SG> un = uo;
  lanes_acc<SG>(un, vn);
  lanes_st<SG>(a.r + rx, zero);
  lanes_st<SG>(a.v + ix, vn);
  lanes_st<SG>(u_out + ix, un);
  float chk = 0.f;
#pragma unroll
  for (int k = 0; k < SG; ++k) chk = fmaf(0.f, un.x[k], chk);
  if (!(chk == 0.f)) atomicOr(a.status, 1);
}

template <int D, int SG, int MODE>
__global__ void __launch_bounds__(128) halo_kernel(const StepArgs a, int plain_blocks) {
  const bool layer = (int)blockIdx.x >= plain_blocks;
  const int ngrp = a.S / SG;
  const int64_t t = (int64_t)(layer ? (int)blockIdx.x - plain_blocks : (int)blockIdx.x) * 128 + threadIdx.x;
  const int64_t i = ngrp == 1 ? t : t / ngrp;
  const int s0 = ngrp == 1 ? 0 : (int)(t - i * ngrp) * SG;
  const int lo = layer ? a.halo_layer : a.h0, hi = layer ? a.h0 + a.hcnt : a.halo_layer;
  if (i < hi - lo) halo_dof<D, SG, MODE>(a, a.u, a.u_out, lo + (int)i, s0, layer);
}

template <int D, int SG>
void launch_halo_t(const StepArgs& a, cudaStream_t st) {
  const int64_t g = a.S / SG;
  const int64_t plain = ((int64_t)(a.halo_layer - a.h0) * g + 127) / 128;
  const int64_t layer = ((int64_t)(a.h0 + a.hcnt - a.halo_layer) * g + 127) / 128;
  if (plain + layer == 0) return;
  if (a.mode == 0) halo_kernel<D, SG, 0><<<(unsigned)(plain + layer), 128, 0, st>>>(a, (int)plain);
  else halo_kernel<D, SG, 1><<<(unsigned)(plain + layer), 128, 0, st>>>(a, (int)plain);
}

}  // namespace fwi
