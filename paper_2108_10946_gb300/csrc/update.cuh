// Per-DoF increment update shared by the element kernels (element-interior DoFs) and the
// node kernel (shared DoFs), and the node kernel itself.
#pragma once
#include "fwi_internal.h"

namespace fwi {

template <int D>
struct LayerCoef {  // offsets inside one layer DoF's coefficient record
  static constexpr int E1 = 0, E2F = D, E2A = 2 * D, PSI2 = 3 * D, E3F = 4 * D, PSI3 = 5 * D,
                       C4 = 6 * D, C5 = 6 * D + 1, DTDET = 6 * D + 2, DTM = 6 * D + 3;
  static constexpr int COUNT = D == 2 ? 4 * D : 6 * D + 4;
};

// Increment-form update of one DoF (shared by the element and node kernels):
//   v' = c1 v - c2 y - c3 u  (- c4 Y^n in the 3D forward, + c5 lam_omega^m in the 3D adjoint)
//   u' = u + v'
// plus the layer auxiliaries of the DoF:
//   forward  P_k' = e1_k P_k - e2f_k sU_k (+ e3f_k sY_k in 3D);  Y' = Y + dt u
//   adjoint  nu_k' = e1_k nu_k - e2a_k sU_k;  lam_w' = lam_w - dt detPsi1 lam + (dt/M) yw
// The update with the DoF's v, c1..c3 and layer index already at hand (chunk kernels
// prefetch them into shared memory).
template <int D>
__device__ __forceinline__ void dof_update_pre(const StepArgs& a, int dof, int s, float y, float uo,
                                               float vo, float c1, float c2, float c3, int pi,
                                               const float* sU, const float* sY, float yw,
                                               const float* po = nullptr) {
  const int S = a.S;
  const size_t i = (size_t)dof * S + s;
  float vn = c1 * vo - c2 * y - c3 * uo;
  if (pi >= 0) {
    typedef LayerCoef<D> L;
    const float* lc = a.lcf + (size_t)pi * L::COUNT;
    if (a.mode == 0) {
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const size_t pk = ((size_t)pi * D + k) * S + s;
        const float pold = po ? po[k] : a.P[pk];
        float pn = __ldg(lc + L::E1 + k) * pold - __ldg(lc + L::E2F + k) * sU[k];
        if constexpr (D == 3) pn += __ldg(lc + L::E3F + k) * sY[k];
        a.P[pk] = pn;
      }
      if constexpr (D == 3) {
        const size_t py = (size_t)pi * S + s;
        const float yo = a.Y[py];
        vn -= __ldg(lc + L::C4) * yo;
        a.Y[py] = yo + a.dt * uo;
      }
    } else {
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const size_t pk = ((size_t)pi * D + k) * S + s;
        const float pold = po ? po[k] : a.P[pk];
        a.P[pk] = __ldg(lc + L::E1 + k) * pold - __ldg(lc + L::E2A + k) * sU[k];
      }
      if constexpr (D == 3) {
        const size_t py = (size_t)pi * S + s;
        const float wo = a.Y[py];
        vn += __ldg(lc + L::C5) * wo;
        a.Y[py] = wo - __ldg(lc + L::DTDET) * uo + __ldg(lc + L::DTM) * yw;
      }
    }
  }
  a.v[i] = vn;
  const float un = uo + vn;
  a.u[i] = un;
  if (!isfinite(un)) atomicOr(a.status, 1);
}

template <int D>
__device__ __forceinline__ void dof_update(const StepArgs& a, int dof, int s, float y, float uo,
                                           const float* sU, const float* sY, float yw) {
  const float c1 = __ldg(a.cf + dof);
  const float c2 = __ldg(a.cf + (size_t)a.N + dof);
  const float c3 = __ldg(a.cf + 2 * (size_t)a.N + dof);
  const float vo = a.v[(size_t)dof * a.S + s];
  const int pi = __ldg(a.pidx + dof);
  dof_update_pre<D>(a, dof, s, y, uo, vo, c1, c2, c3, pi, sU, sY, yw);
}

constexpr int NODE_ITEMS = 4;

// Shared-DoF finish as a separate pass over the DoFs [h0, h0 + hcnt) (the shared DoFs of the plain
// layout; halo.cuh has the chunked layout's), whose element contributions arrived by atomics in
// r[(dof - h0) * S + s].
template <int D>
__global__ void __launch_bounds__(256) node_kernel(const StepArgs a) {
  // NODE_ITEMS (DoF, shot) items per thread, a block-stride apart (coalesced); all their
  // reads are issued before any write, so that each thread has NODE_ITEMS times more
  // memory requests in flight
  const int S = a.S;
  const int64_t total = (int64_t)a.hcnt << a.log2S;
  const int64_t base = (int64_t)blockIdx.x * blockDim.x * NODE_ITEMS + threadIdx.x;
  float uo[NODE_ITEMS], vo[NODE_ITEMS], y[NODE_ITEMS], c1[NODE_ITEMS], c2[NODE_ITEMS],
      c3[NODE_ITEMS];
  int pi[NODE_ITEMS];
#pragma unroll
  for (int k = 0; k < NODE_ITEMS; ++k) {
    const int64_t t = base + (int64_t)k * blockDim.x;
    uo[k] = vo[k] = y[k] = c1[k] = c2[k] = c3[k] = 0.f;
    pi[k] = -1;
    if (t < total) {
      const int64_t i = t >> a.log2S;
      const int dof = a.h0 + (int)i;
      const size_t ix = (size_t)dof * S + (t & (S - 1));
      uo[k] = a.u[ix];
      vo[k] = a.v[ix];
      y[k] = __ldcg(a.r + (size_t)t);
      c1[k] = __ldg(a.cf + dof);
      c2[k] = __ldg(a.cf + (size_t)a.N + dof);
      c3[k] = __ldg(a.cf + 2 * (size_t)a.N + dof);
      pi[k] = __ldg(a.pidx + dof);
    }
  }
#pragma unroll
  for (int k = 0; k < NODE_ITEMS; ++k) {
    const int64_t t = base + (int64_t)k * blockDim.x;
    if (t >= total) continue;
    const int64_t i = t >> a.log2S;
    const int dof = a.h0 + (int)i;
    const int s = (int)(t & (S - 1));
    a.r[(size_t)t] = 0.f;
    float sU[D], sY[D];
    float yw = 0.f;
#pragma unroll
    for (int d = 0; d < D; ++d) sU[d] = sY[d] = 0.f;
    if (pi[k] >= 0) {  // damping layer: the layer sums (a minority of the DoFs)
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const size_t pk = ((size_t)pi[k] * D + d) * S + s;
        sU[d] = __ldcg(a.Pacc + pk);
        a.Pacc[pk] = 0.f;
        if constexpr (D == 3) {
          if (a.mode == 0) {
            sY[d] = __ldcg(a.PaccY + pk);
            a.PaccY[pk] = 0.f;
          }
        }
      }
      if constexpr (D == 3) {
        if (a.mode == 1) {
          const size_t py = (size_t)pi[k] * S + s;
          yw = __ldcg(a.Yacc + py);
          a.Yacc[py] = 0.f;
        }
      }
    }
    dof_update_pre<D>(a, dof, s, y[k], uo[k], vo[k], c1[k], c2[k], c3[k], pi[k], sU, sY, yw);
  }
}

}  // namespace fwi
