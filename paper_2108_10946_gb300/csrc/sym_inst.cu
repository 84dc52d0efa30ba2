// The symmetry-adapted chunk kernels of one KMV element and one group of shots per CTA,
// instantiated once per (dimension, degree, shots): -DKMV_DIM=d -DKMV_K=k -DKMV_SG=1|2|4.
#include <algorithm>

#include "fwi_internal.h"

namespace fwi {
namespace {
constexpr int D = KMV_DIM;
constexpr int NN = D == 2 ? (KMV_K == 2 ? 7 : KMV_K == 3 ? 12 : KMV_K == 4 ? 18 : 30)
                          : (KMV_K == 2 ? 15 : 32);
constexpr int NS = D == 2 ? 3 * KMV_K : (KMV_K == 2 ? 14 : 28);
constexpr int SG = KMV_SG;
constexpr int NSYM = D == 3 && NN == 32 ? 768 : 300;
__constant__ int c_slot[NN];  // slot of every local node (sym_slot_node)
__constant__ float c_sym[NSYM];
__constant__ float2 c_sym2[NSYM];  // every coefficient twice: operands of packed multiply-adds
// Shots per thread of groups of two and four: pairs issue half the instructions, but at KMV5 a
// pair's nodal values leave too few registers for a second pair of warps per scheduler (marine
// mesh, S = 4: 428 us per forward step, 480 us with pairs). KMV4, 250k triangles: 109 us per step
// one by one, 80 us in pairs; KMV3 alike.
#ifndef SYM_LANES
#define SYM_LANES (KMV_K == 5 || KMV_DIM == 3 ? 1 : 2)
#endif
__constant__ float c_w[NN];
}  // namespace
}  // namespace fwi

#include "chunk_sym.cuh"

namespace fwi {
namespace {
constexpr int NT = SymMap<SG>::NT;
// Registers a thread may take: enough CTAs per SM to hide the loads of one behind the arithmetic of
// the others. KMV5 gradient steps hold more at a time and lose less to a fourth CTA less than to
// spills (marine mesh, one gradient of 75 steps: 128.5 ms at 168, 133.1 ms at 128); every other
// kernel is best at 128 (KMV4, S = 4, 250k triangles: 8.0 ms for 100 steps, 10.9 ms at 204; KMV3,
// 120k: 8.9 and 9.8 ms).
template <int MODE, bool LAYER>
constexpr int registers() {
#ifdef SYM_REGS
  return SYM_REGS;
#endif
  if (KMV_DIM == 3 && KMV_K == 3) return LAYER ? 255 : MODE == 2 ? 204 : 168;
  return KMV_K == 5 && MODE == 2 ? 168 : 128;
}

template <int MODE, bool LAYER>
__global__ void __launch_bounds__(NT, 65536 / (registers<MODE, LAYER>() * NT)) k_sym(const StepArgs a) {
  extern __shared__ __align__(16) float smem_sym[];
  if constexpr (D == 2) sym_tri_body<NN, NS, MODE, LAYER, SG>(a, smem_sym);
  else sym_tet_body<NN, NS, MODE, LAYER, SG>(a, smem_sym);
}

template <int MODE, bool LAYER>
int launch_t(const StepArgs& a, int ch0, int nch, cudaStream_t st) {
  if (nch <= 0) return 0;
  const size_t bytes =
      sizeof(float) * (size_t)sym_smem<D, NN, NS, SG, MODE, LAYER>(a.T_max, a.SH_max, a.H_max).total;
  if (bytes > 227 * 1024) return (int)cudaErrorInvalidValue;
  static size_t configured[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  static int wave[64] = {0};  // CTAs that run at a time
  if (dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  if (bytes > configured[dev]) {
    cudaError_t e = cudaFuncSetAttribute(k_sym<MODE, LAYER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    int per = 0, nsm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sym<MODE, LAYER>, NT, bytes);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return (int)e;
    wave[dev] = per * nsm;
    configured[dev] = bytes;
  }
  StepArgs b = a;
  b.ch0 = ch0;
  b.ch1 = ch0 + nch;
  b.wave = wave[dev];
  k_sym<MODE, LAYER><<<dim3((unsigned)nch, (unsigned)(a.S / SG)), NT, bytes, st>>>(b);
  return 0;
}

// chunks [0, nch0) hold no damping-layer element, chunks [nch0, nch) do
int launch(const StepArgs& a, cudaStream_t st, cudaStream_t stl) {
  const int mode = a.mode == 0 ? 0 : (a.ring_u != nullptr ? 2 : 1), nl = a.nch - a.nch0;
  int rc = mode == 0   ? launch_t<0, false>(a, 0, a.nch0, st)
           : mode == 1 ? launch_t<1, false>(a, 0, a.nch0, st)
                       : launch_t<2, false>(a, 0, a.nch0, st);
  if (rc) return rc;
  return mode == 0   ? launch_t<0, true>(a, a.nch0, nl, stl)
         : mode == 1 ? launch_t<1, true>(a, a.nch0, nl, stl)
                     : launch_t<2, true>(a, a.nch0, nl, stl);
}

int upload(const float* w, const float* sym, int nsym) {
  if (nsym > NSYM) return (int)cudaErrorInvalidValue;
  float tab[NSYM] = {0.f}, ws[NN];
  float2 dup[NSYM];
  int slot[NN];
  for (int i = 0; i < nsym; ++i) tab[i] = sym[i];
  if constexpr (D == 3 && NN == 32)  // the rolled loop's table: every axis, [orbit][axis][output][mode]
    for (int o = 0; o < 8; ++o)
      for (int i = 0; i < 96; ++i) {
        const int d = i / 32, z = i / 8 % 4;
        tab[o * 96 + i] = sym[tet_at<NN>(o, d, z, z ^ (d + 1), i % 8)];
      }
#if KMV_DIM == 2
  if (TriSym<NN>::ROLL) {  // X orbits first, then T orbits
    using T = TriSym<NN>;
    int x = 0, t = T::NX * T::XTAB;
    for (int o = 0; o < T::NO; ++o) {
      int& to = T::kind(o) == 'X' ? x : t;
      const int n = T::kind(o) == 'X' ? T::XTAB : T::TTAB;
      for (int i = 0; i < n; ++i) tab[to + i] = sym[T::tab(o) + i];
      to += n;
    }
  }
#endif
  for (int i = 0; i < NSYM; ++i) dup[i] = make_float2(tab[i], tab[i]);
  for (int j = 0; j < NN; ++j) {
    const int q = sym_slot_node(D, NN, j);
    slot[q] = j;
    ws[j] = w[q];
  }
  cudaError_t e = cudaMemcpyToSymbol(c_w, ws, sizeof ws);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_slot, slot, sizeof slot);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_sym, tab, sizeof tab);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_sym2, dup, sizeof dup);
  return (int)e;
}
}  // namespace

#define SYM_CAT2(a, b, c, d) a##b##_##c##_##d
#define SYM_CAT(a, b, c, d) SYM_CAT2(a, b, c, d)
extern const SymKernels SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, KMV_SG) = {upload, launch};
}  // namespace fwi
