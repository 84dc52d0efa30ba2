// Kernels of one KMV element, instantiated once per (dimension, degree): the build compiles
// this file with -DKMV_DIM=d -DKMV_K=k for KMV2..5tri and KMV2..3tet. Nodes per element:
// triangles 7, 12, 18, 30 (6, 9, 12, 15 of them on vertices and edges); tetrahedra 15, 32
// (14, 28 on vertices, edges and faces).
#include <algorithm>
#include <vector>

#include "fwi_internal.h"

#if !defined(KMV_DIM) || !defined(KMV_K)
#error "compile with -DKMV_DIM=<2|3> -DKMV_K=<degree>"
#endif

namespace fwi {
namespace {
constexpr int D = KMV_DIM;
constexpr int NN = D == 2 ? (KMV_K == 2 ? 7 : KMV_K == 3 ? 12 : KMV_K == 4 ? 18 : 30)
                          : (KMV_K == 2 ? 15 : 32);
constexpr int NS = D == 2 ? 3 * KMV_K : (KMV_K == 2 ? 14 : 28);
static_assert((D == 2 && KMV_K >= 2 && KMV_K <= 5) || (D == 3 && KMV_K >= 2 && KMV_K <= 3),
              "KMV elements: triangles k = 2..5, tetrahedra k = 2, 3");
__constant__ float c_dhat[D * NN * NN];
__constant__ float c_w[NN];
}  // namespace
}  // namespace fwi

#include "step_kernel.cuh"
#if KMV_DIM == 2
#include "chunk_tc.cuh"
#endif

#define SYM_CAT2(a, b, c, d) a##b##_##c##_##d
#define SYM_CAT(a, b, c, d) SYM_CAT2(a, b, c, d)
namespace fwi {
extern const SymKernels SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 1), SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 2),
    SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 4);
}

namespace fwi {
namespace {
#if KMV_DIM == 2
// Dhat as the B operands of the tensor-core kernel (hi and lo, canonical layout)
__device__ __align__(16) float g_bimg[TcShape<D, NN>::BIMG];
#endif

__global__ void __launch_bounds__(128) k_step(const StepArgs a) { step_body<D, NN, NS>(a); }

#if KMV_DIM == 2
template <int MODE, bool LAYER>
__global__ void __launch_bounds__(128) k_chunk_tc(const StepArgs a, int nrun) {
  extern __shared__ __align__(128) float smem_tc[];
  chunk_tc_body<D, NN, NS, MODE, LAYER>(a, smem_tc, g_bimg, nrun);
}

// persistent: at most two CTAs per SM (each holds 256 of the SM's 512 tensor-memory
// columns; the shared-memory request is raised so that a third never fits)
template <int MODE, bool LAYER>
int launch_chunk_tc_t(const StepArgs& a, int ch0, int nch, cudaStream_t st) {
  if (nch <= 0) return 0;
  size_t bytes = chunk_tc_smem_floats<D, NN>(a.L_max, a.SG, MODE == 2, LAYER) * sizeof(float);
  if (bytes < 80 * 1024) bytes = 80 * 1024;
  if (bytes > 227 * 1024) return (int)cudaErrorInvalidValue;
  static size_t configured[64] = {0};
  static int nsm[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  if (bytes > configured[dev]) {
    cudaError_t e = cudaFuncSetAttribute(k_chunk_tc<MODE, LAYER>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return (int)e;
    configured[dev] = bytes;
  }
  if (nsm[dev] == 0) {
    cudaError_t e = cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return (int)e;
  }
  StepArgs b = a;
  b.ch0 = ch0;
  dim3 grid((unsigned)std::min(nch, 2 * nsm[dev]), (unsigned)(a.S / a.SG));
  k_chunk_tc<MODE, LAYER><<<grid, a.PE * a.SG, bytes, st>>>(b, nch);
  return 0;
}

#endif

const SymKernels& sym(const StepArgs& a) {
  return a.SG == 4   ? SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 4)
         : a.SG == 2 ? SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 2)
                     : SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 1);
}

// chunks [0, nch0) hold no damping-layer element, chunks [nch0, nch) do
int launch_chunk(const StepArgs& a, cudaStream_t st, cudaStream_t stl) {
  const int mode = a.mode == 0 ? 0 : (a.ring_u != nullptr ? 2 : 1);
  int rc = 0;
#if KMV_DIM == 2
  if (a.tc && mode != 0) {  // the adjoint steps only
    switch (mode) {
      case 1:
        rc = launch_chunk_tc_t<1, false>(a, 0, a.nch0, st);
        if (!rc) rc = launch_chunk_tc_t<1, true>(a, a.nch0, a.nch - a.nch0, stl);
        break;
      default:
        rc = launch_chunk_tc_t<2, false>(a, 0, a.nch0, st);
        if (!rc) rc = launch_chunk_tc_t<2, true>(a, a.nch0, a.nch - a.nch0, stl);
    }
    return rc;
  }
#endif
  return sym(a).launch(a, st, stl);
}
int run(const StepArgs& a, const RunArgs& r, cudaStream_t st) { return sym(a).run(a, r, st); }

int upload(const float* dhat, const float* w, const float* sym, int nsym) {
  cudaError_t e = cudaMemcpyToSymbol(c_dhat, dhat, sizeof(float) * D * NN * NN);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_w, w, sizeof(float) * NN);
#if KMV_DIM == 2
  if (e == cudaSuccess) {
    std::vector<float> img(TcShape<D, NN>::BIMG);
    tc_build_bimg<D, NN>(dhat, img.data());
    e = cudaMemcpyToSymbol(g_bimg, img.data(), sizeof(float) * img.size());
  }
#endif
  int rc = (int)e;
  if (!rc) rc = SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 1).upload(w, sym, nsym);
  if (!rc) rc = SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 2).upload(w, sym, nsym);
  if (!rc) rc = SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, 4).upload(w, sym, nsym);
  return rc;
}

void launch_step(const StepArgs& a, cudaStream_t st) {
  const int64_t threads = (int64_t)a.E * a.S;
  const int bs = 128;
  k_step<<<(unsigned)((threads + bs - 1) / bs), bs, 0, st>>>(a);
}

void launch_record(const StepArgs& a, const int* rec_elem, const float* rec_phi, cudaStream_t st) {
  const int threads = a.R * a.S;
  if (threads == 0) return;
  record_kernel<NN, NS><<<(threads + 127) / 128, 128, 0, st>>>(a, rec_elem, rec_phi);
}
}  // namespace

#define KMV_CAT2(a, b, c, d) a##b##c##d
#define KMV_CAT(a, b, c, d) KMV_CAT2(a, b, c, d)
extern const KernelSet KMV_CAT(kernels_, KMV_DIM, _, KMV_K) = {D,           KMV_K,       NN,
                                                              NS,          NN - NS,     upload,
                                                              launch_step, launch_chunk,
                                                              run,         launch_record};
}  // namespace fwi
