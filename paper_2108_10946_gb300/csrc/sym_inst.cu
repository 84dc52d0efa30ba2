// The symmetry-adapted chunk kernels of one KMV element and one group of shots per CTA,
// instantiated once per (dimension, degree, shots): -DKMV_DIM=d -DKMV_K=k -DKMV_SG=1|2|4.
#include <algorithm>
#include <mutex>

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
#include "halo.cuh"

namespace fwi {
namespace {
constexpr int NT = SymMap<SG, false>::NT, NT_RUN = SymMap<SG, true>::NT;
// Most CTAs of a launch of several steps; two per SM of this chip. Launches per step against one
// launch, ms: KMV2, one shot, 400 steps, 256 CTAs 4.21 / 3.97; 200 steps, 360 CTAs 2.13 / 1.98, 470
// 2.13 / 2.12, 630 2.13 / 2.31 (more CTAs crowd the meetings' counter; 1,560, a KMV5 gradient of 75
// steps: 6.3 / 15.4). Below the line, 12 and 290 CTAs: one shot, KMV5 gradient 4.0 / 3.2 and 3.9 / 3.5,
// KMV3 tetrahedra with a layer 5.8 / 4.3 and 5.8 / 5.3; four shots without a layer, KMV3 gradient 2.5 /
// 2.3 and 2.5 / 2.6. With a layer and four shots launches per step are faster (KMV5 gradient 3.9 / 5.8
// and 4.4 / 7.6): run_chunk's layer instances spill and read their arguments through a pointer.
constexpr int RUN_MAX = 304;

// Registers a thread may take: enough CTAs per SM to hide the loads of one behind the arithmetic of
// the others. KMV5 gradient steps need 168; at 128, with one CTA more per SM, they spill (marine mesh,
// one gradient of 75 steps: 128.5 against 133.1 ms). The other triangle kernels and KMV2 tetrahedra
// are best at 128 (KMV4, S = 4, 250k triangles: 8.0 ms for 100 steps, 10.9 ms at 204; KMV3, 120k: 8.9
// and 9.8 ms), but KMV2 triangles at one shot, which do little with what they load, at 48 (2M
// triangles, 50 steps: 3.54 ms, 3.71 ms at 80). KMV3 tetrahedra keep one or two fields' 32 adapted
// values in registers and take what shared memory leaves: two CTAs per SM of their layer chunks
// have room for 255 registers a thread.
template <int MODE, bool LAYER>
constexpr int registers() {
  if (KMV_DIM == 3 && KMV_K == 3) return LAYER ? 255 : MODE == 2 ? 204 : 168;
  return KMV_K == 5 && MODE == 2 ? 168 : KMV_DIM == 2 && KMV_K == 2 && SG == 1 ? 48 : 128;
}

template <int MODE, bool LAYER>
__global__ void __launch_bounds__(NT, 65536 / (registers<MODE, LAYER>() * NT)) k_sym(const StepArgs a) {
  extern __shared__ __align__(16) float smem_sym[];
  const SymStep x{a.u, a.u_out, a.ring_u, a.n, 0};
  const int c = blockIdx.x + a.ch0, s0 = blockIdx.y * SG;
  if constexpr (D == 2) sym_tri_body<NN, NS, MODE, LAYER, SG, false>(a, x, smem_sym, c, s0);
  else sym_tet_body<NN, NS, MODE, LAYER, SG, false>(a, x, smem_sym, c, s0);
}

// Both kinds of chunks in one launch, the layer's (the longer ones) first.
template <int MODE>
__global__ void __launch_bounds__(NT, 65536 / (registers<MODE, true>() * NT)) k_both(const StepArgs a) {
  extern __shared__ __align__(16) float smem_sym[];
  const SymStep x{a.u, a.u_out, a.ring_u, a.n, 0};
  const int c = a.nch - 1 - blockIdx.x, s0 = blockIdx.y * SG;
  if (c >= a.nch0) {
    if constexpr (D == 2) sym_tri_body<NN, NS, MODE, true, SG, false>(a, x, smem_sym, c, s0);
    else sym_tet_body<NN, NS, MODE, true, SG, false>(a, x, smem_sym, c, s0);
  } else {
    if constexpr (D == 2) sym_tri_body<NN, NS, MODE, false, SG, false>(a, x, smem_sym, c, s0);
    else sym_tet_body<NN, NS, MODE, false, SG, false>(a, x, smem_sym, c, s0);
  }
}

// Several steps in one cooperative launch, for meshes whose steps are shorter than launching them:
// every CTA takes a chunk, all CTAs meet, every thread finishes its halo DoFs, all meet again.
// A chunk and a halo DoF stay with their CTA, so only what crosses CTAs has to come from L2. Both
// kinds of chunks are one kernel here.
__device__ __forceinline__ bool run_meet(unsigned* count, unsigned target, int polls) {
  // (the fields are written as usual and read by bulk copies; the next step's copies come after this
  // step's reads of the tables)
  asm volatile("fence.proxy.async;" ::: "memory");
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    ok = false;
    for (int i = 0; i < polls; ++i) {  // bounded: a CTA that gave up never arrives
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
      if ((int)(v - target) >= 0) {
        ok = true;
        break;
      }
    }
    asm volatile("fence.proxy.async;" ::: "memory");
  }
  return __syncthreads_and(ok);
}

// (Not inlined: the two kinds' code side by side in the step loop would spill.)
template <int MODE, bool LAYER>
__device__ __noinline__ bool run_chunk(const StepArgs& a, const SymStep& x, float* sm, int c, int s0) {
  if constexpr (D == 2) return sym_tri_body<NN, NS, MODE, LAYER, SG, true>(a, x, sm, c, s0);
  else return sym_tet_body<NN, NS, MODE, LAYER, SG, true>(a, x, sm, c, s0);
}

template <int MODE>
__global__ void __launch_bounds__(NT_RUN, 65536 / (registers<MODE, true>() * NT_RUN))
    k_run(const __grid_constant__ StepArgs a, const RunArgs r) {
  extern __shared__ __align__(16) float smem_sym[];
  const int ngrp = a.S / SG, tid = threadIdx.x;
  const int c = a.nch - 1 - blockIdx.x / ngrp, s0 = blockIdx.x % ngrp * SG;  // the layer's chunks, the longer ones, first
  if (tid == 0) sym_bar_init(reinterpret_cast<uint64_t*>(smem_sym));
  // (an earlier launch of the call gave up: its CTAs never met, this one's would poll to the limit)
  if (__syncthreads_or(tid == 0 && (__ldcg(a.status) & 2))) return;
  unsigned target = r.base;
  SymStep x{nullptr, nullptr, nullptr, 0, 0};
  for (int k = 0; k < r.steps; ++k) {
    const int rel = r.rel0 + k * r.dir;  // time level less the segment's first
    x.n = r.n0 + k * r.dir;
    if (MODE == 0) {  // the levels the gradient needs go to the ring, the others stay in u
      x.u = r.ring && rel % r.stride == 0 ? r.ring + (size_t)(rel / r.stride) * r.level : a.u;
      x.u_out = r.ring && (rel + 1) % r.stride == 0 ? r.ring + (size_t)((rel + 1) / r.stride) * r.level : a.u_out;
    } else {
      x.u = a.u;
      x.u_out = a.u_out;
      x.ring_u = r.ring + (size_t)rel * r.level;
    }
    const bool ok = c < a.nch0 ? run_chunk<MODE, false>(a, x, smem_sym, c, s0) : run_chunk<MODE, true>(a, x, smem_sym, c, s0);
    if (!ok) return;
    x.parity ^= 1;
    if (!run_meet(r.count, target += gridDim.x, a.wait_limit)) {
      if (tid == 0) atomicOr(a.status, 2);
      return;
    }
    const int64_t items = (int64_t)a.hcnt * ngrp;
    for (int64_t t = (int64_t)blockIdx.x * NT_RUN + tid; t < items; t += (int64_t)gridDim.x * NT_RUN) {
      const int dof = a.h0 + (int)(t / ngrp);
      halo_dof<D, SG, MODE == 0 ? 0 : 1>(a, x.u, x.u_out, dof, (int)(t % ngrp) * SG, dof >= a.halo_layer);
    }
    if (!run_meet(r.count, target += gridDim.x, a.wait_limit)) {
      if (tid == 0) atomicOr(a.status, 2);
      return;
    }
  }
}

std::mutex g_limits;  // the kernels' shared-memory limits are raised by one thread at a time

// Returns the CTAs of the launch, 0 if the steps are better launched one by one (nothing done), or
// minus a cudaError_t.
template <int MODE>
int run_t(const StepArgs& a, const RunArgs& r, cudaStream_t st) {
  const size_t bytes =
      sizeof(float) * (size_t)(a.nch > a.nch0 ? sym_smem<D, NN, NS, SG, MODE, true>(a.T_max, a.SH_max, a.H_max).total
                                              : sym_smem<D, NN, NS, SG, MODE, false>(a.T_max, a.SH_max, a.H_max).total);
  if (bytes > 227 * 1024) return 0;
  static size_t configured[64] = {0};
  static int nsm[64] = {0};
  int dev = 0, per = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 0;
  cudaError_t e = cudaSuccess;
  std::unique_lock<std::mutex> lk(g_limits);
  if (bytes > configured[dev]) {
    e = cudaFuncSetAttribute(k_run<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return -(int)e;
    configured[dev] = bytes;
  }
  const int sms = nsm[dev];
  lk.unlock();
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_run<MODE>, NT_RUN, bytes);
  if (e != cudaSuccess) return -(int)e;
  const int64_t nwork = (int64_t)a.nch * (a.S / SG);
  const int64_t room = (int64_t)per * sms;
  if (nwork > RUN_MAX || nwork > room) return 0;
  const int grid = (int)nwork;  // (one chunk and shot group per CTA)
  StepArgs b = a;
  RunArgs q = r;
  b.ch0 = 0;
  void* args[] = {&b, &q};
  e = cudaLaunchCooperativeKernel((const void*)k_run<MODE>, dim3((unsigned)grid), dim3(NT_RUN), args, bytes, st);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {  // a part of the device only
    cudaGetLastError();
    return 0;
  }
  return e == cudaSuccess ? grid : -(int)e;
}
int run(const StepArgs& a, const RunArgs& r, cudaStream_t st) { return a.mode == 0 ? run_t<0>(a, r, st) : run_t<2>(a, r, st); }

// One launch of `kernel` over chunks [ch0, ch0 + nch), downwards from the last if down.
int launch_t(void (*kernel)(const StepArgs), int which, size_t bytes, const StepArgs& a, int ch0, int nch, bool down,
             cudaStream_t st) {
  if (nch <= 0) return 0;
  if (bytes > 227 * 1024) return (int)cudaErrorInvalidValue;
  static size_t configured[9][64] = {{0}};
  static int wave[9][64] = {{0}};  // CTAs that run at a time
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  std::unique_lock<std::mutex> lk(g_limits);
  if (bytes > configured[which][dev]) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    int per = 0, nsm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, NT, bytes);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return (int)e;
    wave[which][dev] = per * nsm;
    configured[which][dev] = bytes;
  }
  StepArgs b = a;
  b.ch0 = ch0;
  b.wave = down ? -wave[which][dev] : wave[which][dev];
  lk.unlock();
  kernel<<<dim3((unsigned)nch, (unsigned)(a.S / SG)), NT, bytes, st>>>(b);
  return 0;
}
template <int MODE>
int launch_mode(const StepArgs& a, cudaStream_t st, cudaStream_t stl) {
  const size_t plain = sizeof(float) * (size_t)sym_smem<D, NN, NS, SG, MODE, false>(a.T_max, a.SH_max, a.H_max).total;
  const size_t layer = sizeof(float) * (size_t)sym_smem<D, NN, NS, SG, MODE, true>(a.T_max, a.SH_max, a.H_max).total;
  if (a.both) return launch_t(k_both<MODE>, 6 + MODE, std::max(plain, layer), a, 0, a.nch, true, st);
  const int rc = launch_t(k_sym<MODE, false>, MODE, plain, a, 0, a.nch0, false, st);
  return rc ? rc : launch_t(k_sym<MODE, true>, 3 + MODE, layer, a, a.nch0, a.nch - a.nch0, false, stl);
}

// Chunks [0, nch0) hold no damping-layer element, chunks [nch0, nch) do: one launch each, on st and
// stl, or (a.both) both in one on st.
int launch(const StepArgs& a, cudaStream_t st, cudaStream_t stl) {
  return a.mode == 0             ? launch_mode<0>(a, st, stl)
         : a.ring_u == nullptr ? launch_mode<1>(a, st, stl)
                                 : launch_mode<2>(a, st, stl);
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
extern const SymKernels SYM_CAT(sym_kernels_, KMV_DIM, KMV_K, KMV_SG) = {upload, launch, run};
}  // namespace fwi
