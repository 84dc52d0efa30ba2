// Chunked time step on symmetry-adapted derivatives: one CTA assembles one chunk of
// consecutive elements (Morton order) for a group of SG = min(S, 4) shots, entirely in
// shared memory; a thread takes one element for one shot or for two (SymMap).
//
//   1. load    the chunk's owned DoFs, one contiguous range (bulk copies issued by one thread;
//              copies of one DoF each if the batch has more shots than the group), its halo
//              DoFs and its tables, all at once; the owned ranges of the chunk that will run a
//              wave of CTAs later are brought to L2 meanwhile;
//   2. element the stiffness, layer and gradient arithmetic in adapted coordinates
//              (sym_tri.cuh); every thread writes its nodal sums to places of its own, [node]
//              [element][shot] for shared nodes and the bubble range, so nothing is added by
//              atomics;
//   3. update  each shared DoF adds its elements' sums in the order of an incidence list
//              (bubble DoFs have one) and, if owned, takes its increment update with coalesced
//              writes; halo sums go to global accumulators that the node kernel finishes.
//
// Owned DoFs are read and written by this CTA only; halo DoFs are only read here.
//
// What bounds it: instruction issue, then latency. KMV5 triangles, 4 shots (graded grid of 348k
// triangles, forward step): chunks without layer elements (60 %) 108 us, 3,200 instructions per warp
// of which 1,720 on the FMA pipes, issue slots 65 % full, 279 MB of DRAM traffic (38 % of the copy
// rate); layer chunks 181 us at 40 % (three CTAs per SM for their shared memory). The dense form
// with rows of Dhat from shared memory took 384 and 225 us on a mesh of this size. KMV2, one shot,
// 2M triangles: 71 us per step with the halo kernel's 8, 210 MB; KMV4, 4 shots, 250k: 57 us, 163 MB.
// Chunk sizes (sym_pe): at 32 triangles the KMV2 step spent 115 us, its chunks' fixed chain of loads
// over 96 DoFs each.
#pragma once
#include <type_traits>

#include "lanes.cuh"
#include "sym_tet.cuh"

namespace fwi {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// asynchronous copy of BYTES = 4, 8 or 16 (aligned) bytes
template <int BYTES>
__device__ __forceinline__ void sym_cp(void* dst, const void* src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void sym_cp_wait() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void sym_bar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void sym_bar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// Waits for a phase of the barrier; false if it gave up (after `polls`, each of which the hardware may
// suspend for a while).
__device__ __forceinline__ bool sym_bar_wait(uint64_t* bar, uint32_t parity, int polls) {
  for (int i = 0; i < polls; ++i) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ void sym_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

// A contiguous run of floats as a bulk copy: from the 16-byte boundary at or below its start, so
// it lands `shift` floats past the place it is copied to; whole 16-byte groups, so up to three floats
// past the run come along: arrays that are copied this way are allocated with four floats to spare,
// and in the tables nothing else is written behind a run (SYM_GAP).
struct SymRun {
  const float* src;
  int shift;
  uint32_t bytes;
};
__device__ __forceinline__ int sym_shift(const float* p) { return (int)(((uintptr_t)p >> 2) & 3); }
__device__ __forceinline__ SymRun sym_run(const float* p, int n) {
  SymRun r;
  r.shift = sym_shift(p);
  r.src = p - r.shift;
  r.bytes = n > 0 ? (uint32_t)((n + r.shift + 3) & ~3) * 4u : 0u;
  return r;
}
__device__ __forceinline__ void sym_prefetch(const float* p, int n) {  // to L2
  const SymRun r = sym_run(p, n);
  if (r.bytes) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(r.src), "r"(r.bytes) : "memory");
}

constexpr int SYM_PE = sym_pe(D, NN);  // most elements of a chunk, stride of its tables

// A CTA's threads: one element for LANES shots each. In launches of several steps (RUN: few chunks,
// latency counts) at least 128, those beyond the elements sharing the loads and the update.
template <int SG, bool RUN>
struct SymMap {
  static constexpr int LANES = SYM_LANES < SG ? SYM_LANES : SG, PER = SG / LANES, WORK = SYM_PE * PER;
  static constexpr int NT = RUN && WORK < 128 ? 128 : WORK;
  typedef typename std::conditional<LANES == 2, float2, float>::type V;
};

// What changes from step to step: fields in and out, the forward field (gradient steps), the time
// index, and the parity of the copies' barrier.
struct SymStep {
  const float* u;
  float* u_out;
  const float* ring_u;
  int n;
  uint32_t parity;
};

// Dynamic shared memory of one chunk (offsets in floats). T: largest chunk table (with the gap), SH:
// most shared DoFs (owned and halo), H: longest halo list of a chunk.
struct SymSmem {
  int u, f, c2, ps, om, ys, yb, p1, gs, gb, ws, wb, ss, sb, ids, meta, total;
};
// Floats per DoF of the layer's nodal coefficients in the table: Psi2 c^2 (2D adjoint; the six
// of a 3D DoF are read where they are used, the table would take the second CTA's room).
template <int D, int MODE>
__host__ __device__ constexpr int sym_psi() { return D == 2 && MODE != 0 ? 1 : 0; }

template <int D, int NN, int NS, int SG, int MODE, bool LAYER>
__host__ __device__ inline SymSmem sym_smem(int T, int SH, int H) {
  constexpr int PE = SYM_PE, NI = NN - NS, NE = NS * PE * SG, NB = (NI * PE * SG + 3) / 4 * 4;
  constexpr bool GRAD = MODE == 2, L3 = LAYER && D == 3;
  auto up = [](int n) { return (n + 7) & ~3; };  // a multiple of 4 with room for a run's shift
  auto most = [](int x, int y) { return x > y ? x : y; };
  SymSmem m{};
  int o = 4;  // the mbarrier
  m.u = o, o += up(T * SG);
  m.f = o, o += GRAD && !L3 ? up(T * SG) : 0;
  m.c2 = o, o += up(T);
  m.ps = o, o += LAYER ? up(T * sym_psi<D, MODE>()) : 0;
  // the shared DoFs' layer auxiliaries P lie where the elements' sums go once all have read P (in
  // 2D gradient steps that place holds the forward field's derivatives)
  constexpr bool APART = GRAD && D == 2;
  constexpr int SUMS = (NE + NB) * (L3 && MODE != 0 ? 2 : 1);  // y, and the omega row's (3D adjoint)
  m.ys = o, m.yb = o + NE, m.ws = o + NE + NB, m.wb = m.ws + NE, m.p1 = o + (APART ? SUMS : 0);
  o += !LAYER ? SUMS : APART ? SUMS + up(D * (SH + SYM_GAP) * SG) : most(SUMS, up(D * (SH + SYM_GAP) * SG));
  m.gs = o, o += GRAD ? NE : 0;
  m.gb = o, o += GRAD ? NB : 0;
  // 3D: the second field (the forward field; omega in forward steps) lies where the layer sums go
  m.om = m.ss = o;
  if (L3 && GRAD) m.f = o;
  o += LAYER ? most(D * NE, L3 && MODE != 1 ? up(T * SG) : 0) : 0;
  m.sb = o, o += LAYER ? up(D * NB) : 0;  // bubbles: P, then each (element, shot)'s own layer sums
  m.ids = o, o += up(H);
  m.meta = o, o += up(NS * PE + (SH + 16) / 2);  // table positions, incidence list, its pointers
  m.total = o;
  return m;
}

// Floats per layer DoF of the update's coefficients a.lcs: 2D e1, e2 forward, e2 adjoint, Psi2 c^2
// of the two directions each; 3D e1 and c4, e2 (adjoint) and dt/M, c5 and dt det Psi1.
template <int D>
constexpr int SYM_LCS = D == 2 ? 8 : 12;

struct SymDesc {
  int e0, ne, own, nsh, hp, hn, meta, meta_n, plain, keep;  // keep: an undamped DoF
};
__device__ __forceinline__ SymDesc sym_desc(const StepArgs& a, int c) {
  SymDesc d;
  const int4* p = reinterpret_cast<const int4*>(a.sdesc) + 2 * c;
  const int4 x = __ldg(p), y = __ldg(p + 1);
  d.e0 = x.x, d.ne = x.y & 0xffff, d.keep = x.y >> 16, d.own = x.z, d.nsh = x.w;
  d.hp = y.x, d.hn = y.y, d.meta = y.z, d.meta_n = y.w;
  d.plain = __ldg(a.splain + c);
  return d;
}

// Phase 1 of one chunk. The table: owned shared DoFs [0, nsh), bubbles, SYM_GAP places, halo DoFs (P of
// the shared DoFs: owned, SYM_GAP places, halo). The runs' shifts follow from their addresses
// (sym_shift).
// RUN (several steps in one launch): what other CTAs wrote in an earlier step comes from L2 (copies
// of four and eight bytes would go through L1).
template <int BYTES, bool RUN>
__device__ __forceinline__ void sym_cp_live(float* dst, const float* src) {
  if constexpr (RUN && BYTES < 16) lanes_st<BYTES / 4>(dst, lanes_ldcg<BYTES / 4>(src));
  else sym_cp<BYTES>(dst, src);
}
template <int D, int NN, int NS, int SG, int MODE, bool LAYER, bool RUN>
__device__ __forceinline__ void sym_load(const StepArgs& a, const SymStep& x, const SymDesc& cd, const SymSmem& L,
                                         float* sm, uint64_t* bar, int chunk, int s0, int tid) {
  constexpr int NI = NN - NS, NT = SymMap<SG, RUN>::NT;
  constexpr bool GRAD = MODE == 2, OM = LAYER && D == 3 && MODE == 0;
  constexpr int PSI = LAYER ? sym_psi<D, MODE>() : 0;
  const int S = a.S, on = cd.nsh + cd.ne * NI;
  const size_t i0 = (size_t)cd.own * S + s0;
  const size_t pi0 = (size_t)(cd.own - a.p_own);
  if (tid == 0) {
    // everything that is one run: coefficients, tables, and the fields if the group is the batch
    const SymRun c2 = sym_run(a.c2 + cd.own, on),
                 me = sym_run(reinterpret_cast<const float*>(a.smeta) + cd.meta, cd.meta_n);
    SymRun u{}, f{}, ps{}, om{}, p1{}, p2{};
    if (S == SG) {
      u = sym_run(x.u + i0, on * SG);
      if (GRAD && (D == 3 || cd.keep)) f = sym_run(x.ring_u + i0, on * SG);
    }
    if (LAYER) {
      if (S == SG) {
        p1 = sym_run(a.P + pi0 * D * SG, cd.nsh * D * SG);
        p2 = sym_run(a.P + (pi0 + cd.nsh) * D * SG, cd.ne * NI * D * SG);
      }
      if (PSI) ps = sym_run(a.lpsi + pi0 * PSI, on * PSI);
      if (OM && S == SG) om = sym_run(a.Y + pi0 * SG, on * SG);
    }
    sym_bar_expect(bar, c2.bytes + me.bytes + u.bytes + f.bytes + ps.bytes + om.bytes + p1.bytes + p2.bytes);
    auto go = [&](int at, const SymRun& r) {
      if (r.bytes) sym_bulk(sm + at, r.src, r.bytes, bar);
    };
    go(L.meta, me);
    go(L.u, u);
    go(L.c2, c2);
    if (GRAD) go(L.f, f);
    if (LAYER) {
      go(L.p1, p1);
      go(L.sb, p2);
      go(L.ps, ps);
      go(L.om, om);
    }
    // the update's own reads, to L2 meanwhile
    if (S == SG) sym_prefetch(a.v + i0, on * SG);
    sym_prefetch(a.cf + (size_t)a.N + cd.own, on);
    if (!cd.plain) {
      sym_prefetch(a.cf + cd.own, on);
      sym_prefetch(a.cf + 2 * (size_t)a.N + cd.own, on);
    }
    if (LAYER) sym_prefetch(a.lcs + pi0 * SYM_LCS<D>, on * SYM_LCS<D>);
    if (LAYER && D == 3) {
      sym_prefetch(a.lpsi + pi0 * 4, on * 4);
      sym_prefetch(a.lpsi3 + pi0 * 2, on * 2);
    }
    if (LAYER && D == 3 && S == SG) sym_prefetch(a.Y + pi0 * SG, on * SG);
    // and the ranges of the chunk a wave of CTAs further on
    const int nc = chunk + a.wave;
    if (!RUN && nc >= (LAYER ? a.nch0 : 0) && nc < (LAYER ? a.nch : a.nch0)) {
      const SymDesc nx = sym_desc(a, nc);
      const int nn = nx.nsh + nx.ne * NI;
      sym_prefetch(reinterpret_cast<const float*>(a.smeta) + nx.meta, nx.meta_n);
      sym_prefetch(reinterpret_cast<const float*>(a.halo) + nx.hp, nx.hn);
      sym_prefetch(a.c2 + nx.own, nn);
      if (S == SG) {
        sym_prefetch(x.u + (size_t)nx.own * S, nn * SG);
        if (GRAD) sym_prefetch(x.ring_u + (size_t)nx.own * S, nn * SG);
        if (LAYER) sym_prefetch(a.P + (size_t)(nx.own - a.p_own) * D * SG, nn * D * SG);
      }
    }
  }
  float* us = sm + L.u + sym_shift(x.u + i0);
  float* fs = sm + L.f + (GRAD ? sym_shift(x.ring_u + i0) : 0);
  float* cs = sm + L.c2 + sym_shift(a.c2 + cd.own);
  float *ps = sm + L.ps, *om = sm + L.om, *p1 = sm + L.p1, *p2 = sm + L.sb;
  if (LAYER) {
    if (PSI) ps += sym_shift(a.lpsi + pi0 * PSI);
    if (OM) om += sym_shift(a.Y + pi0 * S + s0);
    p1 += sym_shift(a.P + (pi0 * S + s0) * D);
    p2 += sym_shift(a.P + ((pi0 + cd.nsh) * S + s0) * D);
  }
  if (S != SG) {  // the group's shots are a part of each DoF's run
    for (int l = tid; l < on; l += NT) {
      const size_t dof = (size_t)(cd.own + l);
      sym_cp<4 * SG>(us + l * SG, x.u + dof * S + s0);
      if (GRAD && (D == 3 || cd.keep)) sym_cp<4 * SG>(fs + l * SG, x.ring_u + dof * S + s0);
      if (LAYER)
#pragma unroll
        for (int k = 0; k < D; ++k)
          sym_cp<4 * SG>((l < cd.nsh ? p1 + l * D * SG : p2 + (l - cd.nsh) * D * SG) + k * SG,
                         a.P + ((pi0 + l) * D + k) * S + s0);
      if (OM) sym_cp<4 * SG>(om + l * SG, a.Y + (pi0 + l) * S + s0);
      if (l % (32 / SG) == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.v + dof * S + s0));
    }
  }
  for (int h = tid; h < cd.hn; h += NT) {
    const int id = __ldg(a.halo + cd.hp + h), l = on + SYM_GAP + h;
    reinterpret_cast<int*>(sm + L.ids)[h] = id;
    sym_cp_live<4 * SG, RUN>(us + l * SG, x.u + (size_t)id * S + s0);
    if (GRAD && (D == 3 || cd.keep)) sym_cp<4 * SG>(fs + l * SG, x.ring_u + (size_t)id * S + s0);
    sym_cp<4>(cs + l, a.c2 + id);
    if (LAYER) {
      const size_t pi = (size_t)(id - a.p_halo);
#pragma unroll
      for (int k = 0; k < D; ++k) sym_cp_live<4 * SG, RUN>(p1 + ((cd.nsh + SYM_GAP + h) * D + k) * SG, a.P + (pi * D + k) * S + s0);
      if (PSI) sym_cp<4 * (PSI ? PSI : 1)>(ps + l * PSI, a.lpsi + pi * PSI);
      if (OM) sym_cp_live<4 * SG, RUN>(om + l * SG, a.Y + pi * S + s0);
    }
  }
}

// Sum over the incidence list of a shared DoF of the table t ([node][element][shot]).
template <int SG>
__device__ __forceinline__ Lanes<SG> sym_sum(const float* t, const uint16_t* ge, int b, int e) {
  Lanes<SG> y = lanes_ld<SG>(t + (int)ge[b] * SG);
  for (int i = b + 1; i < e; ++i) lanes_acc<SG>(y, lanes_ld<SG>(t + (int)ge[i] * SG));
  return y;
}

// The update's reads of a round of owned DoFs: increments and coefficients.
template <int SG, int B>
struct SymRound {
  Lanes<SG> v[B];
  float c1[B], c2[B], c3[B];
  __device__ __forceinline__ void load(const StepArgs& a, const SymDesc& cd, int on, int s0, int l0, int nt) {
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const int l = l0 + k * nt;
      if (l < on) {
        const size_t dof = (size_t)(cd.own + l);
        v[k] = lanes_ld<SG>(a.v + dof * a.S + s0);
        c2[k] = __ldg(a.cf + (size_t)a.N + dof);
        c1[k] = cd.plain ? 1.f : __ldg(a.cf + dof);
        c3[k] = cd.plain ? 0.f : __ldg(a.cf + 2 * (size_t)a.N + dof);
      }
    }
  }
};

// Phase 3 of one chunk (after a barrier); cur: its first round's reads, issued before the barrier.
// v' = c1 v - c2 y - c3 u, u' = u + v'. chk collects 0 * u', which stays zero while every value is
// finite.
template <int D, int NN, int NS, int MODE, bool LAYER, int SG, bool RUN, int B>
__device__ __forceinline__ void sym_finish(const StepArgs& a, const SymStep& x, const SymDesc& cd, const SymSmem& L,
                                           const float* sm, int s0, int tid, SymRound<SG, B>& cur, float& chk) {
  constexpr int PE = SYM_PE, NI = NN - NS, NT = SymMap<SG, RUN>::NT;
  constexpr bool GRAD = MODE == 2;
  const int S = a.S, nb = cd.ne * NI, on = cd.nsh + nb;
  const uint16_t* ge = reinterpret_cast<const uint16_t*>(sm + L.meta) + NS * PE;
  const uint16_t* gp = ge + NS * PE;
  const int* ids = reinterpret_cast<const int*>(sm + L.ids);
  const float* us = sm + L.u + sym_shift(x.u + (size_t)cd.own * S + s0);
  for (int l0 = tid; l0 < on; l0 += B * NT) {
    SymRound<SG, B> nxt;
    nxt.load(a, cd, on, s0, l0 + B * NT, NT);
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const int l = l0 + k * NT;
      if (l < on) {
        const Lanes<SG> y = l < cd.nsh ? sym_sum<SG>(sm + L.ys, ge, gp[l], gp[l + 1]) : lanes_ld<SG>(sm + L.yb + (l - cd.nsh) * SG);
        Lanes<SG> un = lanes_ld<SG>(us + l * SG), vn = cur.v[k];
        if (!cd.plain) vn = lanes_fma<SG>(-cur.c3[k], un, lanes_mul<SG>(cur.c1[k], vn));
        vn = lanes_fma<SG>(-cur.c2[k], y, vn);
        if constexpr (LAYER && D == 3) {  // the omega state
          const size_t pi = (size_t)(cd.own + l - a.p_own);
          const float* lc = a.lcs + pi * 12;
          float* Y = a.Y + pi * S + s0;
          const Lanes<SG> Yo = lanes_ld<SG>(Y);
          if constexpr (MODE == 0) {
            vn = lanes_fma<SG>(-__ldg(lc + 3), Yo, vn);
            lanes_st<SG>(Y, lanes_fma<SG>(a.dt, un, Yo));
          } else {
            const Lanes<SG> yw = l < cd.nsh ? sym_sum<SG>(sm + L.ws, ge, gp[l], gp[l + 1]) : lanes_ld<SG>(sm + L.wb + (l - cd.nsh) * SG);
            vn = lanes_fma<SG>(__ldg(lc + 8), Yo, vn);
            lanes_st<SG>(Y, lanes_fma<SG>(__ldg(lc + 7), yw, lanes_fma<SG>(-__ldg(lc + 9), un, Yo)));
          }
        }
        lanes_acc<SG>(un, vn);
#pragma unroll
        for (int j = 0; j < SG; ++j) chk = fmaf(0.f, un.x[j], chk);
        const size_t gi = (size_t)(cd.own + l) * S + s0;
        lanes_st<SG>(a.v + gi, vn);
        lanes_st<SG>(x.u_out + gi, un);
      }
    }
    cur = nxt;
  }
  for (int h = tid; h < cd.hn; h += NT) {
    const int l = cd.nsh + h;
    lanes_add<SG>(a.r + (size_t)(ids[h] - a.N_own) * S + s0, sym_sum<SG>(sm + L.ys, ge, gp[l], gp[l + 1]));
  }
  if constexpr (LAYER) {  // the layer auxiliaries: P' = e1 P - e2 s
    const size_t pi0 = (size_t)(cd.own - a.p_own);
    const float* sb = sm + L.sb + sym_shift(a.P + ((pi0 + cd.nsh) * S + s0) * D);
    constexpr int LC = SYM_LCS<D>, E2 = D == 3 ? 4 : MODE == 0 ? 2 : 4;  // e1 first
    for (int l0 = tid; l0 < on; l0 += 2 * NT) {
      Lanes<SG> P[2][D];
      float e[2][2 * D];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int l = l0 + k * NT;
        if (l < on) {
#pragma unroll
          for (int d = 0; d < D; ++d) {
            P[k][d] = lanes_ld<SG>(a.P + ((pi0 + l) * D + d) * S + s0);
            e[k][d] = __ldg(a.lcs + (pi0 + l) * LC + d);
            e[k][D + d] = __ldg(a.lcs + (pi0 + l) * LC + E2 + d);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int l = l0 + k * NT;
        if (l < on) {
          const int b = l < cd.nsh ? gp[l] : 0, f = l < cd.nsh ? gp[l + 1] : 0;
#pragma unroll
          for (int d = 0; d < D; ++d) {
            const Lanes<SG> s = l < cd.nsh ? sym_sum<SG>(sm + L.ss + d * NS * PE * SG, ge, b, f)
                                           : lanes_ld<SG>(sb + ((l - cd.nsh) * D + d) * SG);
            lanes_st<SG>(a.P + ((pi0 + l) * D + d) * S + s0,
                         lanes_fma<SG>(-e[k][D + d], s, lanes_mul<SG>(e[k][d], P[k][d])));
          }
        }
      }
    }
    for (int h = tid; h < cd.hn; h += NT) {
      const int b = gp[cd.nsh + h], e = gp[cd.nsh + h + 1];
      const size_t pi = (size_t)(ids[h] - a.p_halo);
#pragma unroll
      for (int d = 0; d < D; ++d)
        lanes_add<SG>(a.Pacc + (pi * D + d) * S + s0, sym_sum<SG>(sm + L.ss + d * NS * PE * SG, ge, b, e));
      if constexpr (D == 3 && MODE != 0) lanes_add<SG>(a.Yacc + pi * S + s0, sym_sum<SG>(sm + L.ws, ge, b, e));
    }
  }
  if (GRAD && (D == 3 || cd.keep)) {  // 2 c of the integrand here, once per DoF
    auto put = [&](int dof, const Lanes<SG>& g) {
      const float c = 2.f * __ldg(a.cvel + dof);
      if (a.grad_lanes) {  // one segment accumulator per shot, [S][N]
#pragma unroll
        for (int k = 0; k < SG; ++k) atomicAdd(a.gseg + (size_t)(s0 + k) * a.N + dof, c * g.x[k]);
      } else {  // summed over the shots, [N]
        float t = g.x[0];
#pragma unroll
        for (int k = 1; k < SG; ++k) t += g.x[k];
        atomicAdd(a.gseg + dof, c * t);
      }
    };
    for (int l = tid; l < cd.nsh; l += NT) put(cd.own + l, sym_sum<SG>(sm + L.gs, ge, gp[l], gp[l + 1]));
    for (int l = tid; l < nb; l += NT) put(cd.own + cd.nsh + l, lanes_ld<SG>(sm + L.gb + l * SG));
    for (int h = tid; h < cd.hn; h += NT) put(ids[h], sym_sum<SG>(sm + L.gs, ge, gp[cd.nsh + h], gp[cd.nsh + h + 1]));
  }
}

// Sources and receivers of a chunk (between the element phase and the update, each after a barrier;
// few chunks have any). Their elements' nodal values are still in the table, their sums in the
// threads' places. All threads share the work: one takes a receiver's record of one shot, or a
// node's sum over an element's receivers. (Done by the element's own thread, receiver by receiver,
// this was the longest chain of a step wherever receivers crowd: 4 us with three in an element.)
template <int D, int NN, int NS, int MODE, int SG, bool RUN>
__device__ __forceinline__ void sym_inject(const StepArgs& a, const SymStep& x, const SymDesc& cd, const SymSmem& L,
                                           float* sm, int s0, int tid, int b, int e) {
  constexpr int PE = SYM_PE, NI = NN - NS, NT = SymMap<SG, RUN>::NT;
  const uint16_t* lq = reinterpret_cast<const uint16_t*>(sm + L.meta);
  const float* us = sm + L.u + sym_shift(x.u + (size_t)cd.own * a.S + s0);
  auto place = [&](int q, int el) {
    return sm + (q < NS ? L.ys + (c_slot[q] * PE + el) * SG : L.yb + (el * NI + q - NS) * SG);
  };
  if constexpr (MODE == 0) {
    if (a.rec != nullptr) {
      const int r0 = __ldg(a.rslot_ptr + b), n = (__ldg(a.rslot_ptr + e) - r0) * SG;
      for (int t = tid; t < n; t += NT) {
        const int r = r0 + t / SG, k = t % SG, el = __ldg(a.rslot_elem + r) - cd.e0;
        float acc = 0.f;
#pragma unroll 8
        for (int q = 0; q < NN; ++q) {
          const int l = q < NS ? (int)lq[c_slot[q] * PE + el] : cd.nsh + el * NI + q - NS;
          acc = fmaf(__ldg(a.rslot_phi + (size_t)r * NN + q), us[l * SG + k], acc);
        }
        a.rec[((size_t)(s0 + k) * (a.nt + 1) + x.n) * a.R + __ldg(a.rslot_rec + r)] = acc;
      }
    }
    for (int k = 0; k < SG; ++k) {
      const int el = __ldg(a.src_elem + s0 + k) - cd.e0;
      if (el < 0 || el >= cd.ne) continue;
      const float wv = __ldg(a.wavelet + (size_t)(s0 + k) * a.nt + x.n);
      for (int q = tid; q < NN; q += NT) place(q, el)[k] -= wv * __ldg(a.src_phi + (size_t)(s0 + k) * NN + q);
    }
  } else {
    for (int t = tid; t < (e - b) * NN * SG; t += NT) {
      const int k = t % SG, q = t / SG % NN, slot = b + t / (SG * NN);
      const int rb = __ldg(a.rslot_ptr + slot), re = __ldg(a.rslot_ptr + slot + 1);
      if (rb == re) continue;
      const float* res = a.resid + ((size_t)(s0 + k) * (a.nt + 1) + x.n) * a.R;
      float acc = 0.f;
#pragma unroll 4
      for (int r = rb; r < re; ++r) acc = fmaf(__ldg(res + __ldg(a.rslot_rec + r)), __ldg(a.rslot_phi + (size_t)r * NN + q), acc);
      place(q, __ldg(a.rslot_elem + rb) - cd.e0)[k] += acc;
    }
  }
}

// One orbit of kind K (first slot qb, coefficients at `at`): derivatives, node(q, v, r, t) for each
// node, divergence (of the fluxes that node leaves in r, t; not for a field that is only read).
template <class V, int NN, bool DIV, char K, class F>
__device__ __forceinline__ void sym_tri_orbit(int qb, int at, const TriCoef<V, NN>& U, TriCoef<V, NN>& Y, F node) {
  constexpr int SIDES = K == 'X' ? 2 : 1, NV = K == 'C' ? 1 : 3;
  V r[2][3], t[2][3];
  tri_grad<V, NN, K>(at, U, r, t);
#pragma unroll
  for (int k = 0; k < SIDES; ++k)
#pragma unroll
    for (int v = 0; v < NV; ++v) node(qb + TriSym<NN>::place(K, v, k), v, r[k][v], t[k][v]);
  if constexpr (DIV) tri_div<V, NN, K>(at, r, t, Y);
}
// The element phase's walk over the orbits of a triangle. KMV5's like orbits share their code (its
// seven orbits unrolled are some 3,000 instructions, which miss the instruction caches).
template <class V, int NN, bool DIV, int O, class F>
__device__ __forceinline__ void sym_tri_orbits(const TriCoef<V, NN>& U, TriCoef<V, NN>& Y, F node) {
  using T = TriSym<NN>;
  if constexpr (T::ROLL) {
#pragma unroll 1
    for (int k = 0; k < T::NX; ++k) sym_tri_orbit<V, NN, DIV, 'X'>(T::roll_x(k), k * T::XTAB, U, Y, node);
#pragma unroll 1
    for (int k = 0; k < T::NT; ++k) sym_tri_orbit<V, NN, DIV, 'T'>(T::roll_t(k), T::NX * T::XTAB + k * T::TTAB, U, Y, node);
  } else if constexpr (O < T::NO) {
    constexpr int QB = T::base(O), AT = T::tab(O);
    sym_tri_orbit<V, NN, DIV, T::kind(O)>(QB, AT, U, Y, node);
    sym_tri_orbits<V, NN, DIV, O + 1>(U, Y, node);
  }
}

// One step of a triangle chunk. MODE: 0 forward, 1 adjoint, 2 adjoint with the gradient integrand.
template <int NN, int NS, int MODE, bool LAYER, int SG, bool RUN>
__device__ __forceinline__ bool sym_tri_body(const StepArgs& a, const SymStep& x, float* sm, int chunk, int s0) {
  using M = SymMap<SG, RUN>;
  using V = typename M::V;
  constexpr int NI = NN - NS, PE = SYM_PE;
  constexpr bool ADJ = MODE != 0, GRAD = MODE == 2;
  const int tid = threadIdx.x, S = a.S;
  const SymSmem L = sym_smem<2, NN, NS, SG, MODE, LAYER>(a.T_max, a.SH_max, a.H_max);
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm);
  if (!RUN && tid == 0) sym_bar_init(bar);  // (the thread that issues the barrier's copies)
  const SymDesc cd = sym_desc(a, chunk);
  sym_load<2, NN, NS, SG, MODE, LAYER, RUN>(a, x, cd, L, sm, bar, chunk, s0, tid);
  if (!RUN) __syncthreads();  // the barrier is set up before anyone asks it
  const int el = tid / M::PER, ln = tid % M::PER * M::LANES;  // element, first shot of the group
  const bool act = el < cd.ne;
  const int ee = act ? el : 0, e = cd.e0 + ee, nb = cd.ne * NI;
  const int bub = cd.nsh + ee * NI;
  // a damped chunk's gradient is masked: a plain adjoint step there. (Marine mesh: 87 -> 82 ms a
  // gradient. Tetrahedra lose more to the second path's registers: 22.9 -> 23.8 ms, KMV2.)
  const bool grad = GRAD && (!LAYER || cd.keep);
  const int in0 = __ldg(a.cslot + chunk), in1 = __ldg(a.cslot + chunk + 1);  // sources' and receivers' elements
  const size_t i0 = (size_t)cd.own * S + s0, pi0 = (size_t)(cd.own - a.p_own);
  const uint16_t* lq = reinterpret_cast<const uint16_t*>(sm + L.meta) + ee;
  float H0[3], A0[2][2];
#pragma unroll
  for (int c = 0; c < 3; ++c) H0[c] = __ldg(a.geo + (size_t)c * a.Es + e);
  if constexpr (LAYER)
#pragma unroll
    for (int c = 0; c < 4; ++c) A0[c >> 1][c & 1] = __ldg(a.lgeo + (size_t)c * (a.E - a.E0) + (e - a.E0));
  sym_cp_wait();
  const bool ok = sym_bar_wait(bar, x.parity, a.wait_limit);
  if (__syncthreads_or(!ok)) {  // a copy did not arrive: report it and leave the fields alone
    sym_bar_wait(bar, x.parity, WAIT_POLLS);  // (no CTA ends before its copies)
    if (tid == 0) atomicOr(a.status, 2);
    return false;
  }

  // ---- elements --------------------------------------------------------------------------
  const float* us = sm + L.u + sym_shift(x.u + i0) + ln;
  const float* cs = sm + L.c2 + sym_shift(a.c2 + cd.own);
  // a thread's own places for node q: the sums' ([node][element][shot], bubbles in DoF order), ...
  const int ps = el * SG + ln, pb = el * NI * SG + ln;
  auto at = [&](int q) { return q < NS ? (int)lq[q * PE] : bub + (q - NS); };
  auto ld = [&](const float* p) { return *reinterpret_cast<const V*>(p); };
  auto st = [&](float* p, V v) { *reinterpret_cast<V*>(p) = v; };
  auto own = [&](int s, int b, int q) { return sm + (q < NS ? s + ps + q * PE * SG : b + pb + (q - NS) * SG); };
  TriCoef<V, NN> Y;
  if (act) {
    TriCoef<V, NN> U;
    if (GRAD && grad) {  // the forward field's derivatives wait in places that are filled later
      const float* fs = sm + L.f + sym_shift(x.ring_u + i0) + ln;
      tri_analyse<V, NN>(U, [&](int q) { return ld(fs + at(q) * SG); });
      sym_tri_orbits<V, NN, false, 0>(U, Y, [&](int q, int, V& r, V& t) {
        st(own(L.gs, L.gb, q), r);
        st(own(L.ys, L.yb, q), t);
      });
      asm volatile("" ::: "memory");  // (keeps the two passes' registers apart)
    }
    float H[3][3], A[3][2][2];  // A: rows (radial, tangential) of |J| J^-1 in the three frames
    tri_metric(H0[0], H0[1], H0[2], H);
    if constexpr (LAYER) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        tri_frame<0>(A0[0][c], A0[1][c], A[0][0][c], A[0][1][c]);
        tri_frame<1>(A0[0][c], A0[1][c], A[1][0][c], A[1][1][c]);
        tri_frame<2>(A0[0][c], A0[1][c], A[2][0][c], A[2][1][c]);
      }
    }
    const float* p1 = sm + L.p1 + (LAYER ? sym_shift(a.P + (pi0 * S + s0) * 2) : 0) + ln;
    float* p2 = sm + L.sb + (LAYER ? sym_shift(a.P + ((pi0 + cd.nsh) * S + s0) * 2) : 0) + el * NI * 2 * SG + ln;
    const float* psi = sm + L.ps + (LAYER && ADJ ? sym_shift(a.lpsi + pi0) : 0);
    tri_analyse<V, NN>(U, [&](int q) { return ld(us + at(q) * SG); });
    tri_zero(Y);
    // one node: (r, t) in are the field's derivatives in frame v, out the flux
    sym_tri_orbits<V, NN, true, 0>(U, Y, [&](int q, int v, V& r, V& t) {
      const float w = c_w[q];
      const int l = at(q);
      const V wc = dup<V>(w * cs[l]), gr = r, gt = t;
      const V hr = fma2(dup<V>(H[v][0]), gr, mul2(dup<V>(H[v][1]), gt));
      const V ht = fma2(dup<V>(H[v][1]), gr, mul2(dup<V>(H[v][2]), gt));
      r = mul2(wc, hr);
      t = mul2(wc, ht);
      if (GRAD && grad) {  // w (Ghat grad u_dag) . grad u
        float* g = own(L.gs, L.gb, q);
        st(g, mul2(dup<V>(w), fma2(hr, ld(g), mul2(ht, ld(own(L.ys, L.yb, q))))));
      }
      if constexpr (LAYER) {
        const V sx = mul2(dup<V>(w), fma2(dup<V>(A[v][0][0]), gr, mul2(dup<V>(A[v][1][0]), gt)));
        const V sz = mul2(dup<V>(w), fma2(dup<V>(A[v][0][1]), gr, mul2(dup<V>(A[v][1][1]), gt)));
        V px, pz;
        if (q < NS) {
          const float* p = p1 + (l - (l >= cd.nsh ? nb : 0)) * 2 * SG;
          px = ld(p);
          pz = ld(p + SG);
          st(sm + L.ss + ps + q * PE * SG, sx);
          st(sm + L.ss + ps + (NS + q) * PE * SG, sz);
        } else {  // a bubble's P gives way to its layer sums
          float* p = p2 + (q - NS) * 2 * SG;
          px = ld(p);
          pz = ld(p + SG);
          st(p, sx);
          st(p + SG, sz);
        }
        // Psi2 c^2 (adjoint) is opposite in the two directions
        const float wp = ADJ ? w * psi[l] : w;
        const V zz = dup<V>(ADJ ? -wp : wp), xx = dup<V>(wp);
        px = mul2(xx, px);
        pz = mul2(zz, pz);
        r = fma2(dup<V>(A[v][0][0]), px, fma2(dup<V>(A[v][0][1]), pz, r));
        t = fma2(dup<V>(A[v][1][0]), px, fma2(dup<V>(A[v][1][1]), pz, t));
      }
    });
  }
  if (LAYER && !GRAD) __syncthreads();  // every P of a shared DoF has been read
  if (act) {
    tri_gather_back<V, NN>(Y, [&](int q, V y) { st(own(L.ys, L.yb, q), y); });
  }
  // DoFs per thread whose update reads are in flight at a time. More hide more latency and take
  // registers from CTAs: KMV2, one shot (2M triangles, 50 steps): 4.69 ms with four, 3.71 ms with one;
  // KMV4 segments 6.90 and 6.71 ms with four and two; KMV5, one shot, 6.26 and 6.54 ms.
  constexpr int B = NN == 7 ? 1 : NN == 30 && SG == 1 ? 4 : 2;
  SymRound<SG, B> first;
  first.load(a, cd, cd.nsh + nb, s0, tid, M::NT);
  __syncthreads();
  if (in0 < in1) {
    sym_inject<2, NN, NS, MODE, SG, RUN>(a, x, cd, L, sm, s0, tid, in0, in1);
    __syncthreads();
  }

  float chk = 0.f;
  sym_finish<2, NN, NS, MODE, LAYER, SG, RUN, B>(a, x, cd, L, sm, s0, tid, first, chk);
  if (!(chk == 0.f)) atomicOr(a.status, 1);
  return true;
}

// The walk over the orbits of a tetrahedron: derivatives of N fields, node(q, g) for each node with
// g[field][axis], then the divergence of the fluxes that node leaves in g[0] to Y (and of g[1] to
// Y2, if DIV2).
template <class V, int NN, int N, bool DIV2, int O, class F, class G>
__device__ __forceinline__ void sym_tet_orbits(const TetCoef<V, NN>* const (&U)[N], TetCoef<V, NN>& Y,
                                               TetCoef<V, NN>& Y2, F node, G coefs) {
  if constexpr (O < TetSym<NN>::NO) {
    V g[N > 1 || !DIV2 ? N : 2][3][4];
#pragma unroll
    for (int f = 0; f < N; ++f) {
      tet_grad<V, NN, O, 0>(*U[f], g[f][0]);
      tet_grad<V, NN, O, 1>(*U[f], g[f][1]);
      tet_grad<V, NN, O, 2>(*U[f], g[f][2]);
    }
#pragma unroll
    for (int h = 0; h < TetSize<NN, O>::N; ++h) {
      V x[N > 1 || !DIV2 ? N : 2][3];
#pragma unroll
      for (int f = 0; f < N; ++f)
#pragma unroll
        for (int d = 0; d < 3; ++d) x[f][d] = g[f][d][h];
      node(TetSym<NN>::node(O, h), x, [&] { return coefs(TetSym<NN>::node(O, h)); });
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        g[0][d][h] = x[0][d];
        if constexpr (DIV2) g[1][d][h] = x[1][d];
      }
    }
    tet_div<V, NN, O, 0>(g[0][0], Y);
    tet_div<V, NN, O, 1>(g[0][1], Y);
    tet_div<V, NN, O, 2>(g[0][2], Y);
    if constexpr (DIV2) {
      tet_div<V, NN, O, 0>(g[1][0], Y2);
      tet_div<V, NN, O, 1>(g[1][1], Y2);
      tet_div<V, NN, O, 2>(g[1][2], Y2);
    }
    sym_tet_orbits<V, NN, N, DIV2, O + 1>(U, Y, Y2, node, coefs);
  }
}

// A layer DoF's nodal coefficients: Psi2 c^2 of the three directions, Psi3 c^2.
struct LayerPsi {
  float4 a;  // Psi2, then the first of Psi3
  float2 b;
};

// The same walk rolled (KMV3: all orbits are alike; node slots 4 o + h). coefs(q): the layer's
// coefficients of a node, with EARLY those of an orbit before its derivatives. The unrolled code of
// the layer kernels, some 7,000 instructions, does not fit the instruction caches.
template <class V, int N, bool DIV2, bool EARLY, class F, class G>
__device__ __forceinline__ void sym_tet_roll(const TetCoef<V, 32>* const (&U)[N], TetCoef<V, 32>& Y, TetCoef<V, 32>& Y2,
                                             F node, G coefs) {
  constexpr int NG = N > 1 || !DIV2 ? N : 2;
#pragma unroll 1
  for (int o = 0; o < 8; ++o) {
    const float* t = c_sym + o * 96;  // [axis][output][mode] of this orbit
    LayerPsi ps[4];
    if constexpr (EARLY)
#pragma unroll
      for (int h = 0; h < 4; ++h) ps[h] = coefs(4 * o + h);
    V g[NG][3][4];
#pragma unroll
    for (int f = 0; f < N; ++f)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          V s = mul2(dup<V>(t[(d * 4 + z) * 8]), U[f]->at(z ^ (d + 1), 0));
#pragma unroll
          for (int i = 1; i < 8; ++i) s = fma2(dup<V>(t[(d * 4 + z) * 8 + i]), U[f]->at(z ^ (d + 1), i), s);
          g[f][d][z] = s;
        }
        tet_butterfly(g[f][d]);
      }
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      V x[NG][3];
#pragma unroll
      for (int f = 0; f < N; ++f)
#pragma unroll
        for (int d = 0; d < 3; ++d) x[f][d] = g[f][d][h];
      if constexpr (EARLY) node(4 * o + h, x, [&] { return ps[h]; });
      else node(4 * o + h, x, [&] { return coefs(4 * o + h); });
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        g[0][d][h] = x[0][d];
        if constexpr (DIV2) g[1][d][h] = x[1][d];
      }
    }
#pragma unroll
    for (int f = 0; f < 1 + DIV2; ++f) {
      TetCoef<V, 32>& y = f == 0 ? Y : Y2;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        tet_butterfly(g[f][d]);
#pragma unroll
        for (int z = 0; z < 4; ++z)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            y.at(z ^ (d + 1), i) = fma2(dup<V>(t[(d * 4 + z) * 8 + i]), g[f][d][z], y.at(z ^ (d + 1), i));
      }
    }
  }
}

// One step of a tetrahedra chunk. Fields: u; the forward field (gradient steps); omega (forward
// steps in the layer).
template <int NN, int NS, int MODE, bool LAYER, int SG, bool RUN>
__device__ __forceinline__ bool sym_tet_body(const StepArgs& a, const SymStep& x, float* sm, int chunk, int s0) {
  using M = SymMap<SG, RUN>;
  using V = typename M::V;
  constexpr int NI = NN - NS, PE = SYM_PE;
  constexpr bool ADJ = MODE != 0, GRAD = MODE == 2, OM = LAYER && !ADJ, W = LAYER && ADJ;
  constexpr int NF = 1 + (GRAD || OM);
  const int tid = threadIdx.x, S = a.S;
  const SymSmem L = sym_smem<3, NN, NS, SG, MODE, LAYER>(a.T_max, a.SH_max, a.H_max);
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm);
  if (!RUN && tid == 0) sym_bar_init(bar);  // (the thread that issues the barrier's copies)
  const SymDesc cd = sym_desc(a, chunk);
  sym_load<3, NN, NS, SG, MODE, LAYER, RUN>(a, x, cd, L, sm, bar, chunk, s0, tid);
  if (!RUN) __syncthreads();  // the barrier is set up before anyone asks it
  const int el = tid / M::PER, ln = tid % M::PER * M::LANES;  // element, first shot of the group
  const bool act = el < cd.ne;
  const int ee = act ? el : 0, e = cd.e0 + ee, nb = cd.ne * NI;
  const int bub = cd.nsh + ee * NI;
  const int in0 = __ldg(a.cslot + chunk), in1 = __ldg(a.cslot + chunk + 1);  // sources' and receivers' elements
  const size_t i0 = (size_t)cd.own * S + s0, pi0 = (size_t)(cd.own - a.p_own);
  const uint16_t* lq = reinterpret_cast<const uint16_t*>(sm + L.meta) + ee;
  float G[6], A[3][3];  // |J| J^-1 J^-T and |J| J^-1 in the cube's axes
#pragma unroll
  for (int c = 0; c < 6; ++c) G[c] = __ldg(a.geo + (size_t)c * a.Es + e);
  if constexpr (LAYER)
#pragma unroll
    for (int c = 0; c < 9; ++c) A[c / 3][c % 3] = __ldg(a.lgeo + (size_t)c * (a.E - a.E0) + (e - a.E0));
  sym_cp_wait();
  const bool ok = sym_bar_wait(bar, x.parity, a.wait_limit);
  if (__syncthreads_or(!ok)) {  // a copy did not arrive: report it and leave the fields alone
    sym_bar_wait(bar, x.parity, WAIT_POLLS);  // (no CTA ends before its copies)
    if (tid == 0) atomicOr(a.status, 2);
    return false;
  }

  // ---- elements --------------------------------------------------------------------------
  const float* us = sm + L.u + sym_shift(x.u + i0) + ln;
  const float* cs = sm + L.c2 + sym_shift(a.c2 + cd.own);
  const int ps = el * SG + ln, pb = el * NI * SG + ln;  // a thread's own places (see sym_tri_body)
  // q: a node's slot (sym_slot_node: the local node, at KMV3 orbit by orbit)
  constexpr bool ROLL = NN == 32, EARLY = LAYER;
  auto bi = [](int q) { return ROLL ? NN - 1 - q : q - NS; };  // a bubble's place in its element
  auto at = [&](int q) { return q < NS ? (int)lq[q * PE] : bub + bi(q); };
  auto ld = [&](const float* p) { return *reinterpret_cast<const V*>(p); };
  auto st = [&](float* p, V v) { *reinterpret_cast<V*>(p) = v; };
  auto own = [&](int s, int b, int q) { return sm + (q < NS ? s + ps + q * PE * SG : b + pb + bi(q) * SG); };
  auto slot_of = [](int q) {  // (q and the loop are compile-time once unrolled)
    int j = 0;
#pragma unroll
    for (int i = 0; i < NN; ++i)
      if (sym_slot_node(3, NN, i) == q) j = i;
    return j;
  };
  TetCoef<V, NN> U, F, Y, Y2;
  if (act) {
    if constexpr (GRAD) {
      const float* fs = sm + L.f + sym_shift(x.ring_u + i0) + ln;
      tet_analyse<V, NN>(F, [&](int q) { return ld(fs + at(slot_of(q)) * SG); });
    }
    if constexpr (OM) {
      const float* om = sm + L.om + sym_shift(a.Y + pi0 * S + s0) + ln;
      tet_analyse<V, NN>(F, [&](int q) { return ld(om + at(slot_of(q)) * SG); });
    }
  }
  if (LAYER && NF == 2) __syncthreads();  // the second field's place is the layer sums' from here
  if (act) {
    const float* p1 = sm + L.p1 + (LAYER ? sym_shift(a.P + (pi0 * S + s0) * 3) : 0) + ln;
    float* p2 = sm + L.sb + (LAYER ? sym_shift(a.P + ((pi0 + cd.nsh) * S + s0) * 3) : 0) + el * NI * 3 * SG + ln;
    const int* ids = reinterpret_cast<const int*>(sm + L.ids);
    const float4* psi = reinterpret_cast<const float4*>(a.lpsi);
    const float2* psi3 = reinterpret_cast<const float2*>(a.lpsi3);
    tet_analyse<V, NN>(U, [&](int q) { return ld(us + at(slot_of(q)) * SG); });
    tet_zero(Y);
    if constexpr (W) tet_zero(Y2);
    // one node: x[0] in are the field's derivatives, out the flux (x[1]: the other field's; out, in
    // the layer's adjoint, the omega row's flux)
    auto coefs = [&](int q) {
      const int l = at(q), on = cd.nsh + nb;
      const int pi = l < on ? (int)pi0 + l : ids[l - on - SYM_GAP] - a.p_halo;
      return LayerPsi{__ldg(psi + pi), __ldg(psi3 + pi)};
    };
    auto node = [&](int q, auto& g, auto layer_psi) {
      const float w = c_w[q];
      const int l = at(q);
      const float c2 = cs[l];
      const V wc = dup<V>(w * c2), g0 = g[0][0], g1 = g[0][1], g2 = g[0][2];
      const V h0 = fma2(dup<V>(G[0]), g0, fma2(dup<V>(G[1]), g1, mul2(dup<V>(G[2]), g2)));
      const V h1 = fma2(dup<V>(G[1]), g0, fma2(dup<V>(G[3]), g1, mul2(dup<V>(G[4]), g2)));
      const V h2 = fma2(dup<V>(G[2]), g0, fma2(dup<V>(G[4]), g1, mul2(dup<V>(G[5]), g2)));
      if constexpr (GRAD)  // w (Ghat grad u_dag) . grad u
        st(own(L.gs, L.gb, q), mul2(dup<V>(w), fma2(h0, g[1][0], fma2(h1, g[1][1], mul2(h2, g[1][2])))));
      V f[3] = {mul2(wc, h0), mul2(wc, h1), mul2(wc, h2)};
      if constexpr (LAYER) {
        // (formed in FP64 and rounded once: Psi2 cancels where two directions are damped)
        const LayerPsi lp = layer_psi();
        const float psi2[3] = {lp.a.x, lp.a.y, lp.a.z}, psi3k[3] = {lp.a.w, lp.b.x, lp.b.y};
        float* p = q < NS ? const_cast<float*>(p1) + (l - (l >= cd.nsh ? nb : 0)) * 3 * SG : p2 + bi(q) * 3 * SG;
        V P[3], Q[3], R[3], s[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          P[k] = ld(p + k * SG);
          s[k] = fma2(dup<V>(A[0][k]), g0, fma2(dup<V>(A[1][k]), g1, mul2(dup<V>(A[2][k]), g2)));
          if constexpr (OM) {  // both gradients, each with its Psi c^2
            const V y = fma2(dup<V>(A[0][k]), g[1][0], fma2(dup<V>(A[1][k]), g[1][1], mul2(dup<V>(A[2][k]), g[1][2])));
            s[k] = fma2(dup<V>(-psi3k[k]), y, mul2(dup<V>(psi2[k]), s[k]));
          }
          s[k] = mul2(dup<V>(w), s[k]);
          Q[k] = ADJ ? mul2(dup<V>(w * psi2[k]), P[k]) : mul2(dup<V>(w), P[k]);
          if constexpr (W) R[k] = mul2(dup<V>(w * psi3k[k]), P[k]);
          if (q < NS) st(sm + L.ss + ps + (k * NS + q) * PE * SG, s[k]);
          else st(p + k * SG, s[k]);  // a bubble's P gives way to its layer sums
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          f[d] = fma2(dup<V>(A[d][0]), Q[0], fma2(dup<V>(A[d][1]), Q[1], fma2(dup<V>(A[d][2]), Q[2], f[d])));
          if constexpr (W) g[1][d] = fma2(dup<V>(A[d][0]), R[0], fma2(dup<V>(A[d][1]), R[1], mul2(dup<V>(A[d][2]), R[2])));
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) g[0][d] = f[d];
    };
    if constexpr (NF == 2) {
      const TetCoef<V, NN>* const fields[2] = {&U, &F};
      if constexpr (ROLL) sym_tet_roll<V, 2, W, EARLY>(fields, Y, Y2, node, coefs);
      else sym_tet_orbits<V, NN, 2, W, 0>(fields, Y, Y2, node, coefs);
    } else {
      const TetCoef<V, NN>* const fields[1] = {&U};
      if constexpr (ROLL) sym_tet_roll<V, 1, W, EARLY>(fields, Y, Y2, node, coefs);
      else sym_tet_orbits<V, NN, 1, W, 0>(fields, Y, Y2, node, coefs);
    }
  }
  if (LAYER) __syncthreads();  // every P of a shared DoF has been read
  if (act) {
    tet_gather_back<V, NN>(Y, [&](int q, V y) { st(own(L.ys, L.yb, slot_of(q)), y); });
    if constexpr (W) tet_gather_back<V, NN>(Y2, [&](int q, V y) { st(own(L.ws, L.wb, slot_of(q)), y); });
  }
  constexpr int B = 2;
  SymRound<SG, B> first;
  first.load(a, cd, cd.nsh + nb, s0, tid, M::NT);
  __syncthreads();
  if (in0 < in1) {
    sym_inject<3, NN, NS, MODE, SG, RUN>(a, x, cd, L, sm, s0, tid, in0, in1);
    __syncthreads();
  }

  float chk = 0.f;
  sym_finish<3, NN, NS, MODE, LAYER, SG, RUN, B>(a, x, cd, L, sm, s0, tid, first, chk);
  if (!(chk == 0.f)) atomicOr(a.status, 1);
  return true;
}

}  // namespace fwi
