// Short-axis propagation kernel, FP32 storage (sm_103a): the moving-grid
// split-operator integrator of mg_kernels.cu specialised to tensor grids whose
// D >= 3 axes all have n = 8, 12 or 16 points (the 8D Henon-Heiles grids of
// Sec. III.C).  mg_short64.cu is its counterpart for FP64 storage.
//
// Same method and same persistent structure as k_propagate: kinetic substeps
// U_T,adpt (eq:T_split_substep_adaptive) and potential substeps U_V,adpt
// (Sec. II.G.1) with the grid centres updated from grid-wide reductions
// (eq:eom_qt_case_III_T, eq:eom_pt_solution_case_III_V), composed as in
// eq:comp_TVT, all in one cooperative launch.  What differs is how a
// transform moves through memory:
//  - A pass transforms a group of up to SHORT_MAXG consecutive axes (mg_short.h),
//    so a full transform of an 8D grid takes 3-4 passes over the state
//    instead of 8.
//  - Chunks are copied between global and shared memory with cp.async (8 B
//    per element), nreg-1 chunks ahead of the one being transformed.
//  - Each thread transforms whole lines held in registers: an n-point DFT of
//    compile-time length (8: radix-8 codelet; 12 = 4 x 3 and 16 = 4 x 4 as two
//    codelet stages with the twiddles in between).
//  - The multipliers of the method are applied per line: A_l (with the 1/N_l
//    of the transform pair) before the forward DFT along l, K_l before the
//    inverse DFT.  Between the stages of one launch the state keeps the
//    demodulation factor of its last kinetic substep, so the next forward
//    pass multiplies by A(p) conj(A(p_old)) instead, and only the last kinetic
//    substep of a launch multiplies by conj(A) after its inverse DFTs.
//  - 12-point lines use the Good-Thomas 4 x 3 factorisation (no twiddles).
//  - Each pass is a separate (non-inlined) function, so that its register
//    allocation does not carry the persistent loop's live values.
//  - The potential phase e^{-i sigma V(x^J)/hbar} (eq:U_V_tensor) is a product
//    of per-axis factors e^{-i sigma f_a(x_a)/hbar} and nearest-neighbour pair
//    factors e^{-i sigma h_a(x_a) g_{a+1}(x_{a+1})/hbar}, each tabulated from
//    an FP64 phase argument once per substep; V = sum_a f_a + sum_a h_a g_{a+1}
//    covers the Henon-Heiles and the diagonal harmonic potentials.  Its
//    gradient, needed for <dV/dq>, is accumulated from tabulated f', g, g', h,
//    h' with the line structure: the terms that do not depend on the line's
//    own coordinate are weighted by the line's norm once per line.
//  - FP32 storage: the sums over points are per-line FP32 sums accumulated
//    per thread with an error-free two-sum, then in FP64 across threads and
//    CTAs, like the FP32 kinetic moments of the general kernel.
#include <cuda_runtime.h>
#include <stdint.h>

#include "mg_device.cuh"
#include "mg_short_dev.cuh"
#include "mg_tc.cuh"

namespace mgk {
namespace {

// Lines along any group axis per chunk (12-point lines: a multiple of 3) and
// threads per CTA (one CTA per SM), for FP32 (prec = 1) and FP64 storage.
constexpr int short_lpc(int prec, int n) { return n % 3 == 0 ? (prec ? 576 : 288) : (prec ? 512 : 256); }
// The tensor-core variant (FP32, 16-point lines) holds 256 lines per chunk,
// one per thread: one round of 128-line GEMMs per warpgroup and axis, and
// room in shared memory for the operands beside three chunk regions.
constexpr int short_lpc_tc(int prec, int n, int tc) { return tc ? 256 : short_lpc(prec, n); }
constexpr int short_threads(int prec, int n) { return n % 3 == 0 ? (prec ? 288 : 384) : 256; }

// ---------------------------------------------------------------------------
// n-point DFT of a line held in registers (natural order in and out)
// ---------------------------------------------------------------------------

// x[k] *= W_n^m (W_n = e^{-2 pi i / n}; conjugate for the inverse); m is a
// compile-time constant after unrolling, quarter turns are exact.
template <bool INV, int N, typename V>
__device__ __forceinline__ V twiddle(V t, int m, const V* __restrict__ tw) {
  if (m == 0) return t;
  if (4 * m == N) return mul_si<INV>(t);
  if (2 * m == N) return V{-t.x, -t.y};
  if (4 * m == 3 * N) return mul_si<!INV>(t);
  return INV ? cmulc(t, tw[m]) : cmul(t, tw[m]);
}

// N = R1 * R2 by one decimation step: input index R2 n1 + n2, output k1 + R1 k2.
template <bool INV, int R1, int R2, typename V>
__device__ __forceinline__ void dft2(V* x, const V* __restrict__ tw) {
  constexpr int N = R1 * R2;
  V y[N];
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) {
    V t[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) t[n1] = x[R2 * n1 + n2];
    Dft<INV, R1, V>::run(t);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) y[n2 * R1 + k1] = twiddle<INV, N>(t[k1], (n2 * k1) % N, tw);
  }
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    V t[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) t[n2] = y[n2 * R1 + k1];
    Dft<INV, R2, V>::run(t);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k1 + R1 * k2] = t[k2];
  }
}

template <bool INV, int N, typename V> struct LineDft;
template <bool INV, typename V> struct LineDft<INV, 8, V> {
  static __device__ __forceinline__ void run(V* x, const V*) { Dft<INV, 8, V>::run(x); }
};
// 12 = 4 x 3 with coprime factors (Good-Thomas prime-factor mapping): input
// index (3 n1 + 4 n2) mod 12, output index k with k mod 4 = k1 and k mod 3 =
// k2, i.e. (9 k1 + 4 k2) mod 12; no twiddle factors between the stages.
template <bool INV, typename V> struct LineDft<INV, 12, V> {
  static __device__ __forceinline__ void run(V* x, const V*) {
    V y[12];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
      V t[4];
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) t[n1] = x[(3 * n1 + 4 * n2) % 12];
      Dft<INV, 4, V>::run(t);
#pragma unroll
      for (int k1 = 0; k1 < 4; ++k1) y[n2 * 4 + k1] = t[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      V t[3];
#pragma unroll
      for (int n2 = 0; n2 < 3; ++n2) t[n2] = y[n2 * 4 + k1];
      Dft<INV, 3, V>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) x[(9 * k1 + 4 * k2) % 12] = t[k2];
    }
  }
};
template <bool INV, typename V> struct LineDft<INV, 16, V> {
  static __device__ __forceinline__ void run(V* x, const V* tw) { dft2<INV, 4, 4>(x, tw); }
};

// ---------------------------------------------------------------------------
// Shared memory of the short-axis kernel
// ---------------------------------------------------------------------------

template <typename V, typename T> struct SSm {
  Smem<V> s;  // tw, tA, tAi, tK, sct, fin, sc, red (the fields the shared helpers use)
  V* F;       // [D*n] per-axis potential factors
  V* Pt;      // [(D-1)*n][n+1] pair factors, rows padded (see load_v_short)
  T* col;     // [5][D*n] f', g, g', h, h'
  V* Tp;      // [ngroups][n][n+1] products of the first two multipliers a group's transform meets
  V* reg[3];
  // tensor-core DFT (ShortPlan::tc != 0): B operands of the group's axes,
  // A operands of the two warpgroups, their MMA barriers, the TMEM address
  unsigned char* tcb;
  unsigned char* tca;
  uint64_t* tcbar;
  unsigned* tctm;
};

// Region k of a chunk ring, chosen with selects (a runtime index into the
// pointer array would put the array in local memory).
template <typename V, typename T> __device__ __forceinline__ V* region(const SSm<V, T>& S, int k) {
  return k == 0 ? S.reg[0] : (k == 1 ? S.reg[1] : S.reg[2]);
}

template <typename V, typename T>
__device__ SSm<V, T> carve_short(const Plan& P, const ShortPlan& SP, unsigned char* base) {
  SSm<V, T> m;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    unsigned char* p = base + off;
    off += (bytes + 15) & ~size_t(15);
    return p;
  };
  const int TT = P.tab_total, n = SP.n;
  Smem<V>& s = m.s;
  s.tw = (V*)take(sizeof(V) * TT);
  s.tA = (V*)take(sizeof(V) * TT);
  s.tAi = (V*)take(sizeof(V) * TT);
  s.tK = (V*)take(sizeof(V) * TT);
  s.tv = nullptr;
  s.tc = nullptr;
  s.te = nullptr;
  // no sincos table (expi_prec uses sincosf for FP32); one 16-value record
  // per warp (block_record)
  s.sct = nullptr;
  s.red = (double*)take(sizeof(double) * 16 * (blockDim.x >> 5));
  s.fin = (double*)take(sizeof(double) * PSTRIDE);
  s.sc = (double*)take(sizeof(double) * SC_N);
  s.mbar = (uint64_t*)take(sizeof(uint64_t) * 3);
  s.mphase = (unsigned*)take(sizeof(unsigned) * 4);
  s.tb = nullptr;
  s.li = nullptr;
  m.F = (V*)take(sizeof(V) * TT);
  m.Pt = (V*)take(sizeof(V) * (P.D - 1) * n * (n + 1));
  m.col = (T*)take(sizeof(T) * 5 * TT);
  m.Tp = (V*)take(sizeof(V) * SP.ngroups * n * (n + 1));
  // chunk regions start on 1024-byte boundaries (the period of the 128-byte
  // swizzle of the tensor copies)
  for (int r = 0; r < 3; ++r) {
    if (r < SP.nreg) {
      const uintptr_t a = (uintptr_t)(base + off);
      off += ((a + 1023) & ~(uintptr_t)1023) - a;
      m.reg[r] = (V*)take(sizeof(V) * SP.region_elems);
    } else {
      m.reg[r] = nullptr;
    }
  }
  s.reg[0] = m.reg[0];
  s.reg[1] = m.reg[1];
  s.reg[2] = m.reg[2];
  m.tcb = m.tca = nullptr;
  m.tcbar = nullptr;
  m.tctm = nullptr;
  if (SP.tc) {
    // operands start on 128-byte boundaries (16 bytes would do)
    const uintptr_t a = (uintptr_t)(base + off);
    off += ((a + 127) & ~(uintptr_t)127) - a;
    const int nsp = SP.tc == TC_TF32X3 ? TcShape<TC_TF32X3>::NSPLIT : TcShape<TC_BF16X3>::NSPLIT;
    const int bb = SP.tc == TC_TF32X3 ? TcShape<TC_TF32X3>::B_BYTES : TcShape<TC_BF16X3>::B_BYTES;
    const int ab = SP.tc == TC_TF32X3 ? TcShape<TC_TF32X3>::A_BYTES : TcShape<TC_BF16X3>::A_BYTES;
    m.tcb = take((size_t)SHORT_TC_MAXG * nsp * bb);
    m.tca = take((size_t)2 * nsp * ab);
    m.tcbar = (uint64_t*)take(2 * sizeof(uint64_t));
    m.tctm = (unsigned*)take(16);
  }
  s.end = off;
  return m;
}

template <typename V>
__device__ void load_demod_short(const Plan& P, const ShortPlan& SP, const Smem<V>& S) {
  for (int e = threadIdx.x; e < P.tab_total; e += blockDim.x) {
    S.tA[e] = from_d2<V>(__ldcg(SP.tabB + e));
    S.tAi[e] = from_d2<V>(__ldcg(SP.tabC + e));
  }
}

// A diagonal multiplier along one axis commutes with the DFTs along the
// others, so the multipliers of the first two axes a group's transform meets
// are applied together in the first axis's loop, and the second axis's loop
// multiplies by nothing: one complex multiply per point saved per group of two
// or more axes, each way.  Forward: the group's last axis, then the one before
// it (tables tA); inverse: its first axis, then the next (tables tK).
// Tp[g][jo][r] = t[a1][r] t[a2][jo], a1 the first axis, a2 the second; rows
// padded to n + 1 entries, so that the lines of a warp (one jo each) read
// different banks.
template <typename V, typename T>
__device__ void build_pairs(const ShortPlan& SP, const SSm<V, T>& S, bool inv) {
  const int n = SP.n, nn = n * n;
  const V* t = inv ? S.s.tK : S.s.tA;
  for (int e = threadIdx.x; e < SP.ngroups * nn; e += blockDim.x) {
    const int gi = e / nn, jo = (e - gi * nn) / n, r = e % n;
    const int g = SP.grp[gi].g, l0 = SP.grp[gi].l0;
    if (g < 2) continue;
    const int a1 = inv ? l0 : l0 + g - 1, a2 = inv ? l0 + 1 : l0 + g - 2;
    S.Tp[(gi * n + jo) * (n + 1) + r] = cmul(t[a1 * n + r], t[a2 * n + jo]);
  }
}

template <typename V, typename T>
__device__ void load_v_short(const Plan& P, const ShortPlan& SP, const Bufs& B, const SSm<V, T>& S) {
  const int TT = P.tab_total, n = SP.n;
  const int nP = SP.pairs ? (P.D - 1) * n * n : 0;
  for (int e = threadIdx.x; e < TT; e += blockDim.x) {
    S.F[e] = from_d2<V>(__ldcg(SP.tabF + e));
#pragma unroll
    for (int k = 0; k < 5; ++k) S.col[k * TT + e] = (T)__ldcg(B.tabV + k * TT + e);
  }
  // rows of the pair factors padded to n + 1 entries: the potential sweep's
  // threads read one row each (their own coordinate on axis D-2) at the same
  // column, which falls into different banks this way (unpadded, the rows of
  // a 16-point FP32 table are 128 bytes apart: one bank for all of them)
  for (int e = threadIdx.x; e < nP; e += blockDim.x) S.Pt[e + e / n] = from_d2<V>(__ldcg(SP.tabP + e));
}

// ---------------------------------------------------------------------------
// Chunk copies
// ---------------------------------------------------------------------------

// Chunk copies, element by element (cp.async in, streaming stores out).  The
// element index advances by the CTA size each iteration; the chunk
// coordinates (row of the group block, plane wt) are carried incrementally,
// without a division per element.  Element (wt, row) sits at shared index
// wt * PS + row + row / N (rows padded to N + 1 per last-axis line).
template <int N, bool STORE, typename V>
__device__ __forceinline__ void chunk_copy(const GroupPlan& G, V* __restrict__ gmem, int64_t c, V* reg) {
  int64_t gb;
  int nwt;
  chunk_geom(G, c, gb, nwt);
  const int nt = blockDim.x;
  if (G.contig) {
    // planes are whole blocks, consecutive in memory: element e = wt * ng + row
    int wt = threadIdx.x / G.ng, row = threadIdx.x - wt * G.ng;
    const int dr = nt % G.ng, dw = nt / G.ng;
    V* g = gmem + gb + threadIdx.x;
    while (wt < nwt) {
      V* s = reg + wt * G.PS + row + row / N;
      if (STORE) __stcs(g, *s);
      else cp_async_el(s, g);
      g += nt;
      row += dr;
      wt += dw;
      if (row >= G.ng) {
        row -= G.ng;
        ++wt;
      }
    }
  } else {
    // rows of WT adjacent elements, `inner` apart: element e = row * WT + wt
    int row = threadIdx.x / G.WT, wt = threadIdx.x - row * G.WT;
    const int dw = nt % G.WT, dr = nt / G.WT;
    V* g = gmem + gb + (int64_t)row * G.inner + wt;
    const int64_t gstep = (int64_t)dr * G.inner + dw, gwrap = G.inner - G.WT;
    while (row < G.ng) {
      V* s = reg + wt * G.PS + row + row / N;
      if (STORE) __stcs(g, *s);
      else cp_async_el(s, g);
      g += gstep;
      row += dr;
      wt += dw;
      if (wt >= G.WT) {
        wt -= G.WT;
        ++row;
        g += gwrap;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// One group pass
// ---------------------------------------------------------------------------

// ---------------------------------------------------------------------------
// TMA tensor copies of whole chunks (FP32 storage, 16-point axes)
// ---------------------------------------------------------------------------

__device__ __forceinline__ void tma_load(const void* tm, int rank, void* dst, uint64_t* bar, const int* c) {
  const unsigned d = smem_u32(dst), b = smem_u32(bar);
  if (rank == 2)
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(d), "l"(tm), "r"(c[0]), "r"(c[1]), "r"(b) : "memory");
  else if (rank == 3)
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(d), "l"(tm), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(b) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(d), "l"(tm), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]), "r"(b) : "memory");
}
__device__ __forceinline__ void tma_store(const void* tm, int rank, const void* src, const int* c) {
  const unsigned s = smem_u32(src);
  if (rank == 2)
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(tm), "r"(c[0]), "r"(c[1]), "r"(s) : "memory");
  else if (rank == 3)
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                 ::"l"(tm), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(s) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];"
                 ::"l"(tm), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]), "r"(s) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

// One chunk by tensor copies (issued by one thread).  Group 0: one box of WT
// whole 16x16x16 blocks.  Strided groups: WT / WP boxes of WP adjacent values of
// the trailing index, each landing as its own plane [row][w] of ng x WP.
// `store` = false: load into `reg`, completing on `bar`; true: store `reg`.
template <typename V>
__device__ __forceinline__ void tma_chunk(const ShortPlan& SP, const GroupPlan& G, int gi, int64_t c, V* reg,
                                          uint64_t* bar, bool store) {
  const void* tm = &SP.tmap[gi];
  const int rank = SP.trank[gi];
  int cc[5] = {0, 0, 0, 0, 0};
  if (gi == 0) {
    cc[3] = (int)(c * G.WT);
    if (store) {
      tma_store(tm, rank, reg, cc);
    } else {
      mbar_expect_tx(bar, (unsigned)(G.WT * G.ng * sizeof(V)));
      tma_load(tm, rank, reg, bar, cc);
    }
    return;
  }
  const int WP = G.WT < 256 ? G.WT : 256;
  const int64_t o = c / G.nb, b = c - o * G.nb;
  if (G.l0 > 0) cc[rank - 1] = (int)o;
  if (!store) mbar_expect_tx(bar, (unsigned)(G.WT * G.ng * sizeof(V)));
  for (int p = 0; p * WP < G.WT; ++p) {
    cc[0] = (int)(b * G.WT + p * WP);
    V* dst = reg + p * G.ng * WP;
    if (store) tma_store(tm, rank, dst, cc);
    else tma_load(tm, rank, dst, bar, cc);
  }
}

// ---------------------------------------------------------------------------
// One group pass
// ---------------------------------------------------------------------------

// Shared-memory element of point r of line (wt, hi, lo) along group axis k in
// the 128-byte-swizzled layout of a 16x16x16 block (TMA copies of group 0):
// row R (one last-axis line, 128 bytes), word w, 16-byte chunk w/2 stored at
// chunk (w/2) ^ (R mod 8).
__device__ __forceinline__ int swz(int R, int w) { return R * 16 + ((((w >> 1) ^ R) & 7) << 1) + (w & 1); }

// One pass over the state for group gi.  MODE: SM_NONE (transforms only),
// SM_KIN (forward; kinetic moments on the lines along axis 0), SM_V (inverse;
// potential phase and moments on the lines along the last axis), SM_VONLY
// (potential substep alone).  POST: apply the final conj(A) (inverse passes of
// a launch's last kinetic substep).  TMA: chunks move by tensor copies (FP32,
// 16-point axes; group 0 swizzled, other groups [plane][row][w]); else by
// cp.async into the padded plane layout.
// TCM: the line DFTs run on the tensor cores (mg_tc.cuh; FP32, 16-point
// lines, TMA copies only), with the lines' pre- and post-multipliers folded
// into the DFT matrix; TC_NONE: register DFTs.
template <typename T, int N, bool INV, int MODE, bool POST, bool TMA, int TCM>
__device__ __noinline__ void short_pass(const Plan& P, const ShortPlan& SP, const Bufs& B,
                                       const SSm<typename VT<T>::v, T>& Sref, int gi, int slot) {
  constexpr int mode = MODE;
  using V = typename VT<T>::v;
  // local copies: read through references, the plan (a kernel parameter) and
  // the shared-memory pointers would be reloaded from memory in every loop
  const GroupPlan G = SP.grp[gi];
  const SSm<V, T> S = Sref;
  const int D = P.D, g = G.g, l0 = G.l0;
  const int TT = P.tab_total;
  const int pairs = SP.pairs;
  V* psi = (V*)B.psi;
  const V* tw = S.s.tw;  // forward twiddles of axis 0 (all axes have n points)
  const int nreg = SP.nreg;
  const int64_t mine = blockIdx.x < G.nchunks ? (G.nchunks - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  // layouts: 0 padded planes (cp.async), 1 swizzled blocks, 2 [plane][row][w]
  const int lay = TMA ? (gi == 0 ? 1 : 2) : 0;
  const int WP = lay == 2 ? (G.WT < 256 ? G.WT : 256) : 1;
  unsigned parity = TMA ? *S.s.mphase : 0u;
  LineAcc<T> acc;
  acc.zero();
  // the potential sweep's gradient components of axes D-2 and D-1 (slots 0,
  // 1), whose index is known only at run time: folded into acc once per pass
  LineAcc<T> accv;
  accv.zero();
  unsigned tmem = 0, tcpar = 0;
  if constexpr (TCM != TC_NONE && MODE != SM_VONLY) {
    static_assert(sizeof(T) == 4 && N == 16 && TMA, "tensor-core DFTs: FP32, 16-point lines, TMA copies");
    using TS = TcShape<TCM>;
    // DFT matrices of the group's axes with their multipliers folded in:
    // forward A_l (or the relative demodulation), inverse K_l, and conj(A_l)
    // after the inverse DFT of a launch's last kinetic substep
    for (int k = 0; k < g; ++k) {
      const int a = l0 + k;
      tc_build_b<TCM, INV>(S.tcb + k * TS::NSPLIT * TS::B_BYTES, (INV ? S.s.tK : S.s.tA) + a * N,
                           (INV && POST) ? S.s.tAi + a * N : nullptr);
    }
    if (threadIdx.x == 0) {
      mbar_init(S.tcbar);
      mbar_init(S.tcbar + 1);
      fence_mbar_init();
    }
    fence_proxy_async();  // B operands written by threads, read by the tensor cores
    tc_alloc(S.tctm);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    tmem = *S.tctm;
  }

  // prefetch distance: cp.async copies run nreg - 1 chunks ahead; tensor
  // copies one chunk ahead, so that with three regions the next load never
  // waits for the store issued just before it
  const int pd = TMA ? 1 : nreg - 1;
  for (int s = 0; s < pd; ++s) {
    if (TMA) {
      if (threadIdx.x == 0 && s < mine)
        tma_chunk(SP, G, gi, blockIdx.x + (int64_t)s * gridDim.x, region(S, s), S.s.mbar + s, false);
    } else {
      if (s < mine) chunk_copy<N, false>(G, psi, blockIdx.x + (int64_t)s * gridDim.x, region(S, s));
      cp_commit();
    }
  }
  for (int64_t i = 0; i < mine; ++i) {
    const int ri = (int)(i % nreg);
    {
      const int64_t i2 = i + pd;
      const int r2 = (int)(i2 % nreg);
      if (TMA) {
        if (threadIdx.x == 0 && i2 < mine) {
          // the store that last read region r2 is done with it: with three
          // regions that store was issued two sets ago and the one of the
          // last set may still be reading its own region
          if (nreg == 3) bulk_wait_read1();
          else bulk_wait_read0();
          fence_proxy_async();
          tma_chunk(SP, G, gi, blockIdx.x + i2 * gridDim.x, region(S, r2), S.s.mbar + r2, false);
        }
        wait_chunk(B, S.s.mbar + ri, (parity >> ri) & 1u);
        parity ^= 1u << ri;
      } else {
        if (i2 < mine) chunk_copy<N, false>(G, psi, blockIdx.x + i2 * gridDim.x, region(S, r2));
        cp_commit();
        if (nreg == 3) cp_wait<2>();
        else cp_wait<1>();
        __syncthreads();
      }
    }
    // the chunk, its region, lines and first block / trailing index
    const int64_t c = blockIdx.x + i * gridDim.x;
    V* const reg = region(S, ri);
    int64_t gb;
    int nwt;
    chunk_geom(G, c, gb, nwt);
    const int nl = nwt * ipow<N>(g - 1);  // lines along any group axis
    const unsigned cbase = G.contig ? (unsigned)(c * G.WT) : (unsigned)((c % G.nb) * G.WT);
    const int kend = mode == SM_VONLY ? 0 : g;
    for (int kk = 0; kk < kend; ++kk) {
      // forward: last axis of the group first; inverse: first axis first
      const int k = INV ? kk : g - 1 - kk;
      const int a = l0 + k;
      const bool last = (kk == g - 1);
      const int nlo = ipow<N>(g - 1 - k), nhi = ipow<N>(k);
      const Div16 dlo((unsigned)nlo), dhi((unsigned)nhi), dwp((unsigned)WP);
      const V* pre = (INV ? S.s.tK : S.s.tA) + a * N;
      const V* post = (INV && POST) ? S.s.tAi + a * N : nullptr;
      // multipliers: the pair product (build_pairs) on the group's first axis,
      // none on its second, the axis's own table after that
      const int pm = (g >= 2 && kk < 2) ? kk + 1 : 0;
      const V* tpg = S.Tp + gi * N * (N + 1);
      const Div16 dsec((unsigned)ipow<N>(g >= 2 ? g - 2 : 0));
      // element addressing: linear (base + r * stride) except for the swizzled
      // layout along its last two axes
      const int kind = (lay == 1 && k == g - 1) ? 2 : ((lay == 1 && k == g - 2) ? 1 : 0);
      // tensor-core DFTs: every thread of a warpgroup takes part in every
      // round (one line each, or an empty row)
      const int nrounds = (nl + blockDim.x - 1) / blockDim.x;
      for (int Lset = threadIdx.x, rr = 0; TCM != TC_NONE ? rr < nrounds : Lset < nl; Lset += blockDim.x, ++rr) {
        const bool have = TCM == TC_NONE || Lset < nl;
        const int L = have ? Lset : 0;
        int wt, hi, lo, base = 0, stride = 0;
        if (lay == 2) {
          const int t0 = (int)dwp((unsigned)L), w = L - t0 * WP;
          const int t = (int)dlo((unsigned)t0);
          lo = t0 - t * nlo;
          const int piece = (int)dhi((unsigned)t);
          hi = t - piece * nhi;
          wt = piece * WP + w;
          base = piece * G.ng * WP + (hi * nlo * N + lo) * WP + w;
          stride = nlo * WP;
        } else {
          const int t = (int)dlo((unsigned)L);
          lo = L - t * nlo;
          wt = (int)dhi((unsigned)t);
          hi = t - wt * nhi;
          if (lay == 0) {
            base = wt * G.PS + (k == g - 1 ? hi * (N + 1) : (hi * nlo + lo / N) * (N + 1) + lo % N);
            stride = (k == g - 1) ? 1 : ipow<N>(g - 2 - k) * (N + 1);
          } else if (kind == 0) {  // swizzled, k = 0 of a 3-axis block: rows R = (wt*16 + r)*16 + lo/16
            base = swz((wt * N) * N + (lo >> 4), lo & 15);
            stride = N * N;
          }
        }
        V x[N];
        if (!have) {
#pragma unroll
          for (int r = 0; r < N; ++r) x[r] = V{(T)0, (T)0};
        } else if (kind == 0) {
#pragma unroll
          for (int r = 0; r < N; ++r) x[r] = reg[base + r * stride];
        } else if (kind == 1) {  // rows R = (wt*16 + hi)*16 + r, word lo
          const int rb = (wt * N + hi) * N;
#pragma unroll
          for (int r = 0; r < N; ++r) x[r] = reg[swz(rb + r, lo)];
        } else {  // row R = wt*256 + hi, the whole line: 16-byte pairs
          const int R = wt * N * N + hi;
#pragma unroll
          for (int cp = 0; cp < N / 2; ++cp) {
            const float4 v2 = *reinterpret_cast<const float4*>(reg + swz(R, 2 * cp));
            x[2 * cp] = V{(T)v2.x, (T)v2.y};
            x[2 * cp + 1] = V{(T)v2.z, (T)v2.w};
          }
        }
        if constexpr (TCM != TC_NONE) {
          // the line as row `row` of its warpgroup's A operand; one thread
          // issues the split products, all wait for them and read their row
          using TS = TcShape<TCM>;
          const int wg = threadIdx.x >> 7, row = threadIdx.x & 127;
          unsigned char* ab = S.tca + wg * TS::NSPLIT * TS::A_BYTES;
          tc_stage_line<TCM>(ab, row, reinterpret_cast<const float2*>(x));
          fence_proxy_async();
          __syncthreads();
          // one thread issues both warpgroups' products and one commit (a
          // thread of warp 1: thread 0 issues the chunks' TMA copies)
          if (threadIdx.x == 32) {
            const unsigned char* bk = S.tcb + k * TS::NSPLIT * TS::B_BYTES;
            tc_fence_after();
            tc_issue_products<TCM>(tmem, S.tca, bk);
            tc_issue_products<TCM>(tmem + 32, S.tca + TS::NSPLIT * TS::A_BYTES, bk);
            tc_commit(S.tcbar);
          }
          wait_chunk(B, S.tcbar, tcpar);
          tcpar ^= 1u;
          tc_fence_after();
          float v[32];
          tc_ld32(tmem + ((uint32_t)(32 * ((threadIdx.x >> 5) & 3)) << 16) + wg * 32, v);
          tc_fence_before();
#pragma unroll
          for (int r = 0; r < N; ++r) x[r] = V{(T)v[2 * r], (T)v[2 * r + 1]};
        } else {
          if (pm == 1) {
            // the coordinate of the line along the group's second axis
            const int jo = INV ? (int)dsec((unsigned)lo) : hi % N;
            const V* tp = tpg + jo * (N + 1);
#pragma unroll
            for (int r = 0; r < N; ++r) x[r] = cmul(x[r], tp[r]);
          } else if (pm == 0) {
#pragma unroll
            for (int r = 0; r < N; ++r) x[r] = cmul(x[r], pre[r]);
          }
          LineDft<INV, N, V>::run(x, tw);
          if (post) {
#pragma unroll
            for (int r = 0; r < N; ++r) x[r] = cmul(x[r], post[r]);
          }
        }
        if (!have) continue;
        if (last && mode == SM_KIN) {
          // kinetic moments; the line runs along axis 0 (k = 0, l0 = 0)
          int j[MAXD];
          digits<N>((unsigned)lo, 1, g - 1, j);
          if (!G.contig) digits<N>(cbase + wt, g, D - 1, j);
          T s0 = 0, s1 = 0;
#pragma unroll
          for (int r = 0; r < N; ++r) {
            const T w = x[r].x * x[r].x + x[r].y * x[r].y;
            s0 += w;
            s1 += (T)(r - N / 2) * w;
          }
          acc.add(0, s0);
          acc.add(1, s1);
#pragma unroll
          for (int b = 1; b < MAXD; ++b)
            if (b < D) acc.add(1 + b, (T)(j[b] - N / 2) * s0);
        }
        if (kind == 0) {
#pragma unroll
          for (int r = 0; r < N; ++r) reg[base + r * stride] = x[r];
        } else if (kind == 1) {
          const int rb = (wt * N + hi) * N;
#pragma unroll
          for (int r = 0; r < N; ++r) reg[swz(rb + r, lo)] = x[r];
        } else {
          const int R = wt * N * N + hi;
#pragma unroll
          for (int cp = 0; cp < N / 2; ++cp)
            *reinterpret_cast<float4*>(reg + swz(R, 2 * cp)) =
                make_float4((float)x[2 * cp].x, (float)x[2 * cp].y, (float)x[2 * cp + 1].x, (float)x[2 * cp + 1].y);
        }
      }
      __syncthreads();
    }
    if (mode == SM_V || mode == SM_VONLY) {
      // potential substep on the lines along the last axis (k = g-1, group 0),
      // in a sweep of its own: the transform loop above keeps fewer registers live
      const int nhi = ipow<N>(g - 1);
      const Div16 dhi((unsigned)nhi);
      for (int L = threadIdx.x; L < nl; L += blockDim.x) {
        const int wt = (int)dhi((unsigned)L), hi = L - wt * nhi;
        const int base = wt * G.PS + hi * (N + 1);  // padded layout
        const int R = wt * N * N + hi;              // swizzled layout (3-axis block)
        {
          // potential phase and gradient moments; the line runs along axis D-1
          int j[MAXD];
          if (g >= 2) digits<N>((unsigned)hi, l0, D - 2, j);
          if (l0 > 0) digits<N>(cbase + wt, 0, l0 - 1, j);
          const int jm = pick(j, D - 2), jm2 = pick(j, D - 3 < 0 ? 0 : D - 3);
          const T* cfp = S.col;
          const T* cg = S.col + TT;
          const T* cgp = S.col + 2 * TT;
          const T* ch = S.col + 3 * TT;
          const T* chp = S.col + 4 * TT;
          V lf = S.F[j[0]];
#pragma unroll
          for (int b = 1; b < MAXD - 1; ++b)
            if (b < D - 1) lf = cmul(lf, S.F[b * N + j[b]]);
          const V* prow = nullptr;
          if (pairs) {
#pragma unroll
            for (int b = 0; b < MAXD - 2; ++b)
              if (b < D - 2) lf = cmul(lf, S.Pt[(b * N + j[b]) * (N + 1) + j[b + 1]]);
            prow = S.Pt + ((D - 2) * N + jm) * (N + 1);
          }
          const V* fl = S.F + (D - 1) * N;
          T s0 = 0, sg = 0, sfp = 0, sgp = 0;
          const T* lcg = cg + (D - 1) * N;
          const T* lcfp = cfp + (D - 1) * N;
          const T* lcgp = cgp + (D - 1) * N;
          // one point: its moments and its phase factor (prow already holds
          // the last axis's own factor, build_v_short)
          auto point = [&](int r, V xv) {
            const T w = xv.x * xv.x + xv.y * xv.y;
            s0 += w;
            sg += lcg[r] * w;
            sfp += lcfp[r] * w;
            sgp += lcgp[r] * w;
            return cmul(xv, cmul(lf, prow ? prow[r] : fl[r]));
          };
          if constexpr (TMA) {
            // the whole line in registers (swizzled rows: two points per
            // 16-byte access; 8-byte accesses would put four threads of a
            // warp on each bank), its points independent of one another, the
            // sums over them in two halves
            V xs[N];
#pragma unroll
            for (int cp = 0; cp < N / 2; ++cp) {
              const float4 v2 = *reinterpret_cast<const float4*>(reg + swz(R, 2 * cp));
              xs[2 * cp] = V{(T)v2.x, (T)v2.y};
              xs[2 * cp + 1] = V{(T)v2.z, (T)v2.w};
            }
            T h0 = 0, hg = 0, hfp = 0, hgp = 0;
#pragma unroll
            for (int r = 0; r < N; ++r) {
              const T w = xs[r].x * xs[r].x + xs[r].y * xs[r].y;
              if (r < N / 2) {
                s0 += w;
                sg += lcg[r] * w;
                sfp += lcfp[r] * w;
                sgp += lcgp[r] * w;
              } else {
                h0 += w;
                hg += lcg[r] * w;
                hfp += lcfp[r] * w;
                hgp += lcgp[r] * w;
              }
              xs[r] = cmul(xs[r], cmul(lf, prow ? prow[r] : fl[r]));
            }
            s0 += h0;
            sg += hg;
            sfp += hfp;
            sgp += hgp;
#pragma unroll
            for (int cp = 0; cp < N / 2; ++cp)
              *reinterpret_cast<float4*>(reg + swz(R, 2 * cp)) =
                  make_float4((float)xs[2 * cp].x, (float)xs[2 * cp].y, (float)xs[2 * cp + 1].x,
                              (float)xs[2 * cp + 1].y);
          } else {
#pragma unroll 4
            for (int r = 0; r < N; ++r) reg[base + r] = point(r, reg[base + r]);
          }
          acc.add(0, s0);
          // axes whose derivative does not involve the line's coordinate
#pragma unroll
          for (int b = 0; b < MAXD - 2; ++b)
            if (b < D - 2) {
              T gb2 = cfp[b * N + j[b]] + chp[b * N + j[b]] * cg[(b + 1) * N + j[b + 1]];
              if (b > 0) gb2 += ch[(b - 1) * N + j[b - 1]] * cgp[b * N + j[b]];
              acc.add(1 + b, gb2 * s0);
            }
          {
            const int b = D - 2;  // D >= 3
            const T gb2 = (cfp[b * N + jm] + ch[(b - 1) * N + jm2] * cgp[b * N + jm]) * s0 + chp[b * N + jm] * sg;
            accv.add(0, gb2);
            accv.add(1, sfp + ch[b * N + jm] * sgp);
          }
        }
      }
      __syncthreads();
    }
    if (TMA) {
      // the threads' shared-memory writes before the tensor store reads them
      fence_proxy_async();
      __syncthreads();
      if (threadIdx.x == 0) {
        tma_chunk(SP, G, gi, c, reg, nullptr, true);
        bulk_commit();
      }
    } else {
      chunk_copy<N, true>(G, psi, c, reg);
      __syncthreads();
    }
  }
  if (TMA) {
    if (threadIdx.x == 0) {
      bulk_wait0();  // every store of the pass has reached global memory
      fence_proxy_async_all();
      *S.s.mphase = parity;
    }
    __syncthreads();
  } else {
    cp_wait<0>();
  }
  if constexpr (TCM != TC_NONE && MODE != SM_VONLY) {
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    tc_dealloc(tmem);
  }
  if (MODE == SM_V || MODE == SM_VONLY) {
    acc.merge_rt(D - 1, accv, 0);
    acc.merge_rt(D, accv, 1);
  }
  if (MODE != SM_NONE) block_record<T>(B, S.s.red, slot, acc, D + 1);
}

// ---------------------------------------------------------------------------
// The persistent kernel
// ---------------------------------------------------------------------------

template <typename T, int N, bool TMA, int TCM>
__global__ void __launch_bounds__(short_threads(sizeof(T) == 4, N), 1)
    k_propagate_short(const __grid_constant__ Plan P, const __grid_constant__ Bufs B,
                      const __grid_constant__ Run RN, const __grid_constant__ ShortPlan SP) {
  using V = typename VT<T>::v;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int sflag;
  const SSm<V, T> S = carve_short<V, T>(P, SP, smem_raw);
  const int D = P.D, ng = SP.ngroups;
  if (__ldcg(B.status) != ST_OK) return;
  double* sc = S.s.sc;
  if (threadIdx.x < SC_N) sc[threadIdx.x] = 0.0;
  __syncthreads();
  if (threadIdx.x < D) {
    sc[SC_Q + threadIdx.x] = __ldcg(B.ctrl + threadIdx.x);
    sc[SC_P + threadIdx.x] = __ldcg(B.ctrl + 8 + threadIdx.x);
  }
  load_tables(P, B, S.s, LT_TW);
  if (TMA) init_mbarriers(S.s);
  // the state enters as u: forward multiplier A/N = conj(conj(A)/N), final
  // post-multiplier conj(A), both exact conversions of the context's tables
  for (int e = threadIdx.x; e < P.tab_total; e += blockDim.x) {
    const double2 ai = __ldcg(B.tabAi + e), a = __ldcg(B.tabA + e);
    S.s.tA[e] = from_d2<V>(make_double2(ai.x, -ai.y));
    S.s.tAi[e] = from_d2<V>(make_double2(a.x, -a.y));
  }
  __syncthreads();
  build_pairs(SP, S, false);
  __syncthreads();
  const double* gam = B.gamma;

  if (RN.lead_v) {
    if (threadIdx.x == 0) {
      const double sig = (RN.split == SPLIT_VTV ? 0.5 : 1.0) * gam[0] * RN.dt;
      sc[SC_SIG] = sig;
      sc[SC_SGH] = -sig / P.hbar;
    }
    if (threadIdx.x < D) sc[SC_QN + threadIdx.x] = sc[SC_Q + threadIdx.x];
    __syncthreads();
    build_v_short(P, SP, B, S.s);
    if (!grid_sync(B, &sflag)) return;
    load_v_short(P, SP, B, S);
    __syncthreads();
    short_pass<T, N, false, SM_VONLY, false, TMA, TCM>(P, SP, B, S, 0, 1);
    if (!grid_sync(B, &sflag)) return;
    finish(B, S.s, 1, D + 1);
    centre_after_potential(P, S.s, RN.motion);
    if (sc[SC_ERR] != 0.0) goto done;
    build_demod_short(P, SP, S.s, 0);  // the state is still u
    if (!grid_sync(B, &sflag)) return;
    load_demod_short(P, SP, S.s);
    __syncthreads();
    build_pairs(SP, S, false);
    __syncthreads();
  }

  for (int64_t u = 0; u < RN.n_units; ++u) {
    if (threadIdx.x == 0) {
      double tau, sig;
      bool hasv;
      unit_coeffs(RN, gam, u, tau, sig, hasv);
      sc[SC_TAU] = tau;
      sc[SC_SIG] = sig;
      sc[SC_SGH] = -sig / P.hbar;
      sc[SC_HASV] = hasv ? 1.0 : 0.0;
    }
    __syncthreads();
    const bool hasv = sc[SC_HASV] != 0.0;
    const bool final_unit = (u == RN.n_units - 1);
    // forward transform, group by group from the last axis; kinetic moments
    // in the pass over the group that holds axis 0
    for (int gi = 0; gi < ng; ++gi) {
      if (gi == ng - 1) short_pass<T, N, false, SM_KIN, false, TMA, TCM>(P, SP, B, S, gi, 0);
      else short_pass<T, N, false, SM_NONE, false, TMA, TCM>(P, SP, B, S, gi, 0);
      if (!grid_sync(B, &sflag)) return;
    }
    finish(B, S.s, 0, D + 1);
    centre_after_kinetic(P, S.s, RN.motion);
    if (sc[SC_ERR] != 0.0) goto done;
    build_tables(P, B, S.s, TB_K);
    if (hasv) build_v_short(P, SP, B, S.s);
    if (!grid_sync(B, &sflag)) return;
    load_tables(P, B, S.s, LT_K);
    if (hasv) load_v_short(P, SP, B, S);
    if (threadIdx.x < D) sc[SC_Q + threadIdx.x] = sc[SC_QN + threadIdx.x];
    __syncthreads();
    build_pairs(SP, S, true);
    __syncthreads();
    // inverse transform from the group of axis 0; the potential substep is
    // fused into the pass over the group that holds the last axis
    for (int gi = ng - 1; gi >= 0; --gi) {
      const bool v = (gi == 0 && hasv);
      if (final_unit) {
        if (v) short_pass<T, N, true, SM_V, true, TMA, TCM>(P, SP, B, S, gi, 1);
        else short_pass<T, N, true, SM_NONE, true, TMA, TCM>(P, SP, B, S, gi, 1);
      } else {
        if (v) short_pass<T, N, true, SM_V, false, TMA, TCM>(P, SP, B, S, gi, 1);
        else short_pass<T, N, true, SM_NONE, false, TMA, TCM>(P, SP, B, S, gi, 1);
      }
      if (gi > 0 && !grid_sync(B, &sflag)) return;
    }
    if (hasv) {
      if (!grid_sync(B, &sflag)) return;
      finish(B, S.s, 1, D + 1);
      if (threadIdx.x < D) sc[SC_POLD + threadIdx.x] = sc[SC_P + threadIdx.x];
      __syncthreads();
      centre_after_potential(P, S.s, RN.motion);
      if (sc[SC_ERR] != 0.0) goto done;
      if (!final_unit) {
        build_demod_short(P, SP, S.s, 1);  // the state carries A(p_old)
        if (!grid_sync(B, &sflag)) return;
        load_demod_short(P, SP, S.s);
        __syncthreads();
        build_pairs(SP, S, false);
        __syncthreads();
      }
    }
  }
  // the context's demodulation tables for the final grid centre (read by the
  // next launch and the observables); the kernel's end orders these writes
  build_tables(P, B, S.s, TB_A);
done:
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (int a = 0; a < D; ++a) {
      B.ctrl[a] = sc[SC_Q + a];
      B.ctrl[8 + a] = sc[SC_P + a];
    }
    if (sc[SC_ERR] != 0.0) atomicExch(B.status, (int)sc[SC_ERR]);
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// Host-side lookup (C++ linkage, used by mg_capi.cu)
// ---------------------------------------------------------------------------

// The kernel for axis length n;
// tma: the chunk copies use TMA tensor maps (FP32, n = 16 only).
// tc: the line DFTs on the tensor cores (TC_TF32X3 / TC_BF16X3; FP32, n = 16
// with TMA only).
void* short_kernel(int n, int tma, int tc) {
  if (tma) {
    if (n != 16) return nullptr;
    // The tensor-core rounds inside this persistent kernel are not enabled:
    // their MMA completions did not arrive (the bounded waits ran out) although
    // the same rounds are exact in a kernel of their own (mg_probe_tc_dft16).
    return tc ? nullptr : (void*)k_propagate_short<float, 16, true, TC_NONE>;
  }
  if (tc) return nullptr;
  switch (n) {
    case 8: return (void*)k_propagate_short<float, 8, false, TC_NONE>;
    case 12: return (void*)k_propagate_short<float, 12, false, TC_NONE>;
    case 16: return (void*)k_propagate_short<float, 16, false, TC_NONE>;
  }
  return nullptr;
}

int short_threads_for(int prec, int n) { return short_threads(prec, n); }
int short_lpc_for(int prec, int n, int tc) { return short_lpc_tc(prec, n, tc); }
// Shared-memory bytes of the tensor-core operands (carve_short, with its
// 128-byte alignment): B operands of up to 3 axes, A operands of two
// warpgroups, two mbarriers, the TMEM address slot.
int short_tc_smem_bytes(int tc) {
  if (!tc) return 0;
  const int nsp = tc == TC_TF32X3 ? TcShape<TC_TF32X3>::NSPLIT : TcShape<TC_BF16X3>::NSPLIT;
  const int bb = tc == TC_TF32X3 ? TcShape<TC_TF32X3>::B_BYTES : TcShape<TC_BF16X3>::B_BYTES;
  const int ab = tc == TC_TF32X3 ? TcShape<TC_TF32X3>::A_BYTES : TcShape<TC_BF16X3>::A_BYTES;
  return 128 + SHORT_TC_MAXG * nsp * bb + 2 * nsp * ab + 16 + 16;
}

}  // namespace mgk
