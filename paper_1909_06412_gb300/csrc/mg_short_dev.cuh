// Device helpers of the two short-axis kernels (mg_short.cu, FP32 storage;
// mg_short64.cu, FP64 storage): potential and demodulation tables, index
// arithmetic, asynchronous copies, per-thread accumulators.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "mg_device.cuh"
#include "mg_short.h"

namespace mgk {
namespace {

enum { SM_NONE = 0, SM_KIN = 1, SM_V = 2, SM_VONLY = 3 };
// scalar slots of the short kernel beyond the shared ones: p before the last
// potential substep
constexpr int SC_POLD = 48;

// ---------------------------------------------------------------------------
// Asynchronous global -> shared copies of one element
// ---------------------------------------------------------------------------

__device__ __forceinline__ void cp_async_el(double2* s, const double2* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_el(float2* s, const float2* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K> __device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory");
}

// ---------------------------------------------------------------------------
// Per-thread accumulators of the fused reductions
// ---------------------------------------------------------------------------

template <typename T> struct LineAcc;
template <> struct LineAcc<double> {
  double a[MAXD + 1];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < MAXD + 1; ++i) a[i] = 0.0;
  }
  __device__ __forceinline__ void add(int i, double x) { a[i] += x; }
  __device__ __forceinline__ double get(int i) const { return a[i]; }
  // i known only at run time: predicated adds keep the array in registers
  __device__ __forceinline__ void add_rt(int i, double x) {
#pragma unroll
    for (int k = 0; k < MAXD + 1; ++k)
      if (k == i) a[k] += x;
  }
  // slot k of o into slot i (known only at run time)
  __device__ __forceinline__ void merge_rt(int i, const LineAcc& o, int k) { add_rt(i, o.a[k]); }
};
template <> struct LineAcc<float> {
  float s[MAXD + 1], c[MAXD + 1];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < MAXD + 1; ++i) s[i] = c[i] = 0.f;
  }
  __device__ __forceinline__ void add(int i, float x) { two_sum_acc(s[i], c[i], x); }
  __device__ __forceinline__ double get(int i) const { return (double)s[i] + (double)c[i]; }
  __device__ __forceinline__ void add_rt(int i, float x) {
#pragma unroll
    for (int k = 0; k < MAXD + 1; ++k)
      if (k == i) two_sum_acc(s[k], c[k], x);
  }
  __device__ __forceinline__ void merge_rt(int i, const LineAcc& o, int k) {
    add_rt(i, o.s[k]);
    add_rt(i, o.c[k]);
  }
};

// Sum of acc[0 .. nv-1] over the CTA in a fixed order (warp trees, then warp
// order) into the CTA's record of `slot`, read back by finish().
template <typename T>
__device__ void block_record(const Bufs& B, double* red, int slot, const LineAcc<T>& acc, int nv) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int v = 0; v < MAXD + 1; ++v)
    if (v < nv) {
      const double s = warp_sum(acc.get(v));
      if (lane == 0) red[warp * 16 + v] = s;
    }
  __syncthreads();
  if (warp == 0 && lane < nv) {
    double s = 0;
    for (int w = 0; w < nw; ++w) s += red[w * 16 + lane];
    __stcg(B.part + ((size_t)slot * gridDim.x + blockIdx.x) * PSTRIDE + lane, s);
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Potential tables: V = sum_a f_a(x_a) + sum_{a<D-1} h_a(x_a) g_{a+1}(x_{a+1})
// ---------------------------------------------------------------------------

// f, f', g, g', h, h' of axis a at x.
__device__ __forceinline__ void chain_terms(const Plan& P, int a, double x, double* t) {
  const int D = P.D;
  if (P.pot_kind == POT_HENON_HEILES) {
    const double lam = P.pot[0];
    t[0] = 0.5 * x * x - (a >= 1 ? lam * x * x * x / 3.0 : 0.0);
    t[1] = x - (a >= 1 ? lam * x * x : 0.0);
    t[2] = a >= 1 ? x : 0.0;
    t[3] = a >= 1 ? 1.0 : 0.0;
    t[4] = a <= D - 2 ? lam * x * x : 0.0;
    t[5] = a <= D - 2 ? 2.0 * lam * x : 0.0;
  } else {  // harmonic with a diagonal force-constant matrix
    const double k = P.pot[a * D + a];
    const double d = x - P.pot[D * D + a];
    t[0] = 0.5 * k * d * d;
    t[1] = k * d;
    t[2] = t[3] = t[4] = t[5] = 0.0;
  }
}

// Build the per-axis factors F, the gradient columns (in B.tabV) and the pair
// factors for the grid centred at q_new (scalars SC_QN, SC_SGH of the CTA).
// Tasks of 32 entries, dealt to warp 0 of every CTA first.  A grid barrier
// must follow.
template <typename V>
__device__ void build_v_short(const Plan& P, const ShortPlan& SP, const Bufs& B, const Smem<V>& S) {
  const int TT = P.tab_total, n = SP.n;
  const int nP = SP.pairs ? (P.D - 1) * n * n : 0;
  const int nchF = (TT + 31) / 32, nchP = (nP + 31) / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const double* sc = S.sc;
  const double sgh = sc[SC_SGH];
  for (int t = warp * gridDim.x + blockIdx.x; t < nchF + nchP; t += nwarps * gridDim.x) {
    if (t < nchF) {
      const int e = t * 32 + lane;
      if (e >= TT) continue;
      const int a = e / n, j = e - a * n;
      const double x = fma((double)(j - n / 2), P.dq[a], sc[SC_QN + a]);
      double c[6];
      chain_terms(P, a, x, c);
      double sn, cs;
      expi_prec(P.prec, sgh * c[0], S.sct, sn, cs);
      __stcg(SP.tabF + e, P.prec ? round_unit_f32(cs, sn, 1.0) : make_double2(cs, sn));
#pragma unroll
      for (int k = 0; k < 5; ++k) __stcg(B.tabV + k * TT + e, c[1 + k]);
    } else {
      const int e = (t - nchF) * 32 + lane;
      if (e >= nP) continue;
      const int a = e / (n * n), rem = e - a * n * n;
      const int j = rem / n, j2 = rem - j * n;
      const double x = fma((double)(j - n / 2), P.dq[a], sc[SC_QN + a]);
      const double y = fma((double)(j2 - n / 2), P.dq[a + 1], sc[SC_QN + a + 1]);
      double ca[6], cb[6];
      chain_terms(P, a, x, ca);
      chain_terms(P, a + 1, y, cb);
      // the last pair's factor carries the last axis's own term too: the
      // potential sweep runs along that axis and multiplies by one factor
      const double th = a == P.D - 2 ? fma(ca[4], cb[2], cb[0]) : ca[4] * cb[2];
      double sn, cs;
      expi_prec(P.prec, sgh * th, S.sct, sn, cs);
      __stcg(SP.tabP + e, P.prec ? round_unit_f32(cs, sn, 1.0) : make_double2(cs, sn));
    }
  }
}

// Multipliers of the forward passes and of the final inverse passes.  Between
// stages of one launch the stored state carries the demodulation factor of
// the last kinetic substep, w = A(p) u (A as in mg_kernels.cu), which saves
// the conj(A)/N multiply of every inverse pass but the last:
//  - pre  (global SP.tabB, shared tA): A(p)/N_l if the state is u (rel = 0),
//    else A(p) conj(A(p_old))/N_l = e^{-i (p - p_old) c dq/hbar}/N_l (rel = 1),
//    with p_old the centre before the last potential substep (SC_POLD);
//  - post (global SP.tabC, shared tAi): conj(A(p)), applied by the inverse
//    passes of the launch's last kinetic substep only.
// The 1/N_l of the unitary pair of transforms sits in the forward multiplier.
template <typename V>
__device__ void build_demod_short(const Plan& P, const ShortPlan& SP, const Smem<V>& S, int rel) {
  const int TT = P.tab_total, n = SP.n;
  const int nch = (TT + 31) / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const double* sc = S.sc;
  for (int t = warp * gridDim.x + blockIdx.x; t < 2 * nch; t += nwarps * gridDim.x) {
    const int e = (t % nch) * 32 + lane;
    if (e >= TT) continue;
    const int a = e / n, j = e - a * n;
    const double c = (double)(j - n / 2);
    double sn, cs;
    if (t < nch) {
      const double dp = rel ? sc[SC_P + a] - sc[SC_POLD + a] : sc[SC_P + a];
      expi_prec(P.prec, -dp * c * P.dq[a] / P.hbar, S.sct, sn, cs);
      const double sg = (!rel && (j & 1)) ? -1.0 : 1.0;
      const double re = sg * cs / (double)n, im = sg * sn / (double)n;
      __stcg(SP.tabB + e, P.prec ? round_unit_f32(re, im, 1.0 / ((double)n * (double)n)) : make_double2(re, im));
    } else {
      expi_prec(P.prec, -sc[SC_P + a] * c * P.dq[a] / P.hbar, S.sct, sn, cs);
      const double sg = (j & 1) ? -1.0 : 1.0;
      __stcg(SP.tabC + e, P.prec ? round_unit_f32(sg * cs, -sg * sn, 1.0) : make_double2(sg * cs, -sg * sn));
    }
  }
}

// ---------------------------------------------------------------------------
// Index helpers
// ---------------------------------------------------------------------------

template <int N> __device__ __forceinline__ int ipow(int k) {
  int r = 1;
#pragma unroll
  for (int i = 0; i < SHORT_MAXG; ++i)
    if (i < k) r *= N;
  return r;
}

// Base-N digits of x into j[a] for lo <= a <= hi (j[hi] least significant).
template <int N> __device__ __forceinline__ void digits(unsigned x, int lo, int hi, int (&j)[MAXD]) {
#pragma unroll
  for (int a = MAXD - 1; a >= 0; --a)
    if (a >= lo && a <= hi) {
      const unsigned q = x / N;
      j[a] = (int)(x - q * N);
      x = q;
    }
}

// j[i] for an index known only at run time, without moving j to local memory.
__device__ __forceinline__ int pick(const int (&j)[MAXD], int i) {
  int v = 0;
#pragma unroll
  for (int k = 0; k < MAXD; ++k)
    if (k == i) v = j[k];
  return v;
}

// Global offset of chunk c (first element) and its number of planes.
__device__ __forceinline__ void chunk_geom(const GroupPlan& G, int64_t c, int64_t& gbase, int& nwt) {
  if (G.contig) {
    const int64_t b0 = c * G.WT;
    gbase = b0 * G.ng;
    nwt = (int)(G.nblk - b0 < G.WT ? G.nblk - b0 : G.WT);
  } else {
    const int64_t o = c / G.nb, b = c - o * G.nb;
    gbase = o * (int64_t)G.ng * G.inner + b * G.WT;
    nwt = G.WT;
  }
}

// Wait for the tensor copies of a chunk, bounded like every wait here: gives
// up after the barrier time limit (recording MG_ERR_TIMEOUT), or at once when
// another wait has already failed, so that a failure costs one time limit and
// not one per chunk.
__device__ __forceinline__ void wait_chunk(const Bufs& B, uint64_t* bar, unsigned parity) {
  if (mbar_try_wait(bar, parity)) return;
  const uint64_t t0 = global_ns();
  for (unsigned spins = 1;; ++spins) {
    if (mbar_try_wait(bar, parity)) return;
    if ((spins & 255u) == 0) {
      if (*(volatile int*)B.status != ST_OK) return;
      if (global_ns() - t0 > BARRIER_LIMIT_NS || spins > BARRIER_MAX_SPINS) {
        atomicExch(B.status, ST_TIMEOUT);
        return;
      }
    }
  }
}

}  // namespace
}  // namespace mgk
