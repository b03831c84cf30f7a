// One pass along one axis of the general propagation kernel, FP64 storage:
// the same pass as axis_pass (mg_device.cuh) with its transform on the integer
// units (mg_fixed.cuh).  A chunk is scaled by its norm as it arrives, the
// first Stockham pass converts it and applies the pre-multiplier, the
// epilogue applies the post-multiplier and the potential phase and converts
// back; FP64 is left with that conversion, the phase argument, the gradient
// and the sums.
//
// An FP64 instruction holds its unit for 64 cycles a warp, about 25 of them
// per point bound the FP64 pass; a 64-bit complex multiplication is about 50
// cycles of integer work and a butterfly's additions a few each.  What bounds
// this pass is latency: long dependent chains at 8 warps an SM (a thread needs
// up to 255 registers).  Measured per call, before -> after: 128^3 Duschinsky
// 9.32 -> 6.73 ms, 128 x 2048 Secrest-Johnson 1.96 -> 1.69 ms.  512 threads
// (8.2, 1.81 ms) and two CTAs an SM (10.4 ms on 128^3) spill and lose.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "mg_device.cuh"
#include "mg_fixed.cuh"

namespace mgk {
namespace {

constexpr double INV_2PI = 0.15915494309189535, INV_2PI_LO = -9.839338337591243e-18;
constexpr int PASS_BITS = 61;  // norm bound of a chunk, also after every pass of its transform

extern __shared__ __align__(16) unsigned char smem_raw64[];

// Multiplier words of v 2^s, |v| 2^s <= 1, by integer operations.
__device__ __forceinline__ int4 mult_bits(double2 v, int s) {
  const long long a = to_fixed(__double2hiint(v.x), (unsigned)__double2loint(v.x), 1024 - s, 0) & ~1ll;
  const long long b = to_fixed(__double2hiint(v.y), (unsigned)__double2loint(v.y), 1024 - s, 0) & ~1ll;
  return make_int4((int)(a >> 31), (int)(a & 0x7fffffff), (int)(b >> 31), (int)(b & 0x7fffffff));
}
// floor(log2 n): conj(A)/n is held times 2^this
__device__ __forceinline__ int post_shift(int n) { return 31 - __clz(n); }

// The per-axis tables in multiplier form (in place of load_tables' FP64
// pairs).  Entries that stay in the workspace are turned into words, and
// checked, where a pass reads them.
__device__ void load_mult_tables(const Plan& P, const Bufs& B, const Smem<double2>& S, int what) {
  const int TT = P.tab_total;
  load_tables(P, B, S, what & ~(LT_TW | LT_A | LT_K | LT_SCT));
  if (P.tab_global & TG_MULT) what &= ~(LT_A | LT_K);
  int4* tw = (int4*)S.tw;
  int4* tA = (int4*)S.tA;
  int4* tAi = (int4*)S.tAi;
  int4* tK = (int4*)S.tK;
  for (int e = threadIdx.x; e < TT; e += blockDim.x) {
    double2 w, a, ai, k;
    if (what & LT_TW) w = __ldcg(B.tw + e);
    if (what & LT_A) {
      a = __ldcg(B.tabA + e);
      ai = __ldcg(B.tabAi + e);
    }
    if (what & LT_K) k = __ldcg(B.tabK + e);
    if (what & LT_TW) tw[e] = mult_bits(w, 0);
    if (((what & LT_A) && not_finite(a)) || ((what & LT_K) && not_finite(k))) S.sc[SC_BAD] = 1.0;
    if (what & LT_A) {
      int l = 0;
      while (l + 1 < P.D && e >= P.ax[l + 1].toff) ++l;
      tA[e] = mult_bits(a, 0);
      tAi[e] = mult_bits(ai, post_shift(P.ax[l].n));
    }
    if (what & LT_K) tK[e] = mult_bits(k, 0);
  }
  if (what & LT_SCT) {
    // e^{2 pi i k / 256} and e^{2 pi i k / 65536}, for phase_words
    int4* t = (int4*)S.sct;
    for (int e = threadIdx.x; e < 512; e += blockDim.x) t[e] = __ldcg(B.words + e);
  }
}

// Rounding the factor from radians to turns would shift every phase of a
// substep by the same relative amount, which adds up over the steps (1.5 times
// the error on 64^3 over ten).  It is taken out again: slot SC_TEPS holds the
// relative shift times 2^64 for the potential's factor, KIN_TEPS is that of
// INV_2PI.
constexpr int SC_TEPS = 38;
constexpr float KIN_TEPS = (float)(INV_2PI_LO / INV_2PI * 18446744073709551616.0);
// Potential factor -sigma/hbar in turns, and its SC_TEPS (one thread).
__device__ __forceinline__ double turns_scale(double x, double* sc) {
  const double t = fma(x, INV_2PI, x * INV_2PI_LO);
  sc[SC_TEPS] = t != 0.0 ? (fma(x, INV_2PI, -t) + x * INV_2PI_LO) / t * 18446744073709551616.0 : 0.0;
  return t;
}

// x * e^{2 pi i t (1 + eps 2^-64)} for a phase of t turns.  t modulo 1 as a
// 64-bit fraction (exact); its first two bytes select table factors, the rest
// is a series: a = 2 pi f / 2^16, |f| <= 1/2, sin = a - a^3/6, cos = 1 - a^2/2
// (the next terms are below 2^-61).
__device__ __forceinline__ I2 rotate_turns(I2 x, double t, float eps, const int4* tab, int odd) {
  const int hi = __double2hiint(t);
  const unsigned long long m =
      ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)__double2loint(t);
  // |t| 2^64 = m 2^(e - 1011), modulo 2^64
  const int sh = (int)(((unsigned)hi >> 20) & 0x7ffu) - 1011;
  unsigned long long f = sh >= 0 ? (sh > 63 ? 0ull : m << sh) : (sh < -63 ? 0ull : m >> -sh);
  if (hi < 0) f = 0ull - f;
  // t to 20 bits as a float (below 2^-60 the correction is nothing; above
  // 2^64 turns neither is the phase anything)
  const int e = min(sh + 1011, 1087);
  const float tf = e < 963 ? 0.0f
                           : __int_as_float((int)(((unsigned)hi & 0x80000000u) | ((unsigned)(e - 896) << 23) |
                                                  (((unsigned)hi & 0xfffffu) << 3)));
  f += (unsigned long long)(long long)__float2int_rn(tf * eps);
  f += 1ull << 47;  // the series argument is the signed distance to the nearest 2^-16
  const int4 t1 = tab[(unsigned)(f >> 56)], t2 = tab[256 + ((unsigned)(f >> 48) & 255u)];
  const long long g = (long long)(f & 0xffffffffffffull) - (1ll << 47);
  // a 2^61 = g 2 pi / 8 = g - (1 - pi/4) g
  const long long es = g - mul_c(g, C1MPI4H, C1MPI4L);
  const int eh = (int)(es >> 16);                    // a 2^45, below 2^31
  const long long c2 = wide(eh, eh, 1ll << 29) >> 30;  // a^2 / 2, times 2^61
  const long long cs = (1ll << 61) - c2;
  const int c2h = (int)(c2 >> 8), e3 = eh >> 8;        // a^2 / 2 2^53, a 2^37
  const long long s3 = wide(c2h, e3, 0) >> 29;         // a^3 / 2, times 2^61
  const long long sn = es - mul_c(s3, C13H, C13L);
  const int4 w = make_int4((int)(cs >> 31), (int)(cs & 0x7fffffff), (int)(sn >> 31), (int)(sn & 0x7fffffff));
  return cmul<false, true>(cmul<false, true>(cmul<false, true>(x, t1, odd), t2, -1), w, -1);
}

// One Stockham pass of radix R over L lines of length n (see stockham_pass),
// divided by 2^SC.  The first pass (Ns == 1) converts its FP64 inputs at the
// chunk's scale and applies `pre` (shared) or `preg` (FP64 entries in the
// workspace; one that is not finite is noted in `bad`).
template <bool INV, int R, int SC>
__device__ __forceinline__ void stockham64_pass(const I2* __restrict__ in, I2* __restrict__ out, int n, int L,
                                                Div16 divL, int Ns, const int4* tw, const int4* pre,
                                                const double2* preg, int wsh, int ref, double* bad) {
  const int nR = n / R;
  const int total = L * nR;
  const int ts = n / (Ns * R);
  const int W = 1 << wsh;
  const Div16 divnR((unsigned)nR), divNs((unsigned)Ns);
  for (int b = threadIdx.x; b < total; b += blockDim.x) {
    int j, lbase, ps;
    if (wsh) {
      j = (int)divL((unsigned)b);
      const int line = b - j * L;
      lbase = (line >> wsh) * W * n + (line & (W - 1));
      ps = W;
    } else {
      const int line = (int)divnR((unsigned)b);
      j = b - line * nR;
      lbase = line * n;
      ps = 1;
    }
    const I2* src = in + lbase + j * ps;
    I2* dst = out + lbase;
    I2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = src[r * nR * ps];
    const int k = j - (int)divNs((unsigned)j) * Ns;
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        int4 w = tw[k * r * ts];
        if (INV) {
          w.z = -w.z;
          w.w = -w.w;
        }
        v[r] = cmul<false, true>(v[r], w, -1);
      }
    } else {
      const int tie = tie_of(v[0], v[1]);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = to_fixed(v[r], ref, tie);
      if (pre) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = cmul<false, true>(v[r], pre[j + r * nR]);
      } else if (preg) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const double2 m = __ldcg(preg + j + r * nR);
          if (not_finite(m)) *bad = 1.0;
          v[r] = cmul<false, true>(v[r], mult_bits(m, 0));
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = I2{v[r].x & ~1ll, v[r].y & ~1ll};
      }
    }
    const LineBits lb = line_bits(v[0], v[1]);
    if constexpr (R == 8) {
      idft8_late<INV, SC>(v);
    } else if constexpr (R == 4) {
      idft4<INV, SC>(v[0], v[1], v[2], v[3], lb);
    } else if constexpr (R == 3) {
      idft3<INV>(v[0], v[1], v[2], lb);
#pragma unroll
      for (int r = 0; r < 3; ++r) v[r] = divide<SC>(v[r], lb);
    } else {
      const I2 a = v[0];
      v[0] = iadd(a, v[1]);
      v[1] = isub(a, v[1]);
      if (SC) {
        v[0] = divide<SC>(v[0], lb);
        v[1] = divide<SC>(v[1], lb);
      }
    }
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[(base + r * Ns) * ps] = v[r];
  }
}

// Transform of L lines; returns the buffer with the result and adds the
// divisions to eo.  The norm is below 2^(PASS_BITS + h/2), h 0 or -1: a pass
// multiplies it by sqrt(R) (radix 3 counted as 2) and divides by as little as
// keeps it there.
template <bool INV>
__device__ I2* stockham64(I2* in, I2* out, int L, const AxisPlan& ax, const int4* tw, const int4* pre,
                          const double2* preg, int wsh, BlockScale bs, double* bad, int& eo) {
  const int ref = bs.ref;
  int Ns = 1, h = -bs.spare;
  const int n = ax.n;
  const Div16 divL((unsigned)L);
  for (int pi = 0; pi < ax.nrad; ++pi) {
    const int R = ax.rad[pi];
    h += R == 8 ? 3 : (R == 2 ? 1 : 2);
    const int sc = (h + 1) >> 1;
    h -= 2 * sc;
    eo += sc;
    if (R == 8) {
      if (sc == 1) stockham64_pass<INV, 8, 1>(in, out, n, L, divL, Ns, tw, pre, preg, wsh, ref, bad);
      else stockham64_pass<INV, 8, 2>(in, out, n, L, divL, Ns, tw, pre, preg, wsh, ref, bad);
    } else if (R == 4) {
      stockham64_pass<INV, 4, 1>(in, out, n, L, divL, Ns, tw, pre, preg, wsh, ref, bad);
    } else if (R == 3) {
      stockham64_pass<INV, 3, 1>(in, out, n, L, divL, Ns, tw, pre, preg, wsh, ref, bad);
    } else {
      if (sc == 0) stockham64_pass<INV, 2, 0>(in, out, n, L, divL, Ns, tw, pre, preg, wsh, ref, bad);
      else stockham64_pass<INV, 2, 1>(in, out, n, L, divL, Ns, tw, pre, preg, wsh, ref, bad);
    }
    __syncthreads();
    I2* t = in;
    in = out;
    out = t;
    Ns *= R;
  }
  return in;
}

// A thread's running record of the magnitudes it has seen: largest exponent
// field and the squares relative to it (fx_square).
struct ScanRec {
  int e = FX_EMIN;
  unsigned q = 0;
  __device__ __forceinline__ void add(double2 v) {
    const unsigned m = max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
    const int em = fx_exponent(m);
    if (em > e) {
      const int d = 2 * (em - e);
      q = d < 32 ? (q >> d) + 1u : 1u;
      e = em;
    }
    q += fx_square(m, e);
  }
};
// The chunk's scale from every thread's record (all threads; one barrier).
__device__ __forceinline__ BlockScale chunk_scale(ScanRec s, int* rec) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int E = __reduce_max_sync(0xffffffffu, s.e);
  const int d = 2 * (E - s.e);
  const unsigned q = __reduce_add_sync(0xffffffffu, d < 32 ? (s.q >> d) + 1u : 1u);
  if (lane == 0) {
    rec[2 * warp] = E;
    rec[2 * warp + 1] = (int)q;
  }
  __syncthreads();
  int Em = rec[0];
  for (int w = 1; w < nw; ++w) Em = max(Em, rec[2 * w]);
  unsigned Y = 0;
  for (int w = 0; w < nw; ++w) {
    const int dd = 2 * (Em - rec[2 * w]);
    Y += dd < 32 ? ((unsigned)rec[2 * w + 1] >> dd) + 1u : 1u;
  }
  return block_scale(Em, Y, 2, PASS_BITS);
}

// The arguments as for axis_pass; the phase of RED_V in turns (SC_SGH
// divided by 2 pi).
template <bool INV, int KIND, int DM = MAXD>
__device__ __noinline__ int axis_pass64(const Plan& P, const Bufs& B, const PassArgs& A, int res_in) {
  using V = double2;
  const Smem<V> S = carve<V, true>(P, B, smem_raw64);
  const AxisPlan& ax = P.ax[A.l];
  const int n = ax.n, W = ax.W, D = P.D;
  const bool contig = (A.l == D - 1);
  const int wsh = contig ? 0 : __ffs(W) - 1;
  const int64_t s = ax.stride;
  const unsigned tpo = contig ? 1u : (unsigned)(s / W);  // tiles per outer index
  const int64_t ws = contig ? n : 1;                       // element step between lines of a tile
  const int64_t es = contig ? 1 : s;                       // element step along the axis
  const int4* tw = (const int4*)S.tw + ax.toff;
  const bool gmult = P.tab_global & TG_MULT;
  const V* preT = A.pre == PRE_A ? S.tA + ax.toff : (A.pre == PRE_K ? S.tK + ax.toff : nullptr);
  const V* postT = A.post ? S.tAi + ax.toff : nullptr;
  const int4* pre = gmult ? nullptr : (const int4*)preT;
  const V* preg = gmult ? preT : nullptr;
  const int4* tab = (const int4*)S.sct;
  const double sgh = S.sc[SC_SGH];
  const float teps = (float)S.sc[SC_TEPS];
  int* rec = (int*)S.red;  // free until the pass's own sums

  double acc[DM + 2];
#pragma unroll
  for (int v = 0; v < DM + 2; ++v) acc[v] = 0;

  const int64_t bid = A.nb ? A.bid : (int64_t)blockIdx.x, nb = A.nb ? A.nb : (int64_t)gridDim.x;
  const int64_t mine = bid < ax.ntiles ? (ax.ntiles - bid + nb - 1) / nb : 0;
  const V* src = (const V*)A.src;
  V* dst = (V*)A.dst;
  int res = -1;
  const int chunk = A.from_smem || A.keep ? (int)mine : ax.tpc;
  const bool stream = !P.resident && !A.from_smem && !A.keep && mine > 0;
  int rd = 0, rt = 1, rf = 2;
  unsigned parity = 0;
  if (stream) {
    parity = *S.mphase;
    if (threadIdx.x < 32)
      issue_chunk(ax, contig, src, 0, (int)(mine < chunk ? mine : chunk), S.reg[rd], S.mbar + rd, bid, nb);
  }
  const Div16 divWn((unsigned)(W * n)), divn((unsigned)n);
  for (int64_t c0 = 0; c0 < mine; c0 += chunk) {
    const int nt = (int)(mine - c0 < chunk ? mine - c0 : chunk);
    const int cnt = nt * W * n;
    if (stream && c0 + chunk < mine && threadIdx.x < 32) {
      const int64_t c1 = c0 + chunk;
      issue_chunk(ax, contig, src, c1, (int)(mine - c1 < chunk ? mine - c1 : chunk), S.reg[rf], S.mbar + rf, bid,
                  nb);
    }
    // per-tile offsets and, for the fused reductions, each line's multi-index
    for (int k = threadIdx.x; k < nt; k += blockDim.x) {
      const int64_t t = bid + (c0 + k) * nb;
      const int64_t o = t < (1ll << 32) ? (int64_t)((unsigned)t / tpo) : t / tpo;
      S.tb[k] = contig ? t * W * n : o * n * s + (t - o * tpo) * W;
    }
    if (A.red != RED_NONE) {
      for (int kw = threadIdx.x; kw < nt * W; kw += blockDim.x) {
        const int k = kw / W, w = kw - k * W;
        const int64_t t = bid + (c0 + k) * nb;
        const int64_t o = t < (1ll << 32) ? (int64_t)((unsigned)t / tpo) : t / tpo;
        int idx[DM];
        const unsigned lo = contig ? (unsigned)(t * W + w) : (unsigned)o;
        const unsigned li = contig ? 0u : (unsigned)((t - o * tpo) * W + w);
        decode(P, A.l, lo, li, 0, idx);
        for (int a = 0; a < D; ++a) S.li[kw * D + a] = (uint16_t)idx[a];
      }
    }
    V* cur;
    V* oth;
    ScanRec sr;
    if (A.from_smem || stream) {
      if (A.from_smem) {
        cur = S.reg[res_in];
        oth = S.reg[res_in ^ 1];
      } else {
        wait_region(B, S.mbar + rd, (parity >> rd) & 1u);
        parity ^= 1u << rd;
        cur = S.reg[rd];
        oth = S.reg[rt];
      }
      for (int e = threadIdx.x; e < cnt; e += blockDim.x) sr.add(cur[e]);
    } else {
      // up to LOADS independent global loads in flight per thread
      constexpr int LOADS = 8;
      __syncthreads();  // S.tb ready
      cur = S.reg[0];
      oth = S.reg[1];
      for (int e0 = threadIdx.x; e0 < cnt; e0 += LOADS * blockDim.x) {
        V vals[LOADS];
#pragma unroll
        for (int u = 0; u < LOADS; ++u) {
          const int e = e0 + u * blockDim.x;
          if (e < cnt) {
            const int ti = (int)divWn((unsigned)e);
            const int rem = e - ti * W * n;
            const int w = contig ? (int)divn((unsigned)rem) : rem & (W - 1);
            const int j = contig ? rem - w * n : rem >> wsh;
            vals[u] = __ldcg(src + S.tb[ti] + j * es + w * ws);
          }
        }
#pragma unroll
        for (int u = 0; u < LOADS; ++u) {
          const int e = e0 + u * blockDim.x;
          if (e < cnt) {
            cur[e] = vals[u];
            sr.add(vals[u]);
          }
        }
      }
    }
    const BlockScale bs = chunk_scale(sr, rec);
    int eo = bs.eo;
    I2* ic = (I2*)cur;
    if (A.fft) {
      ic = stockham64<INV>(ic, (I2*)oth, nt * W, ax, tw, pre, preg, wsh, bs, S.sc + SC_BAD, eo);
      cur = (V*)ic;
    }
    if (postT) eo -= post_shift(n);
    const int odd = A.fft ? -1 : 0;
    const bool poison = bs.poison || noted_bad(S.sc);

    // epilogue: element e of the chunk is tile ti, point j, line w
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
      const int ti = (int)divWn((unsigned)e);
      const int rem = e - ti * W * n;
      const int w = contig ? (int)divn((unsigned)rem) : rem & (W - 1);
      const int j = contig ? rem - w * n : rem >> wsh;
      I2 x = ic[e];
      if (!A.fft) x = to_fixed(x, bs.ref, tie_of(x, x));
      bool nan = poison;
      if (postT) {
        int4 m;
        if (gmult) {
          const V f = __ldcg(postT + j);
          if (not_finite(f)) {
            nan = true;
            S.sc[SC_BAD] = 1.0;
          }
          m = mult_bits(f, post_shift(n));
        } else {
          m = ((const int4*)postT)[j];
        }
        x = cmul<false, true>(x, m, odd);
      }
      V v;
      if (A.red != RED_NONE) {
        int idx[DM];
#pragma unroll
        for (int a = 0; a < DM; ++a)
          if (a < D) idx[a] = S.li[(ti * W + w) * D + a];
        idx[A.l] = j;
        if (A.red == RED_KIN) {
          v = from_fixed2(x, eo);
          const double w2 = nan ? __longlong_as_double(0x7ff8000000000000ll) : fma(v.x, v.x, v.y * v.y);
          acc[0] += w2;
#pragma unroll
          for (int a = 0; a < DM; ++a)
            if (a < D) acc[1 + a] = fma(S.tc[P.ax[a].toff + idx[a]], w2, acc[1 + a]);
          if (P.minv_general) {
            // the non-separable part of the kinetic phase (see axis_pass)
            const double th = over_hbar(P, -S.sc[SC_TAU] * kinetic_cross<DM>(P, S.tc, S.sc, idx));
            v = from_fixed2(rotate_turns(x, th * INV_2PI, KIN_TEPS, tab, odd), eo);
            nan = nan || not_finite(th);
          }
        } else {  // RED_V
          double th, g[DM];
          vpoint<KIND, DM>(P, S.tv, idx, sgh, th, g);
          // |x|^2 is the same before and after the phase
          v = from_fixed2(rotate_turns(x, th, teps, tab, odd), eo);
          // an overflowing potential leaves no phase: a NaN, as its sine would be
          nan = nan || not_finite(th);
          const double w2 = nan ? __longlong_as_double(0x7ff8000000000000ll) : fma(v.x, v.x, v.y * v.y);
          acc[0] += w2;
#pragma unroll
          for (int a = 0; a < DM; ++a)
            if (a < D) acc[1 + a] = fma(g[a], w2, acc[1 + a]);
        }
      } else {
        v = from_fixed2(x, eo);
      }
      if (nan) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
      if (A.keep) cur[e] = v;
      else if (dst) __stcg(dst + S.tb[ti] + j * es + w * ws, v);
    }
    __syncthreads();
    if (stream) {
      const int nd = rf;
      rf = rd;
      rd = nd;
      // the transform may have ended in either of the chunk's two regions;
      // both are free again
    } else {
      res = cur == S.reg[0] ? 0 : (cur == S.reg[1] ? 1 : 2);
    }
  }
  if (stream) {
    if (threadIdx.x == 0) *S.mphase = parity;
    __syncthreads();
  }
  if (A.red != RED_NONE) block_partials<V, DM>(B, S, A.slot, acc, D + 1, A.rec ? A.rec + A.slot * PSTRIDE : nullptr);
  return res;
}

}  // namespace
}  // namespace mgk
