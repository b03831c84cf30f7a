// Short-axis propagation kernel for FP64 storage (sm_103a): grids of D >= 3
// axes that all have 8, 12 or 16 points.  The method, the axis groups, the
// order of passes, tables and grid barriers are those of mg_short.cu; what
// differs is the arithmetic inside a pass and how chunks are overlapped.
//
// Arithmetic.  The FP64 units (64 cycles per warp instruction) bound every
// FP64 pass when its transforms run on them.  Here a chunk is turned into
// 64-bit integers with one scale per chunk (mg_fixed.cuh), its multipliers
// and transforms along all axes of the group run on the integer units, and
// only the conversion of the results, the reduced moments (a few values per
// line) and the potential's gradient use the FP64 units.
//
// A chunk's life: FP64 values arrive by cp.async; every thread scans its
// share for the largest magnitudes and the chunk's norm bound is formed from
// them; the lines of the first axis are converted as they are read, those of
// the last axis are converted back as they are written; the chunk is stored.
//
// Overlap.  The CTA is two teams (half of the warps each) that work on
// alternate chunks with their own named barrier, so that one team's copies,
// conversions and barrier waits fall into the other's integer work.  Chunk i
// uses region i mod nreg; the team that has stored chunk i loads chunk
// i + nreg into its region, on an mbarrier that the team taking that chunk
// waits on.
//
// Reductions.  |x|^2 of the integers is summed along a line as integers (each
// component to 2^-57 or 2^-54 of the chunk's norm, without a mean error; the
// squares' high and middle parts in two 64-bit sums, the sums weighted by the
// line's coordinate from running sums of those), and one FP64 value per line
// and moment is formed at the end of the line.
//
// Measured: a 12^8 yoshida4 step 785 -> 276 ms, a 12^4 suzuki4 call 3.96 ->
// 2.06 ms against the same plan on the FP64 units.  What bounds it now is
// latency: 12 (8) warps an SM at up to 168 (255) registers a thread issue 0.30
// instructions a cycle and scheduler; the stalls are the teams' barriers
// (24%), fixed-latency dependences (21%) and shared and global loads (18%).  18
// warps at 112 registers spill (12^7: 25.3 against 21.1 ms a step).
#include <cuda_runtime.h>
#include <stdint.h>

#include "mg_fixed.cuh"
#include "mg_short_dev.cuh"

namespace mgk {
namespace {

__host__ __device__ constexpr int short64_threads(int n) { return n == 12 ? 384 : 256; }
constexpr int TEAMS = 2;

// floor(log2 n^g): forward multipliers A/n^g are stored times 2^this
__device__ __forceinline__ int fwd_shift(int n, int g) {
  return n == 8 ? 3 * g : n == 16 ? 4 * g : (g == 1 ? 3 : g == 2 ? 7 : g == 3 ? 10 : 14);
}
struct S64 {
  Smem<double2> s;  // fin, sc, red, sct, mbar, mphase
  int4* F;     // per-axis potential factors
  int4* Pt;    // pair factors [(D-1) n][n+1]; the last n rows also hold the last axis's own factor
  double* col; // [5][D n] f', g, g', h, h'
  int4* Gh;    // [n^(g-1)] product of the factors among a line's coordinates inside group 0
  double* U;   // [4][n^(g-1)] gradient coefficients of those coordinates (load_v64)
  I2* Lo;      // [2][WT] product of the factors of the axes before group 0
  double* pc;  // [2][WT][SHORT64_PC] gradient coefficients of those axes
  int* jl;     // [2][WT] coordinate on the axis before group 0
  int* es;     // [2][16] norm records of a team's warps
  double* cd;  // r - n/2; then c1, c2 of the last axis (load_v64)
  double2* reg;
  int region_elems;
};

extern __shared__ __align__(16) unsigned char smem64[];

// Every function forms its pointers from the shared array itself, so that
// the compiler sees shared-memory addresses (a pointer handed over through
// memory would be a generic one).
__device__ __forceinline__ S64 carve64(const Plan& P, const ShortPlan& SP, const Bufs& B) {
  unsigned char* base = smem64;
  const Short64Layout L = short64_layout(P.D, SP.n, SP.threads, SP.grp[0].g, SP.grp[0].WT, SP.nreg, SP.region_elems);
  S64 m{};
  m.s.red = (double*)(base + L.red);
  m.s.fin = (double*)(base + L.fin);
  m.s.sc = (double*)(base + L.sc);
  m.s.sct = B.sct;  // read through the caches: a few hundred entries per stage
  m.s.mbar = (uint64_t*)(base + L.mbar);
  m.s.mphase = (unsigned*)(base + L.mphase);
  m.F = (int4*)(base + L.F);
  m.Pt = (int4*)(base + L.Pt);
  m.col = (double*)(base + L.col);
  m.Gh = (int4*)(base + L.Gh);
  m.U = (double*)(base + L.U);
  m.Lo = (I2*)(base + L.Lo);
  m.pc = (double*)(base + L.pc);
  m.jl = (int*)(base + L.jl);
  m.es = (int*)(base + L.es);
  m.cd = (double*)(base + L.cd);
  m.reg = (double2*)(base + L.reg);
  m.region_elems = SP.region_elems;
  return m;
}

// ---------------------------------------------------------------------------
// Tables in multiplier form
// ---------------------------------------------------------------------------

constexpr double M61 = 2305843009213693952.0;  // 2^61

// Multipliers of all points of every group's block.  A diagonal multiplier
// along one axis commutes with the transforms along the others, so a pass
// multiplies once per point, by the product over its group's axes: one phase
// per entry, the sum of the axes' phases.
//   GT_U    A(p) / n^g            (the state is u)
//   GT_REL  A(p) conj(A(p_old)) / n^g  (it carries A(p_old): see build_demod_short)
//   GT_K    K                     (inverse passes)
//   GT_POST conj(A(p))            (after a launch's last inverse passes)
// Tasks of 32 entries, dealt to warp 0 of every CTA first; a grid barrier
// must follow.
enum { GT_U = 0, GT_REL = 1, GT_K = 2, GT_POST = 3 };
template <int N>
__device__ void build_group_table(const Plan& P, const ShortPlan& SP, const Bufs& B, double* sc, int kind, int4* dst) {
  const int total = SP.toff[SP.ngroups], nch = (total + 31) / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  for (int t = warp * gridDim.x + blockIdx.x; t < nch; t += nwarps * gridDim.x) {
    const int e = t * 32 + lane;
    if (e >= total) continue;
    int gi = 0;
    while (e >= SP.toff[gi + 1]) ++gi;
    int row = e - SP.toff[gi], sign = 0;
    double th = 0.0;
    for (int k = SP.grp[gi].g - 1; k >= 0; --k) {
      const int a = SP.grp[gi].l0 + k, j = row % N;
      row /= N;
      const double c = (double)(j - N / 2);
      if (kind == GT_K) {
        const double pk = fma(c, P.dp[a], sc[SC_P + a]);
        th += sc[SC_DELTA + a] * pk - 0.5 * sc[SC_TAU] * P.minv[a] * pk * pk;
      } else {
        th -= (kind == GT_REL ? sc[SC_P + a] - sc[SC_POLD + a] : sc[SC_P + a]) * c * P.dq[a];
        sign ^= j & 1;
      }
    }
    double sn, cs;
    expi_tab(over_hbar(P, th), B.sct, sn, cs);
    if (kind == GT_POST) sn = -sn;
    if (kind == GT_U || kind == GT_REL) {
      const double h = SP.fscale[gi][0], l = SP.fscale[gi][1];
      cs = fma(cs, h, cs * l);
      sn = fma(sn, h, sn * l);
    }
    if ((kind == GT_U || kind == GT_POST) && sign) {
      cs = -cs;
      sn = -sn;
    }
    if (not_finite(make_double2(cs, sn))) {
      sc[SC_BAD] = 1.0;
      __stcg(B.bar + BAR_BAD, 1u);
    }
    __stcg(dst + e, to_mult(make_double2(cs, sn), M61));
  }
}

__device__ __forceinline__ double2 load_factor(const double2* t, double* sc) {
  const double2 f = __ldcg(t);
  if (not_finite(f)) sc[SC_BAD] = 1.0;
  return f;
}

// Last axis along a line: g = g0 + g1 rho, f' = c0 + c1 rho + c2 rho^2, g' and
// h constant factors, rho = r - n/2 (chain_terms as polynomials).
struct LastAxis {
  double g0, g1, c0, c1, c2, gp;
};
__device__ __forceinline__ LastAxis last_axis(const Plan& P, double x, double dq) {
  LastAxis a;
  const int l = P.D - 1;
  if (P.pot_kind == POT_HENON_HEILES) {
    const double lam = P.pot[0];
    a.g0 = x;
    a.g1 = dq;
    a.gp = 1.0;
    a.c0 = x - lam * x * x;
    a.c1 = dq * (1.0 - 2.0 * lam * x);
    a.c2 = -lam * dq * dq;
  } else {
    const double k = P.pot[l * P.D + l];
    a.g0 = a.g1 = a.gp = 0.0;
    a.c0 = k * (x - P.pot[P.D * P.D + l]);
    a.c1 = k * dq;
    a.c2 = 0.0;
  }
  return a;
}

// Potential factors and gradient columns for the grid centred at SC_QN, then
// (after a barrier inside) the products over a line's coordinates inside
// group 0: Gh, and U = [f' + h_(b-1) g'_b + h'_b g_(b+1)] for its first and
// second axis, [c0 + h g'] and h' g1 for the last two (see the sweep).
template <int N> __device__ void load_v64(const Plan& P, const ShortPlan& SP, const Bufs& B, const S64& S) {
  const int TT = P.tab_total, D = P.D;
  for (int e = threadIdx.x; e < TT; e += blockDim.x) {
    S.F[e] = to_mult(load_factor(SP.tabF + e, S.s.sc), M61);
#pragma unroll
    for (int k = 0; k < 5; ++k) S.col[k * TT + e] = __ldcg(B.tabV + k * TT + e);
  }
  for (int e = threadIdx.x; e < (D - 1) * N * N; e += blockDim.x) {
    if (SP.pairs) S.Pt[e + e / N] = to_mult(load_factor(SP.tabP + e, S.s.sc), M61);
    else if (e >= (D - 2) * N * N) S.Pt[e + e / N] = to_mult(__ldcg(SP.tabF + (D - 1) * N + e % N), M61);
  }
  const int g = SP.grp[0].g, l0 = SP.grp[0].l0;
  const int ng1 = ipow<N>(g - 1);
  for (int hi = threadIdx.x; hi < ng1; hi += blockDim.x) {
    int x = hi;
    double2 v = make_double2(1.0, 0.0);
    for (int b = D - 2, prev = -1; b >= l0; --b) {
      const int j = x % N;
      x /= N;
      v = cmul(v, __ldcg(SP.tabF + b * N + j));
      if (prev >= 0 && SP.pairs) v = cmul(v, __ldcg(SP.tabP + (b * N + j) * N + prev));
      prev = j;
    }
    S.Gh[hi] = to_mult(v, M61);
  }
  __syncthreads();
  const double* cfp = S.col;
  const double* cg = S.col + TT;
  const double* cgp = S.col + 2 * TT;
  const double* ch = S.col + 3 * TT;
  const double* chp = S.col + 4 * TT;
  const LastAxis la = last_axis(P, S.s.sc[SC_QN + D - 1], P.dq[D - 1]);
  if (threadIdx.x == 0) {
    S.cd[N] = la.c1;
    S.cd[N + 1] = la.c2;
  }
  for (int hi = threadIdx.x; hi < ng1; hi += blockDim.x) {
    int x = hi, next = 0;
    for (int b = D - 2; b >= l0; --b) {
      const int j = x % N;
      x /= N;
      double u = cfp[b * N + j] + chp[b * N + j] * (b == D - 2 ? la.g0 : cg[(b + 1) * N + next]);
      if (b > l0) u += ch[(b - 1) * N + x % N] * cgp[b * N + j];
      if (b - l0 < 2) S.U[(b - l0) * ng1 + hi] = u;
      if (b == D - 2) {
        S.U[2 * ng1 + hi] = la.c0 + ch[b * N + j] * la.gp;
        S.U[3 * ng1 + hi] = chp[b * N + j] * la.g1;
      }
      next = j;
    }
  }
}

// ---------------------------------------------------------------------------
// Chunk copies: thread L of `lines` moves N elements at constant steps, rows
// L', L' + n^(g-1), ...
// ---------------------------------------------------------------------------

struct CopyPlan {
  int ng1, sstep, contig, WT, PS, ng, lines;
  int64_t inner, gstep;
  Div16 dv;  // by ng1 (contiguous) or WT
  __device__ __forceinline__ CopyPlan(const GroupPlan& G, int ng1_, int n)
      : ng1(ng1_), sstep(ng1_ + ng1_ / n), contig(G.contig), WT(G.WT), PS(G.PS), ng(G.ng), lines(G.WT * ng1_),
        inner(G.inner), gstep(G.contig ? ng1_ : ng1_ * G.inner), dv((unsigned)(G.contig ? ng1_ : G.WT)) {}
};

// Shared and global offset of thread L's first element; false past the chunk.
template <int N>
__device__ __forceinline__ bool copy_start(const CopyPlan& C, int L, int nwt, int64_t gb, int& s, int64_t& g) {
  const int q = (int)C.dv((unsigned)L);
  const int wt = C.contig ? q : L - q * C.WT;
  const int row = C.contig ? L - q * C.ng1 : q;
  s = wt * C.PS + row + row / N;
  g = gb + (C.contig ? (int64_t)(wt * C.ng + row) : (int64_t)row * C.inner + wt);
  return wt < nwt;
}

__device__ __forceinline__ void team_bar(int team, int tt_count) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(tt_count) : "memory");
}
// this thread's outstanding cp.async copies arrive on the mbarrier when done
__device__ __forceinline__ void cp_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_init_count(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

template <int N>
__device__ __forceinline__ void load_chunk(const CopyPlan& C, const GroupPlan& G, const double2* psi, int64_t c,
                                           double2* reg, int tt, int nt, uint64_t* bar) {
  int64_t gb;
  int nwt;
  chunk_geom(G, c, gb, nwt);
  for (int L = tt; L < C.lines; L += nt) {
    int s;
    int64_t g;
    if (!copy_start<N>(C, L, nwt, gb, s, g)) continue;
    double2* sp = reg + s;
    const double2* gp = psi + g;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      cp_async_el(sp, gp);
      sp += C.sstep;
      gp += C.gstep;
    }
  }
  cp_arrive(bar);
}
template <int N>
__device__ __forceinline__ void store_chunk(const CopyPlan& C, const GroupPlan& G, double2* psi, int64_t c,
                                            const double2* reg, int tt, int nt) {
  int64_t gb;
  int nwt;
  chunk_geom(G, c, gb, nwt);
  for (int L = tt; L < C.lines; L += nt) {
    int s;
    int64_t g;
    if (!copy_start<N>(C, L, nwt, gb, s, g)) continue;
    const double2* sp = reg + s;
    double2* gp = psi + g;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      __stcs(gp, *sp);
      sp += C.sstep;
      gp += C.gstep;
    }
  }
}

// ---------------------------------------------------------------------------
// One group pass
// ---------------------------------------------------------------------------

// Integer sums of |x|^2 along a line, and of |x|^2 times the running count
// (twice for W = 2): S_k = sum of S_(k-1).  x is cut into its high word (after
// dropping S bits) and the next B bits, the last of them set: the middle of the
// interval that B - 1 bits leave, so that the values are not low on average.
// |x|^2 = 2^(64 + 2 S) (H + C 2^(1-B)).  The sums are exact modulo 2^64; what
// is taken from them fits: with norm^2 < 2^124.8 (kinetic) or 2^124 the sum of
// the squared high words is below 2^(60.8 - 2 S) or 2^(60 - 2 S), and a weighted
// C below 2^B times its root times that of the sum of the squared weights: 2^62.5
// and 2^61.3 for 12 points, 2^61.7 and 2^61.4 for 16 (norm^2 < 2^122).
template <int W, int S, int B> struct LineSums {
  unsigned long long h0 = 0, h1 = 0, h2 = 0;
  unsigned long long c0 = 0, c1 = 0, c2 = 0;
  static __device__ __forceinline__ int mid(long long v) {
    return (int)((__funnelshift_r((unsigned)v, (unsigned)hi32(v), 32 - B + S) & ((1u << B) - 1)) | 1u);
  }
  __device__ __forceinline__ void add(I2 v) {
    const int xh = hi32(v.x) >> S, yh = hi32(v.y) >> S, xm = mid(v.x), ym = mid(v.y);
    const long long l = wide(xm, xm, wide(ym, ym, 0));
    c0 = (unsigned long long)wide(xh, xm, wide(yh, ym, (long long)c0 + (l >> (B + 1))));
    h0 = (unsigned long long)wide(xh, xh, wide(yh, yh, (long long)h0));
    h1 += h0;
    c1 += c0;
    if (W > 1) {
      h2 += h1;
      c2 += c1;
    }
  }
  // 2^K (H + C 2^(1-B)), rounded, of a weighted sum
  template <int K> static __device__ __forceinline__ long long value(unsigned long long h, unsigned long long c) {
    return (long long)(h << K) + (((long long)c + (1LL << (B - 2 - K))) >> (B - 1 - K));
  }
};
// 2^(30 + S + eo) (NaN for a poisoned chunk): a sum V 2^-k of squares in
// integer units is V * s * s * 2^(4 - k) in the state's units
__device__ __forceinline__ double moment_scale(int eo, int poison) {
  return poison ? __longlong_as_double(0x7ff8000000000000ll) : __hiloint2double((1053 + eo) << 20, 0);
}

template <int N, bool INV, int MODE, bool POST>
__device__ __noinline__ void pass64(const Plan& P, const ShortPlan& SP, const Bufs& B, int gi, int slot) {
  constexpr bool VP = MODE == SM_V || MODE == SM_VONLY;
  // The norm bound is 2^61 after the first multiplication and has to stay
  // below 2^62.8, or 2^62 where a multiplication follows the transforms.
  // 12 points: divisions by 2, 4, 2 (factors 1.73, 0.87, 1.73) or 2, 4, 4;
  // 8 points: by 2 each (factor 1.41) or 2, 4, 2.
  constexpr bool MUL_AFTER = POST || VP;
  const GroupPlan G = SP.grp[gi];
  const S64 S = carve64(P, SP, B);
  const int4* const tabT = SP.tabT + SP.toff[gi];
  const int4* const tabQ = SP.tabQ + SP.toff[gi];
  const int D = P.D, g = G.g, l0 = G.l0, TT = P.tab_total;
  const int nreg = SP.nreg, pairs = SP.pairs;
  double2* psi = (double2*)B.psi;
  const int nt = blockDim.x / TEAMS;
  const int team = threadIdx.x >= nt, tt = threadIdx.x - team * nt;
  const int lane = threadIdx.x & 31, tw = tt >> 5, ntw = nt >> 5;
  const int64_t mine = blockIdx.x < G.nchunks ? (G.nchunks - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  const int ng1 = ipow<N>(g - 1);
  const CopyPlan C(G, ng1, N);
  const unsigned parity0 = *S.s.mphase;
  int* es = S.es + team * 16;
  LineAcc<double> acc, accg;
  acc.zero();
  accg.zero();

  for (int r = team; r < nreg && r < mine; r += TEAMS)
    load_chunk<N>(C, G, psi, blockIdx.x + (int64_t)r * gridDim.x, S.reg + r * S.region_elems, tt, nt, S.s.mbar + r);

  // the launch's last passes have no sum after them that could end it: they ask
  // whether any CTA noted an entry
  const bool bad = noted_bad(S.s.sc) || (POST && __ldcg(B.bar + BAR_BAD) != 0);
  int r = team % nreg;
  unsigned use = team / nreg;
  for (int64_t i = team; i < mine; i += TEAMS) {
    const int64_t c = blockIdx.x + i * gridDim.x;
    int64_t gb;
    int nwt;
    chunk_geom(G, c, gb, nwt);
    const int nl = nwt * ng1;
    const unsigned cbase = G.contig ? (unsigned)(c * G.WT) : (unsigned)((c % G.nb) * G.WT);
    double2* reg = S.reg + r * S.region_elems;
    I2* ireg = reinterpret_cast<I2*>(reg);
    if (VP && tt < nwt) {
      // factors and gradient coefficients of the axes before the group
      int j[MAXD];
      digits<N>(cbase + tt, 0, l0 - 1, j);
      I2 lo = I2{1LL << 60, 0};
      double* pc = S.pc + (team * G.WT + tt) * SHORT64_PC;
      const double* cfp = S.col;
      const double* cg = S.col + TT;
      const double* cgp = S.col + 2 * TT;
      const double* ch = S.col + 3 * TT;
      const double* chp = S.col + 4 * TT;
#pragma unroll
      for (int b = 0; b < MAXD - 2; ++b)
        if (b < l0) {
          lo = cmul_m(lo, S.F[b * N + j[b]]);
          if (pairs && b + 1 < l0) lo = cmul_m(lo, S.Pt[(b * N + j[b]) * (N + 1) + j[b + 1]]);
          double u = cfp[b * N + j[b]];
          if (b + 1 < l0) u = fma(chp[b * N + j[b]], cg[(b + 1) * N + j[b + 1]], u);
          if (b > 0) u = fma(ch[(b - 1) * N + j[b - 1]], cgp[b * N + j[b]], u);
          pc[b] = u;
        }
      const int jl = l0 > 0 ? pick(j, l0 - 1) : 0;
      pc[8] = l0 > 0 ? chp[(l0 - 1) * N + jl] : 0.0;
      pc[9] = l0 > 0 ? ch[(l0 - 1) * N + jl] : 0.0;
      S.Lo[team * G.WT + tt] = lo;
      S.jl[team * G.WT + tt] = jl;
    }
    wait_chunk(B, S.s.mbar + r, ((parity0 >> r) ^ use) & 1u);

    // the chunk's norm bound: the largest |value| of every two points, their
    // squares summed over the warp relative to its largest exponent
    BlockScale bs;
    {
      constexpr int ROUNDS = 2, SUB = N / 2;  // C.lines <= ROUNDS * nt
      unsigned m[ROUNDS][SUB];
      int e = 0;
#pragma unroll
      for (int h = 0; h < ROUNDS; ++h) {
        const int L = tt + h * nt;
        int s = 0;
        int64_t gx;
        const bool have = L < C.lines && copy_start<N>(C, L, nwt, 0, s, gx);
#pragma unroll
        for (int w = 0; w < SUB; ++w) {
          m[h][w] = 0;
          if (have) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const double2 v = reg[s];
              s += C.sstep;
              m[h][w] = max(m[h][w], max((unsigned)__double2hiint(v.x) & 0x7fffffffu,
                                         (unsigned)__double2hiint(v.y) & 0x7fffffffu));
            }
          }
          e = max(e, fx_exponent(m[h][w]));
        }
      }
      e = __reduce_max_sync(0xffffffffu, e);
      unsigned q = 0;
#pragma unroll
      for (int h = 0; h < ROUNDS; ++h)
#pragma unroll
        for (int w = 0; w < SUB; ++w) q += fx_square(m[h][w], e);
      const unsigned sum = __reduce_add_sync(0xffffffffu, q);
      if (lane == 0) {
        es[2 * tw] = e;
        es[2 * tw + 1] = (int)sum;
      }
      team_bar(team, nt);
      int E = es[0];
      for (int w = 1; w < ntw; ++w) E = max(E, es[2 * w]);
      unsigned Y = 0;
      for (int w = 0; w < ntw; ++w) {
        const int d = 2 * (E - es[2 * w]);
        Y += d < 32 ? ((unsigned)es[2 * w + 1] >> d) + 1u : 1u;
      }
      bs = block_scale(E, Y, 4, FX_BITS);
      bs.poison |= bad;
    }
    int eo = bs.eo;

    const int kend = MODE == SM_VONLY ? 1 : g;
    for (int kk = 0; kk < kend; ++kk) {
      // the axes in order; where a reduction needs its lines last, axis 0 (the
      // kinetic moments) or the last axis (the potential) come last
      const int k = MODE == SM_VONLY ? g - 1 : (MODE == SM_KIN ? (kk == g - 1 ? 0 : kk + 1) : kk);
      const bool last = (kk == kend - 1);
      const int nlo = ipow<N>(g - 1 - k), nhi = ipow<N>(k);
      const Div16 dlo((unsigned)nlo), dhi((unsigned)nhi);
      const int stride = (k == g - 1) ? 1 : ipow<N>(g - 2 - k) * (N + 1);
      const bool by2 = N == 8 ? !(MUL_AFTER && kk == 1) : N == 12 && (kk == 0 || (last && !MUL_AFTER));
      if (MODE != SM_VONLY) {
        if (kk == 0) eo += 1 - (INV ? 0 : fwd_shift(N, g));
        eo += by2 ? 1 : 2;
        if (POST && last) eo += 1;
      }
      for (int L = tt; L < nl; L += nt) {
        const int t = (int)dlo((unsigned)L), lo = L - t * nlo;
        const int wt = (int)dhi((unsigned)t), hi = t - wt * nhi;
        const int base = wt * G.PS + (k == g - 1 ? hi * (N + 1) : (hi * nlo + lo / N) * (N + 1) + lo % N);
        const int row = hi * N * nlo + lo;  // of the line's first point in the block
        I2 x[N];
        {
          const I2* p = ireg + base;
#pragma unroll
          for (int q = 0; q < N; ++q) {
            x[q] = *p;
            p += stride;
          }
        }
        if (kk == 0) {
          const int4* mt = tabT + row;
          const int tie = tie_of(x[0], x[N / 2]);
#pragma unroll
          for (int q = 0; q < N; ++q) {
            x[q] = to_fixed(x[q], bs.ref, tie);
            if (MODE != SM_VONLY) {
              x[q] = cmul_half(x[q], __ldcg(mt), 0);
              mt += nlo;
            }
          }
        }
        if (MODE != SM_VONLY) {
          if constexpr (N == 16) {
            IDft<INV, N, 2>::run(x);
          } else {
            if (by2) IDft<INV, N, 1>::run(x);
            else IDft<INV, N, 2>::run(x);
          }
          if (POST && last) {
            const int4* mt = tabQ + row;
#pragma unroll
            for (int q = 0; q < N; ++q) {
              x[q] = cmul_half(x[q], __ldcg(mt), -1);
              mt += nlo;
            }
          }
        }
        if (!last) {
          I2* p = ireg + base;
#pragma unroll
          for (int q = 0; q < N; ++q) {
            *p = x[q];
            p += stride;
          }
          continue;
        }
        int eout = eo;
        if (MODE == SM_KIN) {
          // kinetic moments; the line runs along axis 0 (k = 0, l0 = 0)
          constexpr int SH = 1;
          LineSums<1, SH, 29> m;
#pragma unroll
          for (int q = 0; q < N; ++q) m.add(x[q]);
          const double s = moment_scale(eo + SH, bs.poison);
          const unsigned long long H = N / 2;
          const double w0 = (double)m.template value<3>(m.h0, m.c0) * s * (2.0 * s);
          const double w1 = (double)m.template value<1>(H * m.h0 - m.h1, H * m.c0 - m.c1) * s * (8.0 * s);
          int j[MAXD];
          digits<N>((unsigned)lo, 1, g - 1, j);
          if (!G.contig) digits<N>(cbase + wt, g, D - 1, j);
          acc.add(0, w0);
          acc.add(1, w1);
#pragma unroll
          for (int b = 1; b < MAXD; ++b)
            if (b < D) acc.a[1 + b] = fma(S.cd[j[b]], w0, acc.a[1 + b]);
        }
        if (VP) {
          // potential substep on the line along the last axis: moments, then
          // the phase lf * (last pair's factor at r)
          constexpr int SH = 2;
          LineSums<2, SH, 27> m;
#pragma unroll
          for (int q = 0; q < N; ++q) m.add(x[q]);
          const double s = moment_scale(eo + SH, bs.poison);
          const unsigned long long H = N / 2;
          const double w0 = (double)m.template value<4>(m.h0, m.c0) * s * s;
          constexpr int K1 = MODE == SM_VONLY ? 2 : 4, K2 = MODE == SM_VONLY ? 0 : 2;
          const double s1 = MODE == SM_VONLY ? 4.0 * s : s;
          const double w1 = (double)m.template value<K1>(H * m.h0 - m.h1, H * m.c0 - m.c1) * s * s1;
          const double w2 = (double)m.template value<K2>(H * H * m.h0 - (N + 1) * m.h1 + 2 * m.h2,
                                                   H * H * m.c0 - (N + 1) * m.c1 + 2 * m.c2) * s1 * (4.0 * s);
          const int pw = team * G.WT + wt;
          const double* pc = S.pc + pw * SHORT64_PC;
          const int jm = hi % N, jf = hi / ipow<N>(g >= 2 ? g - 2 : 0);  // coordinates on axes D-2 and l0
          acc.add(0, w0);
#pragma unroll
          for (int b = 0; b < MAXD - 2; ++b)
            if (b < l0) {
              const double u = b == l0 - 1 ? fma(pc[8], S.col[TT + l0 * N + jf], pc[b]) : pc[b];
              acc.a[1 + b] = fma(u, w0, acc.a[1 + b]);
            }
          {
            const double u = fma(pc[9], S.col[2 * TT + l0 * N + jf], S.U[hi]);
            double t0 = u * w0;
            if (g == 2) t0 = fma(S.U[3 * ng1 + hi], w1, t0);
            accg.add(0, t0);
          }
          if (g >= 3) accg.add(1, fma(S.U[3 * ng1 + hi], w1, S.U[ng1 + hi] * w0));
          accg.add(2, fma(S.cd[N + 1], w2, fma(S.cd[N], w1, S.U[2 * ng1 + hi] * w0)));
          I2 lf = S.Lo[pw];
          if (pairs && l0 > 0) lf = cmul_m(lf, S.Pt[((l0 - 1) * N + S.jl[pw]) * (N + 1) + jf]);
          lf = cmul_m(lf, S.Gh[hi]);
          const int4* prow = S.Pt + ((D - 2) * N + jm) * (N + 1);
#pragma unroll
          for (int q = 0; q < N; ++q)
            x[q] = cmul<!POST, true>(x[q], to_mult60(cmul_m(lf, prow[q])), MODE == SM_VONLY ? 0 : -1);
          if (!POST) eout += 1;
        }
        {
          double2* p = reg + base;
#pragma unroll
          for (int q = 0; q < N; ++q) {
            double2 v = from_fixed2(x[q], eout);
            if (bs.poison) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
            *p = v;
            p += stride;
          }
        }
      }
      team_bar(team, nt);
    }
    store_chunk<N>(C, G, psi, c, reg, tt, nt);
    team_bar(team, nt);
    if (i + nreg < mine)
      load_chunk<N>(C, G, psi, c + (int64_t)nreg * gridDim.x, reg, tt, nt, S.s.mbar + r);
    r += TEAMS;
    while (r >= nreg) {
      r -= nreg;
      ++use;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // phases completed by this pass: one per chunk of each region
    unsigned p = parity0;
    for (int q = 0; q < nreg; ++q)
      if (mine > q) p ^= (unsigned)(((mine - q + nreg - 1) / nreg) & 1) << q;
    *S.s.mphase = p;
  }
  if (VP) {
    acc.merge_rt(1 + l0, accg, 0);
    if (g >= 3) acc.merge_rt(2 + l0, accg, 1);
    acc.merge_rt(D, accg, 2);
  }
  if (MODE != SM_NONE && bad) acc.a[0] = __longlong_as_double(0x7ff8000000000000ll);
  if (MODE != SM_NONE) block_record<double>(B, S.s.red, slot, acc, D + 1);
  __syncthreads();
}

// ---------------------------------------------------------------------------
// The persistent kernel
// ---------------------------------------------------------------------------

template <int N>
__global__ void __launch_bounds__(short64_threads(N), 1)
    k_propagate_short64(const __grid_constant__ Plan P, const __grid_constant__ Bufs B, const __grid_constant__ Run RN,
                        const __grid_constant__ ShortPlan SP) {
  __shared__ int sflag;
  const S64 S = carve64(P, SP, B);
  const int D = P.D, ng = SP.ngroups;
  if (__ldcg(B.status) != ST_OK) return;
  double* sc = S.s.sc;
  if (threadIdx.x < SC_N) sc[threadIdx.x] = 0.0;
  if (threadIdx.x < N) S.cd[threadIdx.x] = (double)((int)threadIdx.x - N / 2);
  if (threadIdx.x == 0) {
    for (int q = 0; q < 3; ++q) mbar_init_count(S.s.mbar + q, blockDim.x / TEAMS);
    *S.s.mphase = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x < D) {
    sc[SC_Q + threadIdx.x] = __ldcg(B.ctrl + threadIdx.x);
    sc[SC_P + threadIdx.x] = __ldcg(B.ctrl + 8 + threadIdx.x);
  }
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
    load_v64<N>(P, SP, B, S);
    __syncthreads();
    pass64<N, false, SM_VONLY, false>(P, SP, B, 0, 1);
    if (!grid_sync(B, &sflag)) return;
    finish(B, S.s, 1, D + 1);
    centre_after_potential(P, S.s, RN.motion);
    if (sc[SC_ERR] != 0.0) goto done;
  }
  build_group_table<N>(P, SP, B, sc, GT_U, SP.tabT);
  if (!grid_sync(B, &sflag)) return;

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
      if (gi == ng - 1) pass64<N, false, SM_KIN, false>(P, SP, B, gi, 0);
      else pass64<N, false, SM_NONE, false>(P, SP, B, gi, 0);
      if (!grid_sync(B, &sflag)) return;
    }
    finish(B, S.s, 0, D + 1);
    centre_after_kinetic(P, S.s, RN.motion);
    if (sc[SC_ERR] != 0.0) goto done;
    if (hasv) build_v_short(P, SP, B, S.s);
    build_group_table<N>(P, SP, B, sc, GT_K, SP.tabT);
    if (final_unit) build_group_table<N>(P, SP, B, sc, GT_POST, SP.tabQ);
    if (!grid_sync(B, &sflag)) return;
    if (hasv) load_v64<N>(P, SP, B, S);
    if (threadIdx.x < D) sc[SC_Q + threadIdx.x] = sc[SC_QN + threadIdx.x];
    __syncthreads();
    // inverse transform from the group of axis 0; the potential substep is
    // fused into the pass over the group that holds the last axis
    for (int gi = ng - 1; gi >= 0; --gi) {
      const bool v = (gi == 0 && hasv);
      if (final_unit) {
        if (v) pass64<N, true, SM_V, true>(P, SP, B, gi, 1);
        else pass64<N, true, SM_NONE, true>(P, SP, B, gi, 1);
      } else {
        if (v) pass64<N, true, SM_V, false>(P, SP, B, gi, 1);
        else pass64<N, true, SM_NONE, false>(P, SP, B, gi, 1);
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
        build_group_table<N>(P, SP, B, sc, GT_REL, SP.tabT);
        if (!grid_sync(B, &sflag)) return;
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
    if (sc[SC_ERR] != 0.0) {
      atomicExch(B.status, (int)sc[SC_ERR]);
      // every CTA stopped at the same sum; the one that noted the entry may
      // have had no chunk to mark
      if (__ldcg(B.bar + BAR_BAD) != 0) ((double2*)B.psi)[0].x = __longlong_as_double(0x7ff8000000000000ll);
    }
  }
  if (threadIdx.x == 0 && sc[SC_BAD] != 0.0) atomicExch(B.status, ST_NONFINITE);
}

}  // namespace

// The kernel for axes of n points.
void* short64_kernel(int n) {
  switch (n) {
    case 8: return (void*)k_propagate_short64<8>;
    case 12: return (void*)k_propagate_short64<12>;
    case 16: return (void*)k_propagate_short64<16>;
  }
  return nullptr;
}

}  // namespace mgk
