// Fixed-point arithmetic for the FP64 transforms (sm_103a).
//
// The FP64 units of this GPU take 64 cycles per warp instruction, the integer
// units 2 (measured: DFMA, DADD and every conversion to or from FP64 64
// cycles per warp instruction and sub-partition; 64-bit integer add 4;
// 32 x 32 + 64 multiply-add about 4).  A DFT is mostly additions, so a block
// of the state is carried through its transforms as 64-bit integers with one
// common power-of-two scale: additions are exact, a complex multiplication by
// a table value is 12 multiply-adds, and FP64 appears only where the state is
// read and written.
//
// Scale.  A block is brought to integers whose 2-norm (over the whole block)
// is below 2^FX_BITS, from an upper bound of its norm (block_scale below).
// The transforms are unitary up to known powers of two, so the 2-norm also
// bounds every intermediate modulus: the first multiplication (|m| <= 1)
// returns half the product, so 2^61 bounds the norm after it; later ones keep
// it, and a DFT of n points returns DFT(x) / 2^S: norm factor sqrt(n) / 2^S, at
// most sqrt(12)/2 for S = 1, and at most twice the norm before the division
// (sqrt(8) times it in idft8_late).
// Every rounding of the state is to the integer grid and unbiased: a bias,
// however small beside the rounding noise, is the same vector in every pass over
// a state that changes little between passes, and adds up over thousands of
// passes.  The conversion rounds to nearest, ties and halves are decided by low
// bits of the line's own data (tie_of, LineBits), and products are corrected for
// the mean of the low parts and bits that they drop.  Only a product of two
// multipliers (cmul_m) keeps a mean of 2^-60, far below an FP64 table entry's
// rounding.  Error against 80-bit arithmetic of localised packets on moving
// grids, the FP64 units' passes -> these: 12^4 2.5e-15 -> 1.4e-15, 16^4 3.2e-15
// -> 1.0e-15, 8^5 2.2e-15 -> 1.3e-15, 64^3 2.9e-15 -> 2.4e-15, 512 x 384 1.9e-15
// -> 1.4e-15 (with truncating conversions and uncorrected bits 4.3e-15, 5.4e-15,
// 5.4e-15, 4.3e-15, 2.0e-15).
//
// Multipliers are complex numbers of modulus at most 1 in two 31-bit words
// per component: value = (h 2^31 + l) / 2^61, 0 <= l < 2^31.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mgk {
namespace {

struct I2 {
  long long x, y;
};

__host__ __device__ __forceinline__ I2 iadd(I2 a, I2 b) { return I2{a.x + b.x, a.y + b.y}; }
__host__ __device__ __forceinline__ I2 isub(I2 a, I2 b) { return I2{a.x - b.x, a.y - b.y}; }
__host__ __device__ __forceinline__ I2 ishr(I2 a, int s) { return I2{a.x >> s, a.y >> s}; }
template <bool INV> __host__ __device__ __forceinline__ I2 imul_si(I2 a) {
  return INV ? I2{-a.y, a.x} : I2{a.y, -a.x};
}
// a * b + c, one 32 x 32 + 64 multiply-add (in PTX: from C++ the compiler sees
// which factors cannot be negative and widens the product to 64 x 64)
__host__ __device__ __forceinline__ long long wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (long long)a * b + c;
#endif
}
__host__ __device__ __forceinline__ int hi32(long long a) { return (int)(a >> 32); }
__host__ __device__ __forceinline__ int lo31(long long a) { return (int)((unsigned)a >> 1); }

// (d * (h 2^31 + l)) / 2^63 for constants h, l >= 0.  With d = dh 2^32 + 2 dl + b
// the parts dl * l and b are dropped; their mean (for evenly spread low bits)
// is added with the half for rounding.
__host__ __device__ __forceinline__ long long mul_c(long long d, int h, int l) {
  const int dh = hi32(d), dl = lo31(d);
  const long long c = wide(dl, h, wide(dh, l, (1LL << 30) + (l >> 1) + (h >> 2)));
  return wide(dh, h, c >> 31);
}
constexpr int FX_BITS = 62;

// (a * b) / 2^32 + c
__host__ __device__ __forceinline__ int madhi(int a, int b, int c) {
#ifdef __CUDA_ARCH__
  int d;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
#else
  return (int)(((long long)a * b) >> 32) + c;
#endif
}

// x * m (HALF: half of it) for a multiplier m, |x| < 2^61 (2^62).  Without
// LOW the products of the low words are dropped: positive, one unit (half) on
// average, they cancel in the real part and are added to the imaginary
// part's half for rounding.  The lowest bits of x are dropped: in a value
// that comes from to_fixed that is its rounding (odd = 0), elsewhere (odd = -1)
// it takes one half on average, whose product with m, the same for every x, is
// added (to the sums of the low products; the imaginary one has to stay below
// 2^31, hence the 2^30).
template <bool HALF, bool LOW> __host__ __device__ __forceinline__ I2 cmul(I2 x, int4 m, int odd = 0) {
  constexpr int SH = HALF ? 30 : 29;
  const int rh = m.x, rl = m.y, ih = m.z, il = m.w;
  const int xh = hi32(x.x), xl = lo31(x.x), yh = hi32(x.y), yl = lo31(x.y);
  const int nh = -ih, nl = -il;
  long long cr = 1LL << (SH - 1), ci = (1LL << (SH - 1)) + (LOW ? 1LL << 31 : 1LL << 30);
  if (LOW) {
    ci = wide(madhi(xl, il, madhi(yl, rl, (((rh + ih) >> 3) & odd) - (1 << 30))), 2, ci);
    cr = wide(madhi(xl, rl, madhi(yl, nl, ((rh + nh) >> 3) & odd)), 2, cr);
  }
  cr = wide(yl, nh, wide(yh, nl, wide(xl, rh, wide(xh, rl, cr))));
  ci = wide(yl, rh, wide(yh, rl, wide(xl, ih, wide(xh, il, ci))));
  const int x4 = xh << (31 - SH), y4 = yh << (31 - SH);
  return I2{wide(y4, nh, wide(x4, rh, cr >> SH)), wide(y4, rh, wide(x4, ih, ci >> SH))};
}
// a product of multipliers, which need fewer bits
__host__ __device__ __forceinline__ I2 cmul_m(I2 x, int4 m) { return cmul<false, false>(x, m); }
__host__ __device__ __forceinline__ I2 cmul_half(I2 x, int4 m, int odd) { return cmul<true, true>(x, m, odd); }

// The multiplier words of v, scale = 2^61, and of a product held as integers
// with scale 2^60.
__host__ __device__ __forceinline__ int4 to_mult(double2 v, double scale) {
  const long long a = llrint(v.x * scale), b = llrint(v.y * scale);
  return make_int4((int)(a >> 31), (int)(a & 0x7fffffff), (int)(b >> 31), (int)(b & 0x7fffffff));
}
__host__ __device__ __forceinline__ int4 to_mult60(I2 a) {
  return make_int4((int)(a.x >> 30), (int)(((unsigned)a.x << 1) & 0x7fffffffu), (int)(a.y >> 30),
                   (int)(((unsigned)a.y << 1) & 0x7fffffffu));
}
// ---------------------------------------------------------------------------
// DFTs of a line (natural order in and out): DFT(x) / 2^S, S = 1 or 2 (16 points:
// 2)
// ---------------------------------------------------------------------------

// Low bits of a line's data that decide its ties: px, py are 1 or 2 (added
// before a division by 4: 1.5 on average), bx, by 0 or 1 (before one by 2).
struct LineBits {
  int px, py, bx, by;
};
__host__ __device__ __forceinline__ LineBits line_bits(I2 a, I2 b) {
  const unsigned r = ((unsigned)a.x ^ (unsigned)b.y) >> 1;
  return LineBits{(int)(1 + (r & 1)), (int)(1 + ((r >> 1) & 1)), (int)((r >> 2) & 1), (int)((r >> 3) & 1)};
}
template <int S> __host__ __device__ __forceinline__ I2 divide(I2 a, LineBits b) {
  return S == 2 ? I2{(a.x + b.px) >> 2, (a.y + b.py) >> 2} : I2{(a.x + b.bx) >> 1, (a.y + b.by) >> 1};
}

// four points, divided by 2^S
template <bool INV, int S>
__host__ __device__ __forceinline__ void idft4(I2& v0, I2& v1, I2& v2, I2& v3, LineBits b) {
  if (S) {
    v0.x += S == 2 ? b.px : b.bx;
    v0.y += S == 2 ? b.py : b.by;
  }
  const I2 t0 = iadd(v0, v2), t1 = isub(v0, v2);
  const I2 t2 = iadd(v1, v3), t3 = imul_si<INV>(isub(v1, v3));
  v0 = iadd(t0, t2);
  v2 = isub(t0, t2);
  v1 = iadd(t1, t3);
  v3 = isub(t1, t3);
  if (S) {
    v0 = ishr(v0, S);
    v1 = ishr(v1, S);
    v2 = ishr(v2, S);
    v3 = ishr(v3, S);
  }
}

// 1 - sqrt(3)/2, 1/(2 sqrt(2)), 1/(4 sqrt(2)) and 1 - 1/sqrt(2), times 2^63
constexpr int C3H = 575416509, C3L = 516773425;
// 1 - pi/4 and 1/3, times 2^63 (rotate_turns)
constexpr int C1MPI4H = 921707869, C1MPI4L = 1867226854;
constexpr int C13H = 1431655765, C13L = 715827883;
constexpr int C4H = 1518500249, C4L = 2121767201;
constexpr int C8H = 759250124, C8L = 2134625425;
constexpr int C2H = 1257966796, C2L = 51432894;

// three points, unscaled: v0 +- via sqrt(3)/2 d = d - (1 - sqrt(3)/2) d
template <bool INV> __host__ __device__ __forceinline__ void idft3(I2& v0, I2& v1, I2& v2, LineBits b) {
  const I2 t = iadd(v1, v2), d = isub(v1, v2);
  const I2 m = I2{v0.x - ((t.x + b.bx) >> 1), v0.y - ((t.y + b.by) >> 1)};
  const I2 e = I2{d.x - mul_c(d.x, C3H, C3L), d.y - mul_c(d.y, C3H, C3L)};
  const I2 s = imul_si<INV>(e);
  v0 = iadd(v0, t);
  v1 = iadd(m, s);
  v2 = isub(m, s);
}

template <bool INV, int N, int S> struct IDft;

// 12 = 4 x 3, Good-Thomas (no twiddles): input (3 n1 + 4 n2) mod 12, output
// (9 k1 + 4 k2) mod 12.
template <bool INV, int S> struct IDft<INV, 12, S> {
  static __host__ __device__ __forceinline__ void run(I2* x) {
    const LineBits lb = line_bits(x[1], x[5]);
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2)
      idft4<INV, S>(x[(4 * n2) % 12], x[(3 + 4 * n2) % 12], x[(6 + 4 * n2) % 12], x[(9 + 4 * n2) % 12], lb);
    // x[(3 k1 + 4 n2) % 12] holds output k1 of sub-transform n2
    I2 y[12];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      I2 a = x[(3 * k1) % 12], b = x[(3 * k1 + 4) % 12], c = x[(3 * k1 + 8) % 12];
      idft3<INV>(a, b, c, lb);
      y[(9 * k1) % 12] = a;
      y[(9 * k1 + 4) % 12] = b;
      y[(9 * k1 + 8) % 12] = c;
    }
#pragma unroll
    for (int r = 0; r < 12; ++r) x[r] = y[r];
  }
};

// 8 points, divided at the end: half the rounding noise of the form below, for
// inputs that leave room for the growth of sqrt(8).
template <bool INV, int S> __host__ __device__ __forceinline__ void idft8_late(I2* x) {
  const LineBits lb = line_bits(x[0], x[1]);
  I2 a[4], b[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    a[r] = iadd(x[r], x[r + 4]);
    b[r] = isub(x[r], x[r + 4]);
  }
  const I2 s1 = iadd(b[1], imul_si<INV>(b[1])), s3 = isub(imul_si<INV>(b[3]), b[3]);
  b[1] = I2{s1.x - mul_c(s1.x, C2H, C2L), s1.y - mul_c(s1.y, C2H, C2L)};
  b[3] = I2{s3.x - mul_c(s3.x, C2H, C2L), s3.y - mul_c(s3.y, C2H, C2L)};
  b[2] = imul_si<INV>(b[2]);
  idft4<INV, S>(a[0], a[1], a[2], a[3], lb);
  idft4<INV, S>(b[0], b[1], b[2], b[3], lb);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    x[2 * r] = a[r];
    x[2 * r + 1] = b[r];
  }
}

// 8 by one decimation-in-frequency split.  The shift follows the first
// butterflies; the 1/sqrt(2) rotations carry it in their constant.
template <bool INV, int S> struct IDft<INV, 8, S> {
  static __host__ __device__ __forceinline__ void run(I2* x) {
    const LineBits lb = line_bits(x[1], x[5]);
    I2 a[4], b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      a[r] = iadd(x[r], x[r + 4]);
      b[r] = isub(x[r], x[r + 4]);
      a[r] = divide<S>(a[r], lb);
      if ((r & 1) == 0) b[r] = divide<S>(b[r], lb);
    }
    const I2 s1 = iadd(b[1], imul_si<INV>(b[1])), s3 = isub(imul_si<INV>(b[3]), b[3]);
    constexpr int H = S == 2 ? C8H : C4H, L = S == 2 ? C8L : C4L;
    b[1] = I2{mul_c(s1.x, H, L), mul_c(s1.y, H, L)};
    b[3] = I2{mul_c(s3.x, H, L), mul_c(s3.y, H, L)};
    b[2] = imul_si<INV>(b[2]);
    idft4<INV, 0>(a[0], a[1], a[2], a[3], lb);
    idft4<INV, 0>(b[0], b[1], b[2], b[3], lb);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      x[2 * r] = a[r];
      x[2 * r + 1] = b[r];
    }
  }
};

// e^{-2 pi i m / 16} as multiplier words, m = 0 .. 9
struct Tw16 {
  int rh, rl, ih, il;
};
template <int M> __host__ __device__ __forceinline__ Tw16 tw16() {
  if (M == 1) return Tw16{992008094, 848119337, -410903207, 682315415};
  if (M == 2) return Tw16{759250124, 2134625425, -759250125, 12858223};
  if (M == 3) return Tw16{410903206, 1465168233, -992008095, 1299364311};
  if (M == 6) return Tw16{-759250125, 12858223, -759250125, 12858223};
  return Tw16{-992008095, 1299364311, 410903206, 1465168233};  // M == 9
}
// a * e^{-+2 pi i M / 16} / 4, with the mean of the dropped low parts
// (cmul_m) for these words; the conjugate's words are negated.
template <bool INV, int M> __host__ __device__ __forceinline__ I2 twmul16(I2 a) {
  const Tw16 w = tw16<M>();
  const int rh = w.rh, rl = w.rl, ih = INV ? -w.ih : w.ih, il = INV ? -w.il : w.il;
  const int xh = hi32(a.x), xl = lo31(a.x), yh = hi32(a.y), yl = lo31(a.y);
  const long long kr = (1LL << 30) + (rl - (long long)il) / 2 + (rh - (long long)ih) / 4;
  const long long ki = (1LL << 30) + (rl + (long long)il) / 2 + (rh + (long long)ih) / 4;
  const long long cr = wide(yl, -ih, wide(yh, -il, wide(xl, rh, wide(xh, rl, kr))));
  const long long ci = wide(yl, rh, wide(yh, rl, wide(xl, ih, wide(xh, il, ki))));
  return I2{wide(yh, -ih, wide(xh, rh, cr >> 31)), wide(yh, rh, wide(xh, ih, ci >> 31))};
}

// 16 = 4 x 4 with twiddles, which carry the division by 4.
template <bool INV> struct IDft<INV, 16, 2> {
  static __host__ __device__ __forceinline__ void run(I2* x) {
    const LineBits lb = line_bits(x[1], x[5]);
    // column 0 has no twiddles
    idft4<INV, 2>(x[0], x[4], x[8], x[12], lb);
    idft4<INV, 0>(x[1], x[5], x[9], x[13], lb);
    idft4<INV, 0>(x[2], x[6], x[10], x[14], lb);
    idft4<INV, 0>(x[3], x[7], x[11], x[15], lb);
    // x[n2 + 4 k1]: output k1 of column n2, twiddle W^(n2 k1)
#pragma unroll
    for (int n2 = 1; n2 < 4; ++n2) x[n2] = divide<2>(x[n2], lb);
    x[5] = twmul16<INV, 1>(x[5]);
    x[9] = twmul16<INV, 2>(x[9]);
    x[13] = twmul16<INV, 3>(x[13]);
    x[6] = twmul16<INV, 2>(x[6]);
    x[10] = imul_si<INV>(divide<2>(x[10], lb));
    x[14] = twmul16<INV, 6>(x[14]);
    x[7] = twmul16<INV, 3>(x[7]);
    x[11] = twmul16<INV, 6>(x[11]);
    x[15] = twmul16<INV, 9>(x[15]);
    I2 y[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      I2 a = x[4 * k1], b = x[4 * k1 + 1], c = x[4 * k1 + 2], d = x[4 * k1 + 3];
      idft4<INV, 0>(a, b, c, d, lb);
      y[k1] = a;
      y[k1 + 4] = b;
      y[k1 + 8] = c;
      y[k1 + 12] = d;
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = y[r];
  }
};

// ---------------------------------------------------------------------------
// FP64 <-> integers at a block's scale
// ---------------------------------------------------------------------------

// One word of an FP64 value: hi (sign, exponent, 20 mantissa bits).
constexpr int FX_EMIN = 128;  // smallest exponent field a scale is formed from

// Contribution of a group of values with the largest |hi| word `m` to a
// warp's record: the exponent field and, relative to it, a 9-bit mantissa
// rounded up.  Squares of these summed over a warp bound the warp's norm:
// every value of a group is below (mantissa + 1) 2^(exponent - 1031).
__host__ __device__ __forceinline__ int fx_exponent(unsigned m) {
  const int e = (int)(m >> 20);
  return e < FX_EMIN ? FX_EMIN : e;
}
__host__ __device__ __forceinline__ unsigned fx_square(unsigned m, int emax) {
  const int e = fx_exponent(m);  // an empty or next to empty group adds a unit
  const unsigned a = ((m >> 12) & 0xffu) + 257u;  // 1.mantissa 2^8, rounded up
  const int d = 2 * (emax - e);
  return d < 20 ? ((a * a) >> d) + 1u : 1u;
}

// REF: right-shift of a mantissa moved to bits 10..62 is REF - (its exponent field).
struct BlockScale {
  int ref;     // see to_fixed
  int eo;      // value = integer * 2^eo
  int poison;  // an infinity or NaN is in the block
  int spare;   // the norm is below 2^(bits - spare / 2)
};
// From the largest exponent field E and the sum Y of the groups' squares
// relative to it (each group of `vals` values): norm < 2^(E - 1031 + half).
__host__ __device__ __forceinline__ BlockScale block_scale(int E, unsigned Y, int vals, int bits) {
  const unsigned y = Y * (unsigned)vals;
  int lg = 0;
#ifdef __CUDA_ARCH__
  lg = 32 - __clz((int)y);
#else
  while (lg < 32 && (y >> lg)) ++lg;
#endif
  const int half = (lg + 1) >> 1;
  BlockScale s;
  s.ref = 54 - bits + E + half;
  s.eo = E - 1031 + half - bits;
  s.poison = E >= 2047;
  s.spare = lg & 1;
  return s;
}

// FP64 value (as its two words) to an integer at the block's scale whose lowest
// bit is to be dropped, as the multiplications do: that leaves the nearest even
// integer.  A tie goes away from zero for tie = 0, towards it for tie = 1
// (tie_of: by a low bit of the line's data); the ten spare bits below the
// mantissa keep everything else from being moved by it.  The mean error is zero:
// cut off towards zero, it would be a vector that is the same in every pass, and
// add up.
__host__ __device__ __forceinline__ long long to_fixed(int hi, unsigned lo, int ref, int tie) {
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const long long m = (long long)((((unsigned long long)mh << 32) | lo) << 10);
  // above 63 the value is zero; below zero only for a value above the bound
  // (an infinity or NaN as a multiplier, which its reader notes: SC_BAD)
  unsigned sh = (unsigned)(ref - (int)(((unsigned)hi >> 20) & 0x7ffu));
  sh = sh > 63u ? 63u : sh;
  const long long s = (long long)(hi >> 31);
  return (((m - tie) ^ s) >> sh) + 1;
}
__host__ __device__ __forceinline__ I2 to_fixed(I2 v, int ref, int tie) {
  return I2{to_fixed(hi32(v.x), (unsigned)v.x, ref, tie), to_fixed(hi32(v.y), (unsigned)v.y, ref, tie)};
}
__host__ __device__ __forceinline__ int tie_of(I2 a, I2 b) { return (int)(((unsigned)a.x ^ (unsigned)b.y) & 1u); }
#ifdef __CUDACC__
// An infinity or NaN, which multiplier words cannot carry: where a phase
// overflows its table entries are NaN.  Whoever turns such an entry into words
// notes it in its CTA's SC_BAD, and in word BAR_BAD of the launch's barrier
// block if other CTAs read the words.  From then on its passes write NaN, as
// the products with the entry would be, and its next sum, NaN too, ends the
// launch.
constexpr int SC_BAD = 37;
constexpr int BAR_BAD = 32;
__device__ __forceinline__ bool noted_bad(const double* sc) { return __double2hiint(sc[SC_BAD]) != 0; }
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }
__device__ __forceinline__ bool not_finite(double2 v) { return not_finite(v.x) || not_finite(v.y); }
// integer * 2^eo: converted by the FP64 unit (rounded to nearest), then the
// exponent field is moved; zero stays zero.
__device__ __forceinline__ double from_fixed(long long v, int eo) {
  const double d = (double)v;
  int h = __double2hiint(d);
  if (h != 0) h += eo << 20;
  return __hiloint2double(h, __double2loint(d));
}
__device__ __forceinline__ double2 from_fixed2(I2 v, int eo) {
  return make_double2(from_fixed(v.x, eo), from_fixed(v.y, eo));
}
#endif

}  // namespace
}  // namespace mgk
