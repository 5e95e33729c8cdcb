// 64-bit fixed-point arithmetic of the FP64 forms (host and device).
//
// GB300 issues 1.67 FP64 multiply-adds per clock and SM, but 58 64-bit integer additions, 31
// high products of 32-bit words and 24 32 x 32 + 64 multiply-adds (measured with independent
// chains on every SM).  A transform whose data are 64-bit integers with one exponent per block
// (a plane, a row, a column) therefore runs several times faster than in FP64, and the block as a
// whole is rounded more finely: blocks are scaled from the sum of the magnitudes that enter them, so
// that a unit is about 2^-60 of that sum.  A value far below its block's sum has fewer digits than
// FP64 would give it.  Integer sums are exact, so results do not depend on how the work is split.
//
// Conventions: a block value is X 2^e with X a signed 64-bit integer, |X| < 2^62 wherever a
// complex rotation follows; a block that holds an infinity or a NaN is marked (kFxNan) and
// makes every value computed from it NaN.  Subnormal FP64 inputs count as zero.
#pragma once
#include <stdint.h>

#ifndef PCF_HD
#ifdef __CUDACC__
#define PCF_HD __host__ __device__ __forceinline__
#else
#define PCF_HD inline
#endif
#endif

namespace pcf {

typedef long long fx;
struct alignas(16) fxc {
  fx x, y;
};
// Twiddle c + i s in units of 2^-62, each part split as hi 2^32 + lo (lo signed).
struct alignas(16) fxtw {
  int ch, cl, sh, sl;
};

constexpr int kFxNan = 0x40000000;   // exponent of a block that holds a NaN or an infinity
constexpr int kFxNone = -0x20000000;  // exponent of an all-zero block

PCF_HD int fx_mulhi(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((long long)a * b) >> 32);
#endif
}
// x = hi 2^32 + lo with lo a signed word
PCF_HD int fx_hi(fx x) { return (int)((x + 0x80000000LL) >> 32); }
PCF_HD int fx_lo(fx x) { return (int)(uint32_t)(uint64_t)x; }

// round(x (h 2^32 + l) 2^-62): the cross products are summed in 64 bits and rounded once; the
// product of the low words, left out, is at most one unit and zero on average.
PCF_HD fx fx_mulc(fx x, int h, int l) {
  const int xh = fx_hi(x), xl = fx_lo(x);
  const fx t = (fx)xh * l + (fx)xl * h + (1LL << 29);
  return ((fx)xh * h << 2) + (t >> 30);
}
// (a b) 2^-64 for |a|, |b| < 2^62
PCF_HD fx fx_mul64(fx a, fx b) {
  const int ah = fx_hi(a), al = fx_lo(a), bh = fx_hi(b), bl = fx_lo(b);
  const int t = fx_mulhi(ah, bl) + fx_mulhi(al, bh) + 1;
  return (fx)ah * bh + t;
}
// v w, |v| < 2^62 (the cross products sum to less than 2^63)
PCF_HD fxc fx_cmul(fxc v, fxtw w) {
  const int xh = fx_hi(v.x), xl = fx_lo(v.x), yh = fx_hi(v.y), yl = fx_lo(v.y);
  const fx tr = (fx)xh * w.cl + (fx)xl * w.ch + (fx)yh * -w.sl + (fx)yl * -w.sh + (1LL << 29);
  const fx ti = (fx)xh * w.sl + (fx)xl * w.sh + (fx)yh * w.cl + (fx)yl * w.ch + (1LL << 29);
  return fxc{(((fx)xh * w.ch + (fx)yh * -w.sh) << 2) + (tr >> 30), (((fx)xh * w.sh + (fx)yh * w.ch) << 2) + (ti >> 30)};
}
PCF_HD fxc fx_add(fxc a, fxc b) { return fxc{a.x + b.x, a.y + b.y}; }
PCF_HD fxc fx_sub(fxc a, fxc b) { return fxc{a.x - b.x, a.y - b.y}; }
// +i v (inverse transform) or -i v (forward)
template <bool INV>
PCF_HD fxc fx_i(fxc v) {
  return INV ? fxc{-v.y, v.x} : fxc{v.y, -v.x};
}

// Arithmetic shift right by r in 0..: amounts of 64 and more give 0 (the value is below a unit).
PCF_HD fx fx_sra(fx x, int r) { return r > 63 ? 0 : x >> r; }
// a 2^-r to the nearest, 0 <= a < 2^62, r >= 0; r > 63 gives 0
PCF_HD fx fx_round(fx a, int r) { return r > 63 ? 0 : (a + (fx)((1ULL << r) >> 1)) >> r; }
// r in 0..31: two shifts
PCF_HD fx fx_sra31(fx x, int r) {
#ifdef __CUDA_ARCH__
  const int lo = (int)(uint32_t)(uint64_t)x, hi = (int)(x >> 32);
  return ((fx)(hi >> r) << 32) | __funnelshift_r((unsigned)lo, (unsigned)hi, r);
#else
  return x >> r;
#endif
}
// Bits of the magnitude: |x| < 2^bits from the high word of x ^ (x >> 63).
PCF_HD uint32_t fx_maghi(fx x) {
  const int h = (int)(x >> 32);
  return (uint32_t)(h ^ (h >> 31));
}
PCF_HD int fx_clz32(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}
PCF_HD int fx_clz64(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
// |x| < 2^fx_bits(maghi): 64 - clz of the 64-bit magnitude with a low word of ones
PCF_HD int fx_bits(uint32_t maghi) { return 64 - fx_clz32(maghi); }

// Words of a matrix-vector product, x = h 2^28 + l with |l| <= 2^27: for entries up to 2^57 and columns
// whose magnitudes sum to less than 2^59 both words are 32-bit, and for up to 65 terms the sums of
// h h' (below 2^60) and of h l' + l h' (below 2^63) are exact.  l l' is left out: at most 65 2^54 of
// the 2^116 that the largest entry times the column's sum stand for, 2^-56 of it (random words: 2^-61).
// Split at 29 bits it was 2^-54.
PCF_HD void fx_words(fx x, int* h, int* l) {
  *h = (int)((x + (1 << 27)) >> 28);
  *l = (int)(x - ((fx)*h << 28));
}
// h h' and cross sums -> units of 2^55
PCF_HD fx fx_fold(fx h, fx c) { return (h << 1) + ((c + (1 << 26)) >> 27); }

// Nearest double to x 2^e, by integer instructions (an FP64 conversion and scaling occupy the
// FP64 pipe for as long as 60 integer instructions); exponents outside the normal range give
// zero or infinity.
PCF_HD uint64_t fx_double_bits(fx x, int e) {
  const uint64_t sign = (uint64_t)x & 0x8000000000000000ULL;
  uint64_t a = (uint64_t)(x ^ (x >> 63)) - (uint64_t)(x >> 63);
  if (a == 0) return 0;
  const int lz = fx_clz64(a);
  a <<= lz;
  const uint64_t r = (a >> 11) + ((a >> 10) & 1);  // 53 bits, rounded; bit 52 adds one to the exponent
  const int E = 63 - lz + e + 1022;                // biased exponent - 1
  if (E < 0) return sign;
  if (E > 2045) return sign | 0x7ff0000000000000ULL;
  return sign | (((uint64_t)E << 52) + r);
}

// ------------------------------------------------------------------ small DFTs in registers
// cos, sin in units of 2^-62, split like fxtw
constexpr int kS8h = 759250125, kS8l = -25716447;        // sqrt(1/2)
constexpr int kS3h = 929887697, kS3l = -1332128537;      // sin(pi/3)
constexpr int kC16h = 992008094, kC16l = 1696238673;     // cos(pi/8)
constexpr int kS16h = 410903207, kS16l = -1364630830;    // sin(pi/8)
constexpr int kC91h = 822533958, kC91l = -1633652124;    // cos(2 pi/9)
constexpr int kS91h = 690187940, kS91l = 2016164183;     // sin(2 pi/9)
constexpr int kC92h = 186453311, kC92l = 96060625;       // cos(4 pi/9)
constexpr int kS92h = 1057429273, kS92l = 37236404;      // sin(4 pi/9)
constexpr int kC94h = -1008987269, kC94l = 1537591498;   // cos(8 pi/9)
constexpr int kS94h = 367241333, kS94l = -1978927779;    // sin(8 pi/9)

// v exp(+-i pi/4) and v exp(+-3 i pi/4) (+ for the inverse transform)
template <bool INV>
PCF_HD fxc fx_w8(fxc v) {
  const fx a = INV ? v.x - v.y : v.x + v.y, b = INV ? v.x + v.y : v.y - v.x;
  return fxc{fx_mulc(a, kS8h, kS8l), fx_mulc(b, kS8h, kS8l)};
}
template <bool INV>
PCF_HD fxc fx_w83(fxc v) {
  const fx a = INV ? -v.x - v.y : v.y - v.x, b = INV ? v.x - v.y : -v.x - v.y;
  return fxc{fx_mulc(a, kS8h, kS8l), fx_mulc(b, kS8h, kS8l)};
}

// dft<R, INV>(v): v[k] <- sum_n v[n] exp(+-2 pi i n k/R), natural order, for R = 2, 3, 4, 6, 8, 9,
// 12, 16.  6 and 12 use the prime-factor index maps (no inner twiddles).
template <int R, bool INV>
struct FxDft;
template <bool INV>
struct FxDft<2, INV> {
  static PCF_HD void run(fxc* v) {
    const fxc a = v[0], b = v[1];
    v[0] = fx_add(a, b);
    v[1] = fx_sub(a, b);
  }
};
template <bool INV>
struct FxDft<3, INV> {
  static PCF_HD void run(fxc* v) {
    const fxc s = fx_add(v[1], v[2]), d = fx_sub(v[1], v[2]);
    // m = v0 - s/2, t = +-i sin(pi/3) d
    const fxc m{v[0].x - (s.x >> 1), v[0].y - (s.y >> 1)};
    const fxc t = fx_i<INV>(fxc{fx_mulc(d.x, kS3h, kS3l), fx_mulc(d.y, kS3h, kS3l)});
    v[0] = fx_add(v[0], s);
    v[1] = fx_add(m, t);
    v[2] = fx_sub(m, t);
  }
};
template <bool INV>
struct FxDft<4, INV> {
  static PCF_HD void run(fxc* v) {
    const fxc a = fx_add(v[0], v[2]), b = fx_sub(v[0], v[2]);
    const fxc c = fx_add(v[1], v[3]), d = fx_i<INV>(fx_sub(v[1], v[3]));
    v[0] = fx_add(a, c);
    v[1] = fx_add(b, d);
    v[2] = fx_sub(a, c);
    v[3] = fx_sub(b, d);
  }
};
template <bool INV>
struct FxDft<6, INV> {
  static PCF_HD void run(fxc* v) {
    // n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6)
    fxc a[3] = {v[0], v[2], v[4]}, b[3] = {v[3], v[5], v[1]};
    FxDft<3, INV>::run(a);
    FxDft<3, INV>::run(b);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) {
      v[(4 * k2) % 6] = fx_add(a[k2], b[k2]);
      v[(3 + 4 * k2) % 6] = fx_sub(a[k2], b[k2]);
    }
  }
};
template <bool INV>
struct FxDft<8, INV> {
  static PCF_HD void run(fxc* v) {
    fxc a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = fx_add(v[k], v[k + 4]);
      b[k] = fx_sub(v[k], v[k + 4]);
    }
    b[1] = fx_w8<INV>(b[1]);
    b[2] = fx_i<INV>(b[2]);
    b[3] = fx_w83<INV>(b[3]);
    FxDft<4, INV>::run(a);
    FxDft<4, INV>::run(b);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[2 * k] = a[k];
      v[2 * k + 1] = b[k];
    }
  }
};
template <bool INV>
struct FxDft<9, INV> {
  static PCF_HD void run(fxc* v) {
    // 3 x 3: n = 3 n1 + n2, twiddles exp(+-2 pi i n2 k1/9), k = k1 + 3 k2
    const int sg = INV ? 1 : -1;
    const fxtw w1{kC91h, kC91l, sg * kS91h, sg * kS91l}, w2{kC92h, kC92l, sg * kS92h, sg * kS92l};
    const fxtw w4{kC94h, kC94l, sg * kS94h, sg * kS94l};
    fxc q[3][3];  // [n2][k1]
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 3; ++n1) q[n2][n1] = v[3 * n1 + n2];
      FxDft<3, INV>::run(q[n2]);
    }
    q[1][1] = fx_cmul(q[1][1], w1);
    q[1][2] = fx_cmul(q[1][2], w2);
    q[2][1] = fx_cmul(q[2][1], w2);
    q[2][2] = fx_cmul(q[2][2], w4);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      fxc c[3] = {q[0][k1], q[1][k1], q[2][k1]};
      FxDft<3, INV>::run(c);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = c[k2];
    }
  }
};
template <bool INV>
struct FxDft<12, INV> {
  static PCF_HD void run(fxc* v) {
    // n = 4 n1 + 3 n2, k = 4 k1 + 9 k2 (mod 12)
    fxc q[3][4];
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) {
#pragma unroll
      for (int n2 = 0; n2 < 4; ++n2) q[n1][n2] = v[(4 * n1 + 3 * n2) % 12];
      FxDft<4, INV>::run(q[n1]);
    }
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) {
      fxc c[3] = {q[0][k2], q[1][k2], q[2][k2]};
      FxDft<3, INV>::run(c);
#pragma unroll
      for (int k1 = 0; k1 < 3; ++k1) v[(4 * k1 + 9 * k2) % 12] = c[k1];
    }
  }
};
template <bool INV>
struct FxDft<16, INV> {
  static PCF_HD void run(fxc* v) {
    // 4 x 4: columns n2 = n mod 4, twiddles exp(+-2 pi i n2 k1/16), rows
    const int sg = INV ? 1 : -1;
    const fxtw w1{kC16h, kC16l, sg * kS16h, sg * kS16l}, w3{kS16h, kS16l, sg * kC16h, sg * kC16l};
    const fxtw w9{-kC16h, -kC16l, -sg * kS16h, -sg * kS16l};
    fxc q[4][4];  // [n2][k1]
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) q[n2][n1] = v[4 * n1 + n2];
      FxDft<4, INV>::run(q[n2]);
    }
    q[1][1] = fx_cmul(q[1][1], w1);
    q[1][2] = fx_w8<INV>(q[1][2]);
    q[1][3] = fx_cmul(q[1][3], w3);
    q[2][1] = fx_w8<INV>(q[2][1]);
    q[2][2] = fx_i<INV>(q[2][2]);
    q[2][3] = fx_w83<INV>(q[2][3]);
    q[3][1] = fx_cmul(q[3][1], w3);
    q[3][2] = fx_w83<INV>(q[3][2]);
    q[3][3] = fx_cmul(q[3][3], w9);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      fxc c[4] = {q[0][k1], q[1][k1], q[2][k1], q[3][k1]};
      FxDft<4, INV>::run(c);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = c[k2];
    }
  }
};

// ------------------------------------------------------------------ transforms of a row
// A transform of length L = R S is two passes, in place: DFTs of length R over the elements n,
// n + S, .. (n < S), twiddles, and DFTs of length S over each block of S.  S = 8 wherever R = L/8 is
// one of 2, 4, 6, 8, 12, 16; the other even products of 2 and 3 up to 128 have S = 3, 6 or 9.  R is
// even: neighbouring outputs b = 2 r, 2 r + 1 of the second pass lie in the same S-strided set.
struct FxPlan {
  int R, S;
};
PCF_HD FxPlan fx_plan(int L) {
  switch (L) {
    case 18: return FxPlan{6, 3};
    case 24: return FxPlan{4, 6};
    case 36: return FxPlan{6, 6};
    case 54: return FxPlan{6, 9};
    case 72: return FxPlan{12, 6};
    case 108: return FxPlan{12, 9};
    default: return FxPlan{L >> 3, 8};
  }
}
// Slot of element (block b, member e) in a row.  S = 8: the eight lanes of a shared-memory phase
// meet eight different 16-byte bank groups in both passes without padding.
template <int S>
PCF_HD int fx_slot(int b, int e) {
  return S == 8 ? b * 8 + (e ^ (b & 7)) : b * S + e;
}

}  // namespace pcf
