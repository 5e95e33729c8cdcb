// The per-mode work of the FP64 forms in 64-bit fixed point: Chebyshev analysis, dense Stokes
// solve and Chebyshev synthesis (paper §4, steps 1-5).
//
//   k_yana_fx    CTA (instance, tile of modes, component): coefficients of the products
//   k_ysynth_fx  CTA (instance, tile of modes, field): values and y-derivative values at the
//                Gauss-Lobatto points
//   k_ysolve_fx  CTA (group of instances, mode): right-hand side, dense Stokes operators of both
//                parity groups, xi = -dv/dy, assembly, finite-difference quotient and update
//   k_ystep_fx   CTA (group of instances, mode): the three in one, intermediates in shared memory
//   k_ysolve_f64 CTA (group of instances, mode): the solve of a given right-hand side, in FP64
//
// Every product is a matrix (the same for all columns of a CTA) times columns.  A column's
// values are integers of one exponent, scaled so that the sum of their magnitudes is just below
// 2^59, and split into two words, x = xh 2^28 + xl; a matrix row's entries are at most 2^57, split the
// same way.  A product element is
//   2^56 sum(ah xh) + 2^28 sum(ah xl + al xh)
// with both sums exact in 64 bits for up to 65 terms (fx_words): three 32 x 32 + 64 multiply-adds per
// term, 0.12 clocks of an SM where an FP64 multiply-add takes 0.60.  In units of (largest entry of the
// row) x (sum of the column's magnitudes) the entries are rounded at 2^-58, the column is cut at
// 2^-59, the words' low product is at most 2^-56 (typically 2^-61) and the result's unit is 2^-61:
// finer than FP64's rounding of the largest terms, but the same for every element, so that a
// coefficient far below its column's sum has fewer digits than FP64 would give it.
// Scaling from the sum, and not from K times the largest value, is what keeps the solve's error
// at FP64's: r1 = (u+ - u)/dt cancels the leading digits of u+.  Sums are exact, so every
// organisation gives the same bits.
//
// A thread computes two rows of one complex column (12 multiply-adds per term on one 16-byte
// matrix load, through the read-only cache: the matrices stay in L1 and L2, and one 16-byte
// shared-memory load).  What bounds the kernels at small grids is latency (a handful of
// phases between barriers), at large ones the multiply-adds and, in the solve of a single
// instance, the operators streamed from HBM (16 bytes per two entries).
// Measured (us per launch, FP64 -> now): 32 x 33 x 32, batch 8: analysis 20 -> 12, solves 29 / 30 ->
// 20 / 20, synthesis 28 -> 20; 128 x 97 x 128: 199 -> 68, 289 / 327 (sweeps) -> 139 / 139, 310 -> 121.
#include <algorithm>

#include "pcf_fx.cuh"
#include "pcf_kernels.cuh"

namespace pcf {

namespace {

__device__ __forceinline__ int ec_of(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ fx neg_if(fx a, int hi) {
  const fx m = (fx)(hi >> 31);
  return (a ^ m) - m;
}
// Scale of a column part: the largest biased exponent ecm of its values and S, the sum of their
// magnitudes rounded up in units of 2^(ecm - 1037); q = ecm + bit length of S, so that the sum
// is below 2^(q - 1037).
__device__ __forceinline__ int scale_of(int ecm, int S) { return ecm >= 0x7ff ? kFxNan : ecm + 32 - __clz(S); }
// magnitude of a value (mantissa of the high word hi, times 2n/2^ceil(log2 2n) when n > 0) in those units,
// rounded up; eb: its biased exponent bound
__device__ __forceinline__ int mag(int hi, int n, int eb, int ecm) {
  unsigned m = (((hi & 0xfffff) | 0x100000) >> 6) + 1;
  if (n > 0) m = ((m * (2 * n)) >> (32 - __clz(2 * n - 1))) + 1;
  const int d = ecm - eb;
  return eb <= 0 || d > 27 ? 0 : (int)(m >> d) + 1;
}
// v in units of 2^(q - 1096), to the nearest: the sum of the column's magnitudes is below 2^59
__device__ __forceinline__ fx col_fx(double v, int q) {
  const int hi = __double2hiint(v), ec = (hi >> 20) & 0x7ff, r = q - 15 - ec;
  const fx m = ((fx)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  return neg_if(ec == 0 || r > 63 ? 0 : (m << 6) >> r, hi);
}
// exponent of a product's unit: the column's plus the row's
__device__ __forceinline__ int dot_exp(int q, int row) { return q == kFxNan ? kFxNan : q - 1096 + row; }
__device__ __forceinline__ double fx_out(fx s, int e) {
  return e > kFxNan / 2 ? __longlong_as_double(0x7ff8000000000000LL)
                        : __longlong_as_double((long long)fx_double_bits(s, e));
}
__device__ __forceinline__ int4 limbs(fx re, fx im) {
  int4 w;
  fx_words(re, &w.x, &w.y);
  fx_words(im, &w.z, &w.w);
  return w;
}
// sums of two rows (0, 1) x (re, im): high and cross products
struct Acc {
  fx h0 = 0, h1 = 0, h2 = 0, h3 = 0, c0 = 0, c1 = 0, c2 = 0, c3 = 0;
};
__device__ __forceinline__ void mac(Acc& a, int4 m, int4 x) {
  a.h0 += (fx)m.x * x.x;
  a.c0 += (fx)m.x * x.y;
  a.c0 += (fx)m.y * x.x;
  a.h1 += (fx)m.x * x.z;
  a.c1 += (fx)m.x * x.w;
  a.c1 += (fx)m.y * x.z;
  a.h2 += (fx)m.z * x.x;
  a.c2 += (fx)m.z * x.y;
  a.c2 += (fx)m.w * x.x;
  a.h3 += (fx)m.z * x.z;
  a.c3 += (fx)m.z * x.w;
  a.c3 += (fx)m.w * x.z;
}
// rows 2 rp, 2 rp + 1 of a matrix (column k at A + k hp + rp) times column x (element k at x + k s)
__device__ __forceinline__ Acc dot(const int4* __restrict__ A, int hp, const int4* x, int s, int K) {
  Acc a;
  int k = 0;
  for (; k + 4 <= K; k += 4) {
    int4 m[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) m[u] = __ldg(A + (k + u) * hp);
#pragma unroll
    for (int u = 0; u < 4; ++u) mac(a, m[u], x[(k + u) * s]);
  }
  for (; k < K; ++k) mac(a, __ldg(A + k * hp), x[k * s]);
  return a;
}

// one row and one part: A and x already at the row's and the part's words
__device__ __forceinline__ fx dot_fine(const int2* __restrict__ A, int sa, const int2* x, int s, int K) {
  fx h = 0, c = 0;
  int k = 0;
  for (; k + 4 <= K; k += 4) {
    int2 m[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) m[u] = __ldg(A + (k + u) * sa);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int2 v = x[(k + u) * s];
      h += (fx)m[u].x * v.x;
      c += (fx)m[u].x * v.y;
      c += (fx)m[u].y * v.x;
    }
  }
  for (; k < K; ++k) {
    const int2 m = __ldg(A + k * sa), v = x[k * s];
    h += (fx)m.x * v.x;
    c += (fx)m.x * v.y;
    c += (fx)m.y * v.x;
  }
  return fx_fold(h, c);
}
__device__ __forceinline__ const int2* words(const int4* p, int half) { return reinterpret_cast<const int2*>(p) + half; }

// Tables of one grid (FxCheb): Ae, Ao (analysis), Ce, Co (synthesis), columns k, row pairs
struct FxTab {
  int H, half, hE, hO;
  PCF_HD FxTab(int N) : H(N / 2 + 1), half(N / 2), hE((N / 2 + 2) / 2), hO((N / 2 + 1) / 2) {}
  PCF_HD int Ae() const { return 0; }
  PCF_HD int Ao() const { return H * hE; }
  PCF_HD int Ce() const { return Ao() + half * hO; }
  PCF_HD int Co() const { return Ce() + H * hE; }
};

// Columns of a CTA: element (row n, column col) of an array at n * pitch + col.
struct Cols {
  int n, pitch;  // columns, pitch
  unsigned mul;  // quotients by n
  __device__ __forceinline__ Cols(int n_, int p_) : n(n_), pitch(p_), mul(0xffffffffu / (unsigned)n_ + 1u) {}
  __device__ __forceinline__ int row(int t) const { return n == 1 ? t : (int)__umulhi((unsigned)t, mul); }
};

// Column scales in shared memory: cm[2 col + part] the largest biased exponent, cs[..] the sum.
__device__ __forceinline__ void col_max(int* cm, int col, int er, int ei) {
  if (er > 0) atomicMax(cm + 2 * col, er);
  if (ei > 0) atomicMax(cm + 2 * col + 1, ei);
}
__device__ __forceinline__ void col_sum(const int* cm, int* cs, int col, double2 v, int n, int er, int ei) {
  const int a = mag(__double2hiint(v.x), n, er, cm[2 * col]), b = mag(__double2hiint(v.y), n, ei, cm[2 * col + 1]);
  if (a) atomicAdd(cs + 2 * col, a);
  if (b) atomicAdd(cs + 2 * col + 1, b);
}
__device__ __forceinline__ void clear_max(int* cm, int n) {
  for (int t = threadIdx.x; t < n; t += blockDim.x) cm[t] = 0;
}
// After the maxima of raw values X (rows 0 .. N): their sums, then the scales q in place of cm (a
// barrier on entry, barriers within; deriv: of 2 n a_n).
__device__ __forceinline__ int ec_2n(double a, int n);
__device__ __forceinline__ void col_scales(const double2* X, const Cols& C, int N, int* cm, int* cs, bool deriv) {
  __syncthreads();
  for (int t = threadIdx.x; t < C.n * (N + 1); t += blockDim.x) {
    const int n = C.row(t), col = t - n * C.n;
    const double2 a = X[n * C.pitch + col];
    if (deriv) col_sum(cm, cs, col, a, n, ec_2n(a.x, n), ec_2n(a.y, n));
    else col_sum(cm, cs, col, a, 0, ec_of(a.x), ec_of(a.y));
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * C.n; t += blockDim.x) cm[t] = scale_of(cm[t], cs[t]);
  __syncthreads();
}

// ---------------------------------------------------------------- analysis
// Raw values (row j = node j) -> folded limbs in place: P_j = V_j + V_{N-j} at row j (j <= N/2),
// Q_j = V_j - V_{N-j} at row N - j (their magnitudes sum to at most those of V).  cm: scales.
__device__ __forceinline__ void ana_fold(double2* X, const Cols& C, int N, const int* cm) {
  const int half = N / 2;
  for (int t = threadIdx.x; t < C.n * (half + 1); t += blockDim.x) {
    const int j = C.row(t), col = t - j * C.n;
    double2* p = X + j * C.pitch + col;
    double2* q = X + (N - j) * C.pitch + col;
    const int er = cm[2 * col], ei = cm[2 * col + 1];
    const double2 a = *p;
    const fx ar = col_fx(a.x, er), ai = col_fx(a.y, ei);
    if (j == half) {
      *reinterpret_cast<int4*>(p) = limbs(ar, ai);
    } else {
      const double2 b = *q;
      const fx br = col_fx(b.x, er), bi = col_fx(b.y, ei);
      *reinterpret_cast<int4*>(p) = limbs(ar + br, ai + bi);
      *reinterpret_cast<int4*>(q) = limbs(ar - br, ai - bi);
    }
  }
}
// Coefficient n of column col, part p, goes to out(col, n)[p].  fine: a thread computes one row
// and one part (where a CTA has more threads than row pairs), else two rows and both parts.
template <class OUT>
__device__ __forceinline__ void ana_mac(const double2* X, const Cols& C, int N, const int4* tab, int ea, const int* cm,
                                        bool fine, const OUT& out) {
  const FxTab T(N);
  const int4* x0 = reinterpret_cast<const int4*>(X);
  if (fine) {
    for (int t = threadIdx.x; t < 2 * C.n * (N + 1); t += blockDim.x) {
      const int n = C.row(t >> 1), part = t & 1, col = (t >> 1) - n * C.n, r = n >> 1;
      const fx v = n & 1 ? dot_fine(words(tab + T.Ao() + (r >> 1), r & 1), 2 * T.hO,
                                    words(x0 + N * C.pitch + col, part), -2 * C.pitch, T.half)
                         : dot_fine(words(tab + T.Ae() + (r >> 1), r & 1), 2 * T.hE, words(x0 + col, part), 2 * C.pitch, T.H);
      reinterpret_cast<double*>(out(col, n))[part] = fx_out(v, dot_exp(cm[2 * col + part], ea));
    }
    return;
  }
  for (int t = threadIdx.x; t < C.n * (T.hE + T.hO); t += blockDim.x) {
    const int rs = C.row(t), col = t - rs * C.n;
    const bool even = rs < T.hE;
    const int rp = even ? rs : rs - T.hE;
    // P_j at row j upwards, Q_j at row N - j downwards
    const Acc a = even ? dot(tab + T.Ae() + rp, T.hE, x0 + col, C.pitch, T.H)
                       : dot(tab + T.Ao() + rp, T.hO, x0 + N * C.pitch + col, -C.pitch, T.half);
    const int er = dot_exp(cm[2 * col], ea), ei = dot_exp(cm[2 * col + 1], ea);
    const int n0 = 4 * rp + (even ? 0 : 1), rows = even ? T.H : T.half;
    *out(col, n0) = make_double2(fx_out(fx_fold(a.h0, a.c0), er), fx_out(fx_fold(a.h1, a.c1), ei));
    if (2 * rp + 1 < rows)
      *out(col, n0 + 2) = make_double2(fx_out(fx_fold(a.h2, a.c2), er), fx_out(fx_fold(a.h3, a.c3), ei));
  }
}

// ---------------------------------------------------------------- synthesis
// biased exponent bound of 2 n a
__device__ __forceinline__ int ec_2n(double a, int n) {
  const int e = ec_of(a);
  return e == 0 || n == 0 ? 0 : e == 0x7ff ? 0x7ff : min(e + 32 - __clz(2 * n - 1), 0x7fe);
}
// 2 n v in units of 2^(q - 1098): the magnitudes of the column's 2 n a_n sum to less than 2^61
__device__ __forceinline__ fx deriv_fx(double v, int n, int q) {
  const int hi = __double2hiint(v), ec = (hi >> 20) & 0x7ff, r = q - 23 - ec;
  const fx m = (((fx)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v)) * (2 * n);
  return neg_if(ec == 0 || r > 63 ? 0 : r >= 0 ? m >> r : m << -r, hi);
}
// Coefficients b of d/dy from t_n = 2 n a_n (integers at row n): suffix sums of a parity class,
// one thread per (column, part, class); b_n goes to row n + 1, the chain's own.  bits: largest
// bit length of the sum of |b| / 2^8 per column and part.
__device__ __forceinline__ void deriv_chains(fx* X, const Cols& C, int N, int* bits) {
  const int half = N / 2;
  for (int t = threadIdx.x; t < 4 * C.n; t += blockDim.x) {
    const int q = C.row(t), col = t - q * C.n, part = q & 1, odd = q >> 1;
    fx* x = X + 2 * col + part;
    fx acc = 0, sum = 0;
#pragma unroll 4
    for (int i = half - 1; i >= 0; --i) {
      fx* e = x + 2 * C.pitch * (2 * i + 1 + odd);  // t_{2i+1} -> b_{2i}; t_{2i+2} -> b_{2i+1}
      acc += *e;
      if (i == 0 && !odd) acc >>= 1;  // b_0 counts half
      *e = acc;
      sum += ((acc ^ (acc >> 63)) >> 8) + 1;
    }
    if (bits) atomicMax(bits + 2 * col + part, 64 - fx_clz64((uint64_t)sum));
  }
}
// the right shift that brings the sum of |b| of both classes below 2^59
__device__ __forceinline__ int deriv_shift(int bits) { return max(0, bits + 9 - 59); }
// limbs of plain coefficients in place
__device__ __forceinline__ void syn_limbs(double2* X, const Cols& C, int N, const int* cm) {
  for (int t = threadIdx.x; t < C.n * (N + 1); t += blockDim.x) {
    const int n = C.row(t), col = t - n * C.n;
    double2* p = X + n * C.pitch + col;
    const double2 a = *p;
    *reinterpret_cast<int4*>(p) = limbs(col_fx(a.x, cm[2 * col]), col_fx(a.y, cm[2 * col + 1]));
  }
}
// raw coefficients a -> limbs of the derivative's b in place (three phases); cm: scales of 2 n a_n
__device__ __forceinline__ void syn_deriv(double2* X, const Cols& C, int N, const int* cm, int* bits) {
  for (int t = threadIdx.x; t < C.n * (N + 1); t += blockDim.x) {
    const int n = C.row(t), col = t - n * C.n;
    double2* p = X + n * C.pitch + col;
    const double2 a = *p;
    *reinterpret_cast<longlong2*>(p) = make_longlong2(deriv_fx(a.x, n, cm[2 * col]), deriv_fx(a.y, n, cm[2 * col + 1]));
  }
  __syncthreads();
  deriv_chains(reinterpret_cast<fx*>(X), C, N, bits);
  __syncthreads();
  for (int t = threadIdx.x; t < C.n * (N + 1); t += blockDim.x) {
    const int n = C.row(t), col = t - n * C.n;
    double2* p = X + n * C.pitch + col;
    const longlong2 b = *reinterpret_cast<longlong2*>(p);
    const int sr = deriv_shift(bits[2 * col]), si = deriv_shift(bits[2 * col + 1]);
    *reinterpret_cast<int4*>(p) = limbs((b.x + ((1LL << sr) >> 1)) >> sr, (b.y + ((1LL << si) >> 1)) >> si);
  }
}
// put(col, j, part, value at y_j) for all nodes; deriv: columns of b (row n + 1)
template <class OUT>
__device__ __forceinline__ void syn_mac(const double2* X, const Cols& C, int N, const int4* tab, bool deriv,
                                        const int* cm, const int* bits, bool fine, const OUT& put) {
  const FxTab T(N);
  const int4* x0 = reinterpret_cast<const int4*>(X) + (deriv ? C.pitch : 0);
  // synthesis entries are in units of 2^-57, a product's unit is 2^55; b: 2^(q - 1098) before the shift
  const auto unit = [&](int k) { return dot_exp(cm[k], -2) + (deriv ? deriv_shift(bits[k]) - 2 : 0); };
  const int KE = deriv ? T.half : T.H;
  if (fine) {
    for (int t = threadIdx.x; t < 2 * C.n * T.H; t += blockDim.x) {
      const int j = C.row(t >> 1), part = t & 1, col = (t >> 1) - j * C.n;
      const fx e = dot_fine(words(tab + T.Ce() + (j >> 1), j & 1), 2 * T.hE, words(x0 + col, part), 4 * C.pitch, KE);
      const fx o = dot_fine(words(tab + T.Co() + (j >> 1), j & 1), 2 * T.hE, words(x0 + C.pitch + col, part), 4 * C.pitch, T.half);
      const int u = unit(2 * col + part);
      put(col, j, part, fx_out(e + o, u));
      if (j < T.half) put(col, N - j, part, fx_out(e - o, u));
    }
    return;
  }
  for (int t = threadIdx.x; t < C.n * T.hE; t += blockDim.x) {
    const int rp = C.row(t), col = t - rp * C.n;
    const Acc e = dot(tab + T.Ce() + rp, T.hE, x0 + col, 2 * C.pitch, KE);
    const fx e0 = fx_fold(e.h0, e.c0), e1 = fx_fold(e.h1, e.c1), e2 = fx_fold(e.h2, e.c2), e3 = fx_fold(e.h3, e.c3);
    const Acc o = dot(tab + T.Co() + rp, T.hE, x0 + C.pitch + col, 2 * C.pitch, T.half);
    const fx o0 = fx_fold(o.h0, o.c0), o1 = fx_fold(o.h1, o.c1), o2 = fx_fold(o.h2, o.c2), o3 = fx_fold(o.h3, o.c3);
    const int er = unit(2 * col), ei = unit(2 * col + 1), j = 2 * rp;
    put(col, j, 2, fx_out(e0 + o0, er), fx_out(e1 + o1, ei));
    if (j < T.half) put(col, N - j, 2, fx_out(e0 - o0, er), fx_out(e1 - o1, ei));
    if (j + 1 < T.H) {
      put(col, j + 1, 2, fx_out(e2 + o2, er), fx_out(e3 + o3, ei));
      if (j + 1 < T.half) put(col, N - j - 1, 2, fx_out(e2 - o2, er), fx_out(e3 - o3, ei));
    }
  }
}
// part 0 or 1: the real or imaginary part x; part 2: both
__device__ __forceinline__ void put_part(double2* d, int part, double x, double y) {
  if (part == 2) *d = make_double2(x, y);
  else reinterpret_cast<double*>(d)[part] = x;
}

// ---------------------------------------------------------------- Stokes solve
// -x when neg, on the integer pipe
__device__ __forceinline__ double flip(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}
// One mode, nI instances (columns).  coef(i, c, n, part): Chebyshev coefficient of the products.  C3, R3: [3][ny][nI] arrays; sm_i: 16 nI ints.  done(i, c, n, part, new value) receives
// r1 (PHI), the updated state (PSI_UPDATE) or f.  alive: false in every thread when live is all zero.
template <class COEF, class DONE>
__device__ __forceinline__ void solve_mode(const Inst* insts, int first, int nI, int m, int op, int sig, bool alive, const int* live,
                                           double2* C3, double2* R3, int* sm_i, bool fine, const COEF& coef, const DONE& done) {
  const Inst& I0 = insts[first];
  const int N = I0.N, ny = I0.ny, nm = I0.nmodes, Mz = I0.Mz, Mh = N / 2 + 1, hp = (Mh + 1) / 2;
  const Cols C(nI, nI), CN(ny, ny);
  const int AS = ny * nI;  // between the three arrays
  int* cm = sm_i;            // [3][2 nI] scales of f_v, g, h
  int* ct = sm_i + 6 * nI;   // [2 nI] of 2 n v
  int* cs = sm_i + 8 * nI;   // sums: of the three, then of 2 n v
  clear_max(sm_i, 16 * nI);
  const int ix = m / Mz, pz = m - ix * Mz;
  const double kx = I0.kx[ix], kz = I0.kz[pz];
  const bool mean = m == 0;
  const double ist = sig == 0 ? I0.inv_dt : I0.inv_dtau_hat;
  const bool in_u = op == MODE_PHI;
  if (!__syncthreads_or(alive)) return;
  // S = state/step + product; f_v = S_v, g = i (kx S_u + kz S_w), h = i (kz S_u - kx S_w); mean
  // mode: S_u and S_w (all times nu: the factor 1/nu is in the outputs)
  // One thread per (instance, n, part): an FP64 instruction occupies its quarter of the SM for 77
  // clocks whatever its active lanes, so the parts go to different lanes.
  for (int t = threadIdx.x; t < 2 * nI * ny; t += blockDim.x) {
    const int i = CN.row(t >> 1), part = t & 1, n = (t >> 1) - i * ny;
    const Inst& I = insts[first + i];
    const double* st = reinterpret_cast<const double*>((in_u ? I.uhat : I.rhat) + (size_t)m * ny + n);
    const auto S = [&](int c, int p) { return fma(st[2 * ((size_t)c * nm * ny) + p], ist, coef(i, c, n, p)); };
    double a, g, h;
    if (mean) {
      a = S(0, part);
      g = S(2, part);
      h = 0.0;
    } else {
      const double u = S(0, 1 - part), w = S(2, 1 - part), kxg = flip(kx, !part), kzg = flip(kz, !part);
      a = S(1, part);
      g = fma(kxg, u, kzg * w);
      h = fma(kzg, u, -kxg * w);
    }
    double* o = reinterpret_cast<double*>(C3 + n * nI + i) + part;
    o[0] = a;
    o[2 * AS] = g;
    o[4 * AS] = h;
    int* q = cm + 2 * i + part;
    if (ec_of(a)) atomicMax(q, ec_of(a));
    if (ec_of(g)) atomicMax(q + 2 * nI, ec_of(g));
    if (ec_of(h)) atomicMax(q + 4 * nI, ec_of(h));
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 3 * AS; t += blockDim.x) {
    const int rn = C.row(t), i = t - rn * nI, T = CN.row(rn);
    const double2 a = C3[t];
    col_sum(cm + 2 * nI * T, cs + 2 * nI * T, i, a, 0, ec_of(a.x), ec_of(a.y));
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 6 * nI; t += blockDim.x) cm[t] = scale_of(cm[t], cs[t]);
  __syncthreads();
  for (int t = threadIdx.x; t < 3 * AS; t += blockDim.x) {
    const int rn = C.row(t), i = t - rn * nI, T = CN.row(rn);
    const double2 a = C3[t];
    const int* e = cm + 2 * nI * T + 2 * i;
    reinterpret_cast<int4*>(C3)[t] = limbs(col_fx(a.x, e[0]), col_fx(a.y, e[1]));
  }
  __syncthreads();
  // products: type 0 Av f_v, 1 Ag g, 2 Eh h per parity group; mean mode: Eh S_u, Eh S_w
  const int4* D = I0.fxD[sig] + (size_t)m * 6 * Mh * hp;
  const int* De = I0.fxDe[sig] + (size_t)m * 12 * hp;
  const int4* X = reinterpret_cast<const int4*>(C3);
  const Cols CB(hp, hp);
  for (int t0 = threadIdx.x; t0 < ((mean ? 4 : 6) * hp * nI) << (fine ? 2 : 0); t0 += blockDim.x) {
    const int t = fine ? t0 >> 2 : t0, sub = t0 & 3;
    const int rs = C.row(t), i = t - rs * nI, bl = CB.row(rs), rp = rs - bl * hp, g = bl & 1, T = bl >> 1;
    const int cls = mean ? g : T == 0 ? g : 1 - g;        // class of the input
    const int ocl = mean || T < 2 ? g : 1 - g;             // class of the output
    const int K = (N - cls) / 2 + 1, rows = (N - ocl) / 2 + 1;
    const int4* A = D + (size_t)(g * 3 + (mean ? 2 : T)) * Mh * hp + rp;
    const int4* x = X + T * AS + cls * nI + i;
    longlong2* o = reinterpret_cast<longlong2*>(R3) + T * AS + i + (ocl + 4 * rp) * nI;
    if (fine) {
      if (2 * rp + (sub >> 1) < rows)
        reinterpret_cast<fx*>(o + (sub >> 1) * 2 * nI)[sub & 1] =
            dot_fine(words(A, sub >> 1), 2 * hp, words(x, sub & 1), 4 * nI, K);
      continue;
    }
    if (2 * rp >= rows) continue;
    const Acc a = dot(A, hp, x, 2 * nI, K);
    o[0] = make_longlong2(fx_fold(a.h0, a.c0), fx_fold(a.h1, a.c1));
    if (2 * rp + 1 < rows) o[2 * nI] = make_longlong2(fx_fold(a.h2, a.c2), fx_fold(a.h3, a.c3));
  }
  __syncthreads();
  // v = Av f_v + Ag g at the larger exponent, eta; as doubles in R3[0], R3[2] (mean: u, w)
  for (int t0 = threadIdx.x; t0 < 2 * AS; t0 += blockDim.x) {
    const int t = t0 >> 1, part = t0 & 1, n = C.row(t), i = t - n * nI, g = n & 1, r = n >> 1;
    fx* R = reinterpret_cast<fx*>(R3) + t0;
    const fx a0 = R[0], a1 = R[2 * AS], a2 = R[4 * AS];
    const int e0 = dot_exp(cm[2 * i + part], De[(g * 3 + (mean ? 2 : 0)) * 2 * hp + r]);
    const int e1 = dot_exp(cm[2 * nI + 2 * i + part], De[(g * 3 + (mean ? 2 : 1)) * 2 * hp + r]);
    double v, q;
    if (mean) {
      v = fx_out(a0, e0);
      q = fx_out(a1, e1);
    } else {
      const int e = max(e0, e1);
      v = fx_out((a0 >> min(e - e0, 63)) + (a1 >> min(e - e1, 63)), e);
      q = fx_out(a2, dot_exp(cm[4 * nI + 2 * i + part], De[((1 - g) * 3 + 2) * 2 * hp + r]));
      const int ev = ec_2n(v, n);
      if (ev) atomicMax(ct + 2 * i + part, ev);
    }
    reinterpret_cast<double*>(R3)[t0] = v;
    reinterpret_cast<double*>(R3)[t0 + 4 * AS] = q;
  }
  __syncthreads();
  if (!mean) {  // xi = -dv/dy: suffix sums of 2 n v_n
    col_scales(R3, C, N, ct, cs + 6 * nI, true);
    for (int t = threadIdx.x; t < AS; t += blockDim.x) {
      const int n = C.row(t), i = t - n * nI;
      const double2 v = R3[t];
      reinterpret_cast<longlong2*>(C3)[t] = make_longlong2(deriv_fx(v.x, n, ct[2 * i]), deriv_fx(v.y, n, ct[2 * i + 1]));
    }
    __syncthreads();
    deriv_chains(reinterpret_cast<fx*>(C3), C, N, nullptr);
    __syncthreads();
  }
  // u = -i (kx xi + kz eta)/k^2, w = -i (kz xi - kx eta)/k^2, and the finite-difference quotient.
  // The subtraction goes into the products' chain, d = (w - u) or (r - w) by two fused
  // multiply-adds from the far end: 15 of the 77-clock FP64 instructions per value of three
  // components instead of 22 (first half-step) and 25, and one rounding of u+ less before the
  // cancellation (128 x 97 x 128: 148 and 150 -> 139 us; 32 x 33 x 32, batch 8: 20.5 and 22 -> 20).
  const bool psi = op == MODE_PSI_UPDATE || op == MODE_PSI_GRAD;
  const double ik = I0.ik2nu[m], kxs = kx * ik, kzs = kz * ik, inu = flip(I0.inv_nu, psi);
  for (int t = threadIdx.x; t < 2 * nI * ny; t += blockDim.x) {
    const int i = CN.row(t >> 1), part = t & 1, n = (t >> 1) - i * ny;
    if (!live[i]) continue;
    const Inst& I = insts[first + i];
    const double* R = reinterpret_cast<const double*>(R3 + n * nI + i);
    // component c: ac x + bc y
    double x0, x2, y, a0, a2, b0, b2;
    if (mean) {
      x0 = R[part];
      x2 = R[4 * AS + part];
      a0 = a2 = inu;
      b0 = b2 = y = 0.0;
    } else {
      // the other part of dv/dy and of eta
      const fx bx = n < N ? reinterpret_cast<const fx*>(C3 + (n + 1) * nI + i)[1 - part] : 0;
      y = fx_out(bx, dot_exp(ct[2 * i + 1 - part], -2));
      x0 = x2 = R[4 * AS + 1 - part];
      const bool sg = (part != 0) != psi;
      a0 = flip(kzs, sg);
      b2 = -a0;
      b0 = a2 = flip(kxs, !sg);
    }
    const double x1 = mean ? 0.0 : R[part];
    const size_t gi = 2 * ((size_t)m * ny + n) + part, gc = 2 * (size_t)nm * ny;
    const double* u = reinterpret_cast<const double*>(I.uhat) + gi;
    double* rh = reinterpret_cast<double*>(I.rhat) + gi;
    double d[3], up[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      up[c] = op == MODE_PHI || op == MODE_PSI_UPDATE ? u[c * gc] : 0.0;
      d[c] = op == MODE_PHI ? -up[c] : rh[c * gc];
    }
    d[0] = fma(a0, x0, fma(b0, y, d[0]));
    d[1] = fma(inu, x1, d[1]);
    d[2] = fma(a2, x2, fma(b2, y, d[2]));
    const double step = op == MODE_PSI_UPDATE ? I.dtau * ist : ist;
    double* out = op == MODE_PHI ? rh : reinterpret_cast<double*>(op == MODE_PSI_UPDATE ? I.uhat : I.fhat) + gi;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double o = op == MODE_PSI_UPDATE ? fma(step, d[c], up[c]) : d[c] * step;
      out[c * gc] = o;
      done(i, c, n, part, o);
    }
  }
}

__device__ __forceinline__ int find_group(const GroupLaunch& gl, int cta, int* local) {
  int lo = 0, hi = gl.ngroups - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (gl.prefix[mid] <= cta) lo = mid; else hi = mid - 1;
  }
  *local = cta - gl.prefix[lo];
  return lo;
}

// y-values of mode -m of a state invariant under s2, a_{-m} = e2_c (-1)^m conj(a_m), e2 = (+1, +1, -1)
__device__ __forceinline__ double2 mirror_value(double2 v, int ix, int c) {
  const double s = ((ix & 1) != 0) != (c == 2) ? -1.0 : 1.0;
  return make_double2(s * v.x, -s * v.y);
}
__device__ __forceinline__ int field_comp(int q) { return q < 3 ? q : q == 3 ? 0 : 2; }

}  // namespace

// ---------------------------------------------------------------- kernels
__global__ void __launch_bounds__(320, 3) k_yana_fx(LaunchInfo li, int np, int red, int fine) {
  extern __shared__ __align__(16) double2 smx[];
  int local;
  const int b = find_inst(li, blockIdx.x, &local);
  const Inst& I = li.insts[b];
  if (!inst_active(I)) return;
  const int N = I.N, ny = I.ny, nm = I.nmodes, nrun = red ? (I.Kx + 1) * I.Mz : nm;
  const int tile = local / 3, c = local - 3 * tile, m0 = tile * np;
  const Cols C(np, np + 1);
  double2* X = smx;                   // [ny][np + 1]
  double2* Y = X + ny * C.pitch;      // [np][ny + 1] coefficients on their way out
  int* cm = reinterpret_cast<int*>(Y + np * (ny + 1));
  clear_max(cm, 4 * np);
  __syncthreads();
  const double2* src = I.xz + (size_t)c * ny * nm + m0;
  for (int t = threadIdx.x; t < np * ny; t += blockDim.x) {
    const int j = C.row(t), col = t - j * np;
    double2 v = make_double2(0.0, 0.0);
    if (m0 + col < nrun) v = src[(size_t)j * nm + col];
    X[j * C.pitch + col] = v;
    col_max(cm, col, ec_of(v.x), ec_of(v.y));
  }
  col_scales(X, C, N, cm, cm + 2 * np, false);
  ana_fold(X, C, N, cm);
  __syncthreads();
  ana_mac(X, C, N, I.fxcheb, I.fxcheb_e, cm, fine != 0, [&](int col, int n) { return Y + col * (ny + 1) + n; });
  __syncthreads();
  double2* dst = I.xc + ((size_t)c * nm + m0) * ny;
  for (int t = threadIdx.x; t < min(np, nrun - m0) * ny; t += blockDim.x) {
    const int col = t / ny, n = t - col * ny;
    dst[t] = Y[col * (ny + 1) + n];
  }
}

// Fields 0 .. nf - 1 (nf = 5, or 3 for the values alone).
__global__ void __launch_bounds__(320, 3) k_ysynth_fx(LaunchInfo li, int slot, int nf, int np, int red, int fine) {
  extern __shared__ __align__(16) double2 smx[];
  int local;
  const int b = find_inst(li, blockIdx.x, &local);
  const Inst& I = li.insts[b];
  if (!inst_active(I)) return;
  const int N = I.N, ny = I.ny, nm = I.nmodes, nrun = red ? (I.Kx + 1) * I.Mz : nm;
  const int tile = local / nf, q = local - nf * tile, m0 = tile * np, c = field_comp(q);
  const bool deriv = q >= 3;
  const Cols C(np, np + 1);
  double2* X = smx;  // [ny][np + 1]
  int* cm = reinterpret_cast<int*>(X + ny * C.pitch);
  int* bits = cm + 2 * np;
  int* cs = bits + 2 * np;
  clear_max(cm, 6 * np);
  __syncthreads();
  const double2* src = (slot == 0 ? I.uhat : I.rhat) + ((size_t)c * nm + m0) * ny;
  for (int t = threadIdx.x; t < np * ny; t += blockDim.x) {
    const int col = t / ny, n = t - col * ny;
    double2 v = make_double2(0.0, 0.0);
    if (m0 + col < nrun) v = src[t];
    X[n * C.pitch + col] = v;
    if (deriv) col_max(cm, col, ec_2n(v.x, n), ec_2n(v.y, n));
    else col_max(cm, col, ec_of(v.x), ec_of(v.y));
  }
  col_scales(X, C, N, cm, cs, deriv);
  if (deriv) syn_deriv(X, C, N, cm, bits);
  else syn_limbs(X, C, N, cm);
  __syncthreads();
  double2* dst = I.yv + ((size_t)slot * kFieldsY + q) * ny * nm;
  const int Mz = I.Mz, Mx = I.Mx;
  syn_mac(X, C, N, I.fxcheb, deriv, cm, bits, fine != 0, [&](int col, int j, int part, double x, double y = 0.0) {
    const int m = m0 + col;
    if (m >= nrun) return;
    put_part(dst + (size_t)j * nm + m, part, x, y);
    const int ix = m / Mz;
    if (red && ix > 0) {
      const double2 v = mirror_value(part == 1 ? make_double2(0.0, x) : make_double2(x, y), ix, c);
      put_part(dst + (size_t)j * nm + (Mx - ix) * Mz + (m - ix * Mz), part, part == 1 ? v.y : v.x, v.y);
    }
  });
}

__global__ void __launch_bounds__(256, 3) k_ysolve_fx(GroupLaunch gl, int op, int sig, int fine) {
  extern __shared__ __align__(16) double2 smx[];
  __shared__ int live[kMaxGroup];
  int m;
  const int2 grp = gl.groups[find_group(gl, blockIdx.x, &m)];
  const int first = grp.x, nI = grp.y;
  const Inst& I0 = gl.insts[first];
  bool alive = false;
  if (threadIdx.x < nI) live[threadIdx.x] = alive = inst_active(gl.insts[first + threadIdx.x]);
  const int AS = I0.ny * nI, ny = I0.ny, nm = I0.nmodes;
  int* smi = reinterpret_cast<int*>(smx + 6 * AS);
  solve_mode(gl.insts, first, nI, m, op, sig, alive, live, smx, smx + 3 * AS, smi, fine != 0,
             [&](int i, int c, int n, int part) {
               return reinterpret_cast<const double*>(gl.insts[first + i].xc)[2 * (((size_t)c * nm + m) * ny + n) + part];
             },
             [](int, int, int, int, double) {});
}

// The Stokes solve of a caller's right-hand side (rhat -> fhat).  Its result is the operators' alone:
// no transform's rounding hides the tail of a decaying Chebyshev spectrum, and units of a whole
// column's sum would take its digits (spectrum exp(-n/2), ny = 49: coefficient 46 of v off by
// 1.5e-10 of itself in fixed point, by 6e-14 here).  So the operators are applied in FP64, as stored.
// Bound by the FP64 pipe, which takes a warp's instruction in the same 77 clocks whatever its
// active lanes: one output (row, instance, part) per thread, v rows and eta rows in passes of their
// own, so that a warp's lanes carry chains of about one length.  us, several modes per CTA in FP64
// / fixed point / here: 32 x 33 x 32, batch 8: 30 / 19 / 25; 96 x 31 x 48, batch 3: 56 / 24 / 33;
// 128 x 97 x 128: 980 / 126 / 260.
// X: [3][ny][2 nI] doubles f_v, g, h; V, Q: [ny][2 nI] v and eta (mean mode: u, w); Y: dv/dy.
__global__ void __launch_bounds__(256) k_ysolve_f64(GroupLaunch gl, int sig) {
  extern __shared__ __align__(16) double2 smx[];
  __shared__ int bad[2][2 * kMaxGroup];  // an input of v (u), of eta (w) that is not finite, per column
  int m;
  const int2 grp = gl.groups[find_group(gl, blockIdx.x, &m)];
  const int first = grp.x, nI = grp.y, W = 2 * nI;
  const Inst& I0 = gl.insts[first];
  const int N = I0.N, ny = I0.ny, nm = I0.nmodes, Mz = I0.Mz, H = N / 2 + 1, half = N / 2, AS = ny * W;
  double* X = reinterpret_cast<double*>(smx);
  double *V = X + 3 * AS, *Q = V + AS, *Y = X;  // Y over f_v, once v is done
  const int ix = m / Mz, pz = m - ix * Mz;
  const double kx = I0.kx[ix], kz = I0.kz[pz];
  const bool mean = m == 0;
  const Cols C(W, W), CN(ny, ny);
  for (int t = threadIdx.x; t < 4 * kMaxGroup; t += blockDim.x) (&bad[0][0])[t] = 0;
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * nI * ny; t += blockDim.x) {
    const int i = CN.row(t >> 1), part = t & 1, n = (t >> 1) - i * ny;
    const double* F = reinterpret_cast<const double*>(gl.insts[first + i].rhat + (size_t)m * ny + n);
    const size_t gc = 2 * (size_t)nm * ny;
    double a, g, h;
    if (mean) {
      a = F[part];
      g = 0.0;
      h = F[2 * gc + part];
    } else {
      // g = i (kx F_u + kz F_w), h = i (kz F_u - kx F_w)
      const double u = F[1 - part], w = F[2 * gc + 1 - part], kxg = flip(kx, !part), kzg = flip(kz, !part);
      a = F[gc + part];
      g = fma(kxg, u, kzg * w);
      h = fma(kzg, u, -kxg * w);
    }
    double* o = X + n * W + 2 * i + part;
    o[0] = a;
    o[AS] = g;
    o[2 * AS] = h;
    if (ec_of(a) == 0x7ff || ec_of(g) == 0x7ff) bad[0][2 * i + part] = 1;
    if (ec_of(h) == 0x7ff) bad[1][2 * i + part] = 1;
  }
  __syncthreads();
  const DenseLayout DL(N);
  const double* D = I0.dense[sig] + (size_t)m * DL.per_mode();
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  // sum of an operator row (entries Mh apart) over one parity class of a column
  const auto dot = [&](const double* A, const double* x, int K, double s) {
    int k = 0;
    for (; k + 4 <= K; k += 4) {
      double a[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) a[q] = __ldg(A + (k + q) * H);
#pragma unroll
      for (int q = 0; q < 4; ++q) s = fma(a[q], x[2 * (k + q) * W], s);
    }
    for (; k < K; ++k) s = fma(__ldg(A + k * H), x[2 * k * W], s);
    return s;
  };
  // rows of class 0, then of class 1; neighbouring threads take the columns of one row
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    for (int t = threadIdx.x; t < AS; t += blockDim.x) {
      const int rn = C.row(t), col = t - rn * W, cls = rn >= H, r = cls ? rn - H : rn, n = 2 * r + cls;
      const int own = cls ? half : H, other = cls ? H : half;
      double s;
      if (mean) s = dot(D + DL.at(cls, DL.kEh, r, 0), X + pass * 2 * AS + cls * W + col, own, 0.0);
      else if (pass == 0)
        s = dot(D + DL.at(cls, DL.kAg, r, 0), X + AS + (1 - cls) * W + col, other,
                dot(D + DL.at(cls, DL.kAv, r, 0), X + cls * W + col, own, 0.0));
      else s = dot(D + DL.at(1 - cls, DL.kEh, r, 0), X + 2 * AS + cls * W + col, own, 0.0);
      (pass ? Q : V)[n * W + col] = bad[pass][col] ? nan : s;
    }
  }
  __syncthreads();
  if (!mean) {  // dv/dy: b_n = b_{n+2} + 2 (n+1) v_{n+1}, b_0 half
    for (int t = threadIdx.x; t < 2 * W; t += blockDim.x) {
      const int odd = t >= W, col = t - odd * W;
      double b = bad[0][col] ? nan : 0.0;
      Y[(N - odd) * W + col] = odd ? b = fma(2.0 * N, V[N * W + col], b) : b;
      for (int n = N - odd - 2; n >= 0; n -= 2) {
        b = fma(2.0 * (n + 1), V[(n + 1) * W + col], b);
        Y[n * W + col] = n ? b : 0.5 * b;
      }
    }
    __syncthreads();
  }
  // u = -i (kx xi + kz eta)/(nu k^2), w = -i (kz xi - kx eta)/(nu k^2), xi = -dv/dy
  const double ik = I0.ik2nu[m], kxs = kx * ik, kzs = kz * ik, inu = I0.inv_nu;
  for (int t = threadIdx.x; t < 2 * nI * ny; t += blockDim.x) {
    const int i = CN.row(t >> 1), part = t & 1, n = (t >> 1) - i * ny, at = n * W + 2 * i;
    const size_t gc = 2 * (size_t)nm * ny;
    double* out = reinterpret_cast<double*>(gl.insts[first + i].fhat + (size_t)m * ny + n) + part;
    if (mean) {
      out[0] = inu * V[at + part];
      out[gc] = 0.0;
      out[2 * gc] = inu * Q[at + part];
    } else {
      const double y = Y[at + 1 - part], e = Q[at + 1 - part], a0 = flip(kzs, part != 0), b0 = flip(kxs, part == 0);
      out[0] = fma(a0, e, b0 * y);
      out[gc] = inu * V[at + part];
      out[2 * gc] = fma(b0, e, -a0 * y);
    }
  }
}

__global__ void __launch_bounds__(256, 2) k_ystep_fx(GroupLaunch gl, int op, int synth, int fine) {
  extern __shared__ __align__(16) double2 smx[];
  __shared__ int live[kMaxGroup];
  int m;
  const int2 grp = gl.groups[find_group(gl, blockIdx.x, &m)];
  const int first = grp.x, nI = grp.y;
  const Inst& I0 = gl.insts[first];
  if (threadIdx.x < nI) live[threadIdx.x] = inst_active(gl.insts[first + threadIdx.x]);
  const int N = I0.N, ny = I0.ny, nm = I0.nmodes, AS = ny * nI;
  double2* X = smx;           // [3][ny][nI] (the synthesis: [ny][3 nI], then [ny][2 nI])
  double2* Y = X + 3 * AS;    // [3][ny][nI] coefficients, then the new state
  double2* R = Y + 3 * AS;    // [3][ny][nI]
  int* smi = reinterpret_cast<int*>(R + 3 * AS);
  // analysis of the three components: columns (component, instance)
  const Cols C3(3 * nI, 3 * nI);
  clear_max(smi, 12 * nI);
  __syncthreads();
  for (int t = threadIdx.x; t < 3 * AS; t += blockDim.x) {
    const int j = C3.row(t), col = t - j * C3.n, c = col / nI, i = col - c * nI;
    const double2 v = gl.insts[first + i].xz[((size_t)c * ny + j) * nm + m];
    X[t] = v;
    col_max(smi, col, ec_of(v.x), ec_of(v.y));
  }
  col_scales(X, C3, N, smi, smi + 6 * nI, false);
  ana_fold(X, C3, N, smi);
  __syncthreads();
  ana_mac(X, C3, N, I0.fxcheb, I0.fxcheb_e, smi, fine != 0, [&](int col, int n) {
    const int c = col / nI, i = col - c * nI;
    return Y + c * AS + n * nI + i;
  });
  __syncthreads();
  solve_mode(gl.insts, first, nI, m, op, op == MODE_PHI ? 0 : 1, true, live, X, R, smi, fine != 0,
             [&](int i, int c, int n, int part) { return reinterpret_cast<const double*>(Y + c * AS + n * nI + i)[part]; },
             [&](int i, int c, int n, int part, double v) {
               reinterpret_cast<double*>(Y + c * AS + n * nI + i)[part] = v;
             });
  if (!synth) return;
  __syncthreads();
  // synthesis of the new r1 (PHI) or u: values of the three components, then the y-derivatives of u, w
  const int slot = op == MODE_PHI ? 1 : 0;
#pragma unroll 1
  for (int d = 0; d < 2; ++d) {
    const Cols C(d ? 2 * nI : 3 * nI, d ? 2 * nI : 3 * nI);
    int* bits = smi + 2 * C.n;
    int* cs = bits + 2 * C.n;
    clear_max(smi, 6 * C.n);
    __syncthreads();
    for (int t = threadIdx.x; t < C.n * ny; t += blockDim.x) {
      const int n = C.row(t), col = t - n * C.n, f = col / nI, i = col - f * nI, c = d ? 2 * f : f;
      const double2 v = Y[c * AS + n * nI + i];
      X[t] = v;
      if (d) col_max(smi, col, ec_2n(v.x, n), ec_2n(v.y, n));
      else col_max(smi, col, ec_of(v.x), ec_of(v.y));
    }
    col_scales(X, C, N, smi, cs, d != 0);
    if (d) syn_deriv(X, C, N, smi, bits);
    else syn_limbs(X, C, N, smi);
    __syncthreads();
    syn_mac(X, C, N, I0.fxcheb, d != 0, smi, bits, fine != 0, [&](int col, int j, int part, double x, double y = 0.0) {
      const int f = col / nI, i = col - f * nI;
      if (!live[i]) return;
      put_part(gl.insts[first + i].yv + (((size_t)slot * kFieldsY + (d ? 3 + f : f)) * ny + j) * nm + m, part, x, y);
    });
    __syncthreads();
  }
}

// J = ||r1|| of every active instance from the plane sums of the adjoint product kernel, its
// history entry, and the convergence mask (J < tol: the instance stops before this step's
// update).  One warp per instance.
__global__ void __launch_bounds__(32) k_jnorm(const Inst* insts, int step_index) {
  const Inst& I = insts[blockIdx.x];
  if (!inst_active(I)) return;
  const double J = norm_from_parts(I);
  if (threadIdx.x != 0) return;
  if (I.hist) I.hist[(size_t)step_index * I.hist_stride] = J;
  if (I.tol > 0.0 && J < I.tol && I.active) *I.active = 0;
}

// A matrix entry in units where its row's largest (biased exponent e) is below 2^57, to the nearest
__device__ __forceinline__ fx row_fx(double v, int e) {
  const int hi = __double2hiint(v), ec = (hi >> 20) & 0x7ff, r = e - ec;
  const fx m = ((fx)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  return neg_if(ec == 0 ? 0 : fx_round(m << 4, r), hi);
}
// Dense operators (DenseLayout) of every mode as limbs: block bl of mode m in CTA (bl, m), with
// each row's exponent.
__global__ void __launch_bounds__(128) k_dense_limbs(const double* __restrict__ src, int Mh, int4* dst, int* dexp) {
  const int bl = blockIdx.x, m = blockIdx.y, hp = (Mh + 1) / 2;
  const double* D = src + ((size_t)m * 6 + bl) * Mh * Mh;
  int4* o = dst + ((size_t)m * 6 + bl) * Mh * hp;
  int* oe = dexp + ((size_t)m * 6 + bl) * 2 * hp;
  for (int rp = threadIdx.x; rp < hp; rp += blockDim.x) {
    int e[2] = {0, 0};
    for (int k = 0; k < Mh; ++k)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (2 * rp + h < Mh) e[h] = max(e[h], ec_of(D[k * Mh + 2 * rp + h]));
    for (int k = 0; k < Mh; ++k) {
      fx v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) v[h] = 2 * rp + h < Mh ? row_fx(D[k * Mh + 2 * rp + h], e[h]) : 0;
      o[k * hp + rp] = limbs(v[0], v[1]);
    }
    oe[2 * rp] = e[0] - 1079 + 55;  // entries in units of 2^(e - 1079), products in units of 2^55
    oe[2 * rp + 1] = e[1] - 1079 + 55;
  }
}

// ---------------------------------------------------------------- host
int yfx_tiles(int nmodes, int np) { return (nmodes + np - 1) / np; }
static int one_pass(int tasks, int most) {
  const int passes = (tasks + most - 1) / most;
  return std::max(128, ((tasks + passes - 1) / passes + 31) / 32 * 32);
}
// threads per CTA; fine: one row and one part per thread
int yana_fx_threads(int N, int np, bool fine) {
  return one_pass(fine ? 2 * np * (N + 1) : np * ((N / 2 + 2) / 2 + (N / 2 + 1) / 2), 256);
}
int ysynth_fx_threads(int N, int np, bool fine) { return one_pass(np * (fine ? N + 2 : (N / 2 + 2) / 2), fine ? 320 : 256); }
// many: the launch has at least five CTAs for every SM.  Small CTAs then keep more of their ten
// dependent phases in flight: 96 or 128 threads, whichever leaves fewer lanes idle, while that
// takes at most four passes (128 x 97 x 128: 147 us with 96 threads, 166 with 160; 64 x 65 x 64,
// batch 2: 43 with 128, 48 with 224; 96 x 31 x 48, batch 3: 28 with 96, 35 with 160).  Groups of
// more columns and launches of few CTAs want one pass (32 x 33 x 32, batch 8: 20.5 us with 256
// threads, 24.6 with 96; 24 x 32^3 + 24 x 48^3 + 16 x 64^3 in groups of eight: 358 with 224, 492
// with 96).
int ysolve_fx_threads(int N, int G, bool fine, bool many) {
  const int tasks = 6 * ((N / 2 + 2) / 2) * G * (fine ? 4 : 1);
  if (many && tasks <= 4 * 96) return (tasks + 95) / 96 * 96 <= (tasks + 127) / 128 * 128 ? 96 : 128;
  return one_pass(tasks, 256);
}
size_t smem_yana_fx(int N, int np) { return 16 * ((size_t)(N + 1) * (np + 1) + (size_t)np * (N + 2)) + 16 * (size_t)np; }
size_t smem_ysynth_fx(int N, int np) { return 16 * (size_t)(N + 1) * (np + 1) + 24 * (size_t)np; }
size_t smem_ysolve_fx(int N, int G) { return 16 * 6 * (size_t)(N + 1) * G + 64 * (size_t)G; }
size_t smem_ystep_fx(int N, int G) { return 16 * 9 * (size_t)(N + 1) * G + 72 * (size_t)G; }
void launch_yana_fx(int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int np, int red, int fine) {
  k_yana_fx<<<ctas, threads, smem, s>>>(li, np, red, fine);
}
void launch_ysynth_fx(int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int slot, int nf,
                      int np, int red, int fine) {
  k_ysynth_fx<<<ctas, threads, smem, s>>>(li, slot, nf, np, red, fine);
}
void launch_ysolve_fx(int ctas, int threads, size_t smem, cudaStream_t s, GroupLaunch gl, int op, int sig, int fine) {
  k_ysolve_fx<<<ctas, threads, smem, s>>>(gl, op, sig, fine);
}
// one pass over the columns of a row each for v and for eta
int ysolve_f64_threads(int N, int G) { return one_pass(2 * G * (N + 1), 256); }
size_t smem_ysolve_f64(int N, int G) { return 8 * 5 * (size_t)(N + 1) * 2 * G; }
void launch_ysolve_f64(int ctas, int threads, size_t smem, cudaStream_t s, GroupLaunch gl, int sig) {
  k_ysolve_f64<<<ctas, threads, smem, s>>>(gl, sig);
}
void launch_ystep_fx(int ctas, int threads, size_t smem, cudaStream_t s, GroupLaunch gl, int op, int synth, int fine) {
  k_ystep_fx<<<ctas, threads, smem, s>>>(gl, op, synth, fine);
}
void launch_jnorm(int ninst, cudaStream_t s, const Inst* insts, int step_index) {
  k_jnorm<<<ninst, 32, 0, s>>>(insts, step_index);
}
size_t dense_limbs_len(int N, int nmodes) { return (size_t)nmodes * 6 * (N / 2 + 1) * ((N / 2 + 2) / 2); }
size_t dense_exps_len(int N, int nmodes) { return (size_t)nmodes * 12 * ((N / 2 + 2) / 2); }
void launch_dense_limbs(const double* src, int N, int nmodes, int4* dst, int* dexp) {
  k_dense_limbs<<<dim3(6, nmodes), 64>>>(src, N / 2 + 1, dst, dexp);
}
cudaError_t set_modes_fx_smem(size_t ana, size_t synth, size_t solve, size_t step, size_t solve64) {
  cudaError_t e;
  if ((e = raise_smem_limit((const void*)k_yana_fx, ana))) return e;
  if ((e = raise_smem_limit((const void*)k_ysynth_fx, synth))) return e;
  if ((e = raise_smem_limit((const void*)k_ysolve_fx, solve))) return e;
  if ((e = raise_smem_limit((const void*)k_ysolve_f64, solve64))) return e;
  return raise_smem_limit((const void*)k_ystep_fx, step);
}

}  // namespace pcf
