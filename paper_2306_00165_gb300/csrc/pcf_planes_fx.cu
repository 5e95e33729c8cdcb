// x-z plane kernels of the FP64 forms in 64-bit fixed point (pcf_fx.cuh).
//
//   k_synth_fx  CTA (instance, y-plane, field): inverse x and z transforms of the y-values;
//               writes the plane as integers with one exponent
//   k_prod_fx   CTA (instance, y-plane, component): M(u) or N(q) on the plane, forward z and x
//               transforms, 2/3 truncation, back to FP64; plane sums of q^2 and J
//   k_norm_planes_fx  plane sums of squares
//
// What bounds them: integer issue.  The same transforms in FP64 were bound by the FP64 pipe
// (a 32 x 32 plane needs 11 k FP64 instructions, 6.7 k clocks of an SM); the integer
// butterflies of a plane take under 1 k clocks.
//
// Measured (us per launch, FP64 Stockham passes -> now): 32 x 33 x 32, batch 8: synthesis 75 -> 29,
// products M 41 -> 20, N 55 -> 30; 128 x 97 x 128: 1025 -> 208, 381 -> 105, 529 -> 157.
//
// A transform of length L = R S (fx_plan) is two register passes, thread n of S in the first,
// thread b of R in the second.  Both work in place, so one buffer and one barrier per pass
// suffice; rows have an odd stride for the walks across rows.
#include "pcf_fx.cuh"
#include "pcf_kernels.cuh"

namespace pcf {

namespace {

// Kernels for planes whose sides are 8 R: up to 64, or longer (R = 12, 16 hold more registers); and
// for planes with a side of 18, 24, 36, 54, 72 or 108, which also do the others.
enum FxKind : int { FX_SMALL = 0, FX_BIG = 1, FX_ANY = 2 };
// Threads and resident CTAs the kernels are compiled for: 80 registers for sides up to 64 (768
// threads per SM), 128 registers (512 threads per SM) for the longer transforms.
template <int KIND>
struct FxCfg {
  static constexpr int threads = KIND ? 512 : 256, ctas = KIND ? 1 : 3;
};

// R and S of length n
template <int KIND>
__device__ __forceinline__ FxPlan fx_plan_of(int n) {
  return KIND == FX_ANY ? fx_plan(n) : FxPlan{n >> 3, 8};
}
__device__ __forceinline__ int fx_div(int t, unsigned mul) { return (int)__umulhi((unsigned)t, mul); }
// slot of element i + odd of a row on its way into a transform (i even when odd is 1), and of output
// b + R k
template <int KIND>
__device__ __forceinline__ int fx_in(FxPlan P, int i, int odd = 0) {
  if (KIND == FX_ANY && P.S != 8) return i + odd;  // (i / S) S + i mod S
  return fx_slot<8>(i >> 3, (i & 7) + odd);
}
template <int KIND>
__device__ __forceinline__ int fx_out(FxPlan P, int b, int k) {
  return KIND == FX_ANY && P.S != 8 ? b * P.S + k : fx_slot<8>(b, k);
}

// First pass over nrow rows: ld(row, n) -> element n, result in place in buf.  A row's S threads
// lie in a group of G lanes; the spare lanes (S < G) repeat the last one's loads and store nothing.
template <int R, int S, bool INV, class LD>
__device__ __forceinline__ void fx_first(int nrow, fxc* buf, int LS, const fxtw* __restrict__ tw, const LD& ld) {
  constexpr int LG = S <= 8 ? 3 : 4, G = 1 << LG;
  for (int t = threadIdx.x; t < G * nrow; t += blockDim.x) {
    const int row = t >> LG, lane = t & (G - 1), n = S < G ? min(lane, S - 1) : lane;
    fxc v[R];
    ld(row, n, v);
    if (S < G && lane >= S) continue;
    FxDft<R, INV>::run(v);
    fxc* o = buf + row * LS;
    o[fx_slot<S>(0, n)] = v[0];
#pragma unroll
    for (int k = 1; k < R; ++k) {
      const int4 w = __ldg(reinterpret_cast<const int4*>(tw) + n * k);
      o[fx_slot<S>(k, n)] = fx_cmul(v[k], fxtw{w.x, w.y, w.z, w.w});
    }
  }
}
// Second pass: st(row, b, v): v[k] is output b + R k of the row.
template <int R, int S, bool INV, class ST>
__device__ __forceinline__ void fx_second(int nrow, const fxc* buf, int LS, const ST& st) {
  for (int t = threadIdx.x; t < R * nrow; t += blockDim.x) {
    const int row = t / R, b = t - row * R;
    const fxc* a = buf + row * LS;
    fxc v[S];
#pragma unroll
    for (int e = 0; e < S; ++e) v[e] = a[fx_slot<S>(b, e)];
    FxDft<S, INV>::run(v);
    st(row, b, v);
  }
}

// f(FxRS<R, S>) for the transform length n (uniform in the CTA); the host chooses a KIND that has it
// (planes_fx_kind)
template <int R_, int S_>
struct FxRS {
  static constexpr int R = R_, S = S_;
};
template <int KIND, class F>
__device__ __forceinline__ void fx_length(int n, const F& f) {
  if (KIND == FX_ANY) {
    switch (n) {
      case 18: f(FxRS<6, 3>()); return;
      case 24: f(FxRS<4, 6>()); return;
      case 36: f(FxRS<6, 6>()); return;
      case 54: f(FxRS<6, 9>()); return;
      case 72: f(FxRS<12, 6>()); return;
      case 108: f(FxRS<12, 9>()); return;
    }
  }
  switch (n >> 3) {
    case 2: f(FxRS<2, 8>()); break;
    case 4: f(FxRS<4, 8>()); break;
    case 6: f(FxRS<6, 8>()); break;
    case 12: if (KIND) f(FxRS<12, 8>()); break;
    case 16: if (KIND) f(FxRS<16, 8>()); break;
    default: f(FxRS<8, 8>()); break;  // 64
  }
}

// ------------------------------------------------------------------ FP64 -> fixed point
// Integer view of a nonzero finite factor k: mantissa in [2^61, 2^62) and biased exponent.
struct FxK {
  fx m;
  int e, neg, hi;
};
__device__ __forceinline__ FxK fx_factor(double k) {
  const int hi = __double2hiint(k);
  const fx m = ((fx)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(k);
  return FxK{m << 9, (hi >> 20) & 0x7ff, hi >> 31, hi & 0x7fffffff};
}
__device__ __forceinline__ fx fx_signed(fx a, int neg) {
  const fx m = (fx)neg;
  return (a ^ m) - m;
}
// v 2^-e0 to the nearest, where |v| 2^-e0 < 2^61
__device__ __forceinline__ fx fx_from(double v, int e0) {
  const int hi = __double2hiint(v), ec = (hi >> 20) & 0x7ff;
  const fx m = ((fx)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  return fx_signed(ec == 0 ? 0 : fx_round(m << 8, 1083 + e0 - ec), hi >> 31);
}
// k v 2^-e0, negated when neg
__device__ __forceinline__ fx fx_from_k(double v, const FxK& k, int e0, int neg) {
  const int hi = __double2hiint(v), ec = (hi >> 20) & 0x7ff;
  const fx m = ((fx)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  return fx_signed(ec == 0 || k.e == 0 ? 0 : fx_round(fx_mul64(m << 9, k.m) << 2, 2106 + e0 - ec - k.e),
                   (hi >> 31) ^ k.neg ^ neg);
}
// Exponent of a double: kFxNone (zero, denormal), kFxNan (not finite) or floor(log2 |v|)
__device__ __forceinline__ int fx_bexp(int hi) {
  const int ec = (hi >> 20) & 0x7ff;
  return ec == 0 ? kFxNone : ec == 0x7ff ? kFxNan : ec - 1023;
}
__device__ __forceinline__ float fx_pow2f(int e) { return e < -126 ? 0.f : __int_as_float((e + 127) << 23); }

// Running sum of magnitudes w |v| of doubles of any size, in single precision: a double with
// biased exponent lim counts as 2^33 times its mantissa.  Values up to 2^60 above it are added as
// they are (2^14 of them with weights below 2^8 stay finite), a larger one becomes the new
// reference; values below 2^-160 of it vanish.  Truncated mantissas and the sum's rounding stay
// within the factor 1 + 2^-9 of the bound taken from it.
struct FxSum {
  float acc = 0.f;
  int lim = -4096;
  unsigned top = 0;  // largest |v| (high word) with a weight other than zero
  __device__ __forceinline__ static float mag(int habs, int off) { return __int_as_float(max(habs - off, 0) << 3); }
  __device__ __forceinline__ void add(int hx, int hy, float w) {
    const int m = max(hx, hy), em = m >> 20;
    top = max(top, (unsigned)m);
    if (em > lim + 60) {
      acc *= fx_pow2f(lim - em);
      lim = em;
    }
    const int off = (lim - 160) << 20;
    acc = fmaf(w, mag(hx, off) + mag(hy, off), acc);
  }
};
// The block's sum times g: true when some weighted value is not zero; *bits: sum < 2^bits.  any:
// largest |v| of the thread's values, *all that of the block's.  sh: 4 ints per warp.
__device__ __forceinline__ bool fx_block_bound(FxSum a, float g, unsigned any, int* sh, unsigned* all, int* bits) {
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int L = __reduce_max_sync(0xffffffffu, a.lim);
  float v = a.acc * fx_pow2f(a.lim - L);
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  any = __reduce_max_sync(0xffffffffu, any);
  const unsigned top = __reduce_max_sync(0xffffffffu, a.top);
  if ((threadIdx.x & 31) == 0) {
    sh[4 * warp] = L;
    sh[4 * warp + 1] = __float_as_int(v);
    sh[4 * warp + 2] = (int)any;
    sh[4 * warp + 3] = (int)top;
  }
  __syncthreads();
  int Lm = sh[0];
  unsigned tm = 0, am = 0;
  for (int w = 0; w < nw; ++w) {
    Lm = max(Lm, sh[4 * w]);
    am = max(am, (unsigned)sh[4 * w + 2]);
    tm = max(tm, (unsigned)sh[4 * w + 3]);
  }
  float tot = 0.f;
  for (int w = 0; w < nw; ++w) tot += __int_as_float(sh[4 * w + 1]) * fx_pow2f(sh[4 * w] - Lm);
  tot *= g * (1.f + 0x1p-9f);
  *all = am;
  *bits = (__float_as_int(tot) >> 23) - 126 + Lm - 1056;
  return tm >= 0x00100000u;
}

__device__ __forceinline__ const int2* fx_info(const Inst& I, int slot, int f, int j) {
  return I.pinfo + ((size_t)slot * kFieldsSynth + f) * I.ny + j;
}
// x-storage index i (m = i for i <= Kx, m = i - Mx otherwise) -> FFT bin
__device__ __forceinline__ int xbin(int i, int Kx, int Mx, int nx) { return i <= Kx ? i : nx - (Mx - i); }

}  // namespace

// x rows (one per retained z mode) and z rows (row pairs) in shared memory: the x array whole,
// the z rows `chunk` at a time.
struct FxPlanes {
  int LX, LZ, chunk;
};
// One pass of `threads` threads covers threads/8 row pairs in the first z pass, so more rows
// at a time would only cost shared memory.
__host__ __device__ inline FxPlanes fx_planes(const Inst& I, int threads) {
  FxPlanes p;
  p.LX = I.nx + 1;
  p.LZ = I.nz + 1;
  p.chunk = I.nx / 2 < threads / 8 ? I.nx / 2 : threads / 8 < 16 ? 16 : threads / 8;
  return p;
}
// [x rows | z rows | 64 ints of reduction | exponents of the row pairs and x rows | alignment]
size_t smem_planes_fx(const Inst& I, int threads) {
  const FxPlanes p = fx_planes(I, threads);
  return sizeof(fxc) * ((size_t)I.Mz * p.LX + (size_t)p.chunk * p.LZ) + 4 * (64 + 64 + 64 + 64);
}
// Threads per CTA.  Sides up to 64: the synthesis of small planes keeps two warps busy in every
// pass (32 x 33 x 32, batch 8: 29 us, with 128 threads 32), larger ones four (64 x 65 x 64, batch
// 2: 58 us, with 96 threads 62, with 256 58).  The products take all row pairs of a plane in one
// pass: with few CTAs per SM the loads of their factors are what the time goes to (64 x 65 x 64,
// batch 2: 37 and 51 us with 256 threads, 41 and 67 with 128; 48 x 49 x 48, batch 4: 29 and 41 us
// with 192, 30 and 45 with 128, 35 and 58 with 256; 32 x 33 x 32, batch 8: 20 and 30 us with
// 128, 25 and 36 with 256).  Longer sides: the plane's x rows fill much of the shared memory, so
// the smallest CTA that leaves the SM the most threads (128 x 97 x 128: synthesis 208 us with 512
// threads; before the single-precision bound 233 with 512, 280 with 256, 397 with 128; 96 x 31 x
// 48, batch 3: 56 us with 128); the products take at least 256 (there 40 and 51 us, with 128
// threads 47 and 62).
// Planes with a side that is not 8 R are rare; they take the longer sides' rule.
int planes_fx_kind(const Inst& I) {
  if (fx_plan(I.nx).S != 8 || fx_plan(I.nz).S != 8) return FX_ANY;
  return I.nx > 64 || I.nz > 64 ? FX_BIG : FX_SMALL;
}
int planes_fx_threads(const Inst& I, bool prod) {
  if (planes_fx_kind(I) == FX_SMALL) return prod ? std::max(128, 4 * I.nx) : I.nx * I.nz <= 1024 ? 64 : 128;
  int best = 128, most = 0;
  for (int t = 128; t <= FxCfg<FX_BIG>::threads; t *= 2) {
    const int fit = (int)(228 * 1024 / (smem_planes_fx(I, t) + 1024)), n = t * std::min(fit, 512 / t);
    if (n > most) best = t, most = n;
  }
  return prod ? std::max(best, 256) : best;
}

__constant__ int c_fx_src[kFieldsSynth] = {0, 1, 2, 0, 3, 0, 1, 1, 2, 4, 2};
__constant__ int c_fx_fac[kFieldsSynth] = {0, 0, 0, 1, 0, 2, 1, 2, 1, 0, 2};

// ------------------------------------------------------------------ plane synthesis
// CTA = (instance, y-plane j, field f): u, v, w, u_x, u_y, u_z, v_x, v_z, w_x, w_y, w_z.  The
// plane's exponent e0 comes from the sum B of |Re| + |Im| over the plane's modes (p > 0 twice):
// every intermediate of the two transforms is below 2 B in modulus, and 2 B 2^-e0 < 2^62.  The x
// stage runs each row p (a z mode) at an exponent of its own, from the row's largest value, and its
// results are rounded to e0: at e0 the rounding of the inputs, summed over all the modes, would be
// ten times the rounding of the rest (a flat spectrum at 128 x 33 x 128: modes of r1 off by 2.9e-15 of
// themselves in the median; 6.4e-16 with row exponents, 9.2e-16 in FP64 arithmetic; 32 x 33 x 32, batch
// 8: 28 -> 29 us, 128 x 97 x 128: 205 -> 208).
template <int KIND>
__global__ void __launch_bounds__(FxCfg<KIND>::threads, FxCfg<KIND>::ctas) k_synth_fx(LaunchInfo li, int slot, int nfields) {
  extern __shared__ __align__(16) unsigned char smraw[];
  int local;
  const int b = find_inst(li, blockIdx.x, &local);
  const Inst& I = li.insts[b];
  if (!inst_active(I)) return;
  const int f = local % nfields, j = local / nfields;
  const int nx = I.nx, nz = I.nz, Mz = I.Mz, Kx = I.Kx, Kz = I.Kz, nm = I.nmodes;
  const FxPlanes P = fx_planes(I, blockDim.x);
  fxc* G = reinterpret_cast<fxc*>(smraw);
  fxc* Z = G + Mz * P.LX;
  int* red = reinterpret_cast<int*>(Z + P.chunk * P.LZ);
  int* row = red + 64;  // exponents of the rows p
  const double2* src = I.yv + (((size_t)slot * kFieldsY + c_fx_src[f]) * I.ny + j) * (size_t)nm;
  const int fac = c_fx_fac[f];
  // Bound of the plane: one pass in single precision (a pass for the largest exponent and one
  // in integers took 90 instructions per mode, this one 25)
  const unsigned mzm = I.mz_mul;
  FxSum sum;
  unsigned any = 0;
  for (int p = threadIdx.x; p < Mz; p += blockDim.x) row[p] = 0;
  __syncthreads();
  for (int t0 = threadIdx.x; t0 < nm; t0 += 4 * blockDim.x) {
    double2 s[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = t0 + q * (int)blockDim.x < nm ? src[t0 + q * blockDim.x] : make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = t0 + q * blockDim.x, i = fx_div(t, mzm), p = t - i * Mz;
      const int hx = __double2hiint(s[q].x) & 0x7fffffff, hy = __double2hiint(s[q].y) & 0x7fffffff;
      any = max(any, (unsigned)max(hx, hy));
      // |k| in units of the smallest wavenumber
      const int k = fac == 0 ? 1 : fac == 1 ? (i <= Kx ? i : I.Mx - i) : p;
      if (t < nm && k) {
        sum.add(hx, hy, (float)(p ? 2 * k : k));
        const int m = max(hx, hy) >> 20, e = m + (fac ? 32 - __clz(k) : 0);
        if (m && e > row[p]) atomicMax(row + p, e);
      }
    }
  }
  const int k1 = fac == 0 ? 0x3ff00000 : __double2hiint(fac == 1 ? I.kx[1] : I.kz[1]), ek = fx_bexp(k1);
  int eb;
  const bool live = fx_block_bound(sum, __int_as_float(0x3f800000 | (k1 & 0xfffff) << 3), any, red, &any, &eb);
  const bool bad = any >= 0x7ff00000u || ek == kFxNan;
  int2* info = const_cast<int2*>(fx_info(I, slot, f, j));
  fx* out = reinterpret_cast<fx*>(I.phys) + (((size_t)slot * kFieldsSynth + f) * I.ny + j) * (size_t)nx * nz;
  if (bad || !live) {  // a NaN or an infinity in the plane, or a zero plane (uniform)
    if (!bad)
      for (int t = threadIdx.x; t < nx * nz; t += blockDim.x) out[t] = 0;
    if (threadIdx.x == 0) *info = make_int2(bad ? kFxNan : kFxNone, 0);
    return;
  }
  const int e0 = eb + ek - 61;
  const FxPlan px = fx_plan_of<KIND>(nx);
  // kept for the end of the kernel (in a register it made the 80-register variant spill: uneven batch of
  // 64, 789 us a launch against 768)
  if (KIND == FX_SMALL && threadIdx.x == 0) row[63] = e0;
  // a row's values are below 2^(row - 1022) (times 2^(ek + 1) for a derivative) in each part, and a
  // transform of its Mx modes below 2^cr times that
  const int cr = 32 - __clz((3 * I.Mx) >> 1) - 1022 - 62 + (fac ? ek + 1 : 0);
  for (int p = threadIdx.x; p < Mz; p += blockDim.x) row[p] = max(min(row[p] + cr, e0), e0 - 31);
  __syncthreads();
  // the modes as integers at their x bins (rows p); i k v for the x and z derivatives
  for (int t = threadIdx.x; t < nm; t += blockDim.x) {
    const double2 s = src[t];
    const int i = fx_div(t, mzm), p = t - i * Mz, bin = xbin(i, Kx, I.Mx, nx);
    const int e = row[p];
    fxc v;
    if (fac == 0) {
      v = fxc{fx_from(s.x, e), fx_from(s.y, e)};
    } else {
      const FxK k = fx_factor(fac == 1 ? I.kx[i] : I.kz[p]);
      v = fxc{fx_from_k(s.y, k, e, -1), fx_from_k(s.x, k, e, 0)};
    }
    G[p * P.LX + fx_in<KIND>(px, bin)] = v;
  }
  __syncthreads();
  // x stage, rows p: element = x bin; bins outside |m| <= Kx are zero
  fx_length<KIND>(nx, [&](auto rc) {
    constexpr int R = decltype(rc)::R, S = decltype(rc)::S;
    fx_first<R, S, true>(Mz, G, P.LX, I.twfx_x + nx, [&](int p, int n, fxc* v) {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int bin = n + S * q;
        v[q] = bin <= Kx || bin >= nx - Kx ? G[p * P.LX + fx_slot<S>(q, n)] : fxc{0, 0};
      }
    });
    __syncthreads();
    fx_second<R, S, true>(Mz, G, P.LX, [&](int p, int bk, const fxc* v) {
      fxc* o = G + p * P.LX;
      const int d = e0 - row[p];
      const unsigned h = (1u << d) >> 1;
#pragma unroll
      for (int e = 0; e < S; ++e) o[fx_slot<S>(bk, e)] = fxc{fx_sra31(v[e].x + h, d), fx_sra31(v[e].y + h, d)};
    });
  });
  __syncthreads();
  const int nr = nx / 2, Rx = px.R;
  const unsigned rxm = I.rx_mul;
  unsigned mh = 0;
  for (int r0 = 0; r0 < nr; r0 += P.chunk) {
    const int nrc = min(P.chunk, nr - r0);
    fx_length<KIND>(nz, [&](auto rc) {
      constexpr int R = decltype(rc)::R, S = decltype(rc)::S;
      // row pair (x1, x2 = x1 + 1) -> one complex row G[x1] + i G[x2]
      fx_first<R, S, true>(nrc, Z, P.LZ, I.twfx_z + nz, [&](int r, int n, fxc* v) {
        const int x1 = 2 * (r0 + r), k3 = fx_div(x1, rxm), k1 = x1 - k3 * Rx;
        const int s1 = fx_out<KIND>(px, k1, k3), s2 = fx_out<KIND>(px, k1 + 1, k3);
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int z = n + S * q;
          const bool lo = z <= Kz, hi = z >= nz - Kz;
          v[q] = fxc{0, 0};
          if (lo || hi) {
            const fxc* g = G + (lo ? z : nz - z) * P.LX;
            fxc g1 = g[s1], g2 = g[s2];
            if (z == 0) g1.y = g2.y = 0;
            v[q] = lo ? fxc{g1.x - g2.y, g1.y + g2.x} : fxc{g1.x + g2.y, g2.x - g1.y};
          }
        }
      });
      __syncthreads();
      fx_second<R, S, true>(nrc, Z, P.LZ, [&](int r, int bk, const fxc* v) {
        fx* o = out + (size_t)(2 * (r0 + r)) * nz + bk;
#pragma unroll
        for (int e = 0; e < S; ++e) {
          o[R * e] = v[e].x;
          o[nz + R * e] = v[e].y;
          mh = max(mh, max(fx_maghi(v[e].x), fx_maghi(v[e].y)));
        }
      });
    });
    __syncthreads();  // the next chunk rewrites Z
  }
  mh = __reduce_max_sync(0xffffffffu, mh);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (int)mh;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mh = max(mh, (unsigned)red[w]);
    *info = make_int2(KIND == FX_SMALL ? row[63] : e0, fx_bits(mh));
  }
}

// ------------------------------------------------------------------ products + analysis
namespace {

__device__ __forceinline__ fx fx_shift(fx x, int s) { return s >= 0 ? x << s : x >> min(-s, 63); }
// exponent of a plane scaled to 62 bits (kFxNone: zero, kFxNan: not finite)
__device__ __forceinline__ int fx_e62(int2 inf) { return inf.x == kFxNan || inf.x == kFxNone ? inf.x : inf.x + inf.y - 62; }
// field of the gradient component d of velocity component c; v_y = -(u_x + w_z) is field 3 plus
// field 10 (the sign is the caller's)
__device__ __forceinline__ int fx_grad(int c, int d) {
  return c == 0 ? 3 + d : c == 2 ? 8 + d : d == 0 ? 6 : d == 1 ? 3 : 7;
}

// sum over the block of s 2^e, exact in integers, as a double in thread 0
__device__ double fx_block_sum(unsigned long long s, int e, int* red) {
  // 24-bit parts: 32 lanes of each stay below 2^29
  const unsigned a = (unsigned)s & 0xffffffu, b = (unsigned)(s >> 24) & 0xffffffu, c = (unsigned)(s >> 48);
  const unsigned ra = __reduce_add_sync(0xffffffffu, a), rb = __reduce_add_sync(0xffffffffu, b),
                 rc = __reduce_add_sync(0xffffffffu, c);
  const int warp = threadIdx.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    red[3 * warp] = (int)ra;
    red[3 * warp + 1] = (int)rb;
    red[3 * warp + 2] = (int)rc;
  }
  __syncthreads();
  double v = 0.0;
  if (threadIdx.x == 0) {
    unsigned long long A = 0, B = 0, Cc = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      A += (unsigned)red[3 * w];
      B += (unsigned)red[3 * w + 1];
      Cc += (unsigned)red[3 * w + 2];
    }
    B += A >> 24;
    Cc += B >> 24;
    const unsigned long long lo = (A & 0xffffffu) | ((B & 0xffffffu) << 24);
    v = ldexp((double)Cc, e + 48) + ldexp((double)lo, e);
  }
  return v;
}

}  // namespace

// CTA = (instance, plane j, component c).  Every factor is scaled to 62 bits, the products keep
// their high 64 bits (2^-60 of the largest product) and are summed at the largest term's
// exponent.  The transforms rescale every row pair and then every x row from its own largest
// value, found by shuffles among the lanes that hold the row.
// SUM (M only, the DNS): also the plane sums of u_c^2 and, in an instance's last CTA, the end of
// the DNS step's norm; the planes are in registers here (as a kernel of its own the sums took 4238
// us per 64 steps of four 32 x 33 x 32 fields, now 4047).
template <bool ADJ, int KIND, bool SUM>
__global__ void __launch_bounds__(FxCfg<KIND>::threads, FxCfg<KIND>::ctas) k_prod_fx(LaunchInfo li, int step_index,
                                                                                    DnsInst* dns) {
  extern __shared__ __align__(16) unsigned char smraw[];
  // factors: 0-2 advecting velocity u_b + u; 3-5 gradient of component c of u (M) or q (N);
  // N: 6-8 q, 9-11 derivative c of u's components; 12: the factor of U' (v, or q_0).
  // A factor is plane a 2^sa (+ plane b 2^sb) (+ a constant), below 2^62, with exponent se.
  __shared__ int se[13], ssa[13], ssb[13], ssd[8];
  __shared__ fx sadd[2];
  __shared__ int sh_eP, sh_bad;
  int local;
  const int b = find_inst(li, blockIdx.x, &local);
  const Inst& I = li.insts[b];
  if (!inst_active(I)) return;
  const int c = local % 3, j = local / 3;
  const int nx = I.nx, nz = I.nz, Mx = I.Mx, Mz = I.Mz, Kx = I.Kx;
  const FxPlanes P = fx_planes(I, blockDim.x);
  fxc* X = reinterpret_cast<fxc*>(smraw);
  fxc* Z = X + Mz * P.LX;
  int* red = reinterpret_cast<int*>(Z + P.chunk * P.LZ);
  int* er = red + 64;   // exponents of the row pairs
  int* ep = er + 64;    // exponents of the x rows
  const double dU = I.ubase[I.ny + j];
  // the factors' planes (offsets uniform in the CTA)
  constexpr int NO = ADJ ? 12 : 6;
  const int fs = I.ny * nx * nz;
  const fx* const U = reinterpret_cast<const fx*>(I.phys) + (size_t)j * nx * nz;
  const fx* const Q = U + (ADJ ? (size_t)kFieldsSynth * fs : 0);
  int of[NO];
#pragma unroll
  for (int k = 0; k < NO; ++k) of[k] = fs * (k < 3 ? k : k < 6 ? fx_grad(c, k - 3) : k < 9 ? k - 6 : fx_grad(k - 9, c));
  if (threadIdx.x < 32) {
    const int k = min((int)threadIdx.x, 12);
    const int slot = k == 12 ? ADJ : k < 3 ? 0 : k < 9 ? ADJ : 0;
    const int comp = k < 6 ? c : k - 9, dir = k < 6 ? k - 3 : c;
    const bool grad = (k >= 3 && k < 6) || (k >= 9 && k < 12);
    const int f = k < 3 ? k : k == 12 ? (ADJ ? 0 : 1) : grad ? fx_grad(comp, dir) : k - 6;
    const bool two = grad && comp == 1 && dir == 1;
    const bool used = k < 6 || (ADJ && k < 12) || (k == 12 && c == (ADJ ? 1 : 0));
    const double cst = k < 2 ? I.ubase[2 * k * I.ny + j] : 0.0;
    const int2 ia = used ? *fx_info(I, slot, f, j) : make_int2(kFxNone, 0);
    const int2 ib = two && used ? *fx_info(I, slot, 10, j) : make_int2(kFxNone, 0);
    const int ea = fx_e62(ia), eb = fx_e62(ib), ec = cst != 0.0 ? fx_bexp(__double2hiint(cst)) - 59 : kFxNone;
    int e = max(ea, max(eb, ec));
    if (e != kFxNan && e != kFxNone && (two || ec != kFxNone)) e += 1;  // room for the sum
    const int sa = ia.x == kFxNone || e == kFxNan ? 0 : ia.x - e, sb = ib.x == kFxNone || e == kFxNan ? 0 : ib.x - e;
    // terms: 0-2 advection, 3-5 transposed gradient, 6 the base flow's shear
    const int t = threadIdx.x;
    int x = __shfl_sync(0xffffffffu, e, t < 3 ? t : (3 + t) & 31);
    const int y = __shfl_sync(0xffffffffu, e, t < 3 ? 3 + t : (6 + t) & 31);
    if (t == 6) x = dU != 0.0 ? fx_bexp(__double2hiint(dU)) - 59 : kFxNone;
    const bool term = t < 3 || (ADJ && t < 6) || t == 6;
    const int et = !term || x == kFxNone || y == kFxNone ? kFxNone : x + y + 64;
    const bool nan = term && (x == kFxNan || y == kFxNan) && !(t == 6 && y == kFxNone);
    const int em = __reduce_max_sync(0xffffffffu, nan ? kFxNone : et);
    const bool any = __any_sync(0xffffffffu, nan);
    if (t < 13) {
      se[t] = e;
      ssa[t] = sa;
      ssb[t] = sb;
    }
    if (t < 2) sadd[t] = ec != kFxNone && e != kFxNan ? fx_from(cst, e) : 0;
    if (t < 7) ssd[t] = min(et == kFxNone ? 63 : em - et, 63);
    if (t == 0) {
      sh_eP = em;
      sh_bad = any;
    }
  }
  __syncthreads();
  const bool bad = sh_bad != 0;
  int eP = sh_eP;
  const bool zero = eP < kFxNone / 2;
  unsigned long long sq = 0;
  const int eq = ADJ ? se[6 + c] : kFxNone;
  const bool sqok = ADJ && eq != kFxNan && eq != kFxNone;
  const int nr = nx / 2;
  const unsigned nzm = I.nz_mul;
  const fx dUx = c == (ADJ ? 1 : 0) ? fx_from(dU, fx_bexp(__double2hiint(dU)) - 59) : 0;
  const int lgz = 32 - __clz(nz - 1), lgx = 32 - __clz(nx - 1);
  int sa[NO], sd[7];
#pragma unroll
  for (int k = 0; k < NO; ++k) sa[k] = ssa[k];
#pragma unroll
  for (int k = 0; k < 7; ++k) sd[k] = ssd[k];
  const fx add0 = sadd[0], add1 = sadd[1];
  // One loop over the transform stages, so that the z stage of every chunk of rows and the x
  // stage run the same instructions (the kernel's straight-line code otherwise exceeds the
  // instruction cache): job g < nch is chunk g's products and z stage, job nch the x stage.
  const int nch = !SUM && (bad || (zero && !ADJ)) ? 0 : (nr + P.chunk - 1) / P.chunk;
  const int2 iu = SUM ? *fx_info(I, 0, c, j) : make_int2(kFxNone, 0);
  const int eu = fx_e62(iu);
  const bool suok = SUM && eu != kFxNan && eu != kFxNone;
  const bool live = !bad && !zero;
  int* align = ep + 64;  // right shift of each row pair's values in the x stage (z stage: none)
  if (threadIdx.x < 64) align[threadIdx.x] = 0;
  for (int g = 0; g <= nch; ++g) {
    const bool xs = g == nch;
    const int r0 = g * P.chunk, nrc = xs ? 0 : min(P.chunk, nr - r0), base = 2 * r0 * nz;
    // products of the chunk's rows, two neighbouring points per thread: row 2r in the real
    // part, 2r + 1 in the imaginary part
    for (int t = 2 * threadIdx.x; t < 2 * nrc * nz; t += 2 * blockDim.x) {
      const int row = fx_div(t, nzm), z = t - row * nz, e = base + t;
      longlong2 x[NO];
#pragma unroll
      for (int k = 0; k < NO; ++k)
        x[k] = __ldg(reinterpret_cast<const longlong2*>((k >= 3 && k < 9 ? Q : U) + of[k] + e));
      longlong2 b4 = make_longlong2(0, 0), b10 = b4, pv = b4;
      if (c == 1) {  // v_y = -(u_x + w_z)
        b4 = __ldg(reinterpret_cast<const longlong2*>(Q + 10 * fs + e));
        if (ADJ) b10 = __ldg(reinterpret_cast<const longlong2*>(U + 10 * fs + e));
      }
      const longlong2 uc = c == 0 ? x[0] : c == 1 ? x[1] : x[2];
      if (!ADJ && c == 0) pv = __ldg(reinterpret_cast<const longlong2*>(U + fs + e));
      fx val[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        fx v[NO];
#pragma unroll
        for (int k = 0; k < NO; ++k) {
          v[k] = h ? x[k].y : x[k].x;
          v[k] = k < 2 || k == 4 || k == 10 ? fx_shift(v[k], sa[k]) : v[k] << sa[k];
        }
        v[0] += add0;
        v[1] += add1;
        if (c == 1) {
          v[4] = -(v[4] + fx_shift(h ? b4.y : b4.x, ssb[4]));
          if (ADJ) v[10 % NO] = -(v[10 % NO] + fx_shift(h ? b10.y : b10.x, ssb[10]));
        }
        fx a = (fx_mul64(v[0], v[3]) >> sd[0]) + (fx_mul64(v[1], v[4]) >> sd[1]) + (fx_mul64(v[2], v[5]) >> sd[2]);
        if (suok) {
          const fx q = ((h ? uc.y : uc.x) << (62 - iu.y)) >> 2;  // at most 64 squares below 2^56
          sq += (unsigned long long)fx_mul64(q, q);
        }
        if (!ADJ) {
          if (c == 0) a += fx_mul64(dUx, (h ? pv.y : pv.x) << ssa[12]) >> sd[6];
          a = -a;
        } else {
          a -= (fx_mul64(v[6 % NO], v[9 % NO]) >> sd[3]) + (fx_mul64(v[7 % NO], v[10 % NO]) >> sd[4]) +
               (fx_mul64(v[8 % NO], v[11 % NO]) >> sd[5]);
          if (c == 1) a -= fx_mul64(dUx, v[6 % NO]) >> sd[6];
          const fx qc = (c == 0 ? v[6 % NO] : c == 1 ? v[7 % NO] : v[8 % NO]) >> 2;  // at most 64 squares below 2^56
          sq += (unsigned long long)fx_mul64(qc, qc);
        }
        val[h] = a;
      }
      fxc* o = Z + (row >> 1) * P.LZ;
      reinterpret_cast<fx*>(o + fx_in<KIND>(fx_plan_of<KIND>(nz), z))[row & 1] = val[0];
      reinterpret_cast<fx*>(o + fx_in<KIND>(fx_plan_of<KIND>(nz), z, 1))[row & 1] = val[1];
    }
    if (!live) continue;
    if (xs) {
      int emax = kFxNone;
      for (int r = threadIdx.x & 31; r < nr; r += 32) emax = max(emax, er[r]);
      emax = __reduce_max_sync(0xffffffffu, emax);
      if (threadIdx.x < nr) align[threadIdx.x] = emax - er[threadIdx.x];
      eP = emax;
    }
    __syncthreads();
    fxc* const buf = xs ? X : Z;
    const int LS = xs ? P.LX : P.LZ, rows = xs ? Mz : nrc, lg = xs ? lgx : lgz + 1;
    int* const eo = xs ? ep : er + r0;
    fx_length<KIND>(xs ? nx : nz, [&](auto rc) {
      constexpr int R = decltype(rc)::R, S = decltype(rc)::S, G = S <= 8 ? 8 : 16;
      fx_first<R, S, false>(rows, buf, LS, xs ? I.twfx_x : I.twfx_z, [&](int r, int n, fxc* v) {
        unsigned mh = 0;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const fxc a = buf[r * LS + fx_slot<S>(q, n)];
          const int d = min(align[(n + S * q) >> 1], 63);
          v[q] = fxc{a.x >> d, a.y >> d};
          mh = max(mh, max(fx_maghi(v[q].x), fx_maghi(v[q].y)));
        }
        const unsigned m = ((1u << G) - 1) << (threadIdx.x & 31 & ~(G - 1));
#pragma unroll
        for (int o = 1; o < G; o <<= 1) mh = max(mh, __shfl_xor_sync(m, mh, o));
        // sqrt(2) n max <= 2^61 (z stage: the unpacking adds two values), 2^62 (x stage)
        const int s = fx_bits(mh) + 1 + lg - 62;
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = fxc{fx_shift(v[q].x, -s), fx_shift(v[q].y, -s)};
        if (n == 0) eo[r] = eP + s - (xs ? 0 : 1);
      });
      __syncthreads();
      fx_second<R, S, false>(rows, buf, LS, [&](int r, int bk, const fxc* v) {
        fxc* o = buf + r * LS;
#pragma unroll
        for (int e = 0; e < S; ++e) o[fx_slot<S>(bk, e)] = v[e];
      });
    });
    __syncthreads();
    // rows x1 and x2 of each pair, twice their value: F1 = H_p + conj(H_-p), F2 = -i (H_p - conj(H_-p))
    for (int t = threadIdx.x; t < nrc * Mz; t += blockDim.x) {
      const int r = fx_div(t, I.mz_mul), p = t - r * Mz, pm = p == 0 ? 0 : nz - p;
      const int kp = fx_div(p, I.rz_mul), km = fx_div(pm, I.rz_mul), Rz = fx_plan_of<KIND>(nz).R;
      const fxc hp = Z[r * P.LZ + fx_out<KIND>(fx_plan_of<KIND>(nz), p - kp * Rz, kp)], hm = Z[r * P.LZ + fx_out<KIND>(fx_plan_of<KIND>(nz), pm - km * Rz, km)];
      const int x = 2 * (r0 + r);
      X[p * P.LX + fx_in<KIND>(fx_plan_of<KIND>(nx), x)] = fxc{hp.x + hm.x, hp.y - hm.y};
      X[p * P.LX + fx_in<KIND>(fx_plan_of<KIND>(nx), x, 1)] = fxc{hp.y + hm.y, hm.x - hp.x};
    }
    if (!xs) __syncthreads();
  }
  double2* dst = I.xz + ((size_t)c * I.ny + j) * I.nmodes;
  const int Rx = fx_plan_of<KIND>(nx).R;
  for (int t = threadIdx.x; t < I.nmodes; t += blockDim.x) {
    const int i = fx_div(t, I.mz_mul), p = t - i * Mz, bin = xbin(i, Kx, Mx, nx), k3 = fx_div(bin, I.rx_mul);
    double2 o = make_double2(0.0, 0.0);
    if (bad) o.x = o.y = __longlong_as_double(0x7ff8000000000000LL);
    if (live) {
      fxc a = X[p * P.LX + fx_out<KIND>(fx_plan_of<KIND>(nx), bin - k3 * Rx, k3)];
      if (I.nfx_h) a = fxc{fx_mulc(a.x, I.nfx_h, I.nfx_l), fx_mulc(a.y, I.nfx_h, I.nfx_l)};
      const int e0 = ep[p] + I.nfx_e;
      o = make_double2(__longlong_as_double((long long)fx_double_bits(a.x, e0)),
                       __longlong_as_double((long long)fx_double_bits(a.y, e0)));
    }
    dst[t] = o;
  }
  if (ADJ) {
    const double s = fx_block_sum(sq, sqok ? 2 * eq + 68 : 0, red);
    if (threadIdx.x == 0)
      I.normpart[(size_t)c * I.ny + j] = eq == kFxNan || bad ? __longlong_as_double(0x7ff8000000000000LL) : sqok ? s : 0.0;
  }
  if (ADJ && step_index >= 0) finish_norm(I, step_index);
  if (SUM) {
    const double s = fx_block_sum(sq, suok ? 2 * eu + 68 : 0, red);
    if (threadIdx.x == 0)
      I.normpart[(size_t)c * I.ny + j] = eu == kFxNan ? __longlong_as_double(0x7ff8000000000000LL) : s;
    finish_dns(I, dns[b]);
  }
}

// CTA = (instance, plane j, component c): sum over the plane of the squared velocity component
// c of a slot (0: u, 1: q).
__global__ void __launch_bounds__(128) k_norm_planes_fx(LaunchInfo li, int slot) {
  __shared__ int red[64];
  int local;
  const int b = find_inst(li, blockIdx.x, &local);
  const Inst& I = li.insts[b];
  if (!inst_active(I)) return;
  const int c = local % 3, j = local / 3, n = I.nx * I.nz;
  const int2 inf = *fx_info(I, slot, c, j);
  const int e = fx_e62(inf), sa = 62 - inf.y;
  const bool ok = e != kFxNan && e != kFxNone;
  const fx* a = reinterpret_cast<const fx*>(I.phys) + (((size_t)slot * kFieldsSynth + c) * I.ny + j) * (size_t)n;
  unsigned long long sq = 0;
  if (ok)
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      const fx q = (a[t] << sa) >> 2;  // at most 128 squares below 2^56 per thread
      sq += (unsigned long long)fx_mul64(q, q);
    }
  const double s = fx_block_sum(sq, ok ? 2 * e + 68 : 0, red);
  if (threadIdx.x == 0)
    I.normpart[(size_t)c * I.ny + j] = e == kFxNan ? __longlong_as_double(0x7ff8000000000000LL) : s;
}

void launch_xzsynth_fx(int kind, int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int slot, int nf) {
  if (kind == FX_ANY) k_synth_fx<FX_ANY><<<ctas, threads, smem, s>>>(li, slot, nf);
  else if (kind == FX_BIG) k_synth_fx<FX_BIG><<<ctas, threads, smem, s>>>(li, slot, nf);
  else k_synth_fx<FX_SMALL><<<ctas, threads, smem, s>>>(li, slot, nf);
}
template <int KIND>
static void launch_prod_kind(bool adj, int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int step_index,
                             DnsInst* dns) {
  if (adj) k_prod_fx<true, KIND, false><<<ctas, threads, smem, s>>>(li, step_index, nullptr);
  else if (dns) k_prod_fx<false, KIND, true><<<ctas, threads, smem, s>>>(li, -1, dns);
  else k_prod_fx<false, KIND, false><<<ctas, threads, smem, s>>>(li, -1, nullptr);
}
void launch_prod_fx(int kind, bool adj, int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li,
                    int step_index, DnsInst* dns) {
  (kind == FX_ANY   ? launch_prod_kind<FX_ANY>
   : kind == FX_BIG ? launch_prod_kind<FX_BIG>
                    : launch_prod_kind<FX_SMALL>)(adj, ctas, threads, smem, s, li, step_index, dns);
}
void launch_norm_planes_fx(int ctas, cudaStream_t s, LaunchInfo li, int slot) {
  k_norm_planes_fx<<<ctas, 128, 0, s>>>(li, slot);
}
template <int KIND>
static cudaError_t set_kind_smem(size_t synth, size_t prod) {
  cudaError_t e;
  if ((e = raise_smem_limit((const void*)k_synth_fx<KIND>, synth))) return e;
  if ((e = raise_smem_limit((const void*)k_prod_fx<true, KIND, false>, prod))) return e;
  if ((e = raise_smem_limit((const void*)k_prod_fx<false, KIND, true>, prod))) return e;
  return raise_smem_limit((const void*)k_prod_fx<false, KIND, false>, prod);
}
cudaError_t set_planes_fx_smem(int kind, size_t synth, size_t prod) {
  return kind == FX_ANY   ? set_kind_smem<FX_ANY>(synth, prod)
         : kind == FX_BIG ? set_kind_smem<FX_BIG>(synth, prod)
                          : set_kind_smem<FX_SMALL>(synth, prod);
}

}  // namespace pcf
