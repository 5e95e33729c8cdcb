// Snapshot vector psi and DMD steady-state extrapolation (paper §6.1-6.2).
//
// psi (§6.2, "minimum number of independent variables"): per independent Fourier mode
// (p > 0: every m; p = 0: m > 0) the Chebyshev coefficients 0..N-4 of v and 0..N-2 of
// the wall-normal vorticity eta = i kz u - i kx w (real parts, then imaginary parts),
// followed by the coefficients 0..N-2 of the mean u and w.  The remaining coefficients
// follow from v = dv/dy = 0 and eta = 0 at the walls, u and w from the divergence
// constraint and eta.
//
// DMD: the snapshot matrix S = [s_0 .. s_M] is reduced by a Householder QR on the
// device (S = Q R, Q never formed); Psi = Q R[:, 0:M] and Psi' = Q R[:, 1:M+1], so the
// SVD of Psi, the projected operator A~ = U^T Psi' V Sigma^-1, its eigenpairs and the
// least-squares amplitudes are all computed from the small R on the host; the steady
// state b_1 phi_1 = Psi' (Re(b_1 V Sigma^-1 w_1)) is a combination of the snapshots.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <condition_variable>
#include <cstdio>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include "pcf_ctx.h"
#include "pcf_linalg.h"

namespace pcf {

// ------------------------------------------------------------------ psi <-> uhat
__global__ void k_psi_extract(const double2* __restrict__ uhat, long long state_len, double* __restrict__ psi,
                              long long psi_len, const int* __restrict__ indep, int nindep,
                              const double* __restrict__ kx, const double* __restrict__ kz, int Mz, int ny, int nm,
                              int B) {
  const int N = ny - 1;
  const long long per = (long long)(nindep + 1) * ny;
  const long long total = per * B;
  const int segv = N - 3, sege = N - 1, seg = 2 * segv + 2 * sege;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(t / per);
    const long long r = t - (long long)b * per;
    const int q = (int)(r / ny), n = (int)(r - (long long)q * ny);
    const double2* u = uhat + (size_t)b * state_len;
    double* out = psi + (size_t)b * psi_len;
    if (q < nindep) {
      const int i = indep[2 * q], j = indep[2 * q + 1], m = i * Mz + j;
      double* o = out + (size_t)q * seg;
      const double2 vv = u[((size_t)1 * nm + m) * ny + n];
      if (n < segv) {
        o[n] = vv.x;
        o[segv + n] = vv.y;
      }
      if (n < sege) {
        const double2 uu = u[((size_t)0 * nm + m) * ny + n], ww = u[((size_t)2 * nm + m) * ny + n];
        const double a = kx[i], c = kz[j];
        o[2 * segv + n] = -c * uu.y + a * ww.y;
        o[2 * segv + sege + n] = c * uu.x - a * ww.x;
      }
    } else if (n < sege) {
      double* o = out + (size_t)nindep * seg;
      o[n] = u[((size_t)0 * nm + 0) * ny + n].x;
      o[sege + n] = u[((size_t)2 * nm + 0) * ny + n].x;
    }
  }
}

// One warp per (instance, independent mode or mean): rebuild the mode's u, v, w.  Coefficients
// sit in shared memory; the lanes share the wall sums and the assembly, four lanes run the
// derivative recurrence (parts x parity classes).  One thread per mode with its four
// coefficient columns in local memory took 112 us for 20 states at 32x33x32.
constexpr int kRebuildWarps = 4, kRebuildLen = 132;
__device__ __forceinline__ double warp_sum(double s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
__global__ void __launch_bounds__(32 * kRebuildWarps)
    k_psi_rebuild(const double* __restrict__ psi, long long psi_len, double2* __restrict__ uhat, long long state_len,
                  const int* __restrict__ indep, int nindep, const double* __restrict__ kx,
                  const double* __restrict__ kz, int Mx, int Mz, int ny, int nm, int B) {
  __shared__ double sh[kRebuildWarps][6][kRebuildLen];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kRebuildWarps + warp;
  if (t >= B * (nindep + 1)) return;
  const int b = t / (nindep + 1), q = t - b * (nindep + 1);
  const int N = ny - 1;
  const int segv = N - 3, sege = N - 1, seg = 2 * segv + 2 * sege;
  const double* in = psi + (size_t)b * psi_len;
  double2* u = uhat + (size_t)b * state_len;
  double *vr = sh[warp][0], *vi = sh[warp][1], *er = sh[warp][2], *ei = sh[warp][3], *xr = sh[warp][4], *xi = sh[warp][5];
  // the top coefficient of each parity class from sum a_n = 0
  const auto dirichlet = [&](double* a) {
    for (int par = 0; par < 2; ++par) {
      const int top = (N % 2 == par) ? N : N - 1;
      double s = 0.0;
      for (int n = par + 2 * lane; n < top; n += 64) s += a[n];
      s = warp_sum(s);
      if (lane == 0) a[top] = -s;
    }
    __syncwarp();
  };
  if (q == nindep) {
    // mean u, w: Dirichlet completion, imaginary part zero; v = 0
    const double* o = in + (size_t)nindep * seg;
    for (int c = 0; c < 2; ++c) {
      for (int n = lane; n <= N; n += 32) vr[n] = n < sege ? o[c * sege + n] : 0.0;
      __syncwarp();
      dirichlet(vr);
      const int comp = c == 0 ? 0 : 2;
      for (int n = lane; n <= N; n += 32) u[((size_t)comp * nm + 0) * ny + n] = make_double2(vr[n], 0.0);
      __syncwarp();
    }
    for (int n = lane; n <= N; n += 32) u[((size_t)1 * nm + 0) * ny + n] = make_double2(0.0, 0.0);
    return;
  }
  const int i = indep[2 * q], j = indep[2 * q + 1], m = i * Mz + j;
  const double* o = in + (size_t)q * seg;
  for (int n = lane; n <= N; n += 32) {
    vr[n] = n < segv ? o[n] : 0.0;
    vi[n] = n < segv ? o[segv + n] : 0.0;
    er[n] = n < sege ? o[2 * segv + n] : 0.0;
    ei[n] = n < sege ? o[2 * segv + sege + n] : 0.0;
  }
  __syncwarp();
  // v: for each parity class the two top coefficients from sum a_n = 0, sum n^2 a_n = 0
  for (int par = 0; par < 2; ++par) {
    const int hi = (N % 2 == par) ? N : N - 1, lo = hi - 2;
    for (int part = 0; part < 2; ++part) {
      double* v = part ? vi : vr;
      double s0 = 0, s1 = 0;
      for (int n = par + 2 * lane; n < lo; n += 64) {
        s0 += v[n];
        s1 = fma((double)(n * n), v[n], s1);
      }
      s0 = warp_sum(s0);
      s1 = warp_sum(s1);
      const double h2 = (double)hi * hi, l2 = (double)lo * lo, det = l2 - h2;
      if (lane == 0) {
        v[hi] = (s1 - s0 * l2) / det;
        v[lo] = (s0 * h2 - s1) / det;
      }
    }
  }
  __syncwarp();
  dirichlet(er);
  dirichlet(ei);
  // dv/dy by the coefficient recurrence
  if (lane < 4) {
    const double* v = lane & 1 ? vi : vr;
    double* x = lane & 1 ? xi : xr;
    double acc = 0.0;
    const int n0 = (N - (lane >> 1));  // class of N, or of N - 1
    for (int n = n0; n >= 0; n -= 2) {
      if (n + 1 <= N) acc = fma(2.0 * (n + 1), v[n + 1], acc);
      x[n] = n == 0 ? 0.5 * acc : acc;
    }
  }
  __syncwarp();
  const double a = kx[i], c = kz[j], ik2 = 1.0 / (a * a + c * c);
  const int mconj = (Mx - i) * Mz;  // storage index of (-m, 0)
  for (int n = lane; n <= N; n += 32) {
    const double xre = -xr[n], xim = -xi[n];
    const double2 uu = make_double2((a * xim + c * ei[n]) * ik2, -(a * xre + c * er[n]) * ik2);
    const double2 vv = make_double2(vr[n], vi[n]);
    const double2 ww = make_double2((c * xim - a * ei[n]) * ik2, (-c * xre + a * er[n]) * ik2);
    u[((size_t)0 * nm + m) * ny + n] = uu;
    u[((size_t)1 * nm + m) * ny + n] = vv;
    u[((size_t)2 * nm + m) * ny + n] = ww;
    if (j == 0) {
      u[((size_t)0 * nm + mconj) * ny + n] = make_double2(uu.x, -uu.y);
      u[((size_t)1 * nm + mconj) * ny + n] = make_double2(vv.x, -vv.y);
      u[((size_t)2 * nm + mconj) * ny + n] = make_double2(ww.x, -ww.y);
    }
  }
}

// ------------------------------------------------------------------ Householder QR (R only)
// A: rows x ncol column-major with leading dimension ld (in doubles).
constexpr int kQrBlocks = 64;

__global__ void k_qr_dots(const double* __restrict__ A, long long rows, long long ld, int j, int ncol,
                          double* __restrict__ part) {
  __shared__ double red[32];
  const double* aj = A + (size_t)j * ld;
  for (int k = j; k < ncol; ++k) {
    const double* ak = A + (size_t)k * ld;
    double s = 0.0;
    for (long long i = j + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < rows;
         i += (long long)gridDim.x * blockDim.x)
      s = fma(aj[i], ak[i], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
      part[(size_t)(k - j) * gridDim.x + blockIdx.x] = t;
    }
    __syncthreads();
  }
}

// coef[k] (k > j) = 2 v^T a_k / v^T v for the reflector v = x - alpha e_j; alpha[j] = R_jj.
__global__ void k_qr_reflect(double* __restrict__ A, long long ld, int j, int ncol, const double* __restrict__ part,
                             int G, double* __restrict__ coef, double* __restrict__ alpha) {
  __shared__ double sxj, salpha, svtv;
  if (threadIdx.x == 0) {
    double x2 = 0.0;
    for (int g = 0; g < G; ++g) x2 += part[g];
    const double xj = A[(size_t)j * ld + j];
    const double nrm = sqrt(x2);
    const double al = xj >= 0.0 ? -nrm : nrm;
    sxj = xj;
    salpha = al;
    svtv = 2.0 * (x2 - al * xj);
    alpha[j] = al;
  }
  __syncthreads();
  for (int k = j + 1 + threadIdx.x; k < ncol; k += blockDim.x) {
    double s = 0.0;
    for (int g = 0; g < G; ++g) s += part[(size_t)(k - j) * G + g];
    const double vta = s - salpha * A[(size_t)k * ld + j];
    coef[k] = svtv > 0.0 ? 2.0 * vta / svtv : 0.0;
  }
  __syncthreads();
  if (threadIdx.x == 0) A[(size_t)j * ld + j] = sxj - salpha;
}

__global__ void k_qr_update(double* __restrict__ A, long long rows, long long ld, int j, int ncol,
                            const double* __restrict__ coef) {
  for (long long i = j + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < rows;
       i += (long long)gridDim.x * blockDim.x) {
    const double vi = A[(size_t)j * ld + i];
    for (int k = j + 1; k < ncol; ++k) A[(size_t)k * ld + i] = fma(-coef[k], vi, A[(size_t)k * ld + i]);
  }
}

// Tall-skinny QR, R only: CTA b factors the rows [b RB, (b + 1) RB) of A (n columns, leading
// dimension ld) by Householder reflections in shared memory and writes its R as rows b n ..
// b n + n - 1 of out (leading dimension ldo, zeros below the diagonal); the stacked R's are
// factored again until one CTA is left.  A warp takes a column's projection and update; the
// warp that updates the next pivot column also takes its norm, so that a step has one barrier.
// The column-by-column QR over the whole matrix (three launches per column, each waiting for
// sums over all rows) took 940 us for 20218 x 21; this takes four launches.
constexpr int kTsqrThreads = 512;
__global__ void __launch_bounds__(kTsqrThreads) k_tsqr(const double* __restrict__ A, long long ld, long long rows, int n,
                                                       int RB, double* __restrict__ out, long long ldo) {
  extern __shared__ double q[];  // [n][RB + 1]
  __shared__ double s_alpha, s_f;  // R_jj and 2 / v^T v of the pivot column (0: no reflection)
  const int P = RB + 1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = kTsqrThreads / 32;
  const long long r0 = (long long)blockIdx.x * RB;
  const int m = (int)min((long long)RB, rows - r0);
  for (int t = threadIdx.x; t < n * RB; t += kTsqrThreads) {
    const int k = t / RB, i = t - k * RB;
    q[k * P + i] = i < m ? A[(size_t)k * ld + r0 + i] : 0.0;
  }
  __syncthreads();
  // pivot j: x = a_j[j:], alpha = -sign(x_j) |x|, v = x - alpha e_j in place
  const auto pivot = [&](int j) {
    double* x = q + j * P;
    double s = 0.0;
    for (int i = j + lane; i < RB; i += 32) s = fma(x[i], x[i], s);
    s = warp_sum(s);
    if (lane == 0) {
      const double xj = x[j], nrm = sqrt(s), al = xj >= 0.0 ? -nrm : nrm, vtv = 2.0 * (s - al * xj);
      s_alpha = al;
      s_f = vtv > 0.0 ? 2.0 / vtv : 0.0;
      x[j] = xj - al;
    }
    __syncwarp();
  };
  if (warp == 0) pivot(0);
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const double f = s_f, al = s_alpha;
    __syncthreads();  // the next pivot overwrites them
    const double* v = q + j * P;
    for (int k = j + 1 + warp; k < n; k += nw) {
      double* a = q + k * P;
      double s = 0.0;
      for (int i = j + lane; i < RB; i += 32) s = fma(v[i], a[i], s);
      s = warp_sum(s) * f;
      for (int i = j + lane; i < RB; i += 32) a[i] = fma(-s, v[i], a[i]);
      __syncwarp();
      if (k == j + 1) pivot(k);
    }
    __syncthreads();
    // row j of R: the diagonal, and the updated columns
    for (int k = threadIdx.x; k < n; k += kTsqrThreads) {
      const double d = k < j ? 0.0 : k == j ? al : q[k * P + j];
      out[(size_t)k * ldo + (size_t)blockIdx.x * n + j] = d;
    }
  }
}

// cand[c][i] = sum_k C[c][k] S[i][k+1]  (k < M): steady states as combinations of snapshots, four
// candidates per thread on each load
__global__ void __launch_bounds__(256) k_combine(const double* __restrict__ S, long long rows, long long ld, int M,
                                                 const double* __restrict__ C, int ncand, double* __restrict__ out,
                                                 long long out_ld) {
  const int c0 = 4 * blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < rows;
       i += (long long)gridDim.x * blockDim.x) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k = 0; k < M; ++k) {
      const double x = S[(size_t)(k + 1) * ld + i];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c0 + c < ncand) s[c] = fma(C[(size_t)(c0 + c) * M + k], x, s[c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c0 + c < ncand) out[(size_t)(c0 + c) * out_ld + i] = s[c];
  }
}

}  // namespace pcf

using namespace pcf;

namespace {

thread_local char g_dmd_err[256] = "";

#define DMD_CUDA(call)                                                                    \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) {                                                              \
      snprintf(g_dmd_err, sizeof(g_dmd_err), "%s: %s", #call, cudaGetErrorString(e_));    \
      return PCF_ECUDA;                                                                   \
    }                                                                                     \
  } while (0)

pcf_status ensure_indep(pcf_ctx* c) {
  if (c->d_indep) return PCF_OK;
  std::vector<int> idx;
  for (int i = 0; i < c->Mx; ++i)
    for (int j = 0; j < c->Mz; ++j) {
      const int m = i <= c->Kx ? i : i - c->Mx;
      if (j > 0 || m >= 1) {
        idx.push_back(i);
        idx.push_back(j);
      }
    }
  c->nindep = (int)idx.size() / 2;
  c->psi_len = pcf_psi_len(c->prm.nx, c->prm.ny, c->prm.nz);
  DMD_CUDA(cudaMalloc(&c->d_indep, idx.size() * sizeof(int)));
  c->allocs.push_back(c->d_indep);
  DMD_CUDA(cudaMemcpy(c->d_indep, idx.data(), idx.size() * sizeof(int), cudaMemcpyHostToDevice));
  return PCF_OK;
}

pcf_status ensure_dmd(pcf_ctx* c, int ncol) {
  if (c->dmd_cap >= ncol) return PCF_OK;
  const int cap = std::max(ncol, 32);
  // whole batches of either evaluation context (norms of the masked instances are written too)
  const int ncand = cap + std::max(c->B, 32);
  double *A, *part, *coef, *cpsi, *J, *cc;
  double2* cu;
  DMD_CUDA(cudaMalloc(&A, sizeof(double) * (size_t)c->psi_len * cap));
  DMD_CUDA(cudaMalloc(&part, sizeof(double) * (size_t)kQrBlocks * cap));
  DMD_CUDA(cudaMalloc(&coef, sizeof(double) * 2 * (size_t)cap));
  DMD_CUDA(cudaMalloc(&cpsi, sizeof(double) * (size_t)c->psi_len * ncand));
  DMD_CUDA(cudaMalloc(&cu, sizeof(double2) * (size_t)c->state_len * ncand));
  DMD_CUDA(cudaMalloc(&J, sizeof(double) * (size_t)ncand));
  DMD_CUDA(cudaMalloc(&cc, sizeof(double) * (size_t)cap * ncand));
  for (void* p : {(void*)A, (void*)part, (void*)coef, (void*)cpsi, (void*)cu, (void*)J, (void*)cc})
    c->allocs.push_back(p);
  c->dmd_A = A;
  c->dmd_part = part;
  c->dmd_coef = coef;
  c->dmd_cpsi = cpsi;
  c->dmd_cu = cu;
  c->dmd_J = J;
  c->dmd_c = cc;
  c->dmd_cap = cap;
  c->dmd_ncand_cap = ncand;
  return PCF_OK;
}

pcf_status sync_in(pcf_ctx* c) {
  DMD_CUDA(cudaEventRecord(c->ev_in, c->user));
  DMD_CUDA(cudaStreamWaitEvent(c->cs, c->ev_in, 0));
  return PCF_OK;
}
pcf_status sync_out(pcf_ctx* c) {
  DMD_CUDA(cudaEventRecord(c->ev_out, c->cs));
  DMD_CUDA(cudaStreamWaitEvent(c->user, c->ev_out, 0));
  return PCF_OK;
}

#define DMD_TRY(x)               \
  do {                           \
    pcf_status s_ = (x);         \
    if (s_ != PCF_OK) return s_; \
  } while (0)

// R of the QR of the ncol snapshots (columns of S, leading dimension ld), row-major, on the host.
pcf_status snapshot_r(pcf_ctx* c, const double* S, long long ld, int ncol, std::vector<double>* R) {
  const long long rows = c->psi_len;
  R->assign((size_t)ncol * ncol, 0.0);
  std::vector<double> h((size_t)ncol * ncol);
  const int RB = std::max(256, 2 * ncol);
  const size_t sm = sizeof(double) * (size_t)ncol * (RB + 1);
  const auto blocks = [&](long long r) { return (r + RB - 1) / RB; };
  const long long n1 = blocks(rows) * ncol, n2 = blocks(n1) * ncol;  // rows of the first two levels' outputs
  if (sm <= 227 * 1024 - 64 && n1 + n2 <= rows) {
    // two levels at a time in the workspace (rows x cap): level 1, 3, .. at its start, 2, 4, .. behind it
    DMD_CUDA(raise_smem_limit((const void*)k_tsqr, sm));
    const double* src = S;
    long long r = rows, l = ld;
    for (int level = 0;; ++level) {
      const long long nb = blocks(r), ro = nb * ncol;
      double* dst = level & 1 ? c->dmd_A + n1 * ncol : c->dmd_A;
      k_tsqr<<<(int)nb, kTsqrThreads, sm, c->cs>>>(src, l, r, ncol, RB, dst, ro);
      src = dst;
      r = l = ro;
      if (nb == 1) break;
    }
    DMD_CUDA(cudaGetLastError());
    DMD_CUDA(cudaMemcpyAsync(h.data(), src, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, c->cs));
    DMD_CUDA(cudaStreamSynchronize(c->cs));
    for (int j = 0; j < ncol; ++j)
      for (int k = j; k < ncol; ++k) (*R)[(size_t)j * ncol + k] = h[(size_t)k * ncol + j];
    return PCF_OK;
  }
  // more columns than a CTA's shared memory holds, or few rows: column by column over the whole
  // matrix, copied into the workspace (column-major, ld = rows)
  DMD_CUDA(cudaMemcpy2DAsync(c->dmd_A, sizeof(double) * rows, S, sizeof(double) * ld, sizeof(double) * rows, ncol,
                             cudaMemcpyDeviceToDevice, c->cs));
  double* alpha = c->dmd_coef + c->dmd_cap;
  for (int j = 0; j < ncol; ++j) {
    k_qr_dots<<<kQrBlocks, 256, 0, c->cs>>>(c->dmd_A, rows, rows, j, ncol, c->dmd_part);
    k_qr_reflect<<<1, 128, 0, c->cs>>>(c->dmd_A, rows, j, ncol, c->dmd_part, kQrBlocks, c->dmd_coef, alpha);
    if (j + 1 < ncol) k_qr_update<<<kQrBlocks, 256, 0, c->cs>>>(c->dmd_A, rows, rows, j, ncol, c->dmd_coef);
  }
  DMD_CUDA(cudaGetLastError());
  std::vector<double> al(ncol);
  DMD_CUDA(cudaMemcpy2DAsync(h.data(), sizeof(double) * ncol, c->dmd_A, sizeof(double) * rows,
                             sizeof(double) * ncol, ncol, cudaMemcpyDeviceToHost, c->cs));
  DMD_CUDA(cudaMemcpyAsync(al.data(), alpha, sizeof(double) * ncol, cudaMemcpyDeviceToHost, c->cs));
  DMD_CUDA(cudaStreamSynchronize(c->cs));
  for (int j = 0; j < ncol; ++j) {
    (*R)[(size_t)j * ncol + j] = al[j];
    for (int k = j + 1; k < ncol; ++k) (*R)[(size_t)j * ncol + k] = h[(size_t)k * ncol + j];
  }
  return PCF_OK;
}

// Context that evaluates `want` candidates' residuals, all or many at a time: c itself, or one over
// more instances of the same problem (multiples of four, at most 32, within 1 GiB of plane buffers),
// made on first use and kept with c until it or a call with more candidates ends it.  One candidate
// per pass left the GPU mostly idle: 19 passes of 90 us.
pcf_ctx* eval_ctx(pcf_ctx* c, int want) {
  const long long per = 2LL * kFieldsSynth * c->prm.nx * c->prm.ny * c->prm.nz * 8;
  const int nb = (int)std::min<long long>(std::min((want + 3) / 4 * 4, 32), (1LL << 30) / per);
  if (nb <= c->B) return c;
  if (c->dmd_eval && c->dmd_eval->B < nb) {
    pcf_destroy(c->dmd_eval);
    c->dmd_eval = nullptr;
  }
  if (!c->dmd_eval && pcf_make_child(c, nb, &c->dmd_eval) != PCF_OK) {
    c->dmd_eval = nullptr;
    cudaGetLastError();  // a failed allocation is answered by c itself
  }
  return c->dmd_eval ? c->dmd_eval : c;
}

// The candidates of all ranks: independent small dense problems (about 60 us apiece at 20 snapshots),
// taken one by one by the calling thread and by up to seven helpers.  The call waits for the ranks and
// not for the helpers, which a later call or pcf_destroy joins: on busy cores a helper may get its
// first time slice only milliseconds later (joined at once, a jump of rank 6 at 32 x 33 x 32 took 3.5 ms
// beside threads that spin on every core, and 1.1 ms otherwise).
struct Ranks {
  int ncol = 0, M = 0, rstar = 0;
  std::vector<double> U, s, V, R1, t, C;
  std::vector<char> ok;  // rank rstar - k has coefficients C + k M
  std::atomic<int> next{0};
  std::atomic<bool> failed{false};
  std::mutex lock;
  std::condition_variable all;
  int done = 0;

  bool candidate(int r, double* cv) const {
    std::vector<double> VS((size_t)M * r);  // V_r Sigma_r^-1
    for (int i = 0; i < M; ++i)
      for (int k = 0; k < r; ++k) VS[(size_t)i * r + k] = V[(size_t)i * M + k] / s[k];
    std::vector<double> X((size_t)ncol * r, 0.0);  // R1 V_r Sigma_r^-1
    for (int i = 0; i < ncol; ++i)
      for (int k = 0; k < r; ++k) {
        double a = 0;
        for (int l = 0; l < M; ++l) a += R1[(size_t)i * M + l] * VS[(size_t)l * r + k];
        X[(size_t)i * r + k] = a;
      }
    std::vector<double> At((size_t)r * r, 0.0);  // U_r^T X
    for (int a = 0; a < r; ++a)
      for (int b = 0; b < r; ++b) {
        double v = 0;
        for (int i = 0; i < ncol; ++i) v += U[(size_t)i * M + a] * X[(size_t)i * r + b];
        At[(size_t)a * r + b] = v;
      }
    std::vector<la::cd> lam, W;
    if (!la::eig_general(r, At, lam, W)) return false;
    int q1 = 0;
    double best = 1e300;
    for (int q = 0; q < r; ++q) {
      const double w = std::abs(std::log(lam[q]));
      if (w < best) {
        best = w;
        q1 = q;
      }
    }
    std::vector<double> cp = la::lstsq_svd(ncol, r, X, t);
    std::vector<la::cd> bvec(cp.begin(), cp.end());
    if (!la::csolve(r, W, bvec)) return false;
    const la::cd b1 = bvec[q1];
    for (int l = 0; l < M; ++l) {
      la::cd a = 0;
      for (int k = 0; k < r; ++k) a += VS[(size_t)l * r + k] * W[(size_t)k * r + q1];
      cv[l] = std::real(b1 * a);
    }
    return true;
  }
  void work() noexcept {
    for (int k = next++; k < rstar; k = next++) {
      try {
        ok[k] = candidate(rstar - k, C.data() + (size_t)k * M);
      } catch (...) {
        failed = true;
      }
      const std::lock_guard<std::mutex> g(lock);
      if (++done == rstar) all.notify_all();
    }
  }
  void wait() {
    std::unique_lock<std::mutex> g(lock);
    all.wait(g, [&] { return done == rstar; });
  }
};
// Helpers for P while seven at most run or wait for a core.
void start_helpers(pcf_ctx* c, const std::shared_ptr<Ranks>& P) {
  const auto ended = [](pcf_ctx::Helper& h) {
    if (!h.ended->load()) return false;
    h.thread.join();
    return true;
  };
  c->helpers.erase(std::remove_if(c->helpers.begin(), c->helpers.end(), ended), c->helpers.end());
  try {
    c->helpers.reserve(7);
    const size_t want = std::min(P->rstar, 8) - 1;
    while (c->helpers.size() < want) {
      auto end = std::make_shared<std::atomic<bool>>(false);
      c->helpers.push_back({std::thread([P, end] {
                              P->work();
                              *end = true;
                            }),
                            end});
    }
  } catch (...) {  // no more threads: the others and the caller take the rest
  }
}

}  // namespace

extern "C" {

pcf_status pcf_snapshot(pcf_ctx* c, const double* u_hat, double* psi) {
  if (!c || !u_hat || !psi) return PCF_EINVAL;
  if (!c->uniform) return PCF_ENOTSUP;
  DMD_TRY(ensure_indep(c));
  DMD_TRY(sync_in(c));
  const long long total = (long long)(c->nindep + 1) * c->prm.ny * c->B;
  const int blocks = (int)std::min<long long>((total + 255) / 256, 4096);
  k_psi_extract<<<blocks, 256, 0, c->cs>>>((const double2*)u_hat, c->state_len, psi, c->psi_len, c->d_indep,
                                           c->nindep, c->hinst[0].kx, c->hinst[0].kz, c->Mz, c->prm.ny, c->nm, c->B);
  DMD_CUDA(cudaGetLastError());
  return sync_out(c);
}

pcf_status pcf_from_snapshot(pcf_ctx* c, const double* psi, double* u_hat) {
  if (!c || !u_hat || !psi) return PCF_EINVAL;
  if (!c->uniform) return PCF_ENOTSUP;
  if (c->prm.ny > 129) return PCF_EINVAL;
  DMD_TRY(ensure_indep(c));
  DMD_TRY(sync_in(c));
  const int n = c->B * (c->nindep + 1);
  k_psi_rebuild<<<(n + kRebuildWarps - 1) / kRebuildWarps, 32 * kRebuildWarps, 0, c->cs>>>(psi, c->psi_len, (double2*)u_hat, c->state_len, c->d_indep,
                                                    c->nindep, c->hinst[0].kx, c->hinst[0].kz, c->Mx, c->Mz,
                                                    c->prm.ny, c->nm, c->B);
  DMD_CUDA(cudaGetLastError());
  return sync_out(c);
}

pcf_status pcf_dmd_extrapolate(pcf_ctx* c, const double* S, long long ld, int M, double rank_tol, double* u_out,
                               int* rank_used, double* j_out) {
  if (!c || !S || !u_out || M < 1 || !(rank_tol >= 0)) return PCF_EINVAL;
  if (!c->uniform) return PCF_ENOTSUP;
  DMD_TRY(ensure_indep(c));
  if (ld < c->psi_len) return PCF_EINVAL;
  const int ncol = M + 1;
  DMD_TRY(ensure_dmd(c, ncol));
  DMD_TRY(sync_in(c));
  const long long rows = c->psi_len;
  // R (row-major, ncol x ncol, upper triangular)
  std::vector<double> R;
  DMD_TRY(snapshot_r(c, S, ld, ncol, &R));
  // Psi ~ R0 = R[:, 0:M], Psi' ~ R1 = R[:, 1:M+1], last snapshot t = R[:, M]
  std::vector<double> R0((size_t)ncol * M), R1((size_t)ncol * M), t(ncol);
  for (int i = 0; i < ncol; ++i) {
    for (int k = 0; k < M; ++k) {
      R0[(size_t)i * M + k] = R[(size_t)i * ncol + k];
      R1[(size_t)i * M + k] = R[(size_t)i * ncol + k + 1];
    }
    t[i] = R[(size_t)i * ncol + M];
  }
  auto P = std::make_shared<Ranks>();
  P->ncol = ncol;
  P->M = M;
  la::svd_jacobi(ncol, M, R0, P->U, P->s, P->V);
  int rstar = 0;
  for (int k = 0; k < M; ++k)
    if (P->s[k] > rank_tol * P->s[0]) ++rstar;
  if (rstar == 0) return PCF_ENAN;
  // candidates r = rstar .. 1: coefficient vectors over the snapshots s_1..s_M
  P->rstar = rstar;
  P->R1 = std::move(R1);
  P->t = std::move(t);
  P->C.assign((size_t)rstar * M, 0.0);
  P->ok.assign(rstar, 0);
  std::vector<int> rank_of(rstar);
  start_helpers(c, P);
  P->work();
  P->wait();
  if (P->failed) return PCF_ENOMEM;
  std::vector<double>& Cc = P->C;
  const std::vector<char>& ok = P->ok;
  int ncand = 0;
  for (int k = 0; k < rstar; ++k)
    if (ok[k]) {
      if (ncand < k) std::copy_n(Cc.data() + (size_t)k * M, M, Cc.data() + (size_t)ncand * M);
      rank_of[ncand++] = rstar - k;
    }
  if (ncand == 0) return PCF_ENAN;
  // candidate states on the device; the instances past the last candidate are masked (evaluating
  // copies of it instead, a call of rank 2 took as long as one of rank 20)
  pcf_ctx* ev = eval_ctx(c, ncand);
  DMD_CUDA(cudaMemcpyAsync(c->dmd_c, Cc.data(), sizeof(double) * (size_t)ncand * M, cudaMemcpyHostToDevice, c->cs));
  k_combine<<<dim3((unsigned)std::min<long long>((rows + 255) / 256, 2048), (ncand + 3) / 4), 256, 0, c->cs>>>(
      S, rows, ld, M, c->dmd_c, ncand, c->dmd_cpsi, rows);
  DMD_CUDA(cudaGetLastError());
  {
    const int n = ncand * (c->nindep + 1);
    k_psi_rebuild<<<(n + kRebuildWarps - 1) / kRebuildWarps, 32 * kRebuildWarps, 0, c->cs>>>(
        c->dmd_cpsi, rows, c->dmd_cu, c->state_len, c->d_indep, c->nindep, c->hinst[0].kx, c->hinst[0].kz, c->Mx,
        c->Mz, c->prm.ny, c->nm, ncand);
    DMD_CUDA(cudaGetLastError());
  }
  DMD_CUDA(cudaEventRecord(c->ev_out, c->cs));
  DMD_CUDA(cudaStreamWaitEvent(c->user, c->ev_out, 0));
  std::vector<double> Jc(ncand);
  for (int g = 0; g < ncand; g += ev->B) {
    DMD_TRY(pcf_residual_first(ev, std::min(ev->B, ncand - g), (const double*)(c->dmd_cu + (size_t)g * c->state_len),
                               (double*)ev->r_int, c->dmd_J + g));
  }
  DMD_CUDA(cudaMemcpyAsync(Jc.data(), c->dmd_J, sizeof(double) * ncand, cudaMemcpyDeviceToHost, c->user));
  DMD_CUDA(cudaStreamSynchronize(c->user));
  int bi = -1;
  for (int k = 0; k < ncand; ++k)  // candidates are ordered by decreasing rank: ties keep the larger r
    if (std::isfinite(Jc[k]) && (bi < 0 || Jc[k] < Jc[bi])) bi = k;
  if (bi < 0) return PCF_ENAN;
  DMD_CUDA(cudaMemcpyAsync(u_out, c->dmd_cu + (size_t)bi * c->state_len, sizeof(double2) * c->state_len,
                           cudaMemcpyDeviceToDevice, c->user));
  DMD_CUDA(cudaStreamSynchronize(c->user));
  if (rank_used) *rank_used = rank_of[bi];
  if (j_out) *j_out = Jc[bi];
  return PCF_OK;
}

}  // extern "C"
