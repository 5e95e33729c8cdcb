// Kernel entry points of the pcfadj library (declared for the host launcher).
#pragma once
#include "pcf_internal.h"

namespace pcf {

// Operation of the per-mode kernel.
enum ModeOp : int {
  MODE_SYNTH_ONLY = 0,   // y-synthesis (no solve): sig 0 reads uhat into slot 0, sig 1 rhat into slot 1
  MODE_PHI = 1,          // Stokes step of the NSE, r1 = (u+ - u)/dt, synthesis of r1
  MODE_PSI_UPDATE = 2,   // Stokes step of the dummy dynamics, f, u += dtau f, synthesis of u
  MODE_PSI_GRAD = 3,     // same as MODE_PSI_UPDATE but only writes f
  MODE_SOLVE = 4,        // Stokes step from a coefficient right-hand side (rhat), output fhat
};

struct LaunchInfo {
  const Inst* insts;
  const int* prefix;   // CTA prefix over instances (length ninst + 1)
  int ninst;
  int per = 0;         // CTAs per instance when every instance has the same number, else 0
};

// Launch over groups of consecutive instances that share one grid.
struct GroupLaunch {
  const Inst* insts;
  const int* prefix;   // CTA prefix over groups (length ngroups + 1)
  const int2* groups;  // (first instance, instance count) per group
  int ngroups;
};

__device__ __forceinline__ int find_inst(const LaunchInfo& li, int cta, int* local) {
  if (li.per) {  // no dependent loads on the way to the instance's descriptor
    const int b = cta / li.per;
    *local = cta - b * li.per;
    return b;
  }
  int lo = 0, hi = li.ninst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (li.prefix[mid] <= cta) lo = mid; else hi = mid - 1;
  }
  *local = cta - li.prefix[lo];
  return lo;
}

__device__ __forceinline__ bool inst_active(const Inst& I) { return I.active == nullptr || *I.active != 0; }

// Per-instance state of the DNS that produces guesses (pcf_dns), on the device.
struct DnsInst {
  double* hist;        // ||u_s|| history base (may be null), stride hist_stride
  int hist_stride;
  double2* uprev;      // the state before the current update
  double2* guess;      // guess base (may be null); guess k at guess + k * gstride
  long long gstride;
  int gmax;
  int* count;          // extrema found so far
  int step, slot;      // steps taken in this call; guess slot of this step's capture (-1: none)
  double h1, h2;       // ||u|| of the previous two steps
};

// J = sqrt(0.5 * sum_j w_j * mean_{x,z} |q|^2) from the plane sums, by one full warp (every
// lane returns it): strided partial sums, then a shuffle tree, so that the chain is ny/32 + 5
// additions and not ny.  Every path that computes a norm uses this order.
__device__ __forceinline__ double norm_from_parts(const Inst& I) {
  double s = 0.0;
  for (int q = threadIdx.x & 31; q < I.ny; q += 32) {
    const double pj = __ldcg(I.normpart + q) + __ldcg(I.normpart + I.ny + q) + __ldcg(I.normpart + 2 * I.ny + q);
    s = fma(I.ccw[q], pj, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return sqrt(0.5 * I.inv_nxnz * s);
}

// First warp of a CTA whose thread 0 has written its plane sum: true in the CTA that counts last
// of the instance's 3 ny (thread 0 then resets the counter).
__device__ __forceinline__ bool last_plane(const Inst& I) {
  int last = 0;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(I.jcount, 1) == 3 * I.ny - 1;
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return false;
  __threadfence();
  return true;
}

// End of an adjoint product CTA: the last one computes J, writes the history entry and clears
// the mask when J < tol (the instance stops before this step's update).
__device__ __forceinline__ void finish_norm(const Inst& I, int step_index) {
  if (threadIdx.x >= 32 || !last_plane(I)) return;
  const double J = norm_from_parts(I);
  if (threadIdx.x == 0) {
    if (I.hist) I.hist[(size_t)step_index * I.hist_stride] = J;
    if (I.tol > 0.0 && J < I.tol && I.active) *I.active = 0;
    *I.jcount = 0;
  }
}

// End of a CTA of a DNS step that has written its plane sum of u_c^2: the last one has h_s = ||u_s|| (same arithmetic as the norm
// of r1), writes its history entry and makes the discrete-extremum test of the previous step:
//   (h_{s-1} - h_{s-2}) (h_s - h_{s-1}) < 0  ->  u_{s-1} (held in uprev until this step's update) is
// a guess.  D.step counts the steps of the current call.
__device__ __forceinline__ void finish_dns(const Inst& I, DnsInst& D) {
  if (threadIdx.x >= 32 || !last_plane(I)) return;
  const double h = norm_from_parts(I);
  if (threadIdx.x != 0) return;
  *I.jcount = 0;
  const int step = D.step;
  if (D.hist) D.hist[(size_t)step * D.hist_stride] = h;
  int slot = -1;
  if (step >= 2 && (D.h1 - D.h2) * (h - D.h1) < 0.0) {
    const int k = *D.count;
    if (k < D.gmax) slot = k;
    *D.count = k + 1;
  }
  D.slot = slot;
  D.h2 = D.h1;
  D.h1 = h;
  D.step = step + 1;
}

// Raise the maximum dynamic shared memory of kernel func on the current device to at least
// bytes.  The attribute belongs to the function, not to a context, so it only ever grows: a
// context that needs less must not lower the limit another context launches with.
cudaError_t raise_smem_limit(const void* func, size_t bytes);

// Stokes step by banded tau sweeps, one thread per chain (pcf_sweep.cu): shared memory per
// CTA of `threads` lanes, CTAs for an instance whose launch covers nmodes_run modes, launch
// over a CTA prefix per instance (red: the modes m >= 0 only), and the shared-memory limit.
size_t smem_sweep(int N, int threads);
int sweep_ctas(int nmodes_run, int threads);
void launch_sweep(int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int op, int red);
cudaError_t set_sweep_smem(size_t smem);

// FP32 plane kernels of the mixed form (shared-memory Stockham passes).
// step_index >= 0 (adjoint product only): the last CTA of each instance also computes J from
// the plane sums, its history entry and the convergence mask (in place of launch_jnorm)
// suction: some instance of the launch has a base flow with a wall-normal velocity (ASBL)
void launch_xzsynth(int ctas, size_t smem, cudaStream_t s, LaunchInfo li, int slot, int nf);
void launch_prod(bool adj, bool suction, int ctas, size_t smem, cudaStream_t s, LaunchInfo li, int step_index = -1);
void launch_norm_planes(int ctas, cudaStream_t s, LaunchInfo li, int slot, DnsInst* dns);
cudaError_t set_plane_smem(size_t synth, size_t prod);
// The FP64 forms' plane kernels in 64-bit fixed point (pcf_planes_fx.cu); threads per CTA from
// the largest plane of the launch.
int planes_fx_kind(const Inst& I);  // a launch takes the largest of its instances'
size_t smem_planes_fx(const Inst& I, int threads);
int planes_fx_threads(const Inst& I, bool prod);
void launch_xzsynth_fx(int kind, int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int slot, int nf);
void launch_prod_fx(int kind, bool adj, int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li,
                    int step_index, DnsInst* dns = nullptr);
void launch_norm_planes_fx(int ctas, cudaStream_t s, LaunchInfo li, int slot);
cudaError_t set_planes_fx_smem(int kind, size_t synth, size_t prod);
// Plane kernels of the FP32 form with the x, z transforms in warp registers
// (pcf_planes_warp.cu): nx, nz in {32, 64, 96, 128}.
bool plane_warp_ok(const Inst& I);
size_t smem_plane_warp(const Inst& I, int elem_bytes);
void launch_xzsynth_warp(int ctas, size_t smem, cudaStream_t s, LaunchInfo li, int slot, int nf);
void launch_prod_warp(bool adj, int ctas, size_t smem, cudaStream_t s, LaunchInfo li, int step_index);
cudaError_t set_plane_warp_smem(size_t synth, size_t prod);
__global__ void k_mode(LaunchInfo li, int op, int sig, int mpc);
__global__ void k_norm_final(LaunchInfo li, double* out);
__global__ void k_fp64_probe(double* out, int iters);

size_t smem_plane(const Inst& I, int elem_bytes);
size_t smem_mode(const Inst& I, int mpc);
size_t smem_cheb_tc(int ny);
void launch_cheb_synth_tc(int ctas, size_t smem, cudaStream_t s, LaunchInfo li, int slot);
void launch_cheb_analysis_tc(int ctas, size_t smem, cudaStream_t s, LaunchInfo li);
cudaError_t set_cheb_tc_smem(size_t smem);
// The same contractions on the 5th-generation tensor cores (tcgen05, TMEM accumulator;
// pcf_cheb_tc05.cu), same CTA map.
size_t smem_cheb_tc05(int ny);
void launch_cheb_synth_tc05(int ctas, size_t smem, cudaStream_t s, LaunchInfo li, int slot);
void launch_cheb_analysis_tc05(int ctas, size_t smem, cudaStream_t s, LaunchInfo li);
cudaError_t set_cheb_tc05_smem(size_t smem);
int cheb_tc_tiles(int nmodes);

// Per-mode kernels of the FP64 forms in 64-bit fixed point (pcf_modes_fx.cu): Chebyshev analysis
// and synthesis over tiles of np modes of an instance, dense Stokes solve and the fused half-step
// over groups of instances on one grid (at most kMaxGroup), one CTA per (group, mode).
constexpr int kMaxGroup = 8;
int yfx_tiles(int nmodes, int np);
int yana_fx_threads(int N, int np, bool fine);
int ysynth_fx_threads(int N, int np, bool fine);
int ysolve_fx_threads(int N, int G, bool fine, bool many);
size_t smem_yana_fx(int N, int np);
size_t smem_ysynth_fx(int N, int np);
size_t smem_ysolve_fx(int N, int G);
size_t smem_ystep_fx(int N, int G);
// fine: one matrix row and one part per thread, for launches with few row pairs.
// red: the modes m >= 0 only (a state invariant under s2); the synthesis mirrors their y-values
void launch_yana_fx(int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int np, int red, int fine);
void launch_ysynth_fx(int ctas, int threads, size_t smem, cudaStream_t s, LaunchInfo li, int slot, int nf,
                      int np, int red, int fine);
void launch_ysolve_fx(int ctas, int threads, size_t smem, cudaStream_t s, GroupLaunch gl, int op, int sig, int fine);
// the solve of a given right-hand side (MODE_SOLVE), in FP64
int ysolve_f64_threads(int N, int G);
size_t smem_ysolve_f64(int N, int G);
void launch_ysolve_f64(int ctas, int threads, size_t smem, cudaStream_t s, GroupLaunch gl, int sig);
void launch_ystep_fx(int ctas, int threads, size_t smem, cudaStream_t s, GroupLaunch gl, int op, int synth, int fine);
void launch_jnorm(int ninst, cudaStream_t s, const Inst* insts, int step_index);
cudaError_t set_modes_fx_smem(size_t ana, size_t synth, size_t solve, size_t step, size_t solve64);
// dense operators -> fixed-point words (default stream): lengths of the two arrays, conversion
size_t dense_limbs_len(int N, int nmodes);
size_t dense_exps_len(int N, int nmodes);
void launch_dense_limbs(const double* src, int N, int nmodes, int4* dst, int* dexp);

// Symmetric-subspace projection and the DNS helpers (pcf_sym_dns.cu).
int symmetrize_ctas(const Inst& I);
void launch_symmetrize(int ctas_x, int ninst, cudaStream_t s, const Inst* insts, int mask_override,
                       int reduced = 0);
int dns_ctas(const Inst& I);
void launch_dns_update(int ctas_x, int ninst, cudaStream_t s, const Inst* insts, const DnsInst* dns);

}  // namespace pcf
