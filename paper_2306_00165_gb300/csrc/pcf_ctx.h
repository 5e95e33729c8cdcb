// Context of the pcfadj library (internal; shared by the host translation units).
#pragma once
#include <atomic>
#include <map>
#include <memory>
#include <thread>
#include <vector>

#include "pcf_kernels.cuh"

// Device tables of one grid (shared by every instance on that grid).
struct GridTables {
  double *cheb, *rco, *ccw, *kx, *kz, *y, *ub, *tab0, *tab1, *ik2nu = nullptr;
  double* dense[2] = {nullptr, nullptr};
  int4 *fxcheb = nullptr, *fxD[2] = {nullptr, nullptr};
  int* fxDe[2] = {nullptr, nullptr};
  int fxcheb_e = 0;
  pcf::fxtw *twfx_x = nullptr, *twfx_z = nullptr;
  float2 *twxf = nullptr, *twzf = nullptr;
  uint16_t* tcA = nullptr;
  uint16_t* tcA5 = nullptr;
  double sig[2];
};

struct pcf_ctx {
  pcf_params prm;
  GridTables gt;  // of the first problem
  int N, Kx, Kz, Mx, Mz, nm, B, mpc;
  int sms = 0;          // multiprocessors of the device (152 where the launch rules were measured)
  long long state_len;  // complex values per instance (instance 0; all instances when uniform)
  std::vector<long long> state_off;  // complex offset of each instance's state, [B+1]
  long long total_state = 0;
  bool uniform = true;   // every instance on the same problem
  bool suction = false;  // some instance has a base flow with suction (PCF_ASBL)
  int mode_thr = 128;    // threads per CTA of the single per-mode kernel
  bool mixed = false;    // mixed-precision form (FP32 planes, split-BF16 Chebyshev, FP64 solves)
  // fixed-point plane kernels: threads per CTA, variant (planes_fx_kind)
  int thr_synth = 64, thr_prod = 64, plane_kind = 0;
  bool plane_warp = false;  // FP32 plane kernels with the transforms in warp registers
  bool tc05 = false;        // Chebyshev contractions of the mixed form on tcgen05 (else mma.sync)
  // descent steps in the symmetric subspace run the per-mode kernels on the modes m >= 0 only
  // (every instance enforces s2; split FP64 or float-float kernels); the reduced CTA maps:
  bool reduced = false;
  int* pre_ya_r = nullptr;
  int* pre_yy_r = nullptr;
  int* pre_ys_r = nullptr;
  int cta_ya_r = 0, cta_yy_r = 0, cta_ys_r = 0;
  cudaStream_t user = nullptr, cs = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  std::vector<void*> allocs;
  std::vector<pcf::Inst> hinst;
  pcf::Inst* dinst = nullptr;
  // prefix arrays
  int* pre_synth11 = nullptr;
  int* pre_synth3 = nullptr;
  int* pre_prod = nullptr;
  int* pre_mode = nullptr;
  int* pre_inst = nullptr;
  int* pre_tcs = nullptr;   // tensor-core synthesis (mixed form)
  int* pre_tca = nullptr;   // tensor-core analysis (mixed form)
  int cta_synth11 = 0, cta_synth3 = 0, cta_prod = 0, cta_mode = 0, cta_tcs = 0, cta_tca = 0;
  size_t sm_synth = 0, sm_prod = 0, sm_mode = 0, sm_tc = 0, sm_warp = 0;
  // the FP64 forms' fixed-point per-mode kernels (no problem of solve_kind 1)
  bool split = false;
  int sgrp = 0;                 // largest instances per group of the solve
  int np = 8;                   // modes per tile of the analysis and synthesis
  int ngroups = 0;
  int2* d_groups = nullptr;     // [B] (first, count)
  int* pre_ya = nullptr;        // CTA prefixes over instances: analysis, synthesis
  int* pre_yy = nullptr;
  int* pre_ys = nullptr;        // ... over groups: one CTA per (group, mode)
  int cta_ya = 0, cta_ys = 0, cta_yy = 0;
  int thr_ya = 64, thr_yy = 64, thr_ys = 64, thr_yf = 64, thr_y64 = 64;
  bool fine_y = false, fine_s = false;  // one row and one part per thread (few row pairs)
  size_t sm_ya = 0, sm_ys = 0, sm_yy = 0, sm_yf = 0, sm_y64 = 0;
  // the step runs the fused half-step kernel (k_ystep_fx), with a separate norm kernel (jn)
  bool fused = false, jn = false;
  // the split step's Stokes solve by banded sweeps, one thread per chain (k_sweep), in place
  // of the dense solve: CTA prefixes per instance (full and reduced launches) and geometry
  bool sweep = false;
  int* pre_sw = nullptr;
  int* pre_sw_r = nullptr;
  int cta_sw = 0, cta_sw_r = 0, thr_sw = 32;
  size_t sm_sw = 0;
  double2* r_int = nullptr;    // internal r1 buffer for descent
  double2* u_dev = nullptr;    // device state for the *_host entry point
  double* hist_dev = nullptr;
  int hist_cap = 0;
  int* active = nullptr;  // convergence masks of a run
  int* first = nullptr;   // mask of pcf_residual_first (a run's DMD jump keeps the run's masks)
  std::map<int, cudaGraphExec_t> graphs;
  // symmetric subspace and DNS
  bool any_sym = false;         // some instance enforces a symmetry
  int sym_ctas = 0, dns_ctas = 0;
  pcf::DnsInst* d_dns = nullptr;
  double2* uprev = nullptr;
  int* dns_count = nullptr;
  std::map<int, cudaGraphExec_t> dns_graphs;
  // timing
  int timing = 0;
  double kms[pcf::kNumKernelClasses] = {0};
  long long kcount[pcf::kNumKernelClasses] = {0};
  std::vector<cudaEvent_t> evpool;
  // snapshot vector (psi) and DMD workspace, allocated on first use
  int* d_indep = nullptr;   // (i, j) storage indices of the independent modes
  int nindep = 0;
  long long psi_len = 0;
  double* dmd_A = nullptr;      // Householder QR workspace, psi_len x cap
  double* dmd_part = nullptr;   // partial sums
  double* dmd_coef = nullptr;   // per-column reflector data
  double* dmd_cpsi = nullptr;   // candidate snapshot vectors
  double2* dmd_cu = nullptr;    // candidate states
  double* dmd_J = nullptr;      // candidate norms (batch)
  double* dmd_c = nullptr;      // candidate coefficient vectors (device)
  pcf_ctx* dmd_eval = nullptr;  // context over a batch of candidates on this problem's tables
  // host threads of DMD calls, joined by a later call or with the context
  struct Helper {
    std::thread thread;
    std::shared_ptr<std::atomic<bool>> ended;
  };
  std::vector<Helper> helpers;
  int dmd_cap = 0;              // columns the DMD workspace holds
  int dmd_ncand_cap = 0;
};

// A context over `batch` instances of c's (first) problem that shares c's tables: workspace only.
pcf_status pcf_make_child(pcf_ctx* c, int batch, pcf_ctx** out);
// pcf_residual of the first n instances; the others' outputs are not defined.
pcf_status pcf_residual_first(pcf_ctx* c, int n, const double* u, double* r, double* rnorm);
