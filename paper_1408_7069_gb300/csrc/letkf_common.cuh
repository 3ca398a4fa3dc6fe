// Internal declarations shared by the translation units of libletkf.so.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "letkf.h"

// Device status word bits (set with atomicOr by kernels, read by letkf_sync).
enum : int {
  LK_BIT_NOCONVERGE = 1,
  LK_BIT_NONFINITE = 2,
  LK_BIT_TIMEOUT = 4,
};

// Default node tile of one analysis CTA (TI x TJ nodes); the autotuner may choose
// another of the compiled shapes. The wide class, a warp per node and 170 to 240 registers
// per thread, takes 2 x 2 (shape 2): eight warps of a 2 x 4 tile fill an SM's registers
// alone, of 2 x 2 tiles three fit for 48 columns. Measured on one GB300, four frames
// 2 x 4 -> 2 x 2: 80 x 80, m = 48 417 -> 355 us, m = 40 417 -> 351, m = 64 474 -> 440; 16 x 16,
// m = 56 104 -> 94; 48 systems 2.68 -> 2.36 ms. (The halo cells a node stages grow with it, which
// at a window of 13 still costs less than it gives: 40 x 40, m = 64 517 -> 442.)
constexpr int LK_TILE_I = 2;
constexpr int LK_TILE_J = 4;
// Padding of the slope-anomaly grid: tiles up to this many nodes per side keep
// their halo in bounds.
constexpr int LK_TILE_MAX = 8;
// The compiled analysis tile shapes (id, TI, TJ: nodes per CTA side), for the
// FP32 pair kernel and the FP64 tile kernel alike; letkf_tile_shape enumerates
// them. Each side divides LK_TILE_MAX, so the padded grid covers every halo.
#define LK_FOR_SHAPES(X) X(0, 2, 4) X(1, 4, 4) X(2, 2, 2) X(3, 1, 8) X(4, 1, 2) X(5, 1, 1)
constexpr int LK_NUM_SHAPES = 6;
// CTAs of the residual reduction per instance (fixed, so the sum order is fixed).
constexpr int LK_RES_BLOCKS = 128;
// Threads per CTA of the warp-per-item kernels (observation, forecast, reverse
// gathers): small CTAs spread a 16 m system's few hundred items over all SMs.
constexpr int LK_WARP_CTA = 64;
// Stop cosine of the FP64 sweeps that start from a stored FP32 eigenbasis
// (queued nodes of FP32 handles): the next sweep would rotate by about its
// square, far below what the FP32 outputs resolve.
constexpr double LK_WARM_STOP64 = 1e-8;

// Chebyshev series of (1 + g)^-1/2 and (1 + g)^-1 on [0, ratio] (letkf_cheb.cu):
// classes of ratio LK_CHEB_R0 LK_CHEB_STEP^c, one row of LK_CHEB_LD32 pairs per
// class: (2 / ratio, degree), then the coefficients (a_k, b_k), k = 0 .. degree.
// The step of 1.25 costs at most one product in nine over the exact ratio.
constexpr double LK_CHEB_R0 = 0.25, LK_CHEB_STEP = 1.25;
constexpr int LK_CHEB_CLASSES32 = 33, LK_CHEB_LD32 = 192;
constexpr float LK_CHEB_MAX32 = 300.f;        // below the last class's 315.5
constexpr float LK_CHEB_MAXD = 100.f;         // multi-actuator domains: 94 products
// kappa_hat to which ill-conditioned nodes of FP32 handles take the float-pair
// tridiagonal form (letkf_tri.cuh) instead of FP64 sweeps: the error of its rational
// approximation (15 poles) is 4e-9 there, and 7e-8, more than the sweeps', at 1e6.
// An entry of its list holds the instance in its low LK_TRI_INST bits and above it the
// exponent that bounds the node's kappa_hat.
constexpr float LK_TRI_MAX = 1e5f;
constexpr int LK_TRI_INST = 26;
// Ints of a handle's counters: [0] status bits, [1] FP64 nodes, [2] max and [3]
// total sweeps, [4..6] lengths of the classes' sweep lists, [7..8] of the
// tridiagonal lists of classes 0 and 1 (which fill the same worklists from their ends).
constexpr int LK_COUNTERS = 16, LK_TRI_LIST = 3;   // a class's tridiagonal count sits 3 above its sweep count
// The FP64 table, truncated below FP64 rounding: classes up to 42.4, 128 terms. Beyond,
// the recurrences' rounding in pairs of floats (it grows with the terms' number) is no longer
// below the eigensolve's.
constexpr int LK_CHEB_CLASSES64 = 24, LK_CHEB_LD64 = 136;
constexpr float LK_CHEB_MAX64 = 42.f;

// One AO instance, as the kernels see it (device pointers, by-value copy in a
// device array). The real type of X, Yb, d, y, truth, taper and the outputs is
// float (precision 0) or double (precision 1).
struct LkInst {
  int nsub, m, w, h;        // h = w / 2
  int mp;                   // padded ensemble width of the kernels (16, 32, 48 or 64)
  int n_pts, n_sap, p;
  int gs_rows, gs_cols;     // padded subaperture grid: cell (s+h, t+h) holds subap (s, t)
  const int *pid_map;       // [(nsub+1)^2] node -> point id or -1
  const int2 *pts;          // [n_pts] (i, j)
  const int2 *saps;         // [n_sap] (s, t)
  void *X;                  // [n_pts][2][m]
  void *Ybp;                // [gs_rows][gs_cols][2][m]
  void *dp;                 // [gs_rows][gs_cols][2]
  const void *taper;        // [w*w] tau / sigma2
  float *basis;             // [n_pts][mp][mp] last eigenbasis (FP32 warm start)
  double *basis64;          // FP64 handles: [n_pts][mp][mp] FP64 eigenbasis the reverse mode records
  const float *bank;        // [bank_B][bank_G][bank_G] or NULL
  int bank_B, bank_G;
  double alpha;             // (m - 1) / rho
  double a_ar1, noise_std;
  unsigned long long seed;
  long long y_off;          // offset of this instance in concatenated slopes
  long long node_off;       // ... in concatenated node arrays (truth, mean/spread rows)
  long long noise_off;      // ... in concatenated [n_pts][m] noise
  long long state_off;      // ... in the concatenated ensemble
  // Deformable mirror (letkf_set_dm; dm = 0: none, the pseudo-open-loop form):
  // influence matrix N, command matrix P and D1 N as CSR over the nodes, the
  // commands u [3][n_pts] (slot f % 3 holds the command computed after
  // forecast number f, f the forecast counter *fcount), the predicted phase
  // pmean [n_pts] (written by the forecast) and the correction cor = N u_{k-1}.
  int dm;
  const int *n_ptr, *n_idx, *p_ptr, *p_idx, *dn_ptr, *dn_idx;
  const void *n_val, *p_val, *dn_val;
  void *u, *pmean, *cor;
  const long long *fcount;
};

// Work items.
// One subaperture of the observation kernel: instance, index, cell of the padded grid, node
// ids of its corners (0,0), (1,0), (0,1), (1,1).
struct alignas(16) LkObsItem {
  int inst, k, cell, pad;
  int q00, q10, q01, q11;
};

struct LkTile {             // one analysis CTA: instance, tile origin (node coordinates)
  int inst, i0, j0, cost;
};

struct LkAdjWork;           // reverse-mode workspace (letkf_adjoint.cu)
struct LkDom;               // local-domain tables (letkf_domains.cu)

struct letkf_ctx {
  letkf_config cfg;         // first instance's config (host pointers cleared)
  std::vector<letkf_config> cfgs;   // every instance's config (host pointers cleared)
  cudaStream_t stream = nullptr;
  int device = 0;
  int precision = 0;
  size_t rsz = 4;           // bytes of the real type
  double tol32 = 4e-6, tol64 = 1e-13, fp64_kappa = 300;
  double stop32 = 1e-3;             // FP32 Jacobi stops after a sweep with all cosines <= this
  int max_sweeps = 20;
  float2 *cheb32 = nullptr;         // FP32 Chebyshev table; NULL: every node by Jacobi sweeps
  float4 *cheb64 = nullptr;         // the FP64 one (FP64 handles), in pairs of floats
  double2 *poles = nullptr;         // [16] poles and weights of A^-1/2 (FP32 handles)
  int keep_basis = 0;               // store every node's eigenbasis (reverse mode needs it)
  unsigned char *left64 = nullptr;  // [n_pts] where the FP64 series marks the nodes it leaves

  int n_inst = 0;
  std::vector<LkInst> inst;         // host copies of the descriptors
  LkInst *d_inst = nullptr;         // device copies
  long long n_pts_total = 0, p_total = 0, state_total = 0, noise_total = 0;
  long long sap_total = 0;

  // work lists (device)
  LkObsItem *obs_items = nullptr;   // [sap_total]
  int2 *node_items = nullptr;       // [n_pts_total] (inst, point)
  LkTile *tiles[3] = {nullptr, nullptr, nullptr};   // per width class 16 / 32 / 64
  int n_tiles[3] = {0, 0, 0};
  int tile_shape[3] = {0, 0, 2};    // index into the compiled tile shapes, per class
  int tile_split[3] = {0, 0, 0};    // class 2: leading tiles of MP = 64 instances (MP = 48 after)
  int row_split[3] = {1, 1, 1};     // 2: each column's rows on two lanes (classes 0 and 1, FP32)
  int fp64_warm = 1;                // FP64 handles: FP32 basis pass, then the FP64 sweep from it
  std::vector<LkTile> tiles_host[3];

  // device buffers (single allocations sliced per instance)
  void *X = nullptr, *Ybp = nullptr, *dp = nullptr, *taper = nullptr;
  int *pid_map = nullptr;
  int2 *pts = nullptr, *saps = nullptr;
  float *bank = nullptr, *basis = nullptr;
  double *basis64 = nullptr;        // FP64 handles: the FP64 eigenbases the reverse mode records
  int *counters = nullptr;          // [LK_COUNTERS]
  int2 *worklist = nullptr;         // [n_pts_total] (inst, point) queued for FP64
  long long *frame = nullptr;       // [0] forecast counter, [1] frame index within letkf_run
  double2 *partial = nullptr;       // [n_inst][LK_RES_BLOCKS] residual partial sums
  void *noise_pre = nullptr;        // [noise_total] the frame's forecast noise, drawn ahead
  int *tickets = nullptr;           // [n_inst + 1] last-CTA counters: residual per instance, forecast

  // host copies
  std::vector<int32_t> pts_host, wslopes_host;
  long long frame_host = 0;

  // graph of one closed-loop frame (letkf_run)
  cudaGraphExec_t graph = nullptr;
  const void *graph_y = nullptr, *graph_truth = nullptr;
  const double *graph_resvar = nullptr;
  // graph of a whole run of frames (letkf_run_graph)
  cudaGraphExec_t mgraph = nullptr;
  int mgraph_frames = 0;
  const void *mgraph_y = nullptr, *mgraph_truth = nullptr;
  const double *mgraph_resvar = nullptr;
  const unsigned long long *mgraph_stamps = nullptr;

  LkAdjWork *adj = nullptr;         // letkf_grad buffers and graph, built on first use
  // multi-actuator local domains (cfg.partition > 0): tables, and the host
  // geometry they are rebuilt from when sigma2 or the taper changes
  LkDom *dom = nullptr;
  std::vector<int> dom_pid;
  std::vector<int2> dom_pts, dom_saps;

  // letkf_step: pinned staging and device copies of one frame's inputs and
  // outputs (y, truth, mean, resvar), and its graphs without / with truth
  unsigned char *step_pin = nullptr, *step_dev = nullptr;
  size_t step_off[4] = {0, 0, 0, 0};
  cudaGraphExec_t step_graph[2] = {nullptr, nullptr};

  // Second stream of a handle on a user stream: the residual runs on it beside
  // the observation kernel (fork / join events); ev_out marks a step's
  // downloads, so that letkf_step returns while its forecast still runs.
  cudaStream_t side = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_out = nullptr;

  // deformable-mirror buffers (letkf_set_dm), single allocation per kind
  void *dm_buf = nullptr;           // N, P, D1 N (CSR) and u, pmean, cor
  unsigned char *dm_wfs_y = nullptr;   // letkf_run_dm: the simulated measurement [p]

  std::string err;
};

// Launchers (letkf_kernels.cu / letkf_analysis.cu). All enqueue on h->stream.
// run_idx (device) selects element *run_idx of a sequence (y, truth, resvar);
// NULL means element 0. y, truth, mean, spread and noise are concatenated over
// the instances in instance order.
cudaError_t lk_launch_obs(letkf_ctx *h, const void *y, const long long *run_idx);
// Observation of one frame with, in the same launch, its residual (truth and
// resvar given) and the model noise of the frame's forecast (noise_out given,
// [n_pts][m] at each instance's noise_off). No residual with a deformable mirror, whose
// residual needs N u first; not without subapertures.
cudaError_t lk_launch_obs_residual(letkf_ctx *h, const void *y, const void *truth,
                                   double *resvar, const long long *run_idx, void *noise_out);
cudaError_t lk_launch_analysis(letkf_ctx *h, void *mean, void *spread);
// The forecast inside the analysis (it is local to a node): with the noise already drawn,
// every kernel that writes a node's analysis writes its forecast instead, phi_k to row 1 and
// a phi_k + v to row 0, and the last list kernel advances the counters. `noise` NULL: no.
struct LkCycle {
  const void *noise = nullptr;   // [n_pts][m] at each instance's noise_off
  long long *frame = nullptr;    // the counters to advance, or NULL
};
// Analysis and forecast of a frame in the analysis kernels; *done is false, and nothing
// launched, where the handle's analysis has no such form (domains, row-split or
// FP64-sweep analyses, no list kernels) or no noise is given.
cudaError_t lk_launch_cycle(letkf_ctx *h, const void *noise, bool *done);
cudaError_t lk_launch_analysis_class(letkf_ctx *h, int cls, void *mean, void *spread);
// The forecast also advances the forecast counter and the run index (frame[0..1]).
cudaError_t lk_launch_forecast(letkf_ctx *h, const void *noise);
cudaError_t lk_launch_residual(letkf_ctx *h, const void *truth, double *resvar,
                               const long long *run_idx, double *piston = nullptr);
// The same on another stream of the handle's device.
cudaError_t lk_launch_residual_on(letkf_ctx *h, cudaStream_t stream, const void *truth,
                                  double *resvar, const long long *run_idx, double *piston);
cudaError_t lk_launch_basis_reset(letkf_ctx *h);   // stored eigenbases -> identity
// Deformable mirror (letkf_dm.cu): cor = N u_{k-1} on `stream` (before a
// residual), u_k = P pmean (after a forecast), and the simulated measurement
// y_k = D1 (phi_prev - N u_{k-2}) + w_k of a closed loop (phi_prev NULL: zero).
cudaError_t lk_launch_dm_cor(letkf_ctx *h, cudaStream_t stream);
cudaError_t lk_launch_dm_control(letkf_ctx *h);
cudaError_t lk_launch_dm_wfs(letkf_ctx *h, const void *truth_seq, const void *wnoise_seq,
                             const long long *run_idx, void *y_out);
cudaError_t lk_launch_dm_get(letkf_ctx *h, void *out);
// Writes the global timer (ns) into *dst once the preceding work has completed.
cudaError_t lk_launch_stamp(letkf_ctx *h, unsigned long long *dst);
cudaError_t lk_setup_analysis(letkf_ctx *h);
// FP32 analysis of width class cls, two columns per lane (letkf_pair.cu).
cudaError_t lk_launch_pair(letkf_ctx *h, int cls, void *mean, void *spread, const LkCycle &cy = {});
cudaError_t lk_setup_pair(letkf_ctx *h);
// Inputs and outputs of the reverse mode's node kernels (letkf_adjoint.cu).
struct LkAdjArgs {
  const double *lam_a;   // adjoint of this frame's analysis ensemble
  double *xp_bar, *xbar_bar, *ybw, *dbw, *theta;
  const double *dtap;
  double rho, sigma2;
  int max_sweeps;
  int *counters;
  // [n_pts] nonzero: the node the forward series left to the eigensolve, which the eigensolve
  // form takes here too; NULL: no series, every node by the eigensolve form
  const unsigned char *left;
};
// FP64 node problems by Chebyshev series (letkf_series64.cu): every node of
// width class cls of an FP64 handle, those above LK_CHEB_MAX64 queued in the
// class's worklist and marked in h->left64 (if any); and the adjoint of the nodes
// not marked in a.left.
bool lk_series64(const letkf_ctx *h);     // whether the handle takes this form
cudaError_t lk_launch_series64(letkf_ctx *h, int cls, void *mean, void *spread,
                               const LkCycle &cy = {});
cudaError_t lk_launch_adj_series64(letkf_ctx *h, const LkAdjArgs &a);
cudaError_t lk_setup_series64(letkf_ctx *h);
// Allocates and fills the handle's Chebyshev tables (letkf_cheb.cu).
cudaError_t lk_setup_cheb(letkf_ctx *h);
// FP64 analysis with one CTA of four warps per node (letkf_node64.cu): every
// node of width class cls (0: MP 16, 1: MP 32) of an FP64 handle, or the nodes
// the pair kernel queued in class cls of an FP32 handle.
cudaError_t lk_launch_node64(letkf_ctx *h, int cls, void *mean, void *spread);
cudaError_t lk_launch_list64(letkf_ctx *h, int cls, void *mean, void *spread,
                             const LkCycle &cy = {});
// Shared-memory limit of the wide class's FP64 list kernel (MP = 48 / 64 queue), and
// of the list kernel with the tridiagonal form.
cudaError_t lk_setup_node64w();
cudaError_t lk_setup_list();

// Raises the dynamic shared memory that a kernel may take on the current device to `bytes`.
// The limit belongs to the kernel, which every live handle launches with what its own windows
// need: it is never lowered.
cudaError_t lk_raise_smem_limit(const void *kernel, size_t bytes);
template <typename... KArgs>
cudaError_t lk_raise_smem(void (*kernel)(KArgs...), size_t bytes) {
  return lk_raise_smem_limit(reinterpret_cast<const void *>(kernel), bytes);
}

// Whether width class cls of the handle can take tile shape `shape`: FP32
// handles need whole warps of nodes and, in class 2 (one node per warp), at
// most 8 nodes per tile. (FP64 handles take any shape, which they ignore.)
bool lk_shape_ok(const letkf_ctx *h, int cls, int shape);
bool lk_shape_split_ok(const letkf_ctx *h, int cls, int shape, int split);
cudaError_t lk_launch_pair_basis(letkf_ctx *h, int cls);
int lk_num_tile_shapes();
void lk_tile_shape(int s, int *ti, int *tj);
int lk_width_class(int m);          // 0: m <= 16, 1: m <= 32, 2: m <= 64
void lk_adjoint_release(letkf_ctx *h);  // frees the letkf_grad workspace (and its graph)
// Gaspari & Cohn (1999) 5th-order piecewise rational function of z = r / c.
double lk_gaspari_cohn(double z);
// Local domains (letkf_domains.cu): build / rebuild the tables of a
// single-instance handle with cfg.partition > 0, free them, analyse.
letkf_status lk_domains_build(letkf_ctx *h, const letkf_config &c, const std::vector<int> &pid,
                              const std::vector<int2> &pts, const std::vector<int2> &saps,
                              std::string &err);
letkf_status lk_domains_set_params(letkf_ctx *h, const letkf_config &c,
                                   const std::vector<int> &pid, const std::vector<int2> &pts,
                                   const std::vector<int2> &saps, std::string &err);
void lk_domains_release(letkf_ctx *h);
int lk_domain_count(const letkf_ctx *h);
int lk_domain_of_nodes(const letkf_ctx *h, int *node_dom_host);
int lk_domain_obs_counts(const letkf_ctx *h, int *obs_host);
cudaError_t lk_launch_domains(letkf_ctx *h, void *mean, void *spread);
// The global ETKF for m > 64 (letkf_global.cu): Newton-Schulz root, refined
// mean, matrix-product apply, from the Gram's partial sums. sms: CTAs of the
// cooperative kernel (one per SM).
int lk_ns_tile();
cudaError_t lk_ns_setup();
size_t lk_ns_workspace_bytes(int mpt, long long n_pad);
cudaError_t lk_launch_ns_global(letkf_ctx *h, const double *gpart, const double *cpart,
                                int kchunks, int mpt, int sms, void *ws, void *mean,
                                void *spread);

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------
#ifdef __CUDACC__
template <typename T>
__device__ __forceinline__ T lk_warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Programmatic dependent launch of the per-frame kernels: each is launched
// with lk_launch_pdl, so that it can be scheduled while its predecessor on the
// stream drains; its first statement is lk_pdl_wait(), which returns once the
// predecessor grid has completed and its writes are visible (a no-op for a
// kernel launched without the attribute). The residual, forecast and piston sum
// kernels, the FP64 series and node kernels and the list kernels (but for the one with
// the tridiagonal form) then call lk_pdl_trigger(), letting the next kernel launch at
// once. The observation and FP32 analysis kernels do not: an analysis launched early
// has its CTAs placed on SMs that are still busy, several to an SM, which doubles the
// time of a latency-bound analysis that does not fill the GPU (measured on the
// 16 m system); their dependents launch as their CTAs exit.
__device__ __forceinline__ void lk_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void lk_pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t lk_launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                          cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Ratio class of the Chebyshev tables: the first whose ratio is at least `ratio`
// (rounded up by 2e-5, far above the logarithm's error).
__device__ __forceinline__ int lk_cheb_class(float ratio) {
  constexpr float inv_log2_step = 3.10628372f;               // 1 / log2(LK_CHEB_STEP)
  const float l = __log2f(fmaxf(ratio, 1e-30f) * float(1.0 / LK_CHEB_R0)) * inv_log2_step;
  return max(0, (int)ceilf(l + 1e-4f));
}

// SplitMix64 output after the state advanced counter + 1 steps from seed
// (Steele, Lea & Flood 2014).
__device__ __forceinline__ unsigned long long lk_splitmix64(unsigned long long seed,
                                                            unsigned long long counter) {
  unsigned long long z = seed + (counter + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The AR(1) forecast of member i at node gpt (Section 2.2): a x + v, v the drawn noise.
template <typename S>
__device__ __forceinline__ S lk_ar1(const LkInst &I, const S *__restrict__ noise, int gpt, int i,
                                    S x) {
  return fma(S(I.a_ar1), x, noise[I.noise_off + (long long)gpt * I.m + i]);
}
// The forecast of a node in place, by one warp (lane = member): phi_k to row 1, a phi_k + v
// to row 0; with a deformable mirror the predicted phase, for the command u = P phihat.
template <typename S>
__device__ __forceinline__ void lk_forecast_warp(const LkInst &I, const S *__restrict__ noise,
                                                 int gpt, int lane) {
  S *row0 = static_cast<S *>(I.X) + (size_t)gpt * 2 * I.m;
  S psum = S(0);
  for (int i = lane; i < I.m; i += 32) {
    const S x = row0[i], f = lk_ar1<S>(I, noise, gpt, i, x);
    row0[I.m + i] = x;
    row0[i] = f;
    psum += f;
  }
  if (I.dm) {
    psum = lk_warp_sum(psum);
    if (lane == 0) static_cast<S *>(I.pmean)[gpt] = psum / S(I.m);
  }
}
// Counters of the forecast, by the last list kernel of a frame (nothing in it reads them).
__device__ __forceinline__ void lk_advance(long long *__restrict__ frame) {
  if (frame && blockIdx.x == 0 && threadIdx.x == 0) {
    frame[0] += 1;
    frame[1] += 1;
  }
}
#endif
