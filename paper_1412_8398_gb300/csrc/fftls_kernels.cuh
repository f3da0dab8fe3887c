// Kernel interfaces of the FFT Lippmann-Schwinger iteration (internal header).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "fftls_fft.cuh"

namespace fftls {

// Solver states kept in device memory (Ctrl::state).  Every kernel of an
// iteration reads it on entry, so a captured chunk of iterations stops on the
// device without a host round trip.
enum State : int {
  kRunning = 0,
  kConverged = 1,   // eta test passed: no update this iteration
  kLast = 2,        // max_iter reached: run this iteration's update, then stop
  kStopped = 3,     // set one iteration after kLast
  kDiverged = 4,    // non-finite eta or eta > 1e4 eta_0
  kSwitch = 5,      // hand-over to the next precision phase: no update
};

enum Green : int { kMS = 0, kCentered = 1, kWillot = 2, kRotated = 3 };
// scheme update of the inverse x1 pass
enum Update : int {
  kUpdDirectTau = 0,  // eps <- e                        (eq. ds, tau form)
  kUpdDirectSig = 1,  // eps <- eps + e                  (eq. ds, sigma form)
  kUpdAccel = 2,      // eps <- eps + 2 M (e - eps)      (eq. as)
  kUpdResidual = 3,   // r <- e - eps (eps unchanged)    (defect of the current iterate)
  kUpdCorrDirect = 4, // delta <- r + e                  (correction, direct scheme)
  kUpdCorrAccel = 5,  // delta <- delta + 2 M (r + e - delta) (correction, accelerated)
  kUpdForward = 6,    // x1 turn (register variant) without its inverse transform and update: the spectrum of the iterate
};

// Mutable solver control block (device memory, written by the host between
// phases, advanced by the reduction kernels).
struct Ctrl {
  int state;
  int it;            // eta evaluations so far (all phases)
  int max_it;        // cap on `it`
  int stop_rule;     // 0 = eta, 1 = max delta
  int switch_mode;   // 1: eta <= tol means hand over (kSwitch) instead of kConverged
  int stall;         // iterations since the last 10 % improvement of eta
  int stall_window;  // 0 disables stall detection
  int mean_guard;    // 1: eta test also needs |<eps> - eps_bar| <= tol |eps_bar|
  int phase_it;      // iterations in the current phase
  int phase_max;     // cap on phase_it (0: none); reaching it hands over (kSwitch)
  double tol;
  double eta0;
  double best;
  double last_eta;
  double last_delta;
  double last_mean_err;
  double off_sig[6];   // added to <sigma> and <eps> (correction phases: the FP64 iterate's means)
  double off_eps[6];
  double last_ms[6];   // <sigma>, <eps> of the last eta evaluation (with offsets)
  double last_me[6];
  int fault;           // 1: a tile copy did not complete within its wait limit; the solve was stopped
};

// Geometry: grid n1 x n2 x n3, half spectrum of H = n1/2 + 1 modes along x1,
// stored array-of-structures [x3 pos][x2 pos][x1][component].
struct Geom {
  int n1, n2, n3;
  int H;
  long long N;      // voxels
  long long modes;  // n3 * n2 * H
};

// Per-axis wave-vector table entry for frequency index m (signed s,
// q = 2 pi s / L): {q, sin q, cos q - 1, sin(q/2), cos(q/2), nyquist flag};
// exact zeros at the special modes so that k(q) = 0 is detected exactly.
template <typename T>
struct KTab {
  T q, sn, cm1, sh, ch, nyq;
};

// Coefficients per phase (8 entries, T):
// [0] lambda, [1] 2 mu, [2] lambda - lambda0, [3] 2 (mu - mu0),
// [4] 2 a_mu, [5] 2 (a_kappa - a_mu) / d, [6], [7] unused,
// with a_kappa = kappa0 / (kappa + kappa0), a_mu = mu0 / (mu + mu0).
constexpr int kCoef = 8;

constexpr int kGreenPar = 6;
constexpr int kSmpPar = 8 + kGreenPar;  // doubles per sample in IterArgs::smp_par: lambda0, mu0, eps_bar[6], green_par

template <typename T>
struct IterArgs {
  typedef typename Cplx<T>::type T2;
  Geom g;
  int dim;
  int green;
  int dual;          // 1: forward transform carries tau (buffer A) and sigma (buffer B)
  int update;        // Update
  int corr;          // 1: correction phase (zero mean mode, eta adds d64)
  int want_delta;    // inverse x1 pass computes max |d eps|, |d sigma|
  int write_d64;     // store the FP64 iterate's divergence (FP32) for a later correction phase
  int eta_real;      // 1: eta from the real-space divergence stencil (G^C/W/R, k_eta_stencil, k_eta_2d);
                     //    the forward transform then carries tau only
  int tauform;       // 1: the transformed field is tau (mean mode = eps_bar); 0: sigma
  T* eps;            // n_c x N (the iterate, or the correction delta)
  const uint8_t* phase;
  const T* coef;     // 256 x kCoef
  T2* specA;         // AoS [modes][n_c]: tau_hat (dual) or sigma_hat
  T2* specB;         // AoS [modes][n_c]: sigma_hat (dual)
  const T2* tw[3];   // per axis: e^{-2 pi i t / L}
  const KTab<T>* kt[3];
  const T2* rd[3];     // per axis, by storage position: {a, b} with kr_i = a_i prod_{m != i} b_m
                       // (G^R: a = 2 sin(q/2), b = cos(q/2); G^C: a = sin q, b = 1; G: a = q, b = 1);
                       // G^W: {cos q - 1, sin q}, the axis's k itself
  const float4* tws[3];  // x2, x3: twiddles of the FP32 register passes {w.x, w.x, w.y, w.y} (fftls_strided.cuh)
  const int* perm[3];  // per axis: storage position -> frequency index
  const int* pos[3];   // per axis: frequency index -> storage position
  AxisPlan pl[3];
  double lam0, mu0;
  double eps_bar[6];
  // Constants of Gamma' in T, worked out on the host: GB300 issues one warp-wide FP64 instruction per 16 clocks and
  // SM, so a division and a few conversions per thread cost as much as a small FP32 pass itself (128^3, G's Fourier pass
  // 75 -> 62 us; 100x90x75 G^C 24.5 -> 21.4 us).
  // green_par: lambda0, mu0, -1 / (N mu0), (lambda0 + mu0) / (lambda0 + 2 mu0), 1 / (2 mu0),
  // lambda0 / (2 mu0 (d lambda0 + 2 mu0)); inv_n: 1 / N
  T green_par[kGreenPar], inv_n;
  Ctrl* ctrl;
  double* part_mean;   // [x1_blocks][2 nc]: sums of sigma and eps per block
  double* part_eta;    // [z blocks or eta blocks]: sums of |k*.sigma_hat|^2 per block
  double* part_delta;  // [x5_blocks][2]: max |d eps|, max |d sigma| per block
  double* eta_hist;    // [max_it]
  double* ms_hist;     // [max_it][nc]
  float* rfield;       // n_c x N defect r (written by kUpdResidual, read by corrections)
  float2* d64;         // [modes][3] by frequency index: k*.sigma_hat of the FP64 iterate (phase-free form), or with
                       // eta_real [3][N] floats: its real-space divergence
  // grouped launches (fftls_solve_batched): nsmp samples of one 3D geometry share a
  // launch; sample s finds its fields at these element offsets times s (null fields:
  // offset 0) and its lambda0, mu0, eps_bar[6] and the factors of Gamma' at smp_par[kSmpPar s ..] (device memory).
  // Single solves have nsmp = 1 and use the values above.
  int nsmp;
  long long st_field, st_phase, st_spec, st_coef, st_pmean, st_peta, st_pdelta, st_hist, st_d64;
  const double* smp_par;
  // launch shapes (host-computed)
  int x1_lines, x1_blocks;  // forward x1 pass: lines per batch, blocks (grid-stride over batches)
  int x1_vb;                // forward x1 pass: voxels per thread loaded together (1, 2 or 4; 0: staged by bulk copies)
  int x5_lines, x5_blocks;  // inverse x1 pass
  int x5_vb;                // inverse x1 pass: 1 register loads of eps, 0 staged by bulk copies (FP32)
  int x_threads;
  // x1 turn (fftls_turn.cuh): its twiddles (register variant), blocks (the separate x1 passes run on the
  // same grid, so the partial sums of <sigma>, <eps> have one count), lines per tile or block, threads
  const T2* twt;
  int x_blocks, t_reg, t_lines, t_threads;  // t_reg: the register variant
  size_t t_smem;
  int y_w, y_threads, z_w, z_threads;
  size_t x1_smem, x5_smem, y_smem, z_smem;
  CUtensorMap tm[3];       // FP32 register passes: x2 boxes of specA, of specB, x3 boxes of specA (set per launch)
  int e_planes, e_blocks;  // real-space eta: x3-planes per block, blocks (tiles x slabs)
  size_t e_smem;
};

// Shared memory of the forward x1 pass: twiddles, the tile of G lines, and for the
// staged variant the batch's eps (n_c rows of G n1 floats) and phase ids, 16-byte aligned.
__host__ __device__ inline size_t fwd_x_stage_offset(size_t tw_and_tile) { return (tw_and_tile + 15) & ~(size_t)15; }
__host__ __device__ inline size_t fwd_x_stage_bytes(int G, int n1, int nc) {
  return (size_t)G * n1 * (nc * sizeof(float) + 1);
}

// Threads per block of the strided (x2 / x3) passes with W modes per tile: a
// compile-time count, so that every stage of the tile transforms has a fixed
// trip count.
__host__ __device__ constexpr int strided_threads(int W) { return W == 1 ? 128 : 256; }

// Grouped launches (GRP variants, fftls_kernels_{x,y,z}{32,64}g.cu): the same
// kernels over a.nsmp samples of one 3D geometry; 2D grids are not grouped.
template <typename T> cudaError_t launch_fwd_x_grp(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_eta_stencil_grp(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_mid_y_grp(const IterArgs<T>& a, bool inv, cudaStream_t s);
template <typename T> cudaError_t launch_fourier_z_grp(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_reduce_eta_grp(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_inv_x_grp(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_reduce_delta_grp(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t set_attrs_grp(size_t smax);
template <typename T> cudaError_t set_attrs_xgrp(size_t smax);
template <typename T> cudaError_t set_attrs_ygrp(size_t smax);
template <typename T> cudaError_t set_attrs_zgrp(size_t smax);

// Lengths n1 of the x1 turn's register variant (fftls_turn.cuh).
__host__ __device__ constexpr bool turn_reg_length(int n1) { return ct_length(n1); }
// Entries of the turn's twiddle table: w_L^{j r} at [(r - 1) M + j], r = 1..7, j < M = L / 8, then w_M^{j t}
// at [7 M + (t - 1) R2 + j], t = 1..R1-1, j < R2 (M = R1 R2, R1 = 4 for L = 128, else 8).
__host__ __device__ constexpr int turn_r1(int L) { return L == 128 ? 4 : 8; }
__host__ __device__ constexpr int turn_tw_count(int L) {
  return turn_reg_length(L) ? 7 * (L / 8) + (turn_r1(L) - 1) * (L / 8 / turn_r1(L)) : 0;
}

// Launchers (fftls_kernels.cu).  All return cudaGetLastError().
template <typename T> cudaError_t launch_fwd_x(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_eta_stencil(const IterArgs<T>& a, cudaStream_t s);
// tile of the real-space eta kernel (x1 columns x x2 rows): 64 columns, or 32 where those cover n1 with fewer
// columns to spare (n1 <= 32, 75, 90, 96, ...) and in 2D
constexpr int kEtaTileY = 8;
__host__ __device__ constexpr int eta_tile_x(int dim, int n1) {
  return dim == 2 || (n1 + 31) / 32 * 32 < (n1 + 63) / 64 * 64 ? 32 : 64;
}
template <typename T> cudaError_t launch_mid_y(const IterArgs<T>& a, bool inv, cudaStream_t s);
template <typename T> cudaError_t launch_fourier_z(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_reduce_eta(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_inv_x(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t launch_reduce_delta(const IterArgs<T>& a, cudaStream_t s);
// the x1 turn (fftls_kernels_t32.cu, _t64.cu), its dynamic shared-memory limit and need: `lines` per block of
// the register variant, or per tile of the other (line: bytes of one)
template <typename T> cudaError_t launch_turn(const IterArgs<T>& a, cudaStream_t s);
template <typename T> cudaError_t set_attrs_turn(size_t smax);
template <typename T> size_t turn_smem_reg(int n1, int npairs, int lines);
// Entries of a register pass's twiddle table: w_M^{j r} of stage s at the stage's offset + (r - 1) MR + j
__host__ __device__ constexpr int strided_reg_tw(int L, int s) {
  return s == 0 ? 0 : strided_reg_tw(L, s - 1) + (ct_radix(L, s - 1) - 1) * (ct_msize(L, s - 1) / ct_radix(L, s - 1));
}
// FP32 register passes along x2 and x3 (fftls_strided.cuh, fftls_kernels_yr32.cu, _zr32.cu) and their lengths
__host__ __device__ constexpr bool strided_reg_length(int L) { return ct_length(L); }
cudaError_t launch_y_reg(const IterArgs<float>& a, bool inv, cudaStream_t s);
cudaError_t launch_z_reg(const IterArgs<float>& a, cudaStream_t s);
cudaError_t set_attrs_y_reg();
cudaError_t set_attrs_z_reg();
template <typename T> cudaError_t set_kernel_attributes(const IterArgs<T>& a, size_t smax);
// dynamic shared-memory limits of the x2 and x3 kernels (their own translation units)
template <typename T> cudaError_t set_attrs_y(size_t smax);
template <typename T> cudaError_t set_attrs_z(size_t smax);

// Elementwise helpers.
template <typename T> cudaError_t launch_fill_eps(T* eps, int nc, long long N, const double* eps_bar6, cudaStream_t s);
template <typename TO, typename TI> cudaError_t launch_convert(TO* out, const TI* in, long long n, cudaStream_t s);
// out += in (FP64 += FP32), n values
cudaError_t launch_add_correction(double* out, const float* in, long long n, cudaStream_t s);
// stress = C(x):eps as FP64 (optional), plus FP64 sums of sigma and eps into part[blocks][2 nc]
template <typename T> cudaError_t launch_stress(const T* eps, const uint8_t* phase, const T* coef, int dim,
                                                 long long N, double* stress_out, double* part, int blocks,
                                                 cudaStream_t s);
// largest phase id in the image (atomicMax into *out, zeroed first)
cudaError_t launch_phase_max(const uint8_t* phase, long long N, unsigned int* out, int blocks, cudaStream_t s);
cudaError_t launch_sum_parts(const double* part, int blocks, int width, double* out, cudaStream_t s);

}  // namespace fftls
