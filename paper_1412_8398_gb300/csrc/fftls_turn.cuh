#pragma once
// The x1 turn of the iteration: inverse x1 transform of the strain spectrum, the scheme's update, the
// constitutive law of the new iterate and the forward x1 transform of its polarisation, in one kernel
// (as two passes, the forward one read back from HBM the strain and the phase ids the inverse one had
// just had in registers: 25 of the iteration's 292 bytes per voxel in FP32, one launch and two
// shared-memory stagings of the line more).
//
// Two variants, by the length n1 of the lines:
//  * k_turn_reg, n1 = 64, 128, 256, 512: n1 / 8 threads per line, eight voxels of every component in a
//    thread's registers.  The inverse transform's last stage, the update, the law and the forward
//    transform's first stage all act on voxels x = j + (n1 / 8) r of thread j, so the strain field is
//    updated between two register butterflies and the line goes through shared memory only between
//    stages (at most twice per transform) and for the pairing of modes k and n1 - k.  Lines are
//    independent: their threads synchronise among themselves (a warp, or two warps on a named barrier).
//  * k_turn_gen, any other length, and grids of few lines: tiles of t_lines lines in shared memory, every
//    stage spread over the 256 threads of a block.  A line of k_turn_reg has only n1 / 8 threads, each with a
//    long chain of dependent work, so it pays only while there are enough lines for every SM (turn_reg in
//    fftls_solver.cu: at least 64 threads per SM; FP64 128^2 in 2D, 16 threads a line: 40 us against 20).
// What bounds it at 512^3 (FP32): 97.4 bytes per voxel, 13.1 GB per launch; 2.92 ms (4.48 TB/s, 0.66 of the
// measured copy rate), where the two separate passes took 2.18 + 2.01 ms; 2.74 ms since the sums of <sigma>, <eps>
// take one FP64 conversion and addition per warp and flush instead of twelve (warp_sums).  The rest is the latency of a line's
// chain (12 synchronisations, four register transforms) at 16 warps per SM.  In FP64 the arithmetic bounds it
// (about 250 FP64 instructions per voxel, two lanes per clock and SM): 6.78 against 3.87 + 3.11 ms at 256^3.
// Both take the sample of a grouped launch (fftls_solve_batched) as blockIdx.y; a single solve is one
// sample, so grouped and single solves run the same code and give the same bits.
#include "fftls_kernels_impl.cuh"

namespace fftls {

// sample s of a grouped launch: only what the x1 turn reads
template <typename T>
struct TurnView {
  typedef typename Cplx<T>::type T2;
  T* eps;
  const uint8_t* phase;
  const T* coef;
  T2 *specA, *specB;
  const float* rfield;
  double *part_mean, *part_delta;
};
template <typename T>
__device__ __forceinline__ TurnView<T> turn_view(const IterArgs<T>& a, int s) {
  TurnView<T> v;
  v.eps = a.eps + s * a.st_field;
  v.phase = a.phase + s * a.st_phase;
  v.coef = a.coef + s * a.st_coef;
  v.specA = a.specA + s * a.st_spec;
  v.specB = a.specB + s * a.st_spec;
  v.rfield = a.rfield + s * a.st_field;
  v.part_mean = a.part_mean + s * a.st_pmean;
  v.part_delta = a.part_delta + s * a.st_pdelta;
  return v;
}

// The update of one voxel (eq. ds, tau or sigma form; eq. as; the correction phases): the strain e of
// the inverse transform and the old iterate o give the new iterate n; cf: the phase's coefficients.
template <typename T, int DIM>
__device__ __forceinline__ void turn_update(int upd, const T (&e)[Comp<DIM>::NC], const T (&o)[Comp<DIM>::NC],
                                            const float* rf, long long N, const T* cf, T (&n)[Comp<DIM>::NC]) {
  constexpr int NC = Comp<DIM>::NC;
  if (upd == kUpdAccel || upd == kUpdCorrAccel) {
    T d[NC];
    T trd = (T)0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      d[c] = e[c] - o[c];
      if (upd == kUpdCorrAccel) d[c] += (T)rf[(long long)c * N];
      if (c < DIM) trd += d[c];
    }
    const T am = cf[4], av = cf[5];
#pragma unroll
    for (int c = 0; c < NC; ++c) n[c] = o[c] + am * d[c] + (c < DIM ? av * trd : (T)0);
  } else {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      n[c] = e[c];
      if (upd == kUpdDirectSig) n[c] += o[c];
      else if (upd == kUpdCorrDirect) n[c] += (T)rf[(long long)c * N];
    }
  }
}

// sigma and the transformed field (tau, or sigma in the sigma form) of the new iterate; sums of sigma and eps
template <typename T, int DIM>
__device__ __forceinline__ void turn_law(const T (&n)[Comp<DIM>::NC], const T* cf, bool tauform, T (&s)[Comp<DIM>::NC],
                                         T (&out)[Comp<DIM>::NC]) {
  constexpr int NC = Comp<DIM>::NC;
  const T lam = cf[0], mu2 = cf[1], dlam = cf[2], dmu2 = cf[3];
  T tr = n[0] + n[1];
  if (DIM == 3) tr += n[2];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    s[c] = mu2 * n[c] + (c < DIM ? lam * tr : (T)0);
    out[c] = tauform ? dmu2 * n[c] + (c < DIM ? dlam * tr : (T)0) : s[c];
  }
}

// largest |d eps| and |d sigma| of the update (max-delta stop)
template <typename T, int DIM>
__device__ __forceinline__ void turn_delta(const T (&n)[Comp<DIM>::NC], const T (&o)[Comp<DIM>::NC], const T* cf,
                                           T (&dmax)[2]) {
  constexpr int NC = Comp<DIM>::NC;
  T d[NC];
  T tr = (T)0;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    d[c] = n[c] - o[c];
    if (c < DIM) tr += d[c];
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const T ds = cf[1] * d[c] + (c < DIM ? cf[0] * tr : (T)0);
    dmax[0] = fmax(dmax[0], fabs(d[c]));
    dmax[1] = fmax(dmax[1], fabs(ds));
  }
}

// eight coefficients of a phase (16-byte aligned rows)
__device__ __forceinline__ void load_coef(const float* p, float (&cf)[6]) {
  const float4 u = __ldg(reinterpret_cast<const float4*>(p));
  const float2 v = __ldg(reinterpret_cast<const float2*>(p + 4));
  cf[0] = u.x; cf[1] = u.y; cf[2] = u.z; cf[3] = u.w;
  cf[4] = v.x; cf[5] = v.y;
}
__device__ __forceinline__ void load_coef(const double* p, double (&cf)[6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i) cf[i] = __ldg(p + i);
}

// ---------------------------------------------------------------------------
// lengths 64, 128, 256, 512
// ---------------------------------------------------------------------------
// L = 8 M, M = R1 R2: forward, voxel x = j + M r and mode k = r + 8 (t + R1 u):
//   stage 0: radix 8 over r at fixed j,       twiddle w_L^{j r};
//   stage 1: radix R1 over s, j = j' + R2 s,  twiddle w_M^{j' t};
//   stage 2: radix R2 over j' (none for R2 = 1).
// Thread a of the line's M threads takes j = a in stage 0, the pairs (r, j') = (i / R2, i % R2) with
// i = a + M b in stage 1 and the pairs (r, t), r + 8 t = a + M b in stage 2, so it ends with the modes
// k = a + M v, v = 0..7.  The inverse runs the same steps backwards.  Between stages the line goes
// through shared memory at [r * S1 + j] and [r + 8 t + C2 j'], strides chosen so that the lanes of one
// access (16 in FP32, 8 in FP64) fall in distinct banks on both sides of an exchange.
template <typename T, int L>
struct TurnPlan {
  static constexpr int M = L / 8;
  static constexpr int R1 = turn_r1(L);
  static constexpr int R2 = M / R1;
  static constexpr int NB1 = 8 / R1, NB2 = 8 / R2;
  static constexpr int S1 = R2 == 1 ? 9 : M + (R2 == 8 ? 8 : 4);
  static constexpr int C2 = 8 * R1 + (sizeof(T) == 4 ? (R2 == 8 ? 2 : 4) : (R2 == 8 ? 1 : 2));
  static constexpr int PS = 8 * S1;  // complex values per component pair
  static_assert((R2 - 1) * C2 + 8 * R1 <= PS || R2 == 1, "both exchange layouts fit");
  // complex values of a line (8 mod 16, so that the two or four 8-thread lines of an access at L = 64
  // start in distinct banks)
  __host__ __device__ static constexpr int LS(int np) { return (np * PS) % 16 == 8 ? np * PS : np * PS + 8; }
  static constexpr int TW = turn_tw_count(L);  // twiddles: w_L^{j r}, then w_M^{j' t}
};

template <int R, typename T2>
__device__ __forceinline__ void dft_n(T2* v, bool inv) {
  if (R == 8) dft8(v, inv);
  else if (R == 4) dft4(v, inv);
}

template <int M>
__device__ __forceinline__ void line_sync(int line) {
  if (M <= 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(1 + line), "n"(M) : "memory");
}

// forward transform of the thread's eight voxels of NP component pairs; on return v[p][q] = Z(a + M q)
template <typename T, int L, int NP, typename T2>
__device__ __forceinline__ void line_forward(T2 (&v)[NP][8], T2* buf, const T2* tw, int a, int line) {
  typedef TurnPlan<T, L> P;
#pragma unroll
  for (int p = 0; p < NP; ++p) dft8(v[p], false);
#pragma unroll
  for (int r = 1; r < 8; ++r) {
    const T2 w = tw[(r - 1) * P::M + a];
#pragma unroll
    for (int p = 0; p < NP; ++p) v[p][r] = cmul(v[p][r], w);
  }
#pragma unroll
  for (int p = 0; p < NP; ++p)
#pragma unroll
    for (int r = 0; r < 8; ++r) buf[p * P::PS + r * P::S1 + a] = v[p][r];
  line_sync<P::M>(line);
#pragma unroll
  for (int b = 0; b < P::NB1; ++b) {
    const int i = a + P::M * b, r = i / P::R2, j = i % P::R2;
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int s = 0; s < P::R1; ++s) v[p][b * P::R1 + s] = buf[p * P::PS + r * P::S1 + j + P::R2 * s];
  }
  line_sync<P::M>(line);
#pragma unroll
  for (int b = 0; b < P::NB1; ++b) {
    const int i = a + P::M * b, r = i / P::R2, j = i % P::R2;
#pragma unroll
    for (int p = 0; p < NP; ++p) dft_n<P::R1>(&v[p][b * P::R1], false);
    if (P::R2 > 1) {
#pragma unroll
      for (int t = 1; t < P::R1; ++t) {
        const T2 w = tw[7 * P::M + (t - 1) * P::R2 + j];
#pragma unroll
        for (int p = 0; p < NP; ++p) v[p][b * P::R1 + t] = cmul(v[p][b * P::R1 + t], w);
      }
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int t = 0; t < P::R1; ++t) buf[p * P::PS + r + 8 * t + j * P::C2] = v[p][b * P::R1 + t];
    }
  }
  if (P::R2 > 1) {
    line_sync<P::M>(line);
#pragma unroll
    for (int b = 0; b < P::NB2; ++b)
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        T2 z[P::R2];
#pragma unroll
        for (int u = 0; u < P::R2; ++u) z[u] = buf[p * P::PS + a + P::M * b + u * P::C2];
        dft_n<P::R2>(z, false);
#pragma unroll
        for (int u = 0; u < P::R2; ++u) v[p][b + P::NB2 * u] = z[u];
      }
    line_sync<P::M>(line);
  }
}

// inverse of line_forward (unnormalised): v[p][q] = Z(a + M q) in, voxels a + M r out
template <typename T, int L, int NP, typename T2>
__device__ __forceinline__ void line_inverse(T2 (&v)[NP][8], T2* buf, const T2* tw, int a, int line) {
  typedef TurnPlan<T, L> P;
  if (P::R2 > 1) {
#pragma unroll
    for (int b = 0; b < P::NB2; ++b)
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        T2 z[P::R2];
#pragma unroll
        for (int u = 0; u < P::R2; ++u) z[u] = v[p][b + P::NB2 * u];
        dft_n<P::R2>(z, true);
#pragma unroll
        for (int u = 0; u < P::R2; ++u) buf[p * P::PS + a + P::M * b + u * P::C2] = z[u];
      }
    line_sync<P::M>(line);
#pragma unroll
    for (int b = 0; b < P::NB1; ++b) {
      const int i = a + P::M * b, r = i / P::R2, j = i % P::R2;
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int t = 0; t < P::R1; ++t) v[p][b * P::R1 + t] = buf[p * P::PS + r + 8 * t + j * P::C2];
#pragma unroll
      for (int t = 1; t < P::R1; ++t) {
        const T2 w = tw[7 * P::M + (t - 1) * P::R2 + j];
#pragma unroll
        for (int p = 0; p < NP; ++p) v[p][b * P::R1 + t] = cmulc(v[p][b * P::R1 + t], w);
      }
    }
    line_sync<P::M>(line);
  }
#pragma unroll
  for (int b = 0; b < P::NB1; ++b) {
    const int i = a + P::M * b, r = i / P::R2, j = i % P::R2;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      dft_n<P::R1>(&v[p][b * P::R1], true);
#pragma unroll
      for (int s = 0; s < P::R1; ++s) buf[p * P::PS + r * P::S1 + j + P::R2 * s] = v[p][b * P::R1 + s];
    }
  }
  line_sync<P::M>(line);
#pragma unroll
  for (int p = 0; p < NP; ++p)
#pragma unroll
    for (int r = 0; r < 8; ++r) v[p][r] = buf[p * P::PS + r * P::S1 + a];
#pragma unroll
  for (int r = 1; r < 8; ++r) {
    const T2 w = tw[(r - 1) * P::M + a];
#pragma unroll
    for (int p = 0; p < NP; ++p) v[p][r] = cmulc(v[p][r], w);
  }
#pragma unroll
  for (int p = 0; p < NP; ++p) dft8(v[p], true);
  line_sync<P::M>(line);
}

// components 2p, 2p + 1 of a mode (B = 0 past the last component)
template <int NC>
__device__ __forceinline__ void mode_pair(const float2* m, int p, float2& A, float2& B) {
  if (NC % 2 == 0) {
    const float4 t = *reinterpret_cast<const float4*>(m + 2 * p);
    A = make_float2(t.x, t.y);
    B = make_float2(t.z, t.w);
  } else {
    A = m[2 * p];
    B = 2 * p + 1 < NC ? m[2 * p + 1] : make_float2(0.f, 0.f);
  }
}
template <int NC>
__device__ __forceinline__ void mode_pair(const double2* m, int p, double2& A, double2& B) {
  A = m[2 * p];
  B = 2 * p + 1 < NC ? m[2 * p + 1] : make_double2(0.0, 0.0);
}

// The half spectrum of a line into the thread's modes Z(a + M q) of the packed pairs: z(k) = A + i B and
// z(L - k) = conj(A) + i conj(B); the upper half comes from the thread that loaded mode L - k.
template <typename T, int L, int NC, int NP, typename T2>
__device__ __forceinline__ void line_pack(const T2* spec, T2 (&v)[NP][8], T2* buf, int a, int line) {
  typedef TurnPlan<T, L> P;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = a + P::M * q;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      T2 A, B;
      mode_pair<NC>(spec + (long long)k * NC, p, A, B);
      if (q == 0 && a == 0) { A.y = (T)0; B.y = (T)0; }
      v[p][q] = cmk<T2>(A.x - B.y, A.y + B.x);
      if (q > 0 || a > 0) buf[p * P::PS + L / 2 - k] = cmk<T2>(A.x + B.y, B.x - A.y);
    }
  }
  if (a == 0) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      T2 A, B;
      mode_pair<NC>(spec + (long long)(L / 2) * NC, p, A, B);
      buf[p * P::PS] = cmk<T2>(A.x, B.x);
    }
  }
  line_sync<P::M>(line);
#pragma unroll
  for (int q = 4; q < 8; ++q)
#pragma unroll
    for (int p = 0; p < NP; ++p) v[p][q] = buf[p * P::PS + a + P::M * (q - 4)];
  line_sync<P::M>(line);
}

// Z(k), Z(L - k) of the packed pairs into the half spectrum's modes A = (Z(k) + conj Z(L - k)) / 2,
// B = -i (Z(k) - conj Z(L - k)) / 2
template <typename T, int L, int NC, int NP, typename T2>
__device__ __forceinline__ void line_unpack(T2* spec, const T2 (&v)[NP][8], T2* buf, int a, int line, bool active) {
  typedef TurnPlan<T, L> P;
  const T h = (T)0.5;
#pragma unroll
  for (int q = 4; q < 8; ++q)
#pragma unroll
    for (int p = 0; p < NP; ++p) buf[p * P::PS + a + P::M * (q - 4)] = v[p][q];
  line_sync<P::M>(line);
  auto put = [&](int k, int p, T2 Z, T2 Zm) {
    const T2 A = cmk<T2>(h * (Z.x + Zm.x), h * (Z.y - Zm.y));
    const T2 B = cmk<T2>(h * (Z.y + Zm.y), -h * (Z.x - Zm.x));
    T2* d = spec + (long long)k * NC + 2 * p;
    if (NC % 2 == 0) store_pair(d, A, B);
    else {
      d[0] = A;
      if (2 * p + 1 < NC) d[1] = B;
    }
  };
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = a + P::M * q;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const T2 Z = v[p][q];
      const T2 Zm = (q == 0 && a == 0) ? Z : buf[p * P::PS + L / 2 - k];
      if (active) put(k, p, Z, Zm);
    }
  }
  if (a == 0 && active)
#pragma unroll
    for (int p = 0; p < NP; ++p) put(L / 2, p, v[p][4], v[p][4]);
  line_sync<P::M>(line);
}

// x1 lines per block of k_turn_reg (host and device): 128 threads
__host__ __device__ constexpr int turn_threads() { return 128; }

// FWD (kUpdForward): no inverse transform and no update, the spectrum of the iterate as it is
template <typename T, int DIM, int L, bool FWD>
__global__ void __launch_bounds__(turn_threads(), sizeof(T) == 4 ? 4 : 2)
k_turn_reg(const __grid_constant__ IterArgs<T> a_) {
  typedef typename Cplx<T>::type T2;
  typedef TurnPlan<T, L> P;
  constexpr int NC = Comp<DIM>::NC, NP = (NC + 1) / 2;
  constexpr int FLUSH = 2;  // batches between reductions of the FP32 partial sums (16 voxels per thread)
  const TurnView<T> V = turn_view(a_, blockIdx.y);
  const int st = (a_.ctrl + blockIdx.y)->state;
  if (st != kRunning && st != kLast) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T2* tw = reinterpret_cast<T2*>(smem_raw);
  for (int t = threadIdx.x; t < P::TW; t += blockDim.x) tw[t] = a_.twt[t];
  const int line = threadIdx.x / P::M, a = threadIdx.x % P::M;
  const int lpb = blockDim.x / P::M;
  T2* buf = tw + ((P::TW + 1) & ~1) + line * P::LS(NP);
  const long long N = a_.g.N, nlines = (long long)a_.g.n2 * a_.g.n3;
  const int H = L / 2 + 1;
  const int upd = a_.update;
  const bool tauform = a_.tauform;
  const bool need_o = (upd != kUpdDirectTau && upd != kUpdCorrDirect) || a_.want_delta;  // reads the old iterate
  __shared__ double wacc[turn_threads() / 32][2 * NC];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  T acc[2 * NC];
#pragma unroll
  for (int c = 0; c < 2 * NC; ++c) acc[c] = (T)0;
  T dmax[2] = {(T)0, (T)0};
  int pend = 0;
  double wsum = 0.0;  // the warp's FP64 sum of value lane / sum_lanes(2 NC)
  auto flush = [&]() {
    wsum += (double)warp_sums(acc);
#pragma unroll
    for (int c = 0; c < 2 * NC; ++c) acc[c] = (T)0;
    pend = 0;
  };
  const long long step = (long long)gridDim.x * lpb;
  for (long long l0 = (long long)blockIdx.x * lpb; l0 < nlines; l0 += step) {
    const bool active = l0 + line < nlines;
    const long long ln = active ? l0 + line : nlines - 1;
    {  // the line's strain and phase ids towards L2 while its spectrum is transformed
      constexpr int PER = 128 / sizeof(T);
      if (need_o)
        for (int i = a; i < NC * (L / PER); i += P::M)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(V.eps + (long long)(i / (L / PER)) * N + ln * L + (i % (L / PER)) * PER));
      if (a < (L + 127) / 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(V.phase + ln * L + a * 128));
    }
    T2 v[NP][8];
    if (!FWD) line_pack<T, L, NC, NP>(V.specA + ln * H * NC, v, buf, a, line);
    {  // the next line's spectrum
      const long long nx = ln + step;
      if (!FWD && nx < nlines) {
        const char* base = reinterpret_cast<const char*>(V.specA + nx * H * NC);
        constexpr int bytes = (L / 2 + 1) * NC * (int)sizeof(T2);
        for (int off = a * 128; off < bytes; off += P::M * 128)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(base + off));
      }
    }
    if (!FWD) line_inverse<T, L, NP>(v, buf, tw, a, line);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const long long vox = ln * L + a + P::M * r;
      T e[NC], o[NC], n[NC], s[NC], out[NC], cf[6];
      load_coef(V.coef + (int)V.phase[vox] * kCoef, cf);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (!FWD) e[c] = (c & 1) ? v[c / 2][r].y : v[c / 2][r].x;
        o[c] = need_o ? V.eps[(long long)c * N + vox] : (T)0;
      }
      if constexpr (FWD) {
#pragma unroll
        for (int c = 0; c < NC; ++c) n[c] = o[c];
      } else {
        turn_update<T, DIM>(upd, e, o, V.rfield + vox, N, cf, n);
      }
      turn_law<T, DIM>(n, cf, tauform, s, out);
      if (active) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (!FWD) V.eps[(long long)c * N + vox] = n[c];
          acc[c] += s[c];
          acc[NC + c] += n[c];
        }
        if (a_.want_delta) turn_delta<T, DIM>(n, o, cf, dmax);
      }
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        v[p][r].x = out[2 * p];
        v[p][r].y = 2 * p + 1 < NC ? out[2 * p + 1 < NC ? 2 * p + 1 : 0] : (T)0;
      }
    }
    if (sizeof(T) == 4 && ++pend == FLUSH) flush();
    line_forward<T, L, NP>(v, buf, tw, a, line);
    line_unpack<T, L, NC, NP>(V.specA + ln * H * NC, v, buf, a, line, active);
    if (a_.dual) {  // eta in Fourier space: sigma of the new iterate too (the thread reads back its own stores)
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const long long vox = ln * L + a + P::M * r;
        T n[NC], s[NC], out[NC], cf[6];
        load_coef(V.coef + (int)V.phase[vox] * kCoef, cf);
#pragma unroll
        for (int c = 0; c < NC; ++c) n[c] = V.eps[(long long)c * N + vox];
        turn_law<T, DIM>(n, cf, false, s, out);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          v[p][r].x = s[2 * p];
          v[p][r].y = 2 * p + 1 < NC ? s[2 * p + 1 < NC ? 2 * p + 1 : 0] : (T)0;
        }
      }
      line_forward<T, L, NP>(v, buf, tw, a, line);
      line_unpack<T, L, NC, NP>(V.specB + ln * H * NC, v, buf, a, line, active);
    }
  }
  flush();
  if (lane % sum_lanes(2 * NC) == 0 && lane / sum_lanes(2 * NC) < 2 * NC) wacc[warp][lane / sum_lanes(2 * NC)] = wsum;
  __syncthreads();
  if (threadIdx.x < 2 * NC) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) t += wacc[w][threadIdx.x];
    V.part_mean[(size_t)blockIdx.x * 2 * NC + threadIdx.x] = t;
  }
  if (a_.want_delta) {
    double dm[2] = {(double)dmax[0], (double)dmax[1]};
    block_max<2>(dm);
    if (threadIdx.x == 0) {
      V.part_delta[(size_t)blockIdx.x * 2] = dm[0];
      V.part_delta[(size_t)blockIdx.x * 2 + 1] = dm[1];
    }
  }
}

// ---------------------------------------------------------------------------
// any other length, few lines
// ---------------------------------------------------------------------------
// Tiles of t_lines lines, padded rows of odd stride CP (as the separate x1 passes); DUAL: tau and sigma
// are both transformed, and the inverse transform uses the first columns of the wider rows.
template <typename T, int DIM, bool DUAL>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 1) k_turn_gen(const __grid_constant__ IterArgs<T> a_) {
  typedef typename Cplx<T>::type T2;
  constexpr int NC = Comp<DIM>::NC, NPI = (NC + 1) / 2;
  constexpr int nout = DUAL ? 2 * NC : NC, NP = (nout + 1) / 2, CP = odd_stride(NP);
  const TurnView<T> V = turn_view(a_, blockIdx.y);
  const int st = (a_.ctrl + blockIdx.y)->state;
  if (st != kRunning && st != kLast) return;
  const Geom g = a_.g;
  const int L1 = g.n1, H = g.H;
  T2* tile;
  const T2* tws = load_twiddles(a_.tw[0], L1, kTwX1, &tile);
  const int BS = padded_rows(L1) * CP;
  const int* __restrict__ pos = a_.pos[0];
  const long long N = g.N, nlines = (long long)g.n2 * g.n3;
  const int G = a_.t_lines;
  const int upd = a_.update;
  const bool tauform = a_.tauform;
  __shared__ double wacc[8][2 * NC];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double wsum = 0.0;  // the warp's FP64 sum of value lane / sum_lanes(2 NC)
  T acc[2 * NC];
#pragma unroll
  for (int c = 0; c < 2 * NC; ++c) acc[c] = (T)0;
  T dmax[2] = {(T)0, (T)0};
  const FastDiv fL = make_fastdiv(L1), fH = make_fastdiv(H);
  for (long long l0 = (long long)blockIdx.x * G; l0 < nlines; l0 += (long long)gridDim.x * G) {
    const int nl = (int)min((long long)G, nlines - l0);
    prefetch_voxels<T>(V.eps, V.phase, N, NC, l0 * L1, nl * L1);
    for (int idx = threadIdx.x; idx < nl * H; idx += blockDim.x) {
      const int gl = fdiv(idx, fH), k = idx - gl * H;
      const T2* m = V.specA + ((l0 + gl) * (long long)H + k) * NC;
      const bool edge = k == 0 || 2 * k == L1, mirror = k > 0 && L1 - k >= H;
      T2* r0 = tile + gl * BS + prow(__ldg(&pos[k]), 1) * CP;
      T2* r1 = tile + gl * BS + prow(__ldg(&pos[mirror ? L1 - k : k]), 1) * CP;
#pragma unroll
      for (int p = 0; p < NPI; ++p) {
        T2 A, B;
        mode_pair<NC>(m, p, A, B);
        if (edge) { A.y = (T)0; B.y = (T)0; }
        r0[p] = cmk<T2>(A.x - B.y, A.y + B.x);
        if (mirror) r1[p] = cmk<T2>(A.x + B.y, B.x - A.y);
      }
    }
    __syncthreads();
    tile_fft_ct<CP, NPI, true, true, false>(tile, nl, BS, a_.pl[0], tws);
    for (int idx = threadIdx.x; idx < nl * L1; idx += blockDim.x) {
      const int gl = fdiv(idx, fL), x = idx - gl * L1;
      const long long vox = (l0 + gl) * (long long)L1 + x;
      T2* row = tile + gl * BS + prow(x, 1) * CP;
      T e[NC], o[NC], n[NC], s[NC], out[NC], cf[6];
      load_coef(V.coef + (int)V.phase[vox] * kCoef, cf);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        e[c] = (c & 1) ? row[c / 2].y : row[c / 2].x;
        o[c] = V.eps[(long long)c * N + vox];
      }
      turn_update<T, DIM>(upd, e, o, V.rfield + vox, N, cf, n);
      turn_law<T, DIM>(n, cf, tauform, s, out);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        V.eps[(long long)c * N + vox] = n[c];
        acc[c] += s[c];
        acc[NC + c] += n[c];
      }
      if (a_.want_delta) turn_delta<T, DIM>(n, o, cf, dmax);
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const int c0 = 2 * p, c1 = 2 * p + 1;
        row[p] = cmk<T2>(c0 < NC ? out[c0 % NC] : s[c0 % NC], c1 >= nout ? (T)0 : (c1 < NC ? out[c1 % NC] : s[c1 % NC]));
      }
    }
    if (sizeof(T) == 4) {
      wsum += (double)warp_sums(acc);
#pragma unroll
      for (int c = 0; c < 2 * NC; ++c) acc[c] = (T)0;
    }
    __syncthreads();
    tile_fft_ct<CP, NP, true, false, false>(tile, nl, BS, a_.pl[0], tws);
    for (int idx = threadIdx.x; idx < nl * H; idx += blockDim.x) {
      const int gl = fdiv(idx, fH), k = idx - gl * H;
      const T2* r0 = tile + gl * BS + prow(__ldg(&pos[k]), 1) * CP;
      const T2* r1 = tile + gl * BS + prow(__ldg(&pos[k == 0 ? 0 : L1 - k]), 1) * CP;
      const long long m = (l0 + gl) * (long long)H + k;
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const T2 Z = r0[p], Zm = r1[p];
        const T2 A = cmk<T2>((T)0.5 * (Z.x + Zm.x), (T)0.5 * (Z.y - Zm.y));
        const T2 B = cmk<T2>((T)0.5 * (Z.y + Zm.y), (T)-0.5 * (Z.x - Zm.x));
        const int o0 = 2 * p, o1 = 2 * p + 1;
        T2* d0 = (o0 < NC ? V.specA : V.specB) + m * NC + (o0 % NC);
        if (NC % 2 == 0 && o1 < nout && (o0 < NC) == (o1 < NC)) {
          store_pair(d0, A, B);
        } else {
          *d0 = A;
          if (o1 < nout) (o1 < NC ? V.specA : V.specB)[m * NC + (o1 % NC)] = B;
        }
      }
    }
    __syncthreads();
  }
  if (sizeof(T) == 8) wsum = (double)warp_sums(acc);
  if (lane % sum_lanes(2 * NC) == 0 && lane / sum_lanes(2 * NC) < 2 * NC) wacc[warp][lane / sum_lanes(2 * NC)] = wsum;
  __syncthreads();
  if (threadIdx.x < 2 * NC) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += wacc[w][threadIdx.x];
    V.part_mean[(size_t)blockIdx.x * 2 * NC + threadIdx.x] = t;
  }
  if (a_.want_delta) {
    double dm[2] = {(double)dmax[0], (double)dmax[1]};
    block_max<2>(dm);
    if (threadIdx.x == 0) {
      V.part_delta[(size_t)blockIdx.x * 2] = dm[0];
      V.part_delta[(size_t)blockIdx.x * 2 + 1] = dm[1];
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T, int DIM>
cudaError_t launch_turn_d(const IterArgs<T>& a, cudaStream_t s) {
  const dim3 grid(a.x_blocks, a.nsmp > 1 ? a.nsmp : 1);
  if (a.t_reg) {
    const bool fwd = a.update == kUpdForward;
    switch (a.g.n1) {
      case 64: (fwd ? k_turn_reg<T, DIM, 64, true> : k_turn_reg<T, DIM, 64, false>)<<<grid, a.t_threads, a.t_smem, s>>>(a); break;
      case 128: (fwd ? k_turn_reg<T, DIM, 128, true> : k_turn_reg<T, DIM, 128, false>)<<<grid, a.t_threads, a.t_smem, s>>>(a); break;
      case 256: (fwd ? k_turn_reg<T, DIM, 256, true> : k_turn_reg<T, DIM, 256, false>)<<<grid, a.t_threads, a.t_smem, s>>>(a); break;
      default: (fwd ? k_turn_reg<T, DIM, 512, true> : k_turn_reg<T, DIM, 512, false>)<<<grid, a.t_threads, a.t_smem, s>>>(a); break;
    }
  } else if (a.dual) {
    k_turn_gen<T, DIM, true><<<grid, a.t_threads, a.t_smem, s>>>(a);
  } else {
    k_turn_gen<T, DIM, false><<<grid, a.t_threads, a.t_smem, s>>>(a);
  }
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_turn(const IterArgs<T>& a, cudaStream_t s) {
  return a.dim == 3 ? launch_turn_d<T, 3>(a, s) : launch_turn_d<T, 2>(a, s);
}

template <typename T>
cudaError_t set_attrs_turn(size_t smax) {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* f) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smax);
  };
  set((const void*)k_turn_reg<T, 3, 64, false>);
  set((const void*)k_turn_reg<T, 3, 64, true>);
  set((const void*)k_turn_reg<T, 3, 128, false>);
  set((const void*)k_turn_reg<T, 3, 128, true>);
  set((const void*)k_turn_reg<T, 3, 256, false>);
  set((const void*)k_turn_reg<T, 3, 256, true>);
  set((const void*)k_turn_reg<T, 3, 512, false>);
  set((const void*)k_turn_reg<T, 3, 512, true>);
  set((const void*)k_turn_reg<T, 2, 64, false>);
  set((const void*)k_turn_reg<T, 2, 64, true>);
  set((const void*)k_turn_reg<T, 2, 128, false>);
  set((const void*)k_turn_reg<T, 2, 128, true>);
  set((const void*)k_turn_reg<T, 2, 256, false>);
  set((const void*)k_turn_reg<T, 2, 256, true>);
  set((const void*)k_turn_reg<T, 2, 512, false>);
  set((const void*)k_turn_reg<T, 2, 512, true>);
  set((const void*)k_turn_gen<T, 3, true>);
  set((const void*)k_turn_gen<T, 3, false>);
  set((const void*)k_turn_gen<T, 2, true>);
  set((const void*)k_turn_gen<T, 2, false>);
  return e;
}

// Shared memory of the turn (host): k_turn_reg with lpb lines per block, k_turn_gen with G lines per tile.
template <typename T, int L>
constexpr size_t turn_reg_smem(int np, int lpb) {
  typedef TurnPlan<T, L> P;
  return (size_t)(((P::TW + 1) & ~1) + lpb * P::LS(np)) * 2 * sizeof(T);
}
template <typename T>
size_t turn_smem_reg(int L, int np, int lpb) {
  return L == 64 ? turn_reg_smem<T, 64>(np, lpb) : L == 128 ? turn_reg_smem<T, 128>(np, lpb)
       : L == 256 ? turn_reg_smem<T, 256>(np, lpb) : turn_reg_smem<T, 512>(np, lpb);
}

}  // namespace fftls
