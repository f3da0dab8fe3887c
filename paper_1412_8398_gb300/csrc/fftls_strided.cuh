#pragma once
// FP32 strided passes of the lengths 64, 128, 256, 512 with the transform's butterflies in registers (sm_103a): the x2
// pass (forward or inverse; k_y_reg, k_y_tma) and the x3 pass with Gamma' per mode (k_z_reg, k_z_tma; 3D G^C / G^W /
// G^R with eta from the real-space stencil).
//
// A thread holds eight rows of one 16-byte unit (two complex components of a mode; x2 pass) or of a whole mode (three
// units; x3 pass); a stage is one radix-8 or two radix-4 butterflies on them, and the tile goes through shared memory
// between stages only.  In the x3 pass the last forward stage, Gamma' and the first inverse stage act on the same
// registers.  The two components of a unit run through the same operations as packed pairs (add / sub / mul /
// fma.rn.f32x2), half of the transform's FMA-pipe instructions.  Storage order and per-axis tables are those of the
// tile kernels (AxisPlan), which keep the other lengths, FP64, and G's Fourier pass.
//
// What bounds them: 512^3, 6.47 GB per launch (0.95 ms at the measured copy rate).  x2 pass 1.30 -> 1.09 (forward) and
// 1.31 -> 1.15 ms (inverse), 0.83 - 0.88 of that rate; x3 pass 2.08 -> 1.55 ms, whose tile crosses shared memory twelve
// times (128 bytes per clock and SM: about the time of its HBM traffic) against sixteen before.
#include "fftls_kernels_impl.cuh"

namespace fftls {

// two FP32 values in one 64-bit register pair
struct f2 {
  unsigned long long v;
};
__device__ __forceinline__ f2 f2_make(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_split(f2 a, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// a unit: two complex values (x: real parts, y: imaginary parts)
struct c2 {
  f2 x, y;
};
__device__ __forceinline__ c2 operator+(c2 a, c2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ c2 operator-(c2 a, c2 b) { return {a.x - b.x, a.y - b.y}; }
// -i a (forward), +i a (inverse) added to / subtracted from b
template <bool INV>
__device__ __forceinline__ c2 add_mi(c2 b, c2 a) { return INV ? c2{b.x - a.y, b.y + a.x} : c2{b.x + a.y, b.y - a.x}; }
template <bool INV>
__device__ __forceinline__ c2 sub_mi(c2 b, c2 a) { return INV ? c2{b.x + a.y, b.y - a.x} : c2{b.x - a.y, b.y + a.x}; }

// table entry {w.x, w.x, w.y, w.y}; a w (forward) or a conj(w) (inverse)
template <bool INV>
__device__ __forceinline__ c2 mul_tw(c2 a, f2 wx, f2 wy, f2 nwy) {
  if (INV) return {f2_fma(a.y, wy, a.x * wx), f2_fma(a.x, nwy, a.y * wx)};
  return {f2_fma(a.y, nwy, a.x * wx), f2_fma(a.x, wy, a.y * wx)};
}

template <bool INV>
__device__ __forceinline__ void udft4(c2& v0, c2& v1, c2& v2, c2& v3) {
  const c2 a0 = v0 + v2, a1 = v0 - v2, b0 = v1 + v3, b1 = v1 - v3;
  v0 = a0 + b0;
  v2 = a0 - b0;
  v1 = add_mi<INV>(a1, b1);
  v3 = sub_mi<INV>(a1, b1);
}
// radix 8: two radix-4 halves, the odd one turned by w8^s; the factors 1/sqrt 2 of s = 1, 3 go into the last
// additions as fused multiply-adds
template <bool INV>
__device__ __forceinline__ void udft8(c2* v) {
  c2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  udft4<INV>(e0, e1, e2, e3);
  udft4<INV>(o0, o1, o2, o3);
  const f2 h = f2_make(0.70710678118654752f, 0.70710678118654752f);
  const f2 nh = f2_make(-0.70710678118654752f, -0.70710678118654752f);
  v[0] = e0 + o0;
  v[4] = e0 - o0;
  v[2] = add_mi<INV>(e2, o2);
  v[6] = sub_mi<INV>(e2, o2);
  // w8 o1 = h (o1.x + o1.y, o1.y - o1.x), w8^3 o3 = h (o3.y - o3.x, -(o3.x + o3.y)); conjugate turns in the inverse
  const f2 s1 = o1.x + o1.y, d1 = INV ? o1.x - o1.y : o1.y - o1.x;
  const f2 s3 = o3.x + o3.y, d3 = INV ? o3.x - o3.y : o3.y - o3.x;
  if (INV) {
    v[1] = {f2_fma(d1, h, e1.x), f2_fma(s1, h, e1.y)};
    v[5] = {f2_fma(d1, nh, e1.x), f2_fma(s1, nh, e1.y)};
    v[3] = {f2_fma(s3, nh, e3.x), f2_fma(d3, h, e3.y)};
    v[7] = {f2_fma(s3, h, e3.x), f2_fma(d3, nh, e3.y)};
  } else {
    v[1] = {f2_fma(s1, h, e1.x), f2_fma(d1, h, e1.y)};
    v[5] = {f2_fma(s1, nh, e1.x), f2_fma(d1, nh, e1.y)};
    v[3] = {f2_fma(d3, h, e3.x), f2_fma(s3, nh, e3.y)};
    v[7] = {f2_fma(d3, nh, e3.x), f2_fma(s3, h, e3.y)};
  }
}

// Unit between its memory form (re, im, re', im') and registers
__device__ __forceinline__ c2 unit_in(float4 t) { return {f2_make(t.x, t.z), f2_make(t.y, t.w)}; }
__device__ __forceinline__ float4 unit_out(c2 a) {
  float4 t;
  f2_split(a.x, t.x, t.z);
  f2_split(a.y, t.y, t.w);
  return t;
}
// and between its packed form in shared memory and registers
__device__ __forceinline__ c2 unit_lds(const ulonglong2* p) {
  const ulonglong2 t = *p;
  return {{t.x}, {t.y}};
}
__device__ __forceinline__ void unit_sts(ulonglong2* p, c2 a) { *p = make_ulonglong2(a.x.v, a.y.v); }

// Stage S of length L: radix R, thread a of T = L / 8 takes the butterflies i = a + T b, b < 8 / R, of
// base row (i / MR) M + i % MR and legs r MR; butterfly b keeps leg r in v[b R + r].
template <int L, int S>
struct SPlan {
  static constexpr int T = L / 8, R = ct_radix(L, S), M = ct_msize(L, S), MR = M / R, NB = 8 / R;
  __device__ static __forceinline__ int j(int a, int b) { return (a + T * b) % MR; }
  __device__ static __forceinline__ int row(int a, int b) { return (a + T * b) / MR * M + (a + T * b) % MR; }
  // padded row of leg r (row(a, b) + r MR): MR is a multiple of 8, or 1 in the last stage (rows 8 i + r)
  __device__ static __forceinline__ int prow(int a, int b) { const int e = row(a, b); return e + e / 8; }
  __host__ __device__ static constexpr int pleg(int r) { return MR == 1 ? r : r * MR / 8 * 9; }
};
// twiddles of the stage: float4 {w.x, w.x, w.y, w.y} at strided_reg_tw(L, S) + (r - 1) MR + j
template <int L, int S, bool INV, int NU>
__device__ __forceinline__ void reg_twiddle(c2 (&v)[NU][8], const float4* tw, int a) {
  typedef SPlan<L, S> P;
  if (P::MR == 1) return;
#pragma unroll
  for (int b = 0; b < P::NB; ++b) {
    const float4* t = tw + strided_reg_tw(L, S) + P::j(a, b);
#pragma unroll
    for (int r = 1; r < P::R; ++r) {
      const float4 w = t[(r - 1) * P::MR];
      const f2 wx = f2_make(w.x, w.y), wy = f2_make(w.z, w.w), nwy = f2_make(-w.z, -w.w);
#pragma unroll
      for (int n = 0; n < NU; ++n) v[n][b * P::R + r] = mul_tw<INV>(v[n][b * P::R + r], wx, wy, nwy);
    }
  }
}
template <int L, int S, bool INV, int NU>
__device__ __forceinline__ void reg_butterfly(c2 (&v)[NU][8]) {
  typedef SPlan<L, S> P;
#pragma unroll
  for (int n = 0; n < NU; ++n) {
    if (P::R == 8) udft8<INV>(v[n]);
    else {
#pragma unroll
      for (int b = 0; b < P::NB; ++b) udft4<INV>(v[n][4 * b], v[n][4 * b + 1], v[n][4 * b + 2], v[n][4 * b + 3]);
    }
  }
}
// one exchange through the tile: the legs of stage SW out, the legs of stage SR in (C units per row)
template <int L, int SW, int SR, int C, int NU>
__device__ __forceinline__ void reg_exchange(c2 (&v)[NU][8], ulonglong2* tile, int a) {
  typedef SPlan<L, SW> W;
  typedef SPlan<L, SR> Q;
#pragma unroll
  for (int b = 0; b < W::NB; ++b) {
    ulonglong2* p = tile + W::prow(a, b) * C;
#pragma unroll
    for (int r = 0; r < W::R; ++r)
#pragma unroll
      for (int n = 0; n < NU; ++n) unit_sts(p + W::pleg(r) * C + n, v[n][b * W::R + r]);
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < Q::NB; ++b) {
    const ulonglong2* p = tile + Q::prow(a, b) * C;
#pragma unroll
    for (int r = 0; r < Q::R; ++r)
#pragma unroll
      for (int n = 0; n < NU; ++n) v[n][b * Q::R + r] = unit_lds(p + Q::pleg(r) * C + n);
  }
}
// forward transform up to and with its last butterfly; v holds the legs of stage 0 on entry and those of the last
// stage on return.  A stage reads the rows it later writes, so exchanges need one barrier each.
template <int L, int C, int NU>
__device__ __forceinline__ void reg_forward(c2 (&v)[NU][8], ulonglong2* tile, const float4* tw, int a) {
  constexpr int NST = ct_nst(L);
  reg_butterfly<L, 0, false>(v);
  reg_twiddle<L, 0, false>(v, tw, a);
  reg_exchange<L, 0, 1, C>(v, tile, a);
  reg_butterfly<L, 1, false>(v);
  if constexpr (NST == 3) {
    reg_twiddle<L, 1, false>(v, tw, a);
    reg_exchange<L, 1, 2, C>(v, tile, a);
    reg_butterfly<L, 2, false>(v);
  }
}
// its inverse (unnormalised): legs of the last stage in, of stage 0 out
template <int L, int C, int NU>
__device__ __forceinline__ void reg_inverse(c2 (&v)[NU][8], ulonglong2* tile, const float4* tw, int a) {
  constexpr int NST = ct_nst(L);
  if constexpr (NST == 3) {
    reg_butterfly<L, 2, true>(v);
    reg_exchange<L, 2, 1, C>(v, tile, a);
    reg_twiddle<L, 1, true>(v, tw, a);
  }
  reg_butterfly<L, 1, true>(v);
  reg_exchange<L, 1, 0, C>(v, tile, a);
  reg_twiddle<L, 0, true>(v, tw, a);
  reg_butterfly<L, 0, true>(v);
}

// Tile widths (modes) of the register passes at length L: at most 1024 rows x modes (55 KB of shared memory, three
// blocks of 384 or 128 threads per SM); narrower tiles give small grids more blocks.
__host__ __device__ constexpr int strided_reg_threads_y(int L, int W) { return 3 * W * (L / 8); }
__host__ __device__ constexpr int strided_reg_threads_z(int L, int W) { return W * (L / 8); }
__host__ __device__ constexpr size_t strided_reg_smem(int L, int W) {
  return (size_t)strided_reg_tw(L, ct_nst(L)) * 16 + (size_t)(L + L / 8) * 3 * W * 16;
}

template <int L>
__device__ __forceinline__ void reg_tables(float4* tws, const float4* __restrict__ tw) {
  for (int t = threadIdx.x; t < strided_reg_tw(L, ct_nst(L)); t += blockDim.x) tws[t] = __ldg(tw + t);
}

// x2 pass: W modes x L rows; a thread holds eight rows of one unit, the 3 W units of a row on consecutive threads.
template <int L, int W, bool INV>
__global__ void __launch_bounds__(strided_reg_threads_y(L, W), 960 / strided_reg_threads_y(L, W))
k_y_reg(const __grid_constant__ IterArgs<float> a_, int kinds) {
  constexpr int C = 3 * W, T = L / 8;
  constexpr int SL = ct_nst(L) - 1;
  typedef SPlan<L, 0> P0;
  typedef SPlan<L, SL> PL;
  const int smp = blockIdx.z / kinds, kind = blockIdx.z % kinds;
  const int st = (a_.ctrl + smp)->state;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* tws = reinterpret_cast<float4*>(smem_raw);
  ulonglong2* tile = reinterpret_cast<ulonglong2*>(tws + strided_reg_tw(L, ct_nst(L)));
  const int u = threadIdx.x % C, a = threadIdx.x / C;
  const int x0 = blockIdx.x * W;
  const bool on = x0 + u / 3 < a_.g.H;
  const long long rstride = (long long)a_.g.H * 3;  // in units
  float4* g = reinterpret_cast<float4*>((kind ? a_.specB : a_.specA) + smp * a_.st_spec) +
              ((long long)blockIdx.y * L * a_.g.H + x0) * 3 + u;
  c2 v[1][8];
  float4 raw[8];
  if (on) {
    if (INV) {
#pragma unroll
      for (int r = 0; r < 8; ++r) raw[r] = g[(PL::row(a, 0) + r) * rstride];
    } else {
#pragma unroll
      for (int b = 0; b < P0::NB; ++b)
#pragma unroll
        for (int r = 0; r < P0::R; ++r) raw[b * P0::R + r] = g[(a + T * b + r * P0::MR) * rstride];
    }
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) raw[r] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  reg_tables<L>(tws, a_.tws[1]);
  if (!__syncthreads_or(st == kRunning || st == kLast)) return;  // block-uniform, as strided_begin
#pragma unroll
  for (int r = 0; r < 8; ++r) v[0][r] = unit_in(raw[r]);
  ulonglong2* t = tile + u;
  if (INV) {
    reg_inverse<L, C>(v, t, tws, a);
    if (on) {
#pragma unroll
      for (int b = 0; b < P0::NB; ++b)
#pragma unroll
        for (int r = 0; r < P0::R; ++r) g[(a + T * b + r * P0::MR) * rstride] = unit_out(v[0][b * P0::R + r]);
    }
  } else {
    reg_forward<L, C>(v, t, tws, a);
    if (on) {
#pragma unroll
      for (int r = 0; r < 8; ++r) g[(PL::row(a, 0) + r) * rstride] = unit_out(v[0][r]);
    }
  }
}

// e_hat = -Gamma'(k) : tau_hat / N of G^W at one mode, k_i = e^{i q_i} - 1 (displacement form, a 2 x 2 solve in
// span{k, conj k}, as fourier_mode): b = conj(k) . tau, then u and -(k u + u k) / 2.
__device__ __forceinline__ void green_w_mode(float2 (&X)[6], const float2 (&k)[3], float lam0, float mu0, float invN) {
  const float2 b[3] = {
      cadd(cadd(cmul(cconj(k[0]), X[0]), cmul(cconj(k[1]), X[5])), cmul(cconj(k[2]), X[4])),
      cadd(cadd(cmul(cconj(k[0]), X[5]), cmul(cconj(k[1]), X[1])), cmul(cconj(k[2]), X[3])),
      cadd(cadd(cmul(cconj(k[0]), X[4]), cmul(cconj(k[1]), X[3])), cmul(cconj(k[2]), X[2]))};
  float K = 0.f;
  float2 gk = make_float2(0.f, 0.f), p = gk, r = gk;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    K += k[i].x * k[i].x + k[i].y * k[i].y;
    gk = cadd(gk, cmul(k[i], k[i]));
    p = cadd(p, cmul(k[i], b[i]));
    r = cadd(r, cmul(cconj(k[i]), b[i]));
  }
  const float det = 2.f * mu0 * (lam0 + mu0) * K * K - lam0 * mu0 * (gk.x * gk.x + gk.y * gk.y);
  const float idet = det > 0.f ? recip_pos(det) : 0.f;  // 0 at q = 0 only, set by the caller
  const float2 al = cscale(csub(cscale(p, 2.f * mu0 * K), cscale(cmul(gk, r), mu0)), idet);
  const float2 be = cscale(csub(cscale(r, (lam0 + mu0) * K), cscale(cmul(cconj(gk), p), lam0)), idet);
  const float iu = K > 0.f ? recip_pos(mu0 * K) : 0.f;
  float2 uv[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    float2 t = csub(b[j], cscale(cmul(cconj(k[j]), al), lam0));
    t = csub(t, cscale(cmul(k[j], be), mu0));
    uv[j] = cscale(t, iu);
  }
  const float f = -0.5f * invN;
  X[0] = cscale(cmul(k[0], uv[0]), 2.f * f);
  X[1] = cscale(cmul(k[1], uv[1]), 2.f * f);
  X[2] = cscale(cmul(k[2], uv[2]), 2.f * f);
  X[3] = cscale(cadd(cmul(k[1], uv[2]), cmul(k[2], uv[1])), f);
  X[4] = cscale(cadd(cmul(k[0], uv[2]), cmul(k[2], uv[0])), f);
  X[5] = cscale(cadd(cmul(k[0], uv[1]), cmul(k[1], uv[0])), f);
}

// Gamma' on the thread's eight modes of column (x, py), storage positions pz0 .. pz0 + 7 along x3
template <int L, bool WILLOT>
__device__ __forceinline__ void z_modes(const IterArgs<float>& a_, c2 (&v)[3][8], int x, int py, int pz0, int smp) {
  const double* par = a_.nsmp > 1 ? a_.smp_par + kSmpPar * smp : nullptr;
  const float2 rx = x < a_.g.H ? __ldg(&a_.rd[0][x]) : make_float2(1.f, 1.f), ry = __ldg(&a_.rd[1][py]);
  float gp[4];  // lambda0, mu0 (G^W), -1 / (N mu0), (lambda0 + mu0) / (lambda0 + 2 mu0)
#pragma unroll
  for (int i = 0; i < 4; ++i) gp[i] = par ? (float)par[8 + i] : a_.green_par[i];
  const float bxy = rx.y * ry.y, axy = rx.x * ry.y, bxay = rx.y * ry.x;
  const bool line0 = x == 0 && py == 0;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float2 rz = __ldg(&a_.rd[2][pz0 + r]);
    float2 X[6];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      f2_split(v[n][r].x, X[2 * n].x, X[2 * n + 1].x);
      f2_split(v[n][r].y, X[2 * n].y, X[2 * n + 1].y);
    }
    if (WILLOT) {
      const float2 k[3] = {rx, ry, rz};
      green_w_mode(X, k, gp[0], gp[1], a_.inv_n);
    } else {
      green_rd_mode<float>(X, axy * rz.y, bxay * rz.y, bxy * rz.x, gp[2], gp[3]);
    }
    if (line0 && pz0 + r == 0) {
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        X[c].x = a_.corr ? 0.f : (float)(par ? par[2 + c] : a_.eps_bar[c]);
        X[c].y = 0.f;
      }
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      v[n][r].x = f2_make(X[2 * n].x, X[2 * n + 1].x);
      v[n][r].y = f2_make(X[2 * n].y, X[2 * n + 1].y);
    }
  }
}

// x3 pass of 3D G^C / G^R (real directions, rd = {a, b} per axis) and G^W (WILLOT, rd = k per axis): W modes x L
// rows; a thread holds eight rows of one mode.
template <int L, int W, bool WILLOT>
__global__ void __launch_bounds__(strided_reg_threads_z(L, W), 384 / strided_reg_threads_z(L, W) > 12 ? 12 : 384 / strided_reg_threads_z(L, W))
k_z_reg(const __grid_constant__ IterArgs<float> a_) {
  constexpr int C = 3 * W, T = L / 8;
  constexpr int SL = ct_nst(L) - 1;
  typedef SPlan<L, 0> P0;
  typedef SPlan<L, SL> PL;
  const int smp = blockIdx.z;
  const int st = (a_.ctrl + smp)->state;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* tws = reinterpret_cast<float4*>(smem_raw);
  ulonglong2* tile = reinterpret_cast<ulonglong2*>(tws + strided_reg_tw(L, ct_nst(L)));
  const int w = threadIdx.x % W, a = threadIdx.x / W;
  const int x = blockIdx.x * W + w, py = blockIdx.y;
  const bool on = x < a_.g.H;
  const long long rstride = (long long)a_.g.n2 * a_.g.H * 3;  // in units
  float4* g = reinterpret_cast<float4*>(a_.specA + smp * a_.st_spec) + ((long long)py * a_.g.H + x) * 3;
  c2 v[3][8];
#pragma unroll
  for (int b = 0; b < P0::NB; ++b)
#pragma unroll
    for (int r = 0; r < P0::R; ++r) {
      const float4* q = g + (a + T * b + r * P0::MR) * rstride;
#pragma unroll
      for (int n = 0; n < 3; ++n)
        v[n][b * P0::R + r] = unit_in(on ? q[n] : make_float4(0.f, 0.f, 0.f, 0.f));
    }
  reg_tables<L>(tws, a_.tws[2]);
  if (!__syncthreads_or(st == kRunning || st == kLast)) return;  // block-uniform, as strided_begin
  ulonglong2* t = tile + 3 * w;
  reg_forward<L, C>(v, t, tws, a);
  z_modes<L, WILLOT>(a_, v, x, py, PL::row(a, 0), smp);
  reg_inverse<L, C>(v, t, tws, a);
  if (on) {
#pragma unroll
    for (int b = 0; b < P0::NB; ++b)
#pragma unroll
      for (int r = 0; r < P0::R; ++r) {
        float4* q = g + (a + T * b + r * P0::MR) * rstride;
#pragma unroll
        for (int n = 0; n < 3; ++n) q[n] = unit_out(v[n][b * P0::R + r]);
      }
  }
}

// ---------------------------------------------------------------------------
// tiles moved by tensor-map copies
// ---------------------------------------------------------------------------
// The same transforms on tiles that the copy engine brings in and takes out as boxes of up to 256 rows
// (cp.async.bulk.tensor, one instruction a box): on large grids a row's 96 bytes per tile are far apart, and the
// direct loads above cost a memory request per 16 or 32 of them.
__device__ __forceinline__ void tma_load4(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int s, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(s), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_store4(const CUtensorMap* map, int x, int y, int z, int s, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];\n" ::"l"(map), "r"(x),
               "r"(y), "r"(z), "r"(s), "r"(src)
               : "memory");
}

// Thread 0 alone reads the state (so the block decides as one) and, if the solve goes on, starts the tile's boxes of
// up to 256 rows along axis AX; the block loads its twiddles meanwhile and waits (bounded: a lost copy stops the solve
// with ctl->fault set).  false: nothing to do.
template <int L, int W, int AX>
__device__ __forceinline__ bool tma_tile_load(unsigned char* tile, float4* tws, const float4* tw, const CUtensorMap* map,
                                              int x0, int other, int smp, Ctrl* ctl, uint64_t* bar_word, int* flag) {
  constexpr int BOX = L < 256 ? L : 256;
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(bar_word);
  if (threadIdx.x == 0) {
    const int st = ctl->state;
    const bool go = st == kRunning || st == kLast;
    *flag = go;
    if (go) {
      mbar_init(bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
      mbar_arrive_expect_tx(bar, (uint32_t)(L * W * 48));
#pragma unroll
      for (int r = 0; r < L; r += BOX)
        tma_load4((uint32_t)__cvta_generic_to_shared(tile + (size_t)r * W * 48), map, x0 * 12, AX == 1 ? r : other,
                  AX == 1 ? other : r, smp, bar);
    }
  }
  __syncthreads();
  if (!*flag) return false;  // before anything else: a stopped solve's passes still come to the end of their beat
  reg_tables<L>(tws, tw);
  bool done = false;
  for (long long k = 0; k < kBulkWaitRounds && !done; ++k) done = mbar_try_wait(bar, 0);
  if (__syncthreads_or(!done)) {
    if (threadIdx.x == 0) {
      ctl->fault = 1;
      ctl->state = kStopped;
    }
    // the block's own copies: one more bounded wait before it gives up its shared memory
    for (long long k = 0; k < kBulkWaitRounds && !done; ++k) done = mbar_try_wait(bar, 0);
    return false;
  }
  return true;
}
template <int L, int W, int AX>
__device__ __forceinline__ void tma_tile_store(unsigned char* tile, const CUtensorMap* map, int x0, int other, int smp) {
  constexpr int BOX = L < 256 ? L : 256;
  fence_async_shared();
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int r = 0; r < L; r += BOX)
      tma_store4(map, x0 * 12, AX == 1 ? r : other, AX == 1 ? other : r, smp,
                 (uint32_t)__cvta_generic_to_shared(tile + (size_t)r * W * 48));
    bulk_commit_and_wait();
  }
}

// row e of a tile that the copy engine fills sits at e; between stages at e ^ (e / 8 mod 8), so that the
// butterflies of the last stage, eight rows apart, start in distinct banks
__device__ __forceinline__ int swz_row(int e) { return e ^ ((e >> 3) & 7); }

template <int L, int S, int C, bool SWZ, int NU>
__device__ __forceinline__ void tile_out(c2 (&v)[NU][8], ulonglong2* t, int a) {
  typedef SPlan<L, S> P;
#pragma unroll
  for (int b = 0; b < P::NB; ++b)
#pragma unroll
    for (int r = 0; r < P::R; ++r) {
      const int e = P::row(a, b) + r * P::MR;
      ulonglong2* p = t + (SWZ ? swz_row(e) : e) * C;
#pragma unroll
      for (int n = 0; n < NU; ++n) unit_sts(p + n, v[n][b * P::R + r]);
    }
}
template <int L, int S, int C, bool SWZ, int NU>
__device__ __forceinline__ void tile_in(c2 (&v)[NU][8], const ulonglong2* t, int a) {
  typedef SPlan<L, S> P;
#pragma unroll
  for (int b = 0; b < P::NB; ++b)
#pragma unroll
    for (int r = 0; r < P::R; ++r) {
      const int e = P::row(a, b) + r * P::MR;
      const ulonglong2* p = t + (SWZ ? swz_row(e) : e) * C;
#pragma unroll
      for (int n = 0; n < NU; ++n) v[n][b * P::R + r] = unit_lds(p + n);
    }
}
// memory-form rows in (natural order) and out
template <int L, int C, int NU>
__device__ __forceinline__ void tile_in_mem(c2 (&v)[NU][8], const unsigned char* tile, int u0, int a) {
  typedef SPlan<L, 0> P;
  const float4* t = reinterpret_cast<const float4*>(tile) + u0;
#pragma unroll
  for (int b = 0; b < P::NB; ++b)
#pragma unroll
    for (int r = 0; r < P::R; ++r)
#pragma unroll
      for (int n = 0; n < NU; ++n) v[n][b * P::R + r] = unit_in(t[(P::row(a, b) + r * P::MR) * C + n]);
}
template <int L, int C, int NU>
__device__ __forceinline__ void tile_out_mem(c2 (&v)[NU][8], unsigned char* tile, int u0, int a) {
  typedef SPlan<L, 0> P;
  float4* t = reinterpret_cast<float4*>(tile) + u0;
#pragma unroll
  for (int b = 0; b < P::NB; ++b)
#pragma unroll
    for (int r = 0; r < P::R; ++r)
#pragma unroll
      for (int n = 0; n < NU; ++n) t[(P::row(a, b) + r * P::MR) * C + n] = unit_out(v[n][b * P::R + r]);
}

template <int L, int W>
__host__ __device__ constexpr size_t strided_tma_smem() {
  return (size_t)L * W * 48 + (size_t)strided_reg_tw(L, ct_nst(L)) * 16;
}

// Blocks per SM of k_z_tma: three of 128 threads at 512, whose 164 registers without a spill are worth more than a
// fourth block (1.557 against 1.597 ms); four at the shorter lengths (128^3 31.1 -> 28.9 us, 256^3 188 -> 185 us).
__host__ __device__ constexpr int strided_tma_blocks_z(int L, int W) {
  return (L == 512 ? 384 : 512) / strided_reg_threads_z(L, W) > 12 ? 12 : (L == 512 ? 384 : 512) / strided_reg_threads_z(L, W);
}
template <int L, int W, bool WILLOT>
__global__ void __launch_bounds__(strided_reg_threads_z(L, W), strided_tma_blocks_z(L, W))
k_z_tma(const __grid_constant__ IterArgs<float> a_) {
  constexpr int C = 3 * W;
  constexpr int SL = ct_nst(L) - 1;
  extern __shared__ __align__(128) unsigned char smem_tile[];  // the copy engine's boxes start on 128 bytes
  __shared__ __align__(8) uint64_t bar_word;
  __shared__ int flag;
  unsigned char* tile = smem_tile;
  float4* tws = reinterpret_cast<float4*>(smem_tile + (size_t)L * W * 48);
  const int smp = blockIdx.z, py = blockIdx.y, x0 = blockIdx.x * W;
  if (!tma_tile_load<L, W, 2>(tile, tws, a_.tws[2], &a_.tm[2], x0, py, smp, a_.ctrl + smp, &bar_word, &flag)) return;
  const int w = threadIdx.x % W, a = threadIdx.x / W;
  const int x = x0 + w;
  c2 v[3][8];
  ulonglong2* t = reinterpret_cast<ulonglong2*>(tile) + 3 * w;
  tile_in_mem<L, C>(v, tile, 3 * w, a);
  reg_butterfly<L, 0, false>(v);
  reg_twiddle<L, 0, false>(v, tws, a);
  __syncthreads();  // every row is read: the swizzled rows may overwrite them
  tile_out<L, 0, C, true>(v, t, a);
  __syncthreads();
  tile_in<L, 1, C, true>(v, t, a);
  reg_butterfly<L, 1, false>(v);
  if constexpr (SL == 2) {
    reg_twiddle<L, 1, false>(v, tws, a);
    tile_out<L, 1, C, true>(v, t, a);
    __syncthreads();
    tile_in<L, 2, C, true>(v, t, a);
    reg_butterfly<L, 2, false>(v);
  }
  z_modes<L, WILLOT>(a_, v, x, py, SPlan<L, SL>::row(a, 0), smp);
  if constexpr (SL == 2) {
    reg_butterfly<L, 2, true>(v);
    tile_out<L, 2, C, true>(v, t, a);
    __syncthreads();
    tile_in<L, 1, C, true>(v, t, a);
    reg_twiddle<L, 1, true>(v, tws, a);
  }
  reg_butterfly<L, 1, true>(v);
  tile_out<L, 1, C, true>(v, t, a);
  __syncthreads();
  tile_in<L, 0, C, true>(v, t, a);
  reg_twiddle<L, 0, true>(v, tws, a);
  reg_butterfly<L, 0, true>(v);
  __syncthreads();
  tile_out_mem<L, C>(v, tile, 3 * w, a);
  tma_tile_store<L, W, 2>(tile, &a_.tm[2], x0, py, smp);
}

// x2 pass: 192 threads, two units each in turn; every stage in place in the tile
template <int L, int W, bool INV>
__global__ void __launch_bounds__(strided_reg_threads_y(L, W) / 2, 4)
k_y_tma(const __grid_constant__ IterArgs<float> a_, int kinds) {
  constexpr int C = 3 * W, T = L / 8, NT = strided_reg_threads_y(L, W) / 2;
  constexpr int SL = ct_nst(L) - 1;
  static_assert(NT % C == 0, "whole rows of units per turn");
  constexpr int DA = NT / C;
  extern __shared__ __align__(128) unsigned char smem_tile[];  // the copy engine's boxes start on 128 bytes
  __shared__ __align__(8) uint64_t bar_word;
  __shared__ int flag;
  unsigned char* tile = smem_tile;
  float4* tws = reinterpret_cast<float4*>(smem_tile + (size_t)L * W * 48);
  const int smp = blockIdx.z / kinds, kind = blockIdx.z % kinds, pz = blockIdx.y, x0 = blockIdx.x * W;
  const CUtensorMap* map = &a_.tm[kind];
  if (!tma_tile_load<L, W, 1>(tile, tws, a_.tws[1], map, x0, pz, smp, a_.ctrl + smp, &bar_word, &flag)) return;
  const int u = threadIdx.x % C, a0 = threadIdx.x / C;
  ulonglong2* t = reinterpret_cast<ulonglong2*>(tile) + u;
  c2 v[1][8];
  if (INV) {
#pragma unroll
    for (int h = 0; h < T; h += DA) {
      const int a = a0 + h;
      const float4* q = reinterpret_cast<const float4*>(tile) + SPlan<L, SL>::row(a, 0) * C + u;
#pragma unroll
      for (int r = 0; r < 8; ++r) v[0][r] = unit_in(q[r * C]);
      reg_butterfly<L, SL, true>(v);
      tile_out<L, SL, C, false>(v, t, a);
    }
    __syncthreads();
    if constexpr (SL == 2) {
#pragma unroll
      for (int h = 0; h < T; h += DA) {
        const int a = a0 + h;
        tile_in<L, 1, C, false>(v, t, a);
        reg_twiddle<L, 1, true>(v, tws, a);
        reg_butterfly<L, 1, true>(v);
        tile_out<L, 1, C, false>(v, t, a);
      }
      __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < T; h += DA) {
      const int a = a0 + h;
      tile_in<L, 0, C, false>(v, t, a);
      reg_twiddle<L, 0, true>(v, tws, a);
      reg_butterfly<L, 0, true>(v);
      tile_out_mem<L, C>(v, tile, u, a);
    }
  } else {
#pragma unroll
    for (int h = 0; h < T; h += DA) {
      const int a = a0 + h;
      tile_in_mem<L, C>(v, tile, u, a);
      reg_butterfly<L, 0, false>(v);
      reg_twiddle<L, 0, false>(v, tws, a);
      tile_out<L, 0, C, false>(v, t, a);
    }
    __syncthreads();
    if constexpr (SL == 2) {
#pragma unroll
      for (int h = 0; h < T; h += DA) {
        const int a = a0 + h;
        tile_in<L, 1, C, false>(v, t, a);
        reg_butterfly<L, 1, false>(v);
        reg_twiddle<L, 1, false>(v, tws, a);
        tile_out<L, 1, C, false>(v, t, a);
      }
      __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < T; h += DA) {
      const int a = a0 + h;
      tile_in<L, SL, C, false>(v, t, a);
      reg_butterfly<L, SL, false>(v);
      float4* q = reinterpret_cast<float4*>(tile) + SPlan<L, SL>::row(a, 0) * C + u;
#pragma unroll
      for (int r = 0; r < 8; ++r) q[r * C] = unit_out(v[0][r]);
    }
  }
  tma_tile_store<L, W, 1>(tile, map, x0, pz, smp);
}

// ---------------------------------------------------------------------------
// launchers (FP32)
// ---------------------------------------------------------------------------
// Lengths whose tiles move by tensor maps; 64 loads its rows straight into registers (small grids, where the wait of
// a tile behind the state word is what counts: 64^3, 34.9 against 37.9 us per iteration; at 128^3 the tensor maps give
// 139 against 152 us, at 512^3 the direct loads take 1.42 (x2) and 3.60 ms (x3) against 1.09 - 1.15 and 1.55 ms).
constexpr bool strided_tma(int L) { return L >= 128; }
// Width of the register pass nearest to the schedule's: 512 x 1..2, 256 x 1..4, 128 x 2..8, 64 x 4..16 modes.
__host__ constexpr int strided_reg_width(int L, int w) {
  const int lo = L == 64 ? 4 : L == 128 ? 2 : 1, hi = 1024 / L;
  return w < lo ? lo : w > hi ? hi : w;
}
// Tensor map over a spectrum as (x1 modes x 12 floats, x2, x3, sample) with boxes of W modes x `rows` rows along axis
// ax (1: x2, 2: x3).  The encoder is a driver entry point, looked up once.
inline cudaError_t spectrum_map(CUtensorMap* m, const IterArgs<float>& a, const float2* spec, int W, int rows, int ax) {
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode enc = []() -> Encode {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return (Encode)f;
  }();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t row = (cuuint64_t)a.g.H * 48;
  const cuuint64_t dim[4] = {(cuuint64_t)a.g.H * 12, (cuuint64_t)a.g.n2, (cuuint64_t)a.g.n3, (cuuint64_t)(a.nsmp > 1 ? a.nsmp : 1)};
  const cuuint64_t stride[3] = {row, row * a.g.n2, row * a.g.n2 * a.g.n3};
  const cuuint32_t box[4] = {(cuuint32_t)W * 12, ax == 1 ? (cuuint32_t)rows : 1, ax == 2 ? (cuuint32_t)rows : 1, 1};
  const cuuint32_t one[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float2*>(spec), dim, stride, box, one,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

#define FFTLS_REG_CASES(F) F(64, 4) F(64, 8) F(64, 16)
#define FFTLS_TMA_CASES(F) F(128, 2) F(128, 4) F(128, 8) F(256, 1) F(256, 2) F(256, 4) F(512, 1) F(512, 2)

#ifdef FFTLS_Y_REG
cudaError_t launch_y_reg(const IterArgs<float>& a, bool inv, cudaStream_t s) {
  const int W = strided_reg_width(a.g.n2, a.y_w);
  const int kinds = (!inv && a.dual && !a.eta_real) ? 2 : 1;
  const dim3 grid((a.g.H + W - 1) / W, a.g.n3, kinds * (a.nsmp > 1 ? a.nsmp : 1));
  if (strided_tma(a.g.n2)) {
    IterArgs<float> b = a;
    cudaError_t e = spectrum_map(&b.tm[0], a, a.specA, W, a.g.n2 < 256 ? a.g.n2 : 256, 1);
    if (e == cudaSuccess && kinds > 1) e = spectrum_map(&b.tm[1], a, a.specB, W, a.g.n2 < 256 ? a.g.n2 : 256, 1);
    if (e != cudaSuccess) return e;
#define F(LV, WV)                                                                                                  \
  if (a.g.n2 == LV && W == WV)                                                                                     \
    (inv ? k_y_tma<LV, WV, true> : k_y_tma<LV, WV, false>)<<<grid, strided_reg_threads_y(LV, WV) / 2,              \
                                                             strided_tma_smem<LV, WV>(), s>>>(b, kinds);
    FFTLS_TMA_CASES(F)
#undef F
    return cudaGetLastError();
  }
#define F(LV, WV)                                                                                                  \
  if (a.g.n2 == LV && W == WV)                                                                                     \
    (inv ? k_y_reg<LV, WV, true> : k_y_reg<LV, WV, false>)<<<grid, strided_reg_threads_y(LV, WV),                  \
                                                             strided_reg_smem(LV, WV), s>>>(a, kinds);
  FFTLS_REG_CASES(F)
#undef F
  return cudaGetLastError();
}
cudaError_t set_attrs_y_reg() {
  cudaError_t e = cudaSuccess;
#define F(LV, WV)                                                                                                  \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_y_tma<LV, WV, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                             (int)strided_tma_smem<LV, WV>());                                                     \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_y_tma<LV, WV, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                             (int)strided_tma_smem<LV, WV>());
  FFTLS_TMA_CASES(F)
#undef F
#define F(LV, WV)                                                                                                  \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_y_reg<LV, WV, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                             (int)strided_reg_smem(LV, WV));                                                       \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_y_reg<LV, WV, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                             (int)strided_reg_smem(LV, WV));
  FFTLS_REG_CASES(F)
#undef F
  return e;
}
#endif

#ifdef FFTLS_Z_REG
cudaError_t launch_z_reg(const IterArgs<float>& a, cudaStream_t s) {
  const int W = strided_reg_width(a.g.n3, a.z_w);
  const dim3 grid((a.g.H + W - 1) / W, a.g.n2, a.nsmp > 1 ? a.nsmp : 1);
  const bool will = a.green == kWillot;
  if (strided_tma(a.g.n3)) {
    IterArgs<float> b = a;
    const cudaError_t e = spectrum_map(&b.tm[2], a, a.specA, W, a.g.n3 < 256 ? a.g.n3 : 256, 2);
    if (e != cudaSuccess) return e;
#define F(LV, WV)                                                                                                  \
  if (a.g.n3 == LV && W == WV)                                                                                     \
    (will ? k_z_tma<LV, WV, true> : k_z_tma<LV, WV, false>)<<<grid, strided_reg_threads_z(LV, WV),                 \
                                                              strided_tma_smem<LV, WV>(), s>>>(b);
    FFTLS_TMA_CASES(F)
#undef F
    return cudaGetLastError();
  }
#define F(LV, WV)                                                                                                  \
  if (a.g.n3 == LV && W == WV)                                                                                     \
    (will ? k_z_reg<LV, WV, true> : k_z_reg<LV, WV, false>)<<<grid, strided_reg_threads_z(LV, WV),                 \
                                                              strided_reg_smem(LV, WV), s>>>(a);
  FFTLS_REG_CASES(F)
#undef F
  return cudaGetLastError();
}
cudaError_t set_attrs_z_reg() {
  cudaError_t e = cudaSuccess;
#define F(LV, WV)                                                                                                  \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_z_tma<LV, WV, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                             (int)strided_tma_smem<LV, WV>());                                                     \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_z_tma<LV, WV, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                             (int)strided_tma_smem<LV, WV>());
  FFTLS_TMA_CASES(F)
#undef F
#define F(LV, WV)                                                                                                  \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_z_reg<LV, WV, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                             (int)strided_reg_smem(LV, WV));                                                       \
  if (e == cudaSuccess)                                                                                            \
    e = cudaFuncSetAttribute((const void*)k_z_reg<LV, WV, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                             (int)strided_reg_smem(LV, WV));
  FFTLS_REG_CASES(F)
#undef F
  return e;
}
#endif

}  // namespace fftls
