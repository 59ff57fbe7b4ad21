// FP64 pieces of the Wiener filters and the mass mapping: 2D transforms in FP64 with the pointwise work fused into
// them, for the refinement residual r = A N^-1 (d - A s) - S^-1 s of an FP32 iterate s and its norm ||S r||, the
// application of S = U^dagger diag(P) U, the shear residual and the convergence of a shear field.
//
// The Wiener-filter equation (S^-1 + A N^-1 A) s = A N^-1 d (Eq. 2-3 with a diagonal response A, N^-1 = 0 on missing
// pixels) gives (I + S A N^-1 A) s - S A N^-1 d = -S r, so ||S r|| / ||S A N^-1 d|| is the relative residual used
// everywhere else in the library, here evaluated in FP64.
//
// Complex fields (one real field, or the two components of a shear field, which share their unit) take three kernels:
//   k_rows_fwd   forms z from the caller's arrays and transforms whole rows in shared memory;
//   k_cols       transforms four whole columns in shared memory, then the pointwise step (a norm, or a new spectrum
//                followed by the inverse transform);
//   k_rows_inv   transforms the rows back and forms the caller's outputs.
// The refinement residual has two real fields of different units, the iterate s and N^-1 (d - s), which goes with
// 1 / s: in one complex field the rounding errors of the larger would fall on the smaller. So only their row transforms
// share a complex one, with the second field scaled by a power of two to the first (exact, chosen by each CTA
// from its own rows); k_rows_residual separates the two there and leaves the half spectra (kx <= N/2), and the columns of
// each are transforms of their own: as many columns in all as the packed form has. k_cols_residual forms the norm, k_cols_divp
// and k_rows_half the correction's S^-1 s. Every error is then relative to its own field, in any unit of the data. Against
// both fields packed through the columns too, device us at 1024^2: a residual 217 -> 204, a correction's right-hand side (the
// columns of s alone) 303 -> 208; at 64^2, launch-bound, 21.6 -> 21.5 and 27.2 -> 26.0.
// A norm is two launches and an application of an operator three. The transforms are radix-4 Stockham passes
// (self-sorting; Govindaraju et al., "High performance discrete Fourier transforms on graphics processors", SC'08)
// with the twiddles from a table. Bound: the FP64 rate of this GPU (two lanes per SM and clock) at 512^2 and above, the
// launches below. Against one launch per radix-2 stage (44 launches of a 64^2 residual, each twiddle a sine and cosine in
// FP64, every real field its own complex transform): a refined 64^2 filter 2.00 -> 1.01 ms, the likelihood gradient at
// 256^2 9.5 -> 7.6 ms, the residuals and convergence of a 256^2 shear filter 2.1 -> about 0.2 ms of 20 ms.
#include <cuda_runtime.h>

#include "wf_math.cuh"
#include "wf_refine.h"

namespace wf {

namespace {

// exp(-2 pi i j / 1024), made at compile time
struct Tw64 {
  double2 v[1024];
};
constexpr Tw64 make_tw64() {
  Tw64 t{};
  for (int j = 0; j < 1024; ++j) {
    t.v[j].x = cos2pi(j, 1024);
    t.v[j].y = -sin2pi(j, 1024);
  }
  return t;
}
__device__ const Tw64 g_tw64 = make_tw64();

__device__ __forceinline__ double2 dadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 dsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 dmul(double2 a, double2 w) {
  return make_double2(fma(a.x, w.x, -a.y * w.y), fma(a.x, w.y, a.y * w.x));
}
__device__ __forceinline__ double2 dconj(double2 a) { return make_double2(a.x, -a.y); }

// twiddle exp(-+2 pi i m / n), n a power of two up to 1024
template <bool INV>
__device__ __forceinline__ double2 dtw(int m, int n) {
  const double2 w = __ldg(g_tw64.v + m * (1024 / n));
  return INV ? dconj(w) : w;
}

// One Stockham pass of radix R (4 or 2) from sub-transforms of length Ns to R Ns, on NV vectors of length N at
// buf + v N, by T threads: all inputs into registers, a barrier, all outputs, a barrier.
template <int N, int NV, int T, int R, int Ns, bool INV>
__device__ __forceinline__ void dpass(double2* buf) {
  constexpr int PER = N / R, ITER = NV * PER / T;
  static_assert(ITER >= 1 && ITER * T == NV * PER, "whole butterflies per thread");
  double2 x[ITER][R];
#pragma unroll
  for (int i = 0; i < ITER; ++i) {
    const int id = threadIdx.x + i * T, v = id / PER, j = id % PER, k = j % Ns;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      x[i][r] = buf[v * N + j + r * PER];
      if (Ns > 1 && r > 0) x[i][r] = dmul(x[i][r], dtw<INV>(r * k, R * Ns));
    }
    if constexpr (R == 2) {
      const double2 a = x[i][0], b = x[i][1];
      x[i][0] = dadd(a, b);
      x[i][1] = dsub(a, b);
    } else {
      const double2 s02 = dadd(x[i][0], x[i][2]), d02 = dsub(x[i][0], x[i][2]);
      const double2 s13 = dadd(x[i][1], x[i][3]), d13 = dsub(x[i][1], x[i][3]);
      // -+i d13
      const double2 e = INV ? make_double2(-d13.y, d13.x) : make_double2(d13.y, -d13.x);
      x[i][0] = dadd(s02, s13);
      x[i][1] = dadd(d02, e);
      x[i][2] = dsub(s02, s13);
      x[i][3] = dsub(d02, e);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < ITER; ++i) {
    const int id = threadIdx.x + i * T, v = id / PER, j = id % PER, k = j % Ns;
#pragma unroll
    for (int r = 0; r < R; ++r) buf[v * N + (j / Ns) * Ns * R + k + r * Ns] = x[i][r];
  }
  __syncthreads();
}
template <int N, int NV, int T, int Ns, bool INV>
__device__ __forceinline__ void dpasses(double2* buf) {
  if constexpr (Ns < N) {
    dpass<N, NV, T, 4, Ns, INV>(buf);
    dpasses<N, NV, T, 4 * Ns, INV>(buf);
  }
}
// unnormalised transforms of NV vectors of length N, natural order in and out (CTA barrier at the end)
template <int N, int NV, int T, bool INV>
__device__ __forceinline__ void dfft(double2* buf) {
  if constexpr (ilog2(N) % 2 == 1) {
    dpass<N, NV, T, 2, 1, INV>(buf);
    dpasses<N, NV, T, 2, INV>(buf);
  } else {
    dpasses<N, NV, T, 1, INV>(buf);
  }
}

__device__ __forceinline__ double2* dsmem() {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  return reinterpret_cast<double2*>(smem_raw);
}

// adds the sum of the T threads' values to *out: shuffles, then the warps' sums through shared memory (the CTA's
// buffer, free by now), one atomic per CTA
template <int T>
__device__ __forceinline__ void dadd_block(double v, double* out) {
  constexpr int W = T < 32 ? T : 32;
  constexpr unsigned mask = W == 32 ? 0xffffffffu : (1u << W) - 1u;
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  if constexpr (T > 32) {
    double* red = reinterpret_cast<double*>(dsmem());
    __syncthreads();
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = v;
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
      for (int w = 1; w < T / 32; ++w) v += red[w];
  }
  if (threadIdx.x == 0) atomicAdd(out, v);
}

template <int N>
struct DGeo {
  static constexpr int RB = N >= 512 ? 1 : (N == 16 ? 16 : 512 / N);  // rows per CTA
  static constexpr int TR = RB * N / 4;                               // threads of a row kernel
  static constexpr int TC = N < 256 ? N : 256;                        // threads of a column kernel
  static constexpr int NC = N / 4;                                    // column kernel: CTAs of four columns
};

// the four columns of CTA g: two columns and their mirrors (mirror of entry c: entry mir(g, c)); CTA 0 holds the two
// self-mirrored columns 0 and N/2, and 1 with N - 1
template <int N>
__device__ __forceinline__ int dcol(int g, int c) {
  if (g == 0) return c == 0 ? 0 : (c == 1 ? N / 2 : (c == 2 ? 1 : N - 1));
  return c < 2 ? 2 * g + c : N - 2 * g - (c - 2);
}
__device__ __forceinline__ int dmir(int g, int c) { return g == 0 ? (c < 2 ? c : 5 - c) : (c + 2) % 4; }

// P on the full spectrum from the half table (P depends on |k|: (ky, kx) for kx > W/2 is (-ky, W - kx))
__device__ __forceinline__ double p_full(const float* __restrict__ Pk, int N, int ky, int kx) {
  const int WH = N / 2 + 1;
  return kx <= N / 2 ? double(Pk[ky * WH + kx]) : double(Pk[((N - ky) % N) * WH + (N - kx)]);
}

// rotation (c, s) of the Kaiser-Squires operator at full-spectrum mode (ky, kx), as in the samplers
__device__ __forceinline__ double2 ks_rot_d(int N, int ky, int kx) {
  const int y = ky < N / 2 ? ky : ky - N, x = kx < N / 2 ? kx : kx - N;
  if ((x == 0 && y == 0) || ky == N / 2 || kx == N / 2) return make_double2(1.0, 0.0);
  const double k1 = x, k2 = y, r = 1.0 / (k1 * k1 + k2 * k2);
  return make_double2((k1 * k1 - k2 * k2) * r, 2.0 * k1 * k2 * r);
}

// ---- sources z(field, pixel) of the forward rows ----
struct SrcResidual {  // s, and rpix = A N^-1 (d - A s) on observed pixels with A != 0 (A = 1 when null)
  const float *d, *Nd, *A, *s;
  const uint8_t* mask;
  __device__ __forceinline__ double rpix(int i) const {
    const double a = A ? double(A[i]) : 1.0;
    return (mask[i] || a == 0.0) ? 0.0 : a * (double(d[i]) - a * double(s[i])) / double(Nd[i]);
  }
};
struct SrcRhs {  // A N^-1 d on observed pixels with A != 0
  const float *d, *Nd, *A;
  const uint8_t* mask;
  __device__ __forceinline__ double2 operator()(int, int i) const {
    const double a = A ? double(A[i]) : 1.0;
    return make_double2((mask[i] || a == 0.0) ? 0.0 : a * double(d[i]) / double(Nd[i]), 0.0);
  }
};
struct SrcReal {
  const float* v;
  __device__ __forceinline__ double2 operator()(int, int i) const { return make_double2(double(v[i]), 0.0); }
};
struct SrcPairs {  // fields f of [n][2][H][W]: component 1 + i component 2
  const float* g;
  long long n;
  __device__ __forceinline__ double2 operator()(int f, int i) const {
    return make_double2(double(g[2 * f * n + i]), double(g[(2 * f + 1) * n + i]));
  }
};
struct SrcShear {  // field 0: g1 + i g2 (0 for the right-hand side); field 1: N^-1 (g - d) (rhs: N^-1 d), likewise
  const float *g, *d1, *d2, *N1, *N2;
  const uint8_t* mask;
  long long n;
  int rhs;
  __device__ __forceinline__ double2 operator()(int f, int i) const {
    const double a = rhs ? 0.0 : double(g[i]), b = rhs ? 0.0 : double(g[n + i]);
    if (f == 0) return make_double2(a, b);
    if (mask[i] != 0) return make_double2(0.0, 0.0);
    return make_double2((rhs ? double(d1[i]) : a - double(d1[i])) / double(N1[i]),
                        (rhs ? double(d2[i]) : b - double(d2[i])) / double(N2[i]));
  }
};

// rows of field blockIdx.y of z, transformed, to Z; zero (optional): a sum set to 0 for the next kernel
template <int N, class Src>
__global__ void __launch_bounds__(DGeo<N>::TR) k_rows_fwd(Src src, double2* Z, double* zero) {
  using G = DGeo<N>;
  double2* buf = dsmem();
  const int f = blockIdx.y, base = int(blockIdx.x) * G::RB * N;
  if (zero && blockIdx.x == 0 && threadIdx.x == 0) *zero = 0.0;
  for (int e = threadIdx.x; e < G::RB * N; e += G::TR) buf[e] = src(f, base + e);
  __syncthreads();
  dfft<N, G::RB, G::TR, false>(buf);
  double2* z = Z + (long long)f * N * N + base;
  for (int e = threadIdx.x; e < G::RB * N; e += G::TR) z[e] = buf[e];
}

// ---- pointwise steps of the columns: op.norm or op.map(ky, kx, Z(k)) ----
struct OpPNorm {  // P^2 |z|^2 / n
  static constexpr bool kNorm = true;
  const float* Pk;
  template <int N>
  __device__ __forceinline__ double norm(int ky, int kx, double2 z) const {
    const double p = p_full(Pk, N, ky, kx);
    return p * p * (z.x * z.x + z.y * z.y) * (1.0 / (double(N) * N));
  }
};
struct OpMulP {  // P z / n
  static constexpr bool kNorm = false;
  const float* Pk;
  template <int N>
  __device__ __forceinline__ double2 map(int ky, int kx, double2 z) const {
    const double p = p_full(Pk, N, ky, kx) * (1.0 / (double(N) * N));
    return make_double2(z.x * p, z.y * p);
  }
};
struct OpKsInverse {  // E_hat + i B_hat = (c - i s)(g1_hat + i g2_hat), over n
  static constexpr bool kNorm = false;
  template <int N>
  __device__ __forceinline__ double2 map(int ky, int kx, double2 z) const {
    const double2 r = ks_rot_d(N, ky, kx);
    const double2 o = dmul(z, dconj(r));
    return make_double2(o.x * (1.0 / (double(N) * N)), o.y * (1.0 / (double(N) * N)));
  }
};

// columns 4 g .. 4 g + 3 (g = blockIdx.x) of field blockIdx.y: transform, then the sum of op's norms added to *out, or op's
// new spectrum transformed back in place
template <int N, class Op>
__global__ void __launch_bounds__(DGeo<N>::TC) k_cols(Op op, double2* Z, double* out) {
  using G = DGeo<N>;
  double2* buf = dsmem();
  const int g = blockIdx.x;
  double2* z = Z + (long long)blockIdx.y * N * N;
  for (int e = threadIdx.x; e < 4 * N; e += G::TC) {
    const int c = e % 4, y = e / 4;
    buf[c * N + y] = z[(long long)y * N + 4 * g + c];
  }
  __syncthreads();
  dfft<N, 4, G::TC, false>(buf);
  constexpr int ITER = 4 * N / G::TC;
  if constexpr (Op::kNorm) {
    double acc = 0.0;
#pragma unroll 4
    for (int i = 0; i < ITER; ++i) {
      const int e = threadIdx.x + i * G::TC, c = e / N, ky = e % N;
      acc += op.template norm<N>(ky, 4 * g + c, buf[e]);
    }
    dadd_block<G::TC>(acc, out);
  } else {
    double2 v[ITER];
#pragma unroll
    for (int i = 0; i < ITER; ++i) {
      const int e = threadIdx.x + i * G::TC, c = e / N, ky = e % N;
      v[i] = op.template map<N>(ky, 4 * g + c, buf[e]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITER; ++i) buf[threadIdx.x + i * G::TC] = v[i];
    __syncthreads();
    dfft<N, 4, G::TC, true>(buf);
    for (int e = threadIdx.x; e < 4 * N; e += G::TC) {
      const int c = e % 4, y = e / 4;
      z[(long long)y * N + 4 * g + c] = buf[c * N + y];
    }
  }
}

// Rows of s and of rpix: one complex transform a row, s + i beta rpix with beta a power of two that brings the CTA's
// largest rpix to its largest s, separated into the half spectra Z[0][y][kx] and Z[1][y][kx], kx <= N/2; *zero = 0.
template <int N>
__global__ void __launch_bounds__(DGeo<N>::TR) k_rows_residual(SrcResidual src, double2* Z, double* zero) {
  using G = DGeo<N>;
  constexpr int E = G::RB * N / G::TR, WH = N / 2 + 1, NW = G::TR / 32;
  static_assert(G::TR % 32 == 0, "whole warps");
  __shared__ int top[2][NW];
  double2* buf = dsmem();
  const int base = int(blockIdx.x) * G::RB * N;
  if (zero && blockIdx.x == 0 && threadIdx.x == 0) *zero = 0.0;
  double2 x[E];
  int hs = 0, hr = 0;  // high words of the largest magnitudes
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int at = base + int(threadIdx.x) + i * G::TR;
    x[i] = make_double2(double(src.s[at]), src.rpix(at));
    hs = max(hs, __double2hiint(x[i].x) & 0x7fffffff);
    hr = max(hr, __double2hiint(x[i].y) & 0x7fffffff);
  }
  hs = __reduce_max_sync(0xffffffffu, hs);
  hr = __reduce_max_sync(0xffffffffu, hr);
  if (threadIdx.x % 32 == 0) {
    top[0][threadIdx.x / 32] = hs;
    top[1][threadIdx.x / 32] = hr;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    hs = max(hs, top[0][w]);
    hr = max(hr, top[1][w]);
  }
  const int es = hs >> 20, er = hr >> 20;
  // unscaled if a field is zero or not finite; FP32 inputs keep the difference far below 1000
  int sh = es == 0 || er == 0 || es == 2047 || er == 2047 ? 0 : es - er;
  sh = sh > 1000 ? 1000 : (sh < -1000 ? -1000 : sh);
  const double beta = __hiloint2double((1023 + sh) << 20, 0), half_ib = 0.5 * __hiloint2double((1023 - sh) << 20, 0);
#pragma unroll
  for (int i = 0; i < E; ++i) buf[threadIdx.x + i * G::TR] = make_double2(x[i].x, beta * x[i].y);
  __syncthreads();
  dfft<N, G::RB, G::TR, false>(buf);
  for (int e = threadIdx.x; e < G::RB * WH; e += G::TR) {
    const int v = e / WH, kx = e % WH;
    const double2 a = buf[v * N + kx], b = dconj(buf[v * N + (N - kx) % N]);
    const double2 d = dsub(a, b);  // 2 i beta rpix_hat
    const long long at = ((long long)blockIdx.x * G::RB + v) * WH + kx;
    Z[at] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y + b.y));
    Z[(long long)N * WH + at] = make_double2(half_ib * d.y, -half_ib * d.x);
  }
}

// *out += ||S r||^2: columns kx = 2 g and 2 g + 1 (up to N/2) of both half spectra of k_rows_residual, transformed, then
// |P rpix_hat - s_hat|^2 / n where P > 0, else |s_hat|^2 / n, twice for the columns whose mirror is left out
template <int N>
__global__ void __launch_bounds__(DGeo<N>::TC) k_cols_residual(const float* __restrict__ Pk, const double2* __restrict__ Z,
                                                               double* out) {
  using G = DGeo<N>;
  constexpr int WH = N / 2 + 1;
  double2* buf = dsmem();
  const int k0 = 2 * int(blockIdx.x);
  for (int e = threadIdx.x; e < 4 * N; e += G::TC) {
    const int c = e % 4, y = e / 4, kx = k0 + c % 2;
    buf[c * N + y] = kx <= N / 2 ? __ldg(Z + ((long long)(c / 2) * N + y) * WH + kx) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  dfft<N, 4, G::TC, false>(buf);
  double acc = 0.0;
#pragma unroll 4
  for (int i = 0; i < 2 * N / G::TC; ++i) {
    const int e = threadIdx.x + i * G::TC, kx = k0 + e / N, ky = e % N;
    if (kx > N / 2) continue;
    const double p = double(Pk[ky * WH + kx]);
    const double2 s = buf[e], r = buf[2 * N + e];
    const double2 v = p > 0.0 ? make_double2(p * r.x - s.x, p * r.y - s.y) : s;
    acc += (v.x * v.x + v.y * v.y) * ((kx == 0 || kx == N / 2 ? 1.0 : 2.0) / (double(N) * N));
  }
  dadd_block<G::TC>(acc, out);
}

// q_hat = s_hat / (n P) where P > 0, else 0: columns kx = 4 g .. 4 g + 3 (up to N/2) of the half spectrum of s, transformed,
// divided and transformed back in place
template <int N>
__global__ void __launch_bounds__(DGeo<N>::TC) k_cols_divp(const float* __restrict__ Pk, double2* Z) {
  using G = DGeo<N>;
  constexpr int WH = N / 2 + 1;
  double2* buf = dsmem();
  const int k0 = 4 * int(blockIdx.x);
  for (int e = threadIdx.x; e < 4 * N; e += G::TC) {
    const int c = e % 4, y = e / 4;
    buf[c * N + y] = k0 + c <= N / 2 ? Z[(long long)y * WH + k0 + c] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  dfft<N, 4, G::TC, false>(buf);
#pragma unroll 4
  for (int i = 0; i < 4 * N / G::TC; ++i) {
    const int e = threadIdx.x + i * G::TC, kx = k0 + e / N;
    const double p = kx <= N / 2 ? double(Pk[(e % N) * WH + kx]) : 0.0;
    const double q = p > 0.0 ? 1.0 / (double(N) * N * p) : 0.0;
    buf[e] = p > 0.0 ? make_double2(q * buf[e].x, q * buf[e].y) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  dfft<N, 4, G::TC, true>(buf);
  for (int e = threadIdx.x; e < 4 * N; e += G::TC) {
    const int c = e % 4, y = e / 4;
    if (k0 + c <= N / 2) Z[(long long)y * WH + k0 + c] = buf[c * N + y];
  }
}

// *out += sum_k |G_k + S V_k|^2 / n of the shear residual: G in field 0, V in field 1 of Z, both as component 1 +
// i component 2; S V = rotate(P_E e, P_B b) with e + i b = (c - i s) V, e and b real fields
template <int N>
__global__ void __launch_bounds__(DGeo<N>::TC) k_cols_shear(const float* __restrict__ PE, const float* __restrict__ PB,
                                                            const double2* __restrict__ Z, double* out) {
  using G = DGeo<N>;
  double2* buf = dsmem();
  const int g = blockIdx.x;
  for (int e = threadIdx.x; e < 8 * N; e += G::TC) {
    const int c = e % 4, y = (e / 4) % N, f = e / (4 * N);
    buf[(4 * f + c) * N + y] = __ldg(Z + ((long long)f * N + y) * N + dcol<N>(g, c));
  }
  __syncthreads();
  dfft<N, 8, G::TC, false>(buf);
  const double2* V = buf + 4 * N;
  double acc = 0.0;
#pragma unroll 2
  for (int e = threadIdx.x; e < 4 * N; e += G::TC) {
    const int c = e / N, ky = e % N, kx = dcol<N>(g, c);
    const double2 r = ks_rot_d(N, ky, kx);
    const double2 w = dmul(V[e], dconj(r));
    const double2 m = dconj(dmul(V[dmir(g, c) * N + (N - ky) % N], dconj(r)));  // the rotation is even in k
    const double pe = 0.5 * p_full(PE, N, ky, kx), pb = 0.5 * p_full(PB, N, ky, kx);
    const double2 sv = dmul(make_double2(pe * (w.x + m.x) + pb * (w.x - m.x), pe * (w.y + m.y) + pb * (w.y - m.y)), r);
    const double2 t = dadd(buf[e], sv);
    acc += (t.x * t.x + t.y * t.y) * (1.0 / (double(N) * N));
  }
  dadd_block<G::TC>(acc, out);
}

// ---- destinations dst(field, y, x, z) of the inverse rows ----
template <int N>
struct DstCorrection {  // r = rpix - Re z; (float(r), 1/N_bar) in dn's order (x-major, or row-major with row_major)
  SrcResidual src;
  const float2* dn;
  float2* rtab;
  int row_major;
  __device__ __forceinline__ void operator()(int, int i, double2 z) const {
    const int at = row_major ? i : (i % N) * N + i / N;
    rtab[at] = make_float2(float(src.rpix(i) - z.x), dn[at].y);
  }
};
struct DstReal {
  float* v;
  __device__ __forceinline__ void operator()(int, int i, double2 z) const { v[i] = float(z.x); }
};
struct DstPairs {
  float* k;
  long long n;
  __device__ __forceinline__ void operator()(int f, int i, double2 z) const {
    k[2 * f * n + i] = float(z.x);
    k[(2 * f + 1) * n + i] = float(z.y);
  }
};

template <int N, class Dst>
__global__ void __launch_bounds__(DGeo<N>::TR) k_rows_inv(const double2* __restrict__ Z, Dst dst) {
  using G = DGeo<N>;
  double2* buf = dsmem();
  const int f = blockIdx.y, base = int(blockIdx.x) * G::RB * N;
  const double2* z = Z + (long long)f * N * N + base;
  for (int e = threadIdx.x; e < G::RB * N; e += G::TR) buf[e] = z[e];
  __syncthreads();
  dfft<N, G::RB, G::TR, true>(buf);
  for (int e = threadIdx.x; e < G::RB * N; e += G::TR) dst(f, base + e, buf[e]);
}

// rows of a real field from its half spectrum
template <int N, class Dst>
__global__ void __launch_bounds__(DGeo<N>::TR) k_rows_half(const double2* __restrict__ Z, Dst dst) {
  using G = DGeo<N>;
  constexpr int WH = N / 2 + 1;
  double2* buf = dsmem();
  for (int e = threadIdx.x; e < G::RB * WH; e += G::TR) {
    const int v = e / WH, kx = e % WH;
    const double2 z = __ldg(Z + ((long long)blockIdx.x * G::RB + v) * WH + kx);
    buf[v * N + kx] = z;
    if (kx != 0 && kx != N / 2) buf[v * N + N - kx] = dconj(z);
  }
  __syncthreads();
  dfft<N, G::RB, G::TR, true>(buf);
  const int base = int(blockIdx.x) * G::RB * N;
  for (int e = threadIdx.x; e < G::RB * N; e += G::TR) dst(0, base + e, buf[e]);
}

__global__ void k_add_f32(int n, float* s, const float* __restrict__ e) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) s[i] += e[i];
}

int grid_for(long long n) {
  const long long g = (n + 255) / 256;
  return int(g < 2048 ? (g < 1 ? 1 : g) : 2048);
}

template <class Kern>
cudaError_t smem_attr(Kern kern, int bytes) {
  return bytes > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)
                           : cudaSuccess;
}
template <int N, class Src>
cudaError_t rows_fwd(const Src& src, double2* Z, int fields, double* zero, cudaStream_t st) {
  using G = DGeo<N>;
  k_rows_fwd<N, Src><<<dim3(N / G::RB, fields), G::TR, G::RB * N * 16, st>>>(src, Z, zero);
  return cudaGetLastError();
}
template <int N, class Op>
cudaError_t cols(const Op& op, double2* Z, int fields, double* out, cudaStream_t st) {
  using G = DGeo<N>;
  const cudaError_t e = smem_attr(k_cols<N, Op>, 4 * N * 16);
  if (e != cudaSuccess) return e;
  k_cols<N, Op><<<dim3(G::NC, fields), G::TC, 4 * N * 16, st>>>(op, Z, out);
  return cudaGetLastError();
}
template <int N, class Dst>
cudaError_t rows_inv(const double2* Z, const Dst& dst, int fields, cudaStream_t st) {
  using G = DGeo<N>;
  k_rows_inv<N, Dst><<<dim3(N / G::RB, fields), G::TR, G::RB * N * 16, st>>>(Z, dst);
  return cudaGetLastError();
}

// f(integral constant of the size)
template <class F>
cudaError_t by_size(int N, F&& f) {
  switch (N) {
    case 16: return f(std::integral_constant<int, 16>{});
    case 32: return f(std::integral_constant<int, 32>{});
    case 64: return f(std::integral_constant<int, 64>{});
    case 128: return f(std::integral_constant<int, 128>{});
    case 256: return f(std::integral_constant<int, 256>{});
    case 512: return f(std::integral_constant<int, 512>{});
    case 1024: return f(std::integral_constant<int, 1024>{});
  }
  return cudaErrorInvalidValue;
}

}  // namespace

size_t refine_scratch_bytes(int H, int W) { return size_t(2) * H * (W / 2 + 1) * sizeof(double2); }

cudaError_t refine_bnorm(const RefineArgs& a, cudaStream_t st) {
  auto* Z = static_cast<double2*>(a.scratch);
  return by_size(a.H, [&](auto S) {
    constexpr int N = decltype(S)::value;
    const cudaError_t e = rows_fwd<N>(SrcRhs{a.d, a.Nd, a.A, a.mask}, Z, 1, a.bnorm, st);
    return e != cudaSuccess ? e : cols<N>(OpPNorm{a.Pk}, Z, 1, a.bnorm, st);
  });
}

cudaError_t refine_residual(const RefineArgs& a, cudaStream_t st) {
  auto* Z = static_cast<double2*>(a.scratch);
  return by_size(a.H, [&](auto S) {
    constexpr int N = decltype(S)::value;
    using G = DGeo<N>;
    cudaError_t e = smem_attr(k_cols_residual<N>, 4 * N * 16);
    if (e != cudaSuccess) return e;
    k_rows_residual<N><<<N / G::RB, G::TR, G::RB * N * 16, st>>>(SrcResidual{a.d, a.Nd, a.A, a.s, a.mask}, Z, a.rnorm);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_cols_residual<N><<<N / 4 + 1, G::TC, 4 * N * 16, st>>>(a.Pk, Z, a.rnorm);
    return cudaGetLastError();
  });
}

cudaError_t refine_correction(const RefineArgs& a, cudaStream_t st) {
  auto* Z = static_cast<double2*>(a.scratch);
  return by_size(a.H, [&](auto S) {
    constexpr int N = decltype(S)::value;
    using G = DGeo<N>;
    cudaError_t e = smem_attr(k_cols_divp<N>, 4 * N * 16);
    if (e != cudaSuccess) return e;
    k_cols_divp<N><<<N / 8 + 1, G::TC, 4 * N * 16, st>>>(a.Pk, Z);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_rows_half<N><<<N / G::RB, G::TR, G::RB * N * 16, st>>>(
        Z, DstCorrection<N>{SrcResidual{a.d, a.Nd, a.A, a.s, a.mask}, a.dn, a.rtab, a.row_major});
    return cudaGetLastError();
  });
}

cudaError_t apply_S_f64(const float* v, const float* Pk, int H, int, float* out, void* scratch, cudaStream_t st) {
  auto* Z = static_cast<double2*>(scratch);
  return by_size(H, [&](auto S) {
    constexpr int N = decltype(S)::value;
    cudaError_t e = rows_fwd<N>(SrcReal{v}, Z, 1, nullptr, st);
    if (e == cudaSuccess) e = cols<N>(OpMulP{Pk}, Z, 1, nullptr, st);
    return e != cudaSuccess ? e : rows_inv<N>(Z, DstReal{out}, 1, st);
  });
}

cudaError_t shear_to_convergence_f64(const float* gamma, int fields, int H, int, float* kappa, void* scratch,
                                     cudaStream_t st) {
  auto* Z = static_cast<double2*>(scratch);
  return by_size(H, [&](auto S) {
    constexpr int N = decltype(S)::value;
    constexpr long long n = (long long)N * N;
    cudaError_t e = rows_fwd<N>(SrcPairs{gamma, n}, Z, fields, nullptr, st);
    if (e == cudaSuccess) e = cols<N>(OpKsInverse{}, Z, fields, nullptr, st);
    return e != cudaSuccess ? e : rows_inv<N>(Z, DstPairs{kappa, n}, fields, st);
  });
}

cudaError_t spin2_residual_f64(const float* g, const float* d1, const float* d2, const float* N1, const float* N2,
                               const uint8_t* mask, const float* PE, const float* PB, int H, int, bool with_b,
                               double* out, void* scratch, cudaStream_t st) {
  auto* Z = static_cast<double2*>(scratch);
  return by_size(H, [&](auto S) {
    constexpr int N = decltype(S)::value;
    cudaError_t e = cudaErrorInvalidValue;
    if constexpr (N <= 512) {
      e = smem_attr(k_cols_shear<N>, 8 * N * 16);
      // pass 0: the residual of g; pass 1: the right-hand side S N^-1 d
      for (int rhs = 0; rhs < (with_b ? 2 : 1) && e == cudaSuccess; ++rhs) {
        e = rows_fwd<N>(SrcShear{g, d1, d2, N1, N2, mask, (long long)N * N, rhs}, Z, 2, out + rhs, st);
        if (e != cudaSuccess) break;
        k_cols_shear<N><<<DGeo<N>::NC, DGeo<N>::TC, 8 * N * 16, st>>>(PE, PB, Z, out + rhs);
        e = cudaGetLastError();
      }
    }
    return e;
  });
}

cudaError_t refine_update(int n, float* s, const float* e, cudaStream_t st) {
  k_add_f32<<<grid_for(n), 256, 0, st>>>(n, s, e);
  return cudaGetLastError();
}

}  // namespace wf
