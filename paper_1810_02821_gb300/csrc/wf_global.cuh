// Messenger-field sweeps of fields in global memory: images too large for one SM (N in {256, 512, 1024}), and
// few fields of 128^2 (spin-2, and where clusters cannot run), which one SM each would run with more latency.
//
// The packed half spectrum Z[H][W/2] of every field (kx = 0 and W/2 packed as re/im of column 0) lives in
// global memory (L2-resident when the working set allows). One persistent cooperative kernel runs every
// sweep as two phases separated by a bounded grid barrier:
//   row phase    (CTA = 8 rows of one field): Z rows -> C2R -> s -> [sample write] -> t-draw -> R2C -> Z
//   column phase (CTA = 4 columns of one field): Z columns -> FFT -> s-draw -> inverse FFT -> Z
// (Alg. 1 of the paper with A = I).
//
// Each transform of length n (rows W/2, columns H) is held by n/E threads of E = 2A elements (E = 8 up to 512,
// 16 at 1024: 8 there was 4% faster for one Wiener filter but 25% slower for several chains) and runs in three or four in-place passes, n = 8 R2 [R3] A (decimation in frequency, L1 = n/8):
//   pass 1: 8-point DFTs over m of x[n0 + L1 m], output q1, times W_n^(n0 q1);
//   middle: within each block of length Lb (L1 first), R-point DFTs over m of n1 + (Lb/R) m, output q2 (q3), times
//           W_Lb^(n1 q2);
//   last:   per unit q = q1 + 8 (q2 + R2 q3), the A-point DFT: X[q + (n/A) j].
// A thread owns the units q and n/A - q (0 and n/2A for the first), which hold every mode pair (k, -k), so the
// real-transform passes of a row and the s-draw of a column run on registers, and so does the t-draw between the
// inverse and the forward row transform: Z goes straight from global memory into the first pass's registers and
// back from the last pass's, and only the exchanges inside a transform use shared memory (blocks of L1 + 2 float2
// and the vector strides below leave the accesses free of conflicts). A row's threads share a warp, so its
// exchanges need no CTA barrier.
//
// What bounds it: one field is only N^2/16 (1024: N^2/32) threads, so a phase is the latency of an L2 round trip, two
// transforms whose instructions issue from one or two warps a scheduler, and a grid barrier, not bandwidth.
// Measured at one field (us per sampler sweep / Wiener sweep), against 128-thread items with 8- to 16-point register
// sub-transforms, draws through shared memory and a barrier with a generation word: 256^2 14.7 / 17.7 -> 6.8 / 7.3,
// 512^2 20.5 / 23.3 -> 8.8 / 9.1, 1024^2 27.8 / 33.0 -> 13.1 / 13.8; 31 fields of 256^2 42.4 -> 24.0, 4 of 1024^2
// 88 -> 34. Of a 256^2 sweep's 14K cycles a thread spends about 2.1K in each barrier and 2.5K on loads and stores of
// Z; with 16 elements a thread (half as many warps) the same sweep took 9.6 us.
#pragma once

#include "wf_gibbs.cuh"
#include "wf_units.cuh"

namespace wf {

// RB: rows per CTA
template <int N_, int RB_ = 8>
struct GGeo {
  static constexpr int N = N_, H = N_, W = N_;
  static constexpr int LR = W / 2;           // complex length of a row transform
  static constexpr int E = N_ == 1024 ? 16 : 8, A = E / 2;  // elements per thread, length of the unit transforms
  static constexpr int TR = LR / E, TC = H / E;    // threads per row and per column
  static constexpr int RB = RB_;
  static constexpr int T = RB * TR;                // threads per CTA
  static constexpr int CB = T / TC;                // columns per CTA (RB / 2)
  static constexpr int BR = LR / A, BC = H / A;    // frequency strides of the units
  // float2 strides of a row's and a column's vector: 8 blocks of L1 + 2; short rows TR, columns 4 or 2 modulo 16 apart (a half-warp
  // holds 4 or 8 columns)
  static constexpr int CW = CB < 8 ? CB : 8;
  static constexpr int VROW = LR + 16 + (TR < 8 ? TR : 8), VCOL = H + 16 + 16 / CW;
  static constexpr int VEC = RB * VROW > CB * VCOL ? RB * VROW : CB * VCOL;
  // twiddle tables: T1 [q1][n0] (rows of n/8 + 2), T2 and T3 [q][n1] of the rows and columns, W_W^K (K < LR/2)
  static constexpr int O_T1R = VEC, O_T2R = O_T1R + 8 * (LR / 8 + 2), O_T3R = O_T2R + LR / 8, O_T1C = O_T3R + 16,
                       O_T2C = O_T1C + 8 * (H / 8 + 2), O_T3C = O_T2C + H / 8, O_W = O_T3C + 16, O_EDGE = O_W + LR / 2,
                       SMEM_F2 = O_EDGE + H;
  static constexpr int SMEM = SMEM_F2 * 8;
  static constexpr int ROW_ITEMS = H / RB;  // row-phase work items per field
  static constexpr int COL_ITEMS = LR / CB; // column-phase work items per field
  static constexpr int WH = W / 2 + 1;
  // CTAs per SM the kernels are compiled for: up to 128 registers a thread with 16 elements, 80 with 8
  static constexpr int MIN_CTAS = (E == 16 ? 512 : 768) / T;
  static_assert((CB == 4 || CB % 8 == 0) && TR <= 32 && VCOL % 16 == 16 / CW, "geometry");
};

// middle radices of a transform of length n
template <int n, int E>
struct GRad {
  static constexpr int M = n / (4 * E);  // 1: no middle pass
  static constexpr int R2 = M <= E ? M : 4, R3 = M / R2;
  static constexpr int L1 = n / 8, S = L1 + 2, STEP2 = L1 / R2, STEP3 = STEP2 / R3;
  static_assert(R2 * R3 == M && STEP3 == E / 2 && (R3 == 1 || STEP2 == 16), "passes");
};

__device__ __forceinline__ float2* gsmem() {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  return reinterpret_cast<float2*>(smem_raw);
}

// the twiddle tables, by all threads (ends with a CTA barrier)
template <int N, int RB = 8>
__device__ __forceinline__ void gtab_init() {
  using G = GGeo<N, RB>;
  float2* s = gsmem();
  auto w = [](int j) { return g_tw1024.v[(j * (1024 / N)) & 1023]; };  // exp(-2 pi i j / N)
  for (int i = threadIdx.x; i < 8 * (G::LR / 8); i += G::T) {
    const int q = i / (G::LR / 8), n0 = i % (G::LR / 8);
    s[G::O_T1R + q * (G::LR / 8 + 2) + n0] = w(2 * n0 * q);
  }
  for (int i = threadIdx.x; i < 8 * (G::H / 8); i += G::T) {
    const int q = i / (G::H / 8), n0 = i % (G::H / 8);
    s[G::O_T1C + q * (G::H / 8 + 2) + n0] = w(n0 * q);
  }
  constexpr int SR = GRad<G::LR, G::E>::STEP2, SC = GRad<G::H, G::E>::STEP2;
  for (int i = threadIdx.x; i < G::LR / 8; i += G::T) s[G::O_T2R + i] = w(16 * (i / SR) * (i % SR));
  for (int i = threadIdx.x; i < G::H / 8; i += G::T) s[G::O_T2C + i] = w(8 * (i / SC) * (i % SC));
  for (int i = threadIdx.x; i < 16; i += G::T)  // blocks of length 16
    s[G::O_T3R + i] = s[G::O_T3C + i] = w(N / 16 * (i / 4) * (i % 4));
  for (int i = threadIdx.x; i < G::LR / 2; i += G::T) s[G::O_W + i] = w(i);
  __syncthreads();
}

// twiddle tables of the row (ROW) or column transforms
struct GTab {
  const float2 *t1, *t2, *t3;
};
template <int N, bool ROW, int RB = 8>
__device__ __forceinline__ GTab gtab() {
  using G = GGeo<N, RB>;
  const float2* s = gsmem();
  return ROW ? GTab{s + G::O_T1R, s + G::O_T2R, s + G::O_T3R} : GTab{s + G::O_T1C, s + G::O_T2C, s + G::O_T3C};
}

// position of unit q's first value in a vector of length n, and the unit's twiddles W_Lb^(n1 q2 or q3)
template <int n, int E>
__device__ __forceinline__ int gunit(int q) {
  using R = GRad<n, E>;
  const int r = q / 8;
  return (q % 8) * R::S + (R::R3 == 1 ? (E / 2) * r : R::STEP2 * (r % R::R2) + (E / 2) * (r / R::R2));
}
template <int n, int E>
__device__ __forceinline__ const float2* gunit_tw(int q, const GTab& t) {
  using R = GRad<n, E>;
  return R::R2 == 1 ? t.t1 + R::S * q : R::R3 == 1 ? t.t2 + (E / 2) * (q / 8) : t.t3 + (E / 2) * (q / 8 / R::R2);
}

// pass 1: x[i 8 + m] = element n0 + L1 m, n0 = (E/8) h + i
template <int n, int E>
__device__ __forceinline__ void gfwd1(float2* v, int h, const float2 (&x)[E], const GTab& t) {
  constexpr int S = GRad<n, E>::S, NC = E / 8;
  float2 a[NC][8];
#pragma unroll
  for (int i = 0; i < NC; ++i) {
#pragma unroll
    for (int m = 0; m < 8; ++m) a[i][m] = x[8 * i + m];
    fft<8, false>(a[i]);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if constexpr (NC == 2) {
      if (q > 0) {
        const float4 w = *reinterpret_cast<const float4*>(t.t1 + q * S + 2 * h);
        a[0][q] = cmul(a[0][q], make_float2(w.x, w.y));
        a[1][q] = cmul(a[1][q], make_float2(w.z, w.w));
      }
      *reinterpret_cast<float4*>(v + q * S + 2 * h) = make_float4(a[0][q].x, a[0][q].y, a[1][q].x, a[1][q].y);
    } else {
      v[q * S + h] = q == 0 ? a[0][0] : cmul(a[0][q], t.t1[q * S + h]);
    }
  }
}
template <int n, int E>
__device__ __forceinline__ void ginv1(const float2* v, int h, float2 (&x)[E]) {
  constexpr int S = GRad<n, E>::S, NC = E / 8;
  float2 a[NC][8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if constexpr (NC == 2) {
      const float4 w = *reinterpret_cast<const float4*>(v + q * S + 2 * h);
      a[0][q] = make_float2(w.x, w.y);
      a[1][q] = make_float2(w.z, w.w);
    } else {
      a[0][q] = v[q * S + h];
    }
  }
#pragma unroll
  for (int i = 0; i < NC; ++i) {
    fft<8, true>(a[i]);
#pragma unroll
    for (int m = 0; m < 8; ++m) x[8 * i + m] = a[i][m];
  }
}
// the middle passes (INV: backwards); a butterfly's index puts 8 blocks q1 and two offsets n1 in each half-warp
template <int n, int E, bool INV, class Sync>
__device__ __forceinline__ void gmid(float2* v, int h, const GTab& t, Sync&& sync) {
  using R = GRad<n, E>;
  auto pass2 = [&] {
    if constexpr (R::R2 > 1) {
      constexpr int STEP = R::STEP2;
#pragma unroll
      for (int i = 0; i < E / R::R2; ++i) {
        const int idx = h + (n / E) * i, n1 = (idx & 1) + 2 * (idx >> 4), q1 = (idx >> 1) & 7;
        float2* u = v + q1 * R::S + n1;
        float2 c[R::R2];
#pragma unroll
        for (int m = 0; m < R::R2; ++m) c[m] = u[STEP * m];
        fft<R::R2, INV>(c);
#pragma unroll
        for (int m = 0; m < R::R2; ++m) {
          if (!INV) u[STEP * m] = m == 0 ? c[0] : cmul(c[m], t.t2[STEP * m + n1]);
          else u[STEP * m] = cmul(c[m], cconj(t.t1[q1 * R::S + n1 + STEP * m]));
        }
      }
    }
  };
  auto pass3 = [&] {
    if constexpr (R::R3 > 1) {
      constexpr int STEP = R::STEP3;
#pragma unroll
      for (int i = 0; i < E / R::R3; ++i) {
        const int idx = h + (n / E) * i, r = idx >> 4, q1 = (idx >> 1) & 7;
        const int n1 = (idx & 1) + 2 * (r % (STEP / 2)), q2 = r / (STEP / 2);
        float2* u = v + q1 * R::S + q2 * R::STEP2 + n1;
        float2 c[R::R3];
#pragma unroll
        for (int m = 0; m < R::R3; ++m) c[m] = u[STEP * m];
        fft<R::R3, INV>(c);
#pragma unroll
        for (int m = 0; m < R::R3; ++m) {
          if (!INV) u[STEP * m] = m == 0 ? c[0] : cmul(c[m], t.t3[STEP * m + n1]);
          else u[STEP * m] = cmul(c[m], cconj(t.t2[q2 * R::STEP2 + n1 + STEP * m]));
        }
      }
    }
  };
  if constexpr (R::R2 == 1) {
  } else if constexpr (R::R3 == 1) {
    pass2();
  } else if constexpr (INV) {
    pass3();
    sync();
    pass2();
  } else {
    pass2();
    sync();
    pass3();
  }
}
// last pass: unit q's spectrum X[q + (n/A) j] into p[j]
template <int n, int E>
__device__ __forceinline__ void gfwd_unit(const float2* v, int q, float2 (&p)[E / 2]) {
  const float2* u = v + gunit<n, E>(q);
#pragma unroll
  for (int j = 0; j < E / 2; j += 2) {
    const float4 w = *reinterpret_cast<const float4*>(u + j);
    p[j] = make_float2(w.x, w.y);
    p[j + 1] = make_float2(w.z, w.w);
  }
  fft<E / 2, false>(p);
}
template <int n, int E>
__device__ __forceinline__ void ginv_unit(float2* v, int q, float2 (&p)[E / 2], const GTab& t) {
  fft<E / 2, true>(p);
  ktwiddle<E / 2, true>(p, gunit_tw<n, E>(q, t));
  float2* u = v + gunit<n, E>(q);
#pragma unroll
  for (int j = 0; j < E / 2; j += 2)
    *reinterpret_cast<float4*>(u + j) = make_float4(p[j].x, p[j].y, p[j + 1].x, p[j + 1].y);
}

// Bounded grid barrier for a cooperative launch: every CTA adds one arrival to a running count (a release, so that
// it follows the CTA's stores) and polls with acquire loads until the count reaches its own target, nblocks
// further on at each barrier (target: the caller's, zero at the start of the launch; the comparison is by
// difference, so the count may wrap). The arrival returns nothing, so its way to L2 and the first poll's overlap;
// an atomic that waits for its old value and a generation word cost two more round trips. Gives up after 2^22 polls
// (a few seconds) and raises WF_ERR_TIMEOUT in *err; callers then leave.
struct GridBar {
  unsigned int count;
  unsigned int pad0;
  int err;
  int pad;
};

// the two halves, by one thread of each CTA
__device__ __forceinline__ void grid_arrive(GridBar* gb) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&gb->count), "r"(1u) : "memory");
}
__device__ __forceinline__ bool grid_wait(GridBar* gb, unsigned int target) {
  int ok = 0;
  for (long it = 0; !ok && it < (1L << 22); ++it) {
    unsigned int c;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&gb->count) : "memory");
    ok = int(c - target) >= 0;
    if (!ok && (it & 255) == 255 && *reinterpret_cast<volatile int*>(&gb->err) != 0) break;
  }
  if (!ok) atomicExch(&gb->err, 7);  // WF_ERR_TIMEOUT
  return ok != 0;
}
// opened(): run by thread 0 once the barrier has opened, before the CTA goes on
template <class F>
__device__ __forceinline__ bool grid_barrier(GridBar* gb, unsigned int nblocks, unsigned int& target, F&& opened) {
  __syncthreads();
  __shared__ int s_ok;
  target += nblocks;
  if (threadIdx.x == 0) {
    grid_arrive(gb);
    const bool ok = grid_wait(gb, target);
    if (ok) opened();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}
__device__ __forceinline__ bool grid_barrier(GridBar* gb, unsigned int nblocks, unsigned int& target) {
  return grid_barrier(gb, nblocks, target, [] {});
}

struct GlobalArgs {
  float2* Z;               // [n_fields][H][W/2] packed half spectra (state)
  const float2* aq;        // sampler pixel table [H][W] (a, q)
  const float2* fg;        // sampler mode table [H][W/2+1]
  const float2* dn;        // Wiener-filter pixel table [H][W] (d, 1/N_bar)
  const float* Pk;         // [H][W/2+1]
  const Scalars* sc;
  GridBar* bar;
  // sampler
  const float* init_s;
  long long init_stride;
  float* out;
  long long n_samples;
  int n_fields;
  int n_sweeps;
  int burn_in;
  int thin;
  uint32_t chain0;
  uint32_t step0;
  uint32_t key0, key1;
  // Wiener filter: k_global one field; k_few several, field f on the pixel table dn + f H W, the level norms
  // bnorm2 + f kMaxLevels, out + f H W and bar, acc (2 each) and st from f on
  const double* bnorm2;    // level norms (rhs_mode: one norm for every level)
  double* acc;             // [2] residual accumulators (alternating)
  float2* prev;            // [H][W/2]
  SolveStatus* st;
  double tol, eta, level_tol;
  int max_iter, level_max, check;
  int rhs_mode;            // mode 1: dn holds (r, 1/N_bar), t = lambda tau r + w s (refinement correction)
  int mode;                // 0 sampler, 1 Wiener filter, 2 level norms (fields = levels), 3 weighted power
  int levels;              // mode 2: field f is level f % levels of pixel table f / levels
  double* bnorm_out;       // mode 2: [n_fields / levels][kMaxLevels]
  // mode 3: fields v_f = va_f + vsign * vscale_f * vb_f, tables wts[nw][H][W/2+1], sums into wout[f*nw + j]
  const float* va;
  const float* vb;
  float vsign;
  PairScale vscale;
  const float* wts;
  int nw;
  double* wout;
  int grid_pct;            // host side: percent of the co-resident grid to launch (0 or >= 100: all of it)
  int out_dtype;           // mode 0: OutType of the samples
};

// ---------------------------------------------------------------------------------------------
// row phase: thread tid of a row item holds row tid / TR, unit pair (h, hb), h = tid % TR
// ---------------------------------------------------------------------------------------------
// a row of Z in global memory: ld and st of the entry at kx
struct ZRow {
  float2* p;
  __device__ __forceinline__ float2 ld(int kx) const { return __ldcg(p + kx); }
  __device__ __forceinline__ void st(int kx, float2 v) const { __stcg(p + kx, v); }
};

// the row of z (natural order) -> x (x[8 i + m] = pixel pair (E/8) h + i + (LR/8) m), unnormalised inverse transform
template <int N, int RB = 8, class Z>
__device__ __forceinline__ void grow_inv(const Z& z, float2 (&x)[GGeo<N>::E]) {
  using G = GGeo<N, RB>;
  constexpr int LR = G::LR, BR = G::BR, E = G::E, A = G::A;
  const int h = threadIdx.x % G::TR, hb = h == 0 ? BR / 2 : BR - h;
  const GTab t = gtab<N, true, RB>();
  float2* v = gsmem() + (threadIdx.x / G::TR) * G::VROW;
  {
    float2 p[A], q[A];
#pragma unroll
    for (int j = 0; j < A; ++j) p[j] = z.ld(h + BR * j);
#pragma unroll
    for (int j = 0; j < A; ++j) q[j] = z.ld(hb + BR * j);
    const float2* w = gsmem() + G::O_W;
    if (h == 0) {
      unit0_swap<A>(p, q);
      p[0] = make_float2(p[0].x + p[0].y, p[0].x - p[0].y);
      q[A - 1] = cscale(cconj(q[A - 1]), 2.0f);
    } else {
      k_pre(p[0], q[A - 1], w[h]);
    }
#pragma unroll
    for (int j = 1; j < A / 2; ++j) k_pre(p[j], q[A - 1 - j], w[h + BR * j]);
#pragma unroll
    for (int j = 0; j < A / 2; ++j) k_pre(q[j], p[A - 1 - j], w[hb + BR * j]);
    if (h == 0) unit0_unswap<A>(p, q);
    ginv_unit<LR, E>(v, h, p, t);
    ginv_unit<LR, E>(v, hb, q, t);
  }
  __syncwarp();
  gmid<LR, E, true>(v, h, t, [] { __syncwarp(); });
  __syncwarp();
  ginv1<LR, E>(v, h, x);
}

// x -> half spectrum of the row, to z
template <int N, int RB = 8, class Z>
__device__ __forceinline__ void grow_fwd(const float2 (&x)[GGeo<N>::E], const Z& z) {
  using G = GGeo<N, RB>;
  constexpr int LR = G::LR, BR = G::BR, E = G::E, A = G::A;
  const int h = threadIdx.x % G::TR, hb = h == 0 ? BR / 2 : BR - h;
  const GTab t = gtab<N, true, RB>();
  float2* v = gsmem() + (threadIdx.x / G::TR) * G::VROW;
  gfwd1<LR, E>(v, h, x, t);
  __syncwarp();
  gmid<LR, E, false>(v, h, t, [] { __syncwarp(); });
  __syncwarp();
  float2 p[A], q[A];
  gfwd_unit<LR, E>(v, h, p);
  gfwd_unit<LR, E>(v, hb, q);
  const float2* w = gsmem() + G::O_W;
  if (h == 0) {
    unit0_swap<A>(p, q);
    p[0] = make_float2(p[0].x + p[0].y, p[0].x - p[0].y);  // (R[0], R[LR])
    q[A - 1] = cconj(q[A - 1]);                            // K = LR/2
  } else {
    k_post(p[0], q[A - 1], w[h]);
  }
#pragma unroll
  for (int j = 1; j < A / 2; ++j) k_post(p[j], q[A - 1 - j], w[h + BR * j]);
#pragma unroll
  for (int j = 0; j < A / 2; ++j) k_post(q[j], p[A - 1 - j], w[hb + BR * j]);
  if (h == 0) unit0_unswap<A>(p, q);
#pragma unroll
  for (int j = 0; j < A; ++j) z.st(h + BR * j, p[j]);
#pragma unroll
  for (int j = 0; j < A; ++j) z.st(hb + BR * j, q[j]);
  __syncwarp();  // the row's vector is rewritten by the next item
}

// f(x, e): pixel pair e (pixels 2e and 2e + 1) of the row, for each of the thread's pairs
template <int N, class F>
__device__ __forceinline__ void gpixels(float2 (&x)[GGeo<N>::E], F&& f) {
  using G = GGeo<N>;
  constexpr int NC = G::E / 8;
  const int h = threadIdx.x % G::TR;
#pragma unroll
  for (int m = 0; m < 8; ++m)
#pragma unroll
    for (int i = 0; i < NC; ++i) f(x[8 * i + m], NC * h + i + (G::LR / 8) * m);
}

// a row of a row-major real image (nullptr: zeros)
template <int N>
__device__ __forceinline__ void grow_load(float2 (&x)[GGeo<N>::E], const float* row) {
  gpixels<N>(x, [&](float2& v, int e) {
    v = row != nullptr ? __ldg(reinterpret_cast<const float2*>(row) + e) : make_float2(0.f, 0.f);
  });
}
// x to row y of an image of element type ot
template <int N>
__device__ __forceinline__ void grow_store(float2 (&x)[GGeo<N>::E], void* img, long long y, int ot) {
  gpixels<N>(x, [&](float2& v, int e) { store_pair(img, y * (N / 2) + e, v, ot); });
}

// Pixel update of row y (pixel tables row-major):
//   mode 0: sampler t-draw t = (1 - w) d + sqrt(w) (sqrt(w) s + sqrt(tau) xi) with the (a, q) table, Philox
//           counter (pixel group (y W + x) / 4, step, chain, stream);
//   mode 4: its mean t = a + q^2 s (no draw);
//   mode 1: Wiener-filter t-update t = w (s - d) + d, w = 1 / (1 + lambda tau / N_bar) from the (d, 1/N_bar)
//           table (rhs_mode: t = w s + lambda tau r with r in place of d);
//   mode 2: the level right-hand side N_lambda^-1 d with N_lambda = N_bar + lt2 (s ignored).
// The two pairs of a Philox group are in one thread (E = 16), or in neighbouring lanes (E = 8): there each lane
// draws half of the groups and the two exchange the halves they need. tab(e): the table's entries of pixels 2e and
// 2e + 1; draw(i, z): the normals of the thread's i-th group (pixel_group).
template <int N>
__device__ __forceinline__ uint32_t pixel_group(int y, int i) {
  using G = GGeo<N>;
  const int h = threadIdx.x % G::TR;
  if constexpr (G::E == 16) return uint32_t(y * (G::W / 4) + h + (G::LR / 16) * i);
  else return uint32_t(y * (G::W / 4) + (h + (G::LR / 8) * ((h & 1) ? 4 + i : i)) / 2);
}
template <int N, class T, class D>
__device__ __forceinline__ void pixel_update(int mode, float2 (&x)[GGeo<N>::E], T&& tab, D&& draw, float sqrt_tau,
                                             float ltau, int rhs_mode, float lt2) {
  using G = GGeo<N>;
  if (mode == 0) {
    const int h = threadIdx.x % G::TR;
    auto upd = [&](float2& v, float4 c, float z0, float z1) {
      v.x = fmaf(c.y, fmaf(c.y, v.x, sqrt_tau * z0), c.x);
      v.y = fmaf(c.w, fmaf(c.w, v.y, sqrt_tau * z1), c.z);
    };
    if constexpr (G::E == 16) {
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int e = 2 * h + (G::LR / 8) * m;
        const float4 c0 = tab(e), c1 = tab(e + 1);
        float z[4];
        draw(m, z);
        upd(x[m], c0, z[0], z[1]);
        upd(x[8 + m], c1, z[2], z[3]);
      }
    } else {
      const bool odd = h & 1;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e0 = h + (G::LR / 8) * i, e1 = h + (G::LR / 8) * (4 + i);
        const float4 c0 = tab(e0), c1 = tab(e1);
        float z[4];  // even lanes: the group of pair e0, odd lanes: that of e1
        draw(i, z);
        const float r0 = __shfl_xor_sync(0xffffffffu, odd ? z[0] : z[2], 1);
        const float r1 = __shfl_xor_sync(0xffffffffu, odd ? z[1] : z[3], 1);
        upd(x[i], c0, odd ? r0 : z[0], odd ? r1 : z[1]);
        upd(x[4 + i], c1, odd ? z[2] : r0, odd ? z[3] : r1);
      }
    }
  } else if (mode == 4) {
    gpixels<N>(x, [&](float2& v, int e) {
      const float4 c = tab(e);
      v.x = fmaf(c.y, c.y * v.x, c.x);
      v.y = fmaf(c.w, c.w * v.y, c.z);
    });
  } else if (mode == 1) {
    const float g = rhs_mode ? 0.0f : 1.0f, hh = rhs_mode ? ltau : 1.0f;
    auto upd = [&](float& v, float dv, float inb) {
      const float w = wf_weight(ltau, inb);
      v = fmaf(w, fmaf(-g, dv, v), hh * dv);
    };
    gpixels<N>(x, [&](float2& v, int e) {
      const float4 c = tab(e);
      upd(v.x, c.x, c.y);
      upd(v.y, c.z, c.w);
    });
  } else {
    auto rhs = [&](float dv, float inb) { return dv / ((inb > 0.0f ? wf_rcp(inb) : wf_inf()) + lt2); };
    gpixels<N>(x, [&](float2& v, int e) {
      const float4 c = tab(e);
      v = make_float2(rhs(c.x, c.y), rhs(c.z, c.w));
    });
  }
}

// with the tables in global memory and the draws on the spot
template <int N>
__device__ __forceinline__ void pixel_update(int mode, float2 (&x)[GGeo<N>::E], int y, const float2* __restrict__ aq,
                                             const float2* __restrict__ dn, uint32_t step, uint32_t chain,
                                             uint32_t key0, uint32_t key1, float sqrt_tau, float ltau, int rhs_mode,
                                             float lt2, uint32_t stream = 0u) {
  const float4* tab =
      reinterpret_cast<const float4*>((mode == 0 || mode == 4 ? aq : dn) + (long long)y * GGeo<N>::W);
  pixel_update<N>(
      mode, x, [&](int e) { return __ldg(tab + e); },
      [&](int i, float (&z)[4]) { normals4(pixel_group<N>(y, i), step, chain, stream, key0, key1, z); }, sqrt_tau,
      ltau, rhs_mode, lt2);
}

// Row phase on one work item: rows y0 .. y0+RB-1 of field f. first: start from the real state s0.
template <int N>
__device__ void row_item(const GlobalArgs& a, int f, int y0, int done, bool first, bool emit_only, float ltau,
                         const Scalars& sc) {
  using G = GGeo<N>;
  const int y = y0 + int(threadIdx.x) / G::TR;
  const ZRow z{a.Z + ((long long)f * G::H + y) * G::LR};
  float2 x[G::E];
  if (!first) {
    grow_inv<N>(z, x);
  } else if (a.mode == 3) {
    const long long o = ((long long)f * G::H + y) * G::W;
    grow_load<N>(x, a.va + o);
    if (a.vb) {
      const float sgn = a.vsign * pair_scale(a.vscale, f);
      gpixels<N>(x, [&](float2& v, int e) {
        const float2 u = __ldg(reinterpret_cast<const float2*>(a.vb + o) + e);
        v = make_float2(fmaf(sgn, u.x, v.x), fmaf(sgn, u.y, v.y));
      });
    }
  } else {
    grow_load<N>(x, a.mode == 0 && a.init_s ? a.init_s + f * a.init_stride + (long long)y * G::W : nullptr);
  }
  // x holds the row's pixels (unnormalised transforms, the 1/n and 1/sqrt(2n) factors are in the Fourier-space
  // tables)
  if (a.mode == 0 && !first) {
    const int d1 = done;  // sweeps completed
    if (d1 > a.burn_in && (d1 - a.burn_in) % a.thin == 0) {
      const long long ms = (d1 - a.burn_in) / a.thin - 1;
      grow_store<N>(x, a.out, ((long long)f * a.n_samples + ms) * G::H + y, a.out_dtype);
    }
  }
  if (emit_only) {
    if (a.mode == 1) grow_store<N>(x, a.out, y, kOutF32);  // Wiener filter: final state to out
    return;
  }
  if (a.mode != 3)  // mode 3 transforms the field as loaded
    pixel_update<N>(a.mode, x, y, a.aq, a.mode == 2 ? a.dn + (long long)(f / a.levels) * G::H * G::W : a.dn, a.step0 + uint32_t(done), a.chain0 + uint32_t(f), a.key0, a.key1,
                    sc.sqrt_tau, ltau, a.rhs_mode, a.mode == 2 ? float(level_lambda(sc, f % a.levels, a.eta) * sc.tau) : 0.f);
  grow_fwd<N>(x, z);
}

// ---------------------------------------------------------------------------------------------
// column phase: thread tid of a column item holds column c0 + tid % CB, unit pair (h, hb), h = tid / CB
// ---------------------------------------------------------------------------------------------
// the CTA's columns of Z in global memory: at(y0, c): column c from row y0, with ld and st of row y0 + dy
template <int N>
struct ZCols {
  float2* p;  // of column 0
  struct Col {
    float2* p;
    __device__ __forceinline__ float2 ld(int dy) const { return __ldcg(p + (long long)dy * (N / 2)); }
    __device__ __forceinline__ void st(int dy, float2 v) const { __stcg(p + (long long)dy * (N / 2), v); }
  };
  __device__ __forceinline__ Col at(int y0, int c) const { return Col{p + (long long)y0 * (N / 2) + c}; }
};
// Columns c0 .. c0 + CB - 1 of z: forward transform, f(p, q) on the thread's units (after unit0_swap: mode
// pairs (p[j], q[A-1-j]) at ky1 = h + BC j and (q[j], p[A-1-j]) at ky1 = hb + BC j, j < A/2), and with INV the inverse
// transform back to Z.
template <int N, bool INV, int RB = 8, class Z, class F>
__device__ __forceinline__ void gcol(const Z& z, int c0, F&& f) {
  using G = GGeo<N, RB>;
  constexpr int H = G::H, BC = G::BC, E = G::E, A = G::A, NC = E / 8;
  const int c = threadIdx.x % G::CB, h = threadIdx.x / G::CB, hb = h == 0 ? BC / 2 : BC - h;
  const GTab t = gtab<N, false, RB>();
  float2* v = gsmem() + c * G::VCOL;
  const auto zc = z.at(NC * h, c);
  {
    float2 x[E];
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
      for (int i = 0; i < NC; ++i) x[8 * i + m] = zc.ld(H / 8 * m + i);
    gfwd1<H, E>(v, h, x, t);
  }
  __syncthreads();
  gmid<H, E, false>(v, h, t, [] { __syncthreads(); });
  __syncthreads();
  {
    float2 p[A], q[A];
    gfwd_unit<H, E>(v, h, p);
    gfwd_unit<H, E>(v, hb, q);
    if (h == 0) unit0_swap<A>(p, q);
    f(p, q, c0 + c, h, hb);
    if (!INV) {
      __syncthreads();  // the vectors are rewritten by the next item
      return;
    }
    if (h == 0) unit0_unswap<A>(p, q);
    ginv_unit<H, E>(v, h, p, t);
    ginv_unit<H, E>(v, hb, q, t);
  }
  __syncthreads();
  gmid<H, E, true>(v, h, t, [] { __syncthreads(); });
  __syncthreads();
  {
    float2 x[E];
    ginv1<H, E>(v, h, x);
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
      for (int i = 0; i < NC; ++i) zc.st(H / 8 * m + i, x[8 * i + m]);
  }
  __syncthreads();
}

// inter(y1, y2, ky1, ky2) on the mode pairs of an interior column; the H/2 pairs of the packed edge column (column
// 0: kx = 0 as A and kx = W/2 as B in Y = A + i B) are shared out over all threads of its CTA
template <int N, int RB = 8, class I, class X>
__device__ __forceinline__ void gpairs(float2 (&p)[GGeo<N>::A], float2 (&q)[GGeo<N>::A], int col, int h, int hb,
                                       int c0, I&& inter, X&& edge) {
  using G = GGeo<N, RB>;
  constexpr int H = G::H, BC = G::BC, A = G::A;
  float2* e = gsmem() + G::O_EDGE;
  if (c0 == 0) {  // the same in every thread of the CTA
    if (col == 0) {
#pragma unroll
      for (int j = 0; j < A / 2; ++j) {
        e[2 * (h + BC * j)] = p[j];
        e[2 * (h + BC * j) + 1] = q[A - 1 - j];
        e[2 * (hb + BC * j)] = q[j];
        e[2 * (hb + BC * j) + 1] = p[A - 1 - j];
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < H / 2; k += G::T) {
      float2 y1 = e[2 * k], y2 = e[2 * k + 1];
      edge(y1, y2, k, k == 0 ? H / 2 : H - k);
      e[2 * k] = y1;
      e[2 * k + 1] = y2;
    }
  }
  if (col != 0) {
#pragma unroll
    for (int j = 0; j < A / 2; ++j) {
      const int ky1 = h + BC * j;
      inter(p[j], q[A - 1 - j], ky1, ky1 == 0 ? H / 2 : H - ky1);
    }
#pragma unroll
    for (int j = 0; j < A / 2; ++j) inter(q[j], p[A - 1 - j], hb + BC * j, H - hb - BC * j);
  }
  if (c0 == 0) {
    __syncthreads();
    if (col == 0) {
#pragma unroll
      for (int j = 0; j < A / 2; ++j) {
        p[j] = e[2 * (h + BC * j)];
        q[A - 1 - j] = e[2 * (h + BC * j) + 1];
        q[j] = e[2 * (hb + BC * j)];
        p[A - 1 - j] = e[2 * (hb + BC * j) + 1];
      }
    }
  }
}

// Column-phase spectral update of columns c0 .. c0+CB-1 (tables in natural order):
//   mode 0: sampler s-draw s_hat = f t_hat + g zeta with the (f/n, g/sqrt(2n)) table and Philox counter
//           (column pair group col H/2 + j, step, chain, stream 1; edge column as in the on-chip kernel);
//   mode 1: Wiener-filter update s_hat = P/(P + lambda tau) t_hat / n; with cmp, returns this thread's part of
//           sum_k |s_hat - prev|^2 ((P + lambda tau)/(lambda tau))^2 (the residual from consecutive
//           iterates); with store, keeps s_hat in prev;
//   mode 2: returns this thread's part of sum_k P^2 |t_hat|^2 of the level right-hand side (Z unchanged).
// Per-mode terms and a thread's partial sum in FP32, the CTA and grid sums in FP64.
// z: the CTA's columns; fg(ky, kx), Pk(ky, kx), prev(ky, kx): the tables; draw(i, g, z): the normals of the thread's
// i-th pair, group g; edraw(ky, z): those of a pair of the edge column.
template <int N, int RB = 8, class Z, class FG, class PK, class PV, class D, class X>
__device__ __forceinline__ float gcol_update(int mode, const Z& z, int c0, FG&& fg, PK&& Pk, PV&& prev, D&& draw,
                                             X&& edraw, float ltau, bool cmp, bool store) {
  using G = GGeo<N, RB>;
  constexpr int H = G::H, EW = G::W / 2;
  constexpr float INV_N = 1.0f / float(G::H * G::W);
  float acc = 0.0f;
  if (mode == 0) {
    gcol<N, true, RB>(z, c0, [&](float2 (&p)[G::A], float2 (&q)[G::A], int col, int h, int hb) {
      int i = 0;
      gpairs<N, RB>(
          p, q, col, h, hb, c0,
          [&](float2& y1, float2& y2, int ky1, int ky2) {
            const float2 m1 = fg(ky1, col), m2 = fg(ky2, col);
            float z[4];
            draw(i++, uint32_t(col * (H / 2) + ky1), z);
            y1 = make_float2(fmaf(m1.x, y1.x, m1.y * z[0]), fmaf(m1.x, y1.y, m1.y * z[1]));
            y2 = make_float2(fmaf(m2.x, y2.x, m2.y * z[2]), fmaf(m2.x, y2.y, m2.y * z[3]));
          },
          [&](float2& y1, float2& y2, int ky1, int ky2) {
            const float2 a1 = fg(ky1, 0), b1 = fg(ky1, EW);
            float z[4];
            edraw(ky1, z);
            if (ky1 == 0) {
              const float2 a2 = fg(ky2, 0), b2 = fg(ky2, EW);
              constexpr float R2 = 1.41421356237309505f;
              y1 = make_float2(fmaf(a1.x, y1.x, R2 * a1.y * z[0]), fmaf(b1.x, y1.y, R2 * b1.y * z[2]));
              y2 = make_float2(fmaf(a2.x, y2.x, R2 * a2.y * z[1]), fmaf(b2.x, y2.y, R2 * b2.y * z[3]));
            } else {
              const float2 y2c = cconj(y2);
              const float2 A = cscale(cadd(y1, y2c), 0.5f);
              const float2 B = cmul_mi(cscale(csub(y1, y2c), 0.5f));
              const float2 Ap = make_float2(fmaf(a1.x, A.x, a1.y * z[0]), fmaf(a1.x, A.y, a1.y * z[1]));
              const float2 Bp = make_float2(fmaf(b1.x, B.x, b1.y * z[2]), fmaf(b1.x, B.y, b1.y * z[3]));
              y1 = cadd(Ap, cmul_i(Bp));
              y2 = cadd(cconj(Ap), cmul_i(cconj(Bp)));
            }
          });
    });
  } else if (mode == 1) {
    const float inv_lt = cmp ? 1.0f / ltau : 0.0f;
    auto wres = [&](float P, float dre, float dim) -> float {
      const float g = fmaf(P, inv_lt, 1.0f);
      return fmaf(dre, dre, dim * dim) * (g * g);
    };
    auto fcoef = [&](float P) { return wf_fdiv(P, P + ltau) * INV_N; };
    gcol<N, true, RB>(z, c0, [&](float2 (&p)[G::A], float2 (&q)[G::A], int col, int h, int hb) {
      gpairs<N, RB>(
          p, q, col, h, hb, c0,
          [&](float2& y1, float2& y2, int ky1, int ky2) {
            const float P1 = Pk(ky1, col), P2 = Pk(ky2, col);
            y1 = cscale(y1, fcoef(P1));
            y2 = cscale(y2, fcoef(P2));
            if (cmp) {
              const float2 o1 = prev(ky1, col), o2 = prev(ky2, col);
              acc += 2.0f * (wres(P1, y1.x - o1.x, y1.y - o1.y) + wres(P2, y2.x - o2.x, y2.y - o2.y));
            }
            if (store) {
              prev(ky1, col) = y1;
              prev(ky2, col) = y2;
            }
          },
          [&](float2& y1, float2& y2, int ky1, int ky2) {
            const float Pa1 = Pk(ky1, 0), Pb1 = Pk(ky1, EW);
            const float fa1 = fcoef(Pa1), fb1 = fcoef(Pb1);
            if (ky1 == 0) {
              const float Pa2 = Pk(ky2, 0), Pb2 = Pk(ky2, EW);
              y1 = make_float2(fa1 * y1.x, fb1 * y1.y);
              y2 = make_float2(fcoef(Pa2) * y2.x, fcoef(Pb2) * y2.y);
              if (cmp) {
                const float2 o1 = prev(0, 0), o2 = prev(ky2, 0);
                acc += wres(Pa1, y1.x - o1.x, 0.f) + wres(Pb1, y1.y - o1.y, 0.f) + wres(Pa2, y2.x - o2.x, 0.f) +
                       wres(Pb2, y2.y - o2.y, 0.f);
              }
            } else {
              const float2 y2c = cconj(y2);
              const float2 A = cscale(cscale(cadd(y1, y2c), 0.5f), fa1);
              const float2 B = cscale(cmul_mi(cscale(csub(y1, y2c), 0.5f)), fb1);
              y1 = cadd(A, cmul_i(B));
              y2 = cadd(cconj(A), cmul_i(cconj(B)));
              if (cmp) {
                const float2 o1 = prev(ky1, 0), o2c = cconj(prev(ky2, 0));
                const float2 oA = cscale(cadd(o1, o2c), 0.5f);
                const float2 oB = cmul_mi(cscale(csub(o1, o2c), 0.5f));
                acc += 2.0f * (wres(Pa1, A.x - oA.x, A.y - oA.y) + wres(Pb1, B.x - oB.x, B.y - oB.y));
              }
            }
            if (store) {
              prev(ky1, 0) = y1;
              prev(ky2, 0) = y2;
            }
          });
    });
  } else {
    auto p2 = [](float P, float re, float im) -> float { return fmaf(P * re, P * re, (P * im) * (P * im)); };
    gcol<N, false, RB>(z, c0, [&](float2 (&p)[G::A], float2 (&q)[G::A], int col, int h, int hb) {
      gpairs<N, RB>(
          p, q, col, h, hb, c0,
          [&](float2& y1, float2& y2, int ky1, int ky2) {
            acc += 2.0f * (p2(Pk(ky1, col), y1.x, y1.y) + p2(Pk(ky2, col), y2.x, y2.y));
          },
          [&](float2& y1, float2& y2, int ky1, int ky2) {
            if (ky1 == 0) {
              acc += p2(Pk(0, 0), y1.x, 0.f) + p2(Pk(0, EW), y1.y, 0.f) +
                     p2(Pk(ky2, 0), y2.x, 0.f) + p2(Pk(ky2, EW), y2.y, 0.f);
            } else {
              const float2 y2c = cconj(y2);
              const float2 A = cscale(cadd(y1, y2c), 0.5f);
              const float2 B = cmul_mi(cscale(csub(y1, y2c), 0.5f));
              acc += 2.0f * (p2(Pk(ky1, 0), A.x, A.y) + p2(Pk(ky1, EW), B.x, B.y));
            }
          });
    });
  }
  return acc;
}

// with the tables in global memory and the draws on the spot
template <int N>
__device__ __forceinline__ float gcol_update(int mode, float2* Z, int c0, const float2* __restrict__ fg,
                                             const float* __restrict__ Pk, float2* prev, uint32_t step,
                                             uint32_t chain, uint32_t key0, uint32_t key1, float ltau, bool cmp,
                                             bool store) {
  constexpr int L = N / 2, WH = N / 2 + 1;
  auto draw = [&](uint32_t g, float (&z)[4]) { normals4(g, step, chain, 1u, key0, key1, z); };
  return gcol_update<N>(
      mode, ZCols<N>{Z + c0}, c0, [&](int ky, int kx) { return __ldg(fg + ky * WH + kx); },
      [&](int ky, int kx) { return __ldg(Pk + ky * WH + kx); },
      [&](int ky, int kx) -> float2& { return prev[ky * L + kx]; },
      [&](int, uint32_t g, float (&z)[4]) { draw(g, z); }, [&](int ky, float (&z)[4]) { draw(uint32_t(ky), z); }, ltau,
      cmp, store);
}

// mode 3: weighted power sums of CB columns of field f into acc[j], j < nw
template <int N>
__device__ void col_wpower(const GlobalArgs& a, int f, int c0, double (&acc)[4]) {
  using G = GGeo<N>;
  constexpr int WH = G::WH, TS = G::H * G::WH;
  auto sq = [](float p, float q) -> double { return double(p) * p + double(q) * q; };
  gcol<N, false>(ZCols<N>{a.Z + (long long)f * G::H * G::LR + c0}, c0, [&](float2 (&p)[G::A], float2 (&q)[G::A], int col, int h, int hb) {
    gpairs<N>(
        p, q, col, h, hb, c0,
        [&](float2& y1, float2& y2, int ky1, int ky2) {
          for (int t = 0; t < a.nw; ++t) {
            const float* wt = a.wts + t * TS;
            acc[t] += 2.0 * (__ldg(wt + ky1 * WH + col) * sq(y1.x, y1.y) + __ldg(wt + ky2 * WH + col) * sq(y2.x, y2.y));
          }
        },
        [&](float2& y1, float2& y2, int ky1, int ky2) {
          for (int t = 0; t < a.nw; ++t) {
            const float* wt = a.wts + t * TS;
            if (ky1 == 0) {
              acc[t] += __ldg(wt) * sq(y1.x, 0.f) + __ldg(wt + G::W / 2) * sq(y1.y, 0.f) +
                        __ldg(wt + ky2 * WH) * sq(y2.x, 0.f) + __ldg(wt + ky2 * WH + G::W / 2) * sq(y2.y, 0.f);
            } else {
              const float2 y2c = cconj(y2);
              const float2 A = cscale(cadd(y1, y2c), 0.5f);
              const float2 B = cmul_mi(cscale(csub(y1, y2c), 0.5f));
              acc[t] += 2.0 * (__ldg(wt + ky1 * WH) * sq(A.x, A.y) + __ldg(wt + ky1 * WH + G::W / 2) * sq(B.x, B.y));
            }
          }
        });
  });
}

// CTA sum in a fixed order, valid in the first warp: the threads' values through shared memory (T doubles), one warp
// adds them (with every thread in the shuffle tree the SM's two FP64 lanes are busy for several hundred cycles)
template <int T>
__device__ __forceinline__ double gblock_sum(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
#pragma unroll
    for (int w = 0; w < T / 32; ++w) s += red[32 * w + threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  __syncthreads();
  return s;
}

// schedule of the cooled solve, decided by one thread per CTA (every CTA the same way) and shared
struct GSolveState {
  double rho2;  // of the last check (-1: none)
  float ltau;
  int lev, k, status;
};

template <int N>
__global__ void __launch_bounds__(GGeo<N>::T, GGeo<N>::MIN_CTAS) k_global(const __grid_constant__ GlobalArgs a) {
  using G = GGeo<N>;
  __shared__ double red[G::T];
  __shared__ GSolveState dec;
  const Scalars sc = *a.sc;
  if (sc.status != 0) {
    if (a.mode == 1 && blockIdx.x == 0 && threadIdx.x == 0) a.st->status = sc.status;
    return;
  }
  gtab_init<N>();
  const unsigned int nb = gridDim.x;
  unsigned int target = 0;  // of the grid barrier
  const int row_items = G::ROW_ITEMS * a.n_fields, col_items = G::COL_ITEMS * a.n_fields;

  auto rows = [&](int done, bool first, bool emit_only, float ltau) {
    for (int it = blockIdx.x; it < row_items; it += nb) {
      const int f = it / G::ROW_ITEMS;
      if (a.mode == 2 && f % a.levels >= sc.n_levels) continue;  // level fields past the schedule
      row_item<N>(a, f, (it % G::ROW_ITEMS) * G::RB, done, first, emit_only, ltau, sc);
    }
  };
  auto col = [&](int f, int it, int done, float ltau, bool cmp, bool store) -> float {
    return gcol_update<N>(a.mode, a.Z + (long long)f * G::H * G::LR, (it % G::COL_ITEMS) * G::CB, a.fg, a.Pk, a.prev,
                          a.step0 + uint32_t(done), a.chain0 + uint32_t(f), a.key0, a.key1, ltau, cmp, store);
  };
  auto cols = [&](int done, float ltau, bool cmp, bool store) -> double {
    double acc = 0.0;
    for (int it = blockIdx.x; it < col_items; it += nb) {
      const float v = col(it / G::COL_ITEMS, it, done, ltau, cmp, store);
      if (cmp) acc += double(v);
    }
    return acc;
  };

  if (a.mode == 0) {
    rows(0, true, false, 0.f);
    for (int i = 0; i < a.n_sweeps; ++i) {
      if (!grid_barrier(a.bar, nb, target)) return;
      cols(i, 0.f, false, false);
      if (!grid_barrier(a.bar, nb, target)) return;
      rows(i + 1, false, i + 1 == a.n_sweeps, 0.f);
    }
    return;
  }
  if (a.mode == 3) {  // weighted power of given fields
    rows(0, true, false, 0.f);
    if (!grid_barrier(a.bar, nb, target)) return;
    for (int it = blockIdx.x; it < col_items; it += nb) {
      const int f = it / G::COL_ITEMS;
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      col_wpower<N>(a, f, (it % G::COL_ITEMS) * G::CB, acc);
      for (int t = 0; t < a.nw; ++t) {
        const double s = gblock_sum<G::T>(acc[t], red);
        if (threadIdx.x == 0) atomicAdd(a.wout + f * a.nw + t, s / double(G::H * G::W));
      }
    }
    return;
  }
  if (a.mode == 2) {  // level norms, fields = levels
    rows(0, true, false, 0.f);
    if (!grid_barrier(a.bar, nb, target)) return;
    for (int it = blockIdx.x; it < col_items; it += nb) {
      const int f = it / G::COL_ITEMS;
      if (f % a.levels >= sc.n_levels) continue;
      const double s = gblock_sum<G::T>(col(f, it, 0, 0.f, false, false), red);
      if (threadIdx.x == 0)
        atomicAdd(a.bnorm_out + (f / a.levels) * kMaxLevels + f % a.levels, s / double(G::H * G::W));
    }
    return;
  }
  // Wiener filter with lambda-cooling, one field; every CTA follows the same schedule
  const int last_level = sc.n_levels - 1;
  int lev = 0, it = 0, k = 0, status = 1, parity = 0;
  float ltau = float(sc.lam0 * sc.tau);
  double rho2 = -1.0;
  rows(0, true, false, ltau);
  while (true) {
    ++k;
    ++it;
    const bool cmp = (k % a.check == 0) && k >= 2;
    const bool store = ((k + 1) % a.check == 0);
    if (!grid_barrier(a.bar, nb, target)) return;
    const double mine = cols(it, ltau, cmp, store);
    if (cmp) {
      const double part = gblock_sum<G::T>(mine, red);
      if (threadIdx.x == 0) atomicAdd(a.acc + parity, part);
    }
    // a check's decision by the thread that waits for the barrier: rho = sqrt(tot / bn) against the tolerances,
    // without the division and the root (run by every thread these took about 4000 cycles a check)
    const bool open = grid_barrier(a.bar, nb, target, [&] {
      if (!cmp) return;
      const double tot = __ldcg(a.acc + parity) * double(G::H * G::W);
      const double bn = a.bnorm2[a.rhs_mode ? 0 : lev], ref = bn > 0.0 ? bn : 1.0;
      if (blockIdx.x == 0) a.acc[parity ^ 1] = 0.0;  // next check's accumulator
      GSolveState d{tot, ltau, lev, k, 1};
      if (residual_nonfinite(tot, ref)) {
        d.status = 6;  // non-finite residual
      } else if (lev < last_level) {
        if (tot < a.level_tol * a.level_tol * ref || k >= a.level_max) {
          ++d.lev;
          d.ltau = float(level_lambda(sc, d.lev, a.eta) * sc.tau);
          d.k = 0;
        }
      } else if (tot < a.tol * a.tol * ref) {
        d.status = 0;
      }
      if (blockIdx.x == 0) d.rho2 = tot / ref;
      dec = d;
    });
    if (!open) return;
    if (cmp) {
      parity ^= 1;
      rho2 = dec.rho2;
      lev = dec.lev;
      ltau = dec.ltau;
      k = dec.k;
      status = dec.status;
    }
    if (status == 1 && it >= a.max_iter) status = 5;  // not converged
    rows(it, false, status != 1, ltau);
    if (status != 1) break;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.st->status = status;
    a.st->iters = it;
    a.st->resid = rho2 >= 0.0 ? sqrt(rho2) : rho2;
  }
}

}  // namespace wf
