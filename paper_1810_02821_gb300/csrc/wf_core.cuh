// Messenger-field sweeps of one field (32^2, 64^2 or 128^2) by several threads per row (Alg. 1 of the paper,
// A = I, and its G -> 0 form with lambda-cooling, §2.2). The field stays in one SM's shared memory.
//
// Geometry. The packed half spectrum [H][L] (L = W/2 float2; kx = 0 and W/2 packed in column 0) is held by
// T = H L / E threads with E = 2 A elements each. A transform of length B A (rows: L = BR A, columns:
// H = BC A) is two register passes, decimation in frequency:
//   pass 1: the thread owns A-strided subsequences n0 + A m: B-point DFTs over m (output q), times W^(n0 q);
//   pass 2: the thread owns two units q, the A-point DFTs over n0: X[q + B j], j < A.
// Both passes work in place (pass 1 leaves (q, n0) at A q + n0, pass 2 leaves X[q + B j] at A q + j), so the
// spectrum is in digit-reversed slot order; the inverse runs the passes backwards. The two units of a thread
// are q and B - q (0 and B/2 for the first thread), which hold every mode pair (k, -k): the real-transform
// post and pre passes along rows and the s-draw along columns run on registers between the transforms, and the
// t-draw runs on registers between the inverse and the forward row transform.
//
// Threads. The lanes of a warp are 32 rows (row passes) or 32 column slots (column passes) with one unit pair
// each, so the twiddles are warp-uniform (shared-memory broadcasts), a row stride of L + 1 float2 makes both
// access patterns free of bank conflicts, and the tables are read along lanes ([x][y] pixel tables, mode tables
// in slot order). Pass 1 and pass 2 exchange within the TR (TC) warps of a row (column) group: four group
// barriers (six with the edge column) and two CTA barriers per sweep.
//
// Why this split: with one thread per row (64-point register transforms, 128 data registers) a 128^2 field is 4
// warps, so a single chain leaves three quarters of an SM's issue slots empty and a full SM holds 12 warps and issues
// in 59% of its cycles. With E = 16 a field is 16 warps of 64 registers, two fields an SM. Measured (us per sweep):
// one 128^2 chain 14.7 -> 9.6, 1000 chains 65.4 -> 60.0; one 64^2 chain 7.4 -> 4.2; one 32^2 chain 4.1 -> 2.0. A full
// SM now runs at 64% issue with eligible warps waiting: the bound is the dispatch of the instructions themselves
// (49K warp instructions a 128^2 sweep, a third of them the Philox draws, 64-bit integer products and paired FP32
// operations taking more than one dispatch slot), no longer latency.
#pragma once

#include "wf_bphase.cuh"
#include "wf_units.cuh"

namespace wf {

// sizes with these kernels, and the mode tables' slot order for them (mode_pos with cm = BR; 0: natural order)
WF_HD constexpr bool core_size(int N) { return N == 32 || N == 64 || N == 128; }
WF_HD constexpr int core_cm(int N) { return N == 128 ? 8 : (N == 32 || N == 64 ? 4 : 0); }

template <int N_>
struct KGeo {
  static constexpr int N = N_, H = N_, W = N_, L = N_ / 2;
  static constexpr int A = N_ >= 64 ? 8 : 4;   // length of the unit transforms
  static constexpr int E = 2 * A;              // elements per thread
  static constexpr int BR = L / A, BC = H / A; // strided radices of the row and column transforms
  static constexpr int TR = BR / 2, TC = BC / 2;  // threads per row and per column
  static constexpr int T = H * TR;
  static constexpr int NR = E / BR, NC = E / BC;  // strided subsequences per thread
  static constexpr int SP = L + 1;
  static constexpr int FIELD_BYTES = (H * SP * 8 + 15) / 16 * 16;
  // twiddle tables: W_L^(n0 q) by n0 and by q, W_H^(n0 q) by n0 and by q, W_W^K at [q][j], K = q + BR j, j < A/2
  static constexpr int O_R = 0, O_RT = O_R + A * BR, O_C = O_RT + A * BR, O_CT = O_C + A * BC, O_P = O_CT + A * BC;
  static constexpr int NTW = O_P + BR * (A / 2);
  static constexpr int GT = L >= 32 ? TC * 32 : T;  // threads of a column group
  static constexpr int EDGE = H;                    // parked modes of the packed edge column
  static constexpr int SMEM = FIELD_BYTES + (NTW + EDGE) * 8;  // (+ 33 doubles for the solve's sums)
  static_assert(core_cm(N) == BR, "slot order of the mode tables");
  static_assert(T == L * TC && BR >= 2 && NR % 2 == 0 && NC >= 1 && T % 32 == 0, "geometry");
};

template <int ID, int THREADS, int GROUPS>
__device__ __forceinline__ void group_bar(int g) {
  if (ID == GROUPS || g == ID - 1) {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
  } else if constexpr (ID < GROUPS) {
    group_bar<ID + 1, THREADS, GROUPS>(g);
  }
}
// Barrier of one group of warps (group g of GROUPS in the CTA), or of the whole CTA. The barrier numbers are
// literals: a kernel with a run-time barrier number reserves all 16, of which an SM has 64, so four CTAs.
template <int THREADS, int FIELD, int GROUPS>
__device__ __forceinline__ void group_sync(int g) {
  if constexpr (THREADS == 32) {
    __syncwarp();
  } else if constexpr (THREADS == FIELD) {
    __syncthreads();
  } else {
    static_assert(GROUPS <= 8, "barrier numbers 1 .. 8");
    group_bar<1, THREADS, GROUPS>(g);
  }
}

// The thread's coordinates, formed anew in every pass: the thread index is read through a volatile
// statement at 128^2, so that the compiler does not keep the passes' addresses in registers across the whole sweep
// (64 registers a thread, half of them data).
__device__ __forceinline__ unsigned char* kfield_smem() {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  return smem_raw;
}
template <int N>
__device__ __forceinline__ int ktid() {
  if constexpr (N < 128) return int(threadIdx.x);
  int v;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(v));
  return v;
}
// thread index within its field, the field of the CTA (of NF, T threads each) and its buffer
template <int N, int NF>
struct KField {
  using G = KGeo<N>;
  int lt, f;
  __device__ __forceinline__ KField() {
    lt = ktid<N>();
    f = 0;
    if constexpr (NF > 1) {
      f = lt / G::T;
      lt %= G::T;
    }
  }
  __device__ __forceinline__ float2* S() const {
    return reinterpret_cast<float2*>(kfield_smem() + (NF > 1 ? f * G::FIELD_BYTES : 0));
  }
  static __device__ __forceinline__ float2* tables() {
    return reinterpret_cast<float2*>(kfield_smem() + NF * G::FIELD_BYTES);
  }
};
template <int N, int NF = 1>
struct KRow {  // row y, unit pair (h, hb) of row group g
  using G = KGeo<N>;
  int y, h, hb, g;
  float2* row;
  const float2* tw;
  __device__ __forceinline__ KRow() {
    const KField<N, NF> k;
    const int w = __shfl_sync(0xffffffffu, k.lt / 32, 0);  // the same in every lane, known to the compiler
    g = w / G::TR;
    h = w % G::TR;
    hb = h == 0 ? G::BR / 2 : G::BR - h;
    y = g * 32 + k.lt % 32;
    if constexpr (NF > 1) g += __shfl_sync(0xffffffffu, k.f, 0) * (G::T / (G::TR * 32));
    row = k.S() + y * G::SP;
    tw = KField<N, NF>::tables();
  }
  __device__ __forceinline__ void sync() const { group_sync<G::TR * 32, G::T, NF * (G::T / (G::TR * 32))>(g); }
};
template <int N, int NF = 1>
struct KCol {  // column slot, unit pair (h, hb) of column group g
  using G = KGeo<N>;
  int slot, h, hb, g, f, gl;  // f: field of the CTA, gl: thread index within the group
  float2* col;
  const float2* tw;
  __device__ __forceinline__ KCol() {
    const KField<N, NF> k;
    f = k.f;
    if constexpr (G::L >= 32) {
      const int w = __shfl_sync(0xffffffffu, k.lt / 32, 0);
      g = w / G::TC;
      h = w % G::TC;
      slot = g * 32 + k.lt % 32;
    } else {
      g = 0;
      h = k.lt / G::L;
      slot = k.lt % G::L;
    }
    hb = h == 0 ? G::BC / 2 : G::BC - h;
    gl = G::L >= 32 ? h * 32 + k.lt % 32 : k.lt;
    col = k.S() + slot;
    tw = KField<N, NF>::tables();
  }
  __device__ __forceinline__ float2* edge() const { return KField<N, NF>::tables() + G::NTW; }
  __device__ __forceinline__ int kx() const { return slot / G::A + G::BR * (slot % G::A); }
  __device__ __forceinline__ void sync() const {
    group_sync<G::GT, G::T, NF * (G::T / G::GT)>(g + (NF > 1 ? f * (G::T / G::GT) : 0));
  }
};
// the twiddle tables, by all threads (ends with a CTA barrier)
template <int N, int NF = 1>
__device__ __forceinline__ void ktw_init() {
  using G = KGeo<N>;
  float2* t = KField<N, NF>::tables();
  for (int i = threadIdx.x; i < G::NTW; i += NF * G::T) {
    int k;  // exponent over N
    if (i < G::O_RT) k = 2 * (i / G::BR) * (i % G::BR);
    else if (i < G::O_C) k = 2 * ((i - G::O_RT) / G::A) * ((i - G::O_RT) % G::A);
    else if (i < G::O_CT) k = ((i - G::O_C) / G::BC) * ((i - G::O_C) % G::BC);
    else if (i < G::O_P) k = ((i - G::O_CT) / G::A) * ((i - G::O_CT) % G::A);
    else k = (i - G::O_P) / (G::A / 2) + G::BR * ((i - G::O_P) % (G::A / 2));
    t[i] = g_tw1024.v[k * (1024 / N)];
  }
  __syncthreads();
}

// B twiddles of a table row (16-byte aligned), two per load
template <int B>
__device__ __forceinline__ void kload_tw(float2 (&o)[B], const float2* w) {
#pragma unroll
  for (int k = 0; k < B; k += 2) {
    const float4 v = *reinterpret_cast<const float4*>(w + k);
    o[k] = make_float2(v.x, v.y);
    o[k + 1] = make_float2(v.z, v.w);
  }
}

// Forward row transforms: x[i BR + m] = pixel pair n0 + A m (n0 = hr NR + i) of row y -> half spectrum in the
// row's slots. Ends without a CTA barrier.
template <int N, int NF = 1>
__device__ __forceinline__ void krow_fwd(float2 (&x)[KGeo<N>::E]) {
  using G = KGeo<N>;
  const KRow<N, NF> t;
  constexpr int A = G::A, BR = G::BR;
  float2* row = t.row;
#pragma unroll
  for (int i = 0; i < G::NR; ++i) {
    float2 c[BR];
#pragma unroll
    for (int m = 0; m < BR; ++m) c[m] = x[i * BR + m];
    fft<BR, false>(c);
    const int n0 = t.h * G::NR + i;
    ktwiddle<BR, false>(c, t.tw + G::O_R + n0 * BR);
#pragma unroll
    for (int q = 0; q < BR; ++q) row[n0 + A * q] = c[q];
  }
  t.sync();
  float2 p[A], q[A];
#pragma unroll
  for (int j = 0; j < A; ++j) p[j] = row[A * t.h + j];
#pragma unroll
  for (int j = 0; j < A; ++j) q[j] = row[A * t.hb + j];
  fft<A, false>(p);
  fft<A, false>(q);
  float2 wp[A / 2], wq[A / 2];
  kload_tw<A / 2>(wp, t.tw + G::O_P + t.h * (A / 2));
  kload_tw<A / 2>(wq, t.tw + G::O_P + t.hb * (A / 2));
  if (t.h == 0) {
    unit0_swap<A>(p, q);
    p[0] = make_float2(p[0].x + p[0].y, p[0].x - p[0].y);  // (R[0], R[L])
    q[A - 1] = cconj(q[A - 1]);                            // K = L/2
  } else {
    k_post(p[0], q[A - 1], wp[0]);
  }
#pragma unroll
  for (int j = 1; j < A / 2; ++j) k_post(p[j], q[A - 1 - j], wp[j]);
#pragma unroll
  for (int j = 0; j < A / 2; ++j) k_post(q[j], p[A - 1 - j], wq[j]);
  if (t.h == 0) unit0_unswap<A>(p, q);
#pragma unroll
  for (int j = 0; j < A; ++j) row[A * t.h + j] = p[j];
#pragma unroll
  for (int j = 0; j < A; ++j) row[A * t.hb + j] = q[j];
}

// Inverse row transforms: half spectrum in the row's slots -> x (pixel pairs), unnormalised.
template <int N, int NF = 1>
__device__ __forceinline__ void krow_inv(float2 (&x)[KGeo<N>::E]) {
  using G = KGeo<N>;
  const KRow<N, NF> t;
  constexpr int A = G::A, BR = G::BR;
  float2* row = t.row;
  {
    float2 p[A], q[A];
#pragma unroll
    for (int j = 0; j < A; ++j) p[j] = row[A * t.h + j];
#pragma unroll
    for (int j = 0; j < A; ++j) q[j] = row[A * t.hb + j];
    float2 wp[A / 2], wq[A / 2];
    kload_tw<A / 2>(wp, t.tw + G::O_P + t.h * (A / 2));
    kload_tw<A / 2>(wq, t.tw + G::O_P + t.hb * (A / 2));
    if (t.h == 0) {
      unit0_swap<A>(p, q);
      p[0] = make_float2(p[0].x + p[0].y, p[0].x - p[0].y);
      q[A - 1] = cscale(cconj(q[A - 1]), 2.0f);
    } else {
      k_pre(p[0], q[A - 1], wp[0]);
    }
#pragma unroll
    for (int j = 1; j < A / 2; ++j) k_pre(p[j], q[A - 1 - j], wp[j]);
#pragma unroll
    for (int j = 0; j < A / 2; ++j) k_pre(q[j], p[A - 1 - j], wq[j]);
    if (t.h == 0) unit0_unswap<A>(p, q);
    fft<A, true>(p);
    fft<A, true>(q);
    ktwiddle<A, true>(p, t.tw + G::O_RT + t.h * A);
    ktwiddle<A, true>(q, t.tw + G::O_RT + t.hb * A);
#pragma unroll
    for (int j = 0; j < A; ++j) row[A * t.h + j] = p[j];
#pragma unroll
    for (int j = 0; j < A; ++j) row[A * t.hb + j] = q[j];
  }
  t.sync();
#pragma unroll
  for (int i = 0; i < G::NR; ++i) {
    float2 c[BR];
    const int n0 = t.h * G::NR + i;
#pragma unroll
    for (int q = 0; q < BR; ++q) c[q] = row[n0 + A * q];
    fft<BR, true>(c);
#pragma unroll
    for (int m = 0; m < BR; ++m) x[i * BR + m] = c[m];
  }
}

// Column transforms of the whole field with `f(p, q)` between them on the mode pairs of this thread's column:
// pairs (p[j], q[A-1-j]) at ky1 = hc + BC j and (q[j], p[A-1-j]) at ky1 = hcb + BC j, j < A/2, ky2 = H - ky1
// (H/2 for ky1 = 0). Called after a CTA barrier; with INV the inverse transform is left in the rows.
template <int N, bool INV, int NF = 1, class F>
__device__ __forceinline__ void kcol(F&& f) {
  using G = KGeo<N>;
  constexpr int A = G::A, BC = G::BC, SP = G::SP;
  const KCol<N, NF> t;
  float2* col = t.col;
#pragma unroll
  for (int i = 0; i < G::NC; ++i) {
    float2 c[BC];
    const int n0 = t.h * G::NC + i;
#pragma unroll
    for (int m = 0; m < BC; ++m) c[m] = col[(n0 + A * m) * SP];
    fft<BC, false>(c);
    ktwiddle<BC, false>(c, t.tw + G::O_C + n0 * BC);
#pragma unroll
    for (int q = 0; q < BC; ++q) col[(n0 + A * q) * SP] = c[q];
  }
  t.sync();
  {
    float2 p[A], q[A];
#pragma unroll
    for (int j = 0; j < A; ++j) p[j] = col[(A * t.h + j) * SP];
#pragma unroll
    for (int j = 0; j < A; ++j) q[j] = col[(A * t.hb + j) * SP];
    fft<A, false>(p);
    fft<A, false>(q);
    if (t.h == 0) unit0_swap<A>(p, q);
    f(t, p, q);
    if (!INV) return;
    if (t.h == 0) unit0_unswap<A>(p, q);
    fft<A, true>(p);
    fft<A, true>(q);
    ktwiddle<A, true>(p, t.tw + G::O_CT + t.h * A);
    ktwiddle<A, true>(q, t.tw + G::O_CT + t.hb * A);
#pragma unroll
    for (int j = 0; j < A; ++j) col[(A * t.h + j) * SP] = p[j];
#pragma unroll
    for (int j = 0; j < A; ++j) col[(A * t.hb + j) * SP] = q[j];
  }
  t.sync();
#pragma unroll
  for (int i = 0; i < G::NC; ++i) {
    float2 c[BC];
    const int n0 = t.h * G::NC + i;
#pragma unroll
    for (int q = 0; q < BC; ++q) c[q] = col[(n0 + A * q) * SP];
    fft<BC, true>(c);
#pragma unroll
    for (int m = 0; m < BC; ++m) col[(n0 + A * m) * SP] = c[m];
  }
}

// Run inter(y1, y2, ky1, ky2) on the thread's mode pairs of an interior column. The H/2 pairs of the packed edge
// column (slot 0, kx = 0 as A and kx = W/2 as B in Y = A + i B) are parked by their threads and handed one per
// lane to the last warps of the column group, edge(y1, y2, ky1, ky2), so that one or two warps run the edge code
// once instead of all TC warps for one lane each (64^2, 1216 chains: 5% of the sampler's instructions).
template <int N, class I, class X>
__device__ __forceinline__ void kpairs(const KCol<N>& t, float2 (&p)[KGeo<N>::A], float2 (&q)[KGeo<N>::A],
                                       I&& inter, X&& edge) {
  using G = KGeo<N>;
  constexpr int A = G::A;
  float2* e = t.edge();
  if (t.g == 0) {
    if (t.slot == 0) {
#pragma unroll
      for (int j = 0; j < A / 2; ++j) {
        e[2 * (t.h + G::BC * j)] = p[j];
        e[2 * (t.h + G::BC * j) + 1] = q[A - 1 - j];
        e[2 * (t.hb + G::BC * j)] = q[j];
        e[2 * (t.hb + G::BC * j) + 1] = p[A - 1 - j];
      }
    }
    t.sync();
  }
  if (t.slot != 0) {
#pragma unroll
    for (int j = 0; j < A / 2; ++j) {
      const int ky1 = t.h + G::BC * j;
      inter(p[j], q[A - 1 - j], ky1, j == 0 && t.h == 0 ? G::H / 2 : G::H - ky1);
    }
#pragma unroll
    for (int j = 0; j < A / 2; ++j) {
      const int ky1 = t.hb + G::BC * j;
      inter(q[j], p[A - 1 - j], ky1, G::H - ky1);
    }
  }
  if (t.g == 0) {
    const int ky1 = G::GT - 1 - t.gl;  // the group's last H/2 threads
    if (ky1 < G::H / 2) {
      float2 y1 = e[2 * ky1], y2 = e[2 * ky1 + 1];
      edge(y1, y2, ky1, ky1 == 0 ? G::H / 2 : G::H - ky1);
      e[2 * ky1] = y1;
      e[2 * ky1 + 1] = y2;
    }
    t.sync();
    if (t.slot == 0) {
#pragma unroll
      for (int j = 0; j < A / 2; ++j) {
        p[j] = e[2 * (t.h + G::BC * j)];
        q[A - 1 - j] = e[2 * (t.h + G::BC * j) + 1];
        q[j] = e[2 * (t.hb + G::BC * j)];
        p[A - 1 - j] = e[2 * (t.hb + G::BC * j) + 1];
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// pointwise updates on registers
// ---------------------------------------------------------------------------------------------
// t-draw (t_draw_staged): x[i BR + m], x[(i+1) BR + m] (i even) are the four pixels of group n / 2
template <int N, int NF = 1, bool DRAW = true>
__device__ __forceinline__ void kt_draw(float2 (&x)[KGeo<N>::E], const float2* __restrict__ aq,
                                        float sqrt_tau, uint32_t step, uint32_t chain, uint32_t k0, uint32_t k1,
                                        uint32_t stream) {
  using G = KGeo<N>;
  const KRow<N, NF> t;
  const float2* tab = aq + 2 * t.h * G::NR * G::H + t.y;
  const uint32_t grp = uint32_t(t.y * (G::W / 4) + t.h * (G::NR / 2));
#pragma unroll
  for (int a = 0; a < G::NR / 2; ++a)
#pragma unroll
    for (int m = 0; m < G::BR; ++m) {
      const int n = 2 * a + G::A * m;  // pixel pair relative to the thread's first
      const float2 c0 = __ldg(tab + (2 * n) * G::H), c1 = __ldg(tab + (2 * n + 1) * G::H);
      const float2 c2 = __ldg(tab + (2 * n + 2) * G::H), c3 = __ldg(tab + (2 * n + 3) * G::H);
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      if (DRAW) normals4(grp + uint32_t(n / 2), step, chain, stream, k0, k1, z);
      float2& p0 = x[2 * a * G::BR + m];
      float2& p1 = x[(2 * a + 1) * G::BR + m];
      p0.x = fmaf(c0.y, fmaf(c0.y, p0.x, sqrt_tau * z[0]), c0.x);
      p0.y = fmaf(c1.y, fmaf(c1.y, p0.y, sqrt_tau * z[1]), c1.x);
      p1.x = fmaf(c2.y, fmaf(c2.y, p1.x, sqrt_tau * z[2]), c2.x);
      p1.y = fmaf(c3.y, fmaf(c3.y, p1.y, sqrt_tau * z[3]), c3.x);
    }
}

// Wiener-filter t-update at level lambda (t_update_wf_staged)
template <int N, int NF = 1>
__device__ __forceinline__ void kt_update_wf(float2 (&x)[KGeo<N>::E],
                                             const float2* __restrict__ dn, float lt_, bool rhs) {
  using G = KGeo<N>;
  const KRow<N, NF> t;
  const float2* tab = dn + 2 * t.h * G::NR * G::H + t.y;
  const float g = rhs ? 0.0f : 1.0f, h = rhs ? lt_ : 1.0f;
#pragma unroll
  for (int i = 0; i < G::NR; ++i)
#pragma unroll
    for (int m = 0; m < G::BR; ++m) {
      const int n = i + G::A * m;
      const float2 c0 = __ldg(tab + (2 * n) * G::H), c1 = __ldg(tab + (2 * n + 1) * G::H);
      const float w0 = wf_weight(lt_, c0.y), w1 = wf_weight(lt_, c1.y);
      float2& v = x[i * G::BR + m];
      v.x = fmaf(w0, fmaf(-g, c0.x, v.x), h * c0.x);
      v.y = fmaf(w1, fmaf(-g, c1.x, v.y), h * c1.x);
    }
}

// right-hand side of the level-lambda Wiener equation, d / (N_bar + lambda tau) (rhs_row)
template <int N>
__device__ __forceinline__ void kt_rhs(float2 (&x)[KGeo<N>::E], const float2* __restrict__ dn,
                                       float lt_) {
  using G = KGeo<N>;
  const KRow<N> t;
  const float2* tab = dn + 2 * t.h * G::NR * G::H + t.y;
#pragma unroll
  for (int i = 0; i < G::NR; ++i)
#pragma unroll
    for (int m = 0; m < G::BR; ++m) {
      const int n = i + G::A * m;
      const float2 c0 = __ldg(tab + (2 * n) * G::H), c1 = __ldg(tab + (2 * n + 1) * G::H);
      const float nb0 = c0.y > 0.0f ? wf_rcp(c0.y) : wf_inf(), nb1 = c1.y > 0.0f ? wf_rcp(c1.y) : wf_inf();
      x[i * G::BR + m] = make_float2(c0.x / (nb0 + lt_), c1.x / (nb1 + lt_));
    }
}

// Mode coefficients by slot-order index (ky L + slot; kx = W/2 at H L + ky): the per-call table, or the per-band
// table of the hierarchical sampler with the band statistics (as TableCoef and BandCoef)
struct KTabCoef {
  static constexpr bool kBand = false;
  const float2* __restrict__ fg;
  __device__ __forceinline__ float2 m(int i) const { return __ldg(fg + i); }
  __device__ __forceinline__ void put(int, float, float) const {}
};
struct KBandCoef {
  static constexpr bool kBand = true;
  const float2* __restrict__ fg;
  const int2* __restrict__ bmap;
  const float2* cb;
  float2* buf;
  float n;
  __device__ __forceinline__ float2 m(int i) const {
    const int b = __ldg(bmap + i).x;
    return b < 0 ? __ldg(fg + i) : cb[b];
  }
  __device__ __forceinline__ void put(int i, float s2, float x2) const {
    const int pos = __ldg(bmap + i).y;
    if (pos >= 0) __stcg(buf + pos, make_float2(s2 * n, x2));
  }
};

// the s-draw of Alg. 1 on the thread's mode pairs (counter layout of s_draw_interior and s_draw_edge)
template <int N, class C>
__device__ __forceinline__ void ks_draw(const KCol<N>& t, float2 (&p)[KGeo<N>::A], float2 (&q)[KGeo<N>::A],
                                        const C& cf, uint32_t step, uint32_t chain, uint32_t k0, uint32_t k1) {
  using G = KGeo<N>;
  constexpr int L = G::L, HL = G::H * G::L;
  auto sq = [](float2 v) { return fmaf(v.x, v.x, v.y * v.y); };
  kpairs<N>(
      t, p, q,
      [&](float2& y1, float2& y2, int ky1, int ky2) {
        const int i1 = ky1 * L + t.slot, i2 = ky2 * L + t.slot;
        const float2 m1 = cf.m(i1), m2 = cf.m(i2);
        const uint32_t grp = uint32_t(t.kx() * (G::H / 2) + ky1);
        float z[4];
        normals4(grp, step, chain, 1u, k0, k1, z);
        y1 = make_float2(fmaf(m1.x, y1.x, m1.y * z[0]), fmaf(m1.x, y1.y, m1.y * z[1]));
        y2 = make_float2(fmaf(m2.x, y2.x, m2.y * z[2]), fmaf(m2.x, y2.y, m2.y * z[3]));
        if constexpr (C::kBand) {  // both modes have their mirror in the other half plane: weight 2
          float zb[4];
          normals4(grp, step, chain, 6u, k0, k1, zb);
          cf.put(i1, 2.0f * sq(y1), fmaf(zb[0], zb[0], zb[1] * zb[1]));
          cf.put(i2, 2.0f * sq(y2), fmaf(zb[2], zb[2], zb[3] * zb[3]));
        }
      },
      [&](float2& y1, float2& y2, int ky1, int ky2) {
        float z[4], zb[4] = {0.f, 0.f, 0.f, 0.f};
        normals4(uint32_t(ky1), step, chain, 1u, k0, k1, z);
        if constexpr (C::kBand) normals4(uint32_t(ky1), step, chain, 6u, k0, k1, zb);
        const float2 a1 = cf.m(ky1 * L), b1 = cf.m(HL + ky1);
        if (ky1 == 0) {  // the four self-conjugate modes, real with variance g^2
          const float2 a2 = cf.m(ky2 * L), b2 = cf.m(HL + ky2);
          constexpr float R2 = 1.41421356237309505f;
          y1 = make_float2(fmaf(a1.x, y1.x, R2 * a1.y * z[0]), fmaf(b1.x, y1.y, R2 * b1.y * z[2]));
          y2 = make_float2(fmaf(a2.x, y2.x, R2 * a2.y * z[1]), fmaf(b2.x, y2.y, R2 * b2.y * z[3]));
          if constexpr (C::kBand) {  // one real degree of freedom each
            cf.put(0, y1.x * y1.x, zb[0] * zb[0]);
            cf.put(HL, y1.y * y1.y, zb[2] * zb[2]);
            cf.put(ky2 * L, y2.x * y2.x, zb[1] * zb[1]);
            cf.put(HL + ky2, y2.y * y2.y, zb[3] * zb[3]);
          }
        } else {
          const float2 y2c = cconj(y2);
          const float2 Am = cscale(cadd(y1, y2c), 0.5f);
          const float2 Bm = cmul_mi(cscale(csub(y1, y2c), 0.5f));
          const float2 Ap = make_float2(fmaf(a1.x, Am.x, a1.y * z[0]), fmaf(a1.x, Am.y, a1.y * z[1]));
          const float2 Bp = make_float2(fmaf(b1.x, Bm.x, b1.y * z[2]), fmaf(b1.x, Bm.y, b1.y * z[3]));
          y1 = cadd(Ap, cmul_i(Bp));
          y2 = cadd(cconj(Ap), cmul_i(cconj(Bp)));
          if constexpr (C::kBand) {  // (ky1, 0) and (ky1, W/2) with their mirrors at H - ky1: weight 2
            cf.put(ky1 * L, 2.0f * sq(Ap), fmaf(zb[0], zb[0], zb[1] * zb[1]));
            cf.put(HL + ky1, 2.0f * sq(Bp), fmaf(zb[2], zb[2], zb[3] * zb[3]));
          }
        }
      });
}

// Wiener-filter s-update at level lambda with its residual bookkeeping (s_update_wf_parked): P in slot order
// (pks), previous iterate prev[ky L + slot]; returns the thread's share of the residual sum
template <int N>
__device__ __forceinline__ float ks_update_wf(const KCol<N>& t, float2 (&p)[KGeo<N>::A], float2 (&q)[KGeo<N>::A],
                                               const float* __restrict__ pks, float lt_, float2* __restrict__ prev,
                                               bool cmp, bool store) {
  using G = KGeo<N>;
  constexpr int L = G::L, HL = G::H * G::L;
  constexpr float INV_N = 1.0f / float(G::H * G::W);
  const float inv_lt = cmp ? 1.0f / lt_ : 0.0f;
  float acc = 0.0f;
  auto wres = [&](float P, float dre, float dim) -> float {
    const float g = fmaf(P, inv_lt, 1.0f);
    return fmaf(dre, dre, dim * dim) * (g * g);
  };
  auto fcoef = [&](float P) { return wf_fdiv(P, P + lt_) * INV_N; };
  kpairs<N>(
      t, p, q,
      [&](float2& y1, float2& y2, int ky1, int ky2) {
        const int i1 = ky1 * L + t.slot, i2 = ky2 * L + t.slot;
        const float P1 = __ldg(pks + i1), P2 = __ldg(pks + i2);
        y1 = cscale(y1, fcoef(P1));
        y2 = cscale(y2, fcoef(P2));
        if (cmp) {
          const float2 o1 = prev[i1], o2 = prev[i2];
          acc += 2.0f * (wres(P1, y1.x - o1.x, y1.y - o1.y) + wres(P2, y2.x - o2.x, y2.y - o2.y));
        }
        if (store) {
          prev[i1] = y1;
          prev[i2] = y2;
        }
      },
      [&](float2& y1, float2& y2, int ky1, int ky2) {
        const float Pa1 = __ldg(pks + ky1 * L), Pb1 = __ldg(pks + HL + ky1);
        const float fa1 = fcoef(Pa1), fb1 = fcoef(Pb1);
        if (ky1 == 0) {  // the four self-conjugate modes
          const float Pa2 = __ldg(pks + ky2 * L), Pb2 = __ldg(pks + HL + ky2);
          y1 = make_float2(fa1 * y1.x, fb1 * y1.y);
          y2 = make_float2(fcoef(Pa2) * y2.x, fcoef(Pb2) * y2.y);
          if (cmp) {
            const float2 o1 = prev[0], o2 = prev[ky2 * L];
            acc += wres(Pa1, y1.x - o1.x, 0.f) + wres(Pb1, y1.y - o1.y, 0.f) + wres(Pa2, y2.x - o2.x, 0.f) +
                   wres(Pb2, y2.y - o2.y, 0.f);
          }
        } else {
          const float2 y2c = cconj(y2);
          const float2 Am = cscale(cscale(cadd(y1, y2c), 0.5f), fa1);
          const float2 Bm = cscale(cmul_mi(cscale(csub(y1, y2c), 0.5f)), fb1);
          y1 = cadd(Am, cmul_i(Bm));
          y2 = cadd(cconj(Am), cmul_i(cconj(Bm)));
          if (cmp) {
            const float2 o1 = prev[ky1 * L], o2c = cconj(prev[ky2 * L]);
            const float2 oA = cscale(cadd(o1, o2c), 0.5f);
            const float2 oB = cmul_mi(cscale(csub(o1, o2c), 0.5f));
            // modes ky1 and H - ky1 of each edge column have equal magnitude: weight 2
            acc += 2.0f * (wres(Pa1, Am.x - oA.x, Am.y - oA.y) + wres(Pb1, Bm.x - oB.x, Bm.y - oB.y));
          }
        }
        if (store) {
          prev[ky1 * L] = y1;
          prev[ky2 * L] = y2;
        }
      });
  return acc;
}

// the thread's share of sum_k P^2 |V|^2 over the full spectrum (p2_power)
template <int N>
__device__ __forceinline__ float ks_p2(const KCol<N>& t, float2 (&p)[KGeo<N>::A], float2 (&q)[KGeo<N>::A],
                                        const float* __restrict__ pks) {
  using G = KGeo<N>;
  constexpr int L = G::L, HL = G::H * G::L;
  float acc = 0.0f;
  auto p2 = [](float P, float re, float im) -> float { return fmaf(P * re, P * re, (P * im) * (P * im)); };
  kpairs<N>(
      t, p, q,
      [&](float2& y1, float2& y2, int ky1, int ky2) {
        acc += 2.0f * (p2(__ldg(pks + ky1 * L + t.slot), y1.x, y1.y) + p2(__ldg(pks + ky2 * L + t.slot), y2.x, y2.y));
      },
      [&](float2& y1, float2& y2, int ky1, int ky2) {
        if (ky1 == 0) {
          acc += p2(__ldg(pks), y1.x, 0.f) + p2(__ldg(pks + HL), y1.y, 0.f) + p2(__ldg(pks + ky2 * L), y2.x, 0.f) +
                 p2(__ldg(pks + HL + ky2), y2.y, 0.f);
        } else {
          const float2 y2c = cconj(y2);
          const float2 Am = cscale(cadd(y1, y2c), 0.5f);
          const float2 Bm = cmul_mi(cscale(csub(y1, y2c), 0.5f));
          acc += 2.0f * (p2(__ldg(pks + ky1 * L), Am.x, Am.y) + p2(__ldg(pks + HL + ky1), Bm.x, Bm.y));
        }
      });
  return acc;
}

// ---------------------------------------------------------------------------------------------
// field input and output
// ---------------------------------------------------------------------------------------------
// the thread's pixel pairs of a row-major [H][W] image (nullptr: zeros), through the field buffer so that the
// loads coalesce; NC false: an image that another CTA wrote during this launch
template <int N, int NF = 1, bool NC = true>
__device__ __forceinline__ void kload(float2 (&x)[KGeo<N>::E], const float* src) {
  using G = KGeo<N>;
  if (src == nullptr) {
#pragma unroll
    for (int e = 0; e < G::E; ++e) x[e] = make_float2(0.f, 0.f);
    return;
  }
  const KField<N, NF> k;
  for (int e = k.lt; e < G::H * G::L; e += G::T)
    k.S()[(e / G::L) * G::SP + e % G::L] =
        NC ? __ldg(reinterpret_cast<const float2*>(src) + e) : __ldcg(reinterpret_cast<const float2*>(src) + e);
  __syncthreads();
  const KRow<N, NF> t;
  const float2* row = t.row + t.h * G::NR;
#pragma unroll
  for (int i = 0; i < G::NR; ++i)
#pragma unroll
    for (int m = 0; m < G::BR; ++m) x[i * G::BR + m] = row[i + G::A * m];
  __syncthreads();
}
// x to an image of element type ot (CTA barriers on both sides of the copy)
template <int N, int NF = 1>
__device__ __forceinline__ void kstore(const float2 (&x)[KGeo<N>::E], void* out, int ot) {
  using G = KGeo<N>;
  {
    const KRow<N, NF> t;
    float2* row = t.row + t.h * G::NR;
#pragma unroll
    for (int i = 0; i < G::NR; ++i)
#pragma unroll
      for (int m = 0; m < G::BR; ++m) row[i + G::A * m] = x[i * G::BR + m];
  }
  __syncthreads();
  const KField<N, NF> k;
#pragma unroll 4
  for (int e = k.lt; e < G::H * G::L; e += G::T) {
    const float2 v = k.S()[(e / G::L) * G::SP + e % G::L];
    if (ot == kOutF32) __stcs(reinterpret_cast<float2*>(out) + e, v);
    else store_pair(out, e, v, ot);
  }
  __syncthreads();
}

// Sampler sweeps d0 .. d1 - 1 of a chain from the state in x. Per sweep: t-draw, forward rows, column transforms
// around the s-draw, inverse rows; post() after the column barrier (the band draw), emit(m) after sample m has been stored to
// out + m H W elements (CTA barriers before and after the store).
template <int N, class C, class Post, class Emit>
__device__ __forceinline__ void ksweeps(float2 (&x)[KGeo<N>::E], const float2* __restrict__ aq,
                                        const C& cf, float sqrt_tau, uint32_t step0, uint32_t chain, uint32_t k0,
                                        uint32_t k1, int d0, int d1, int burn_in, int thin, void* out, int ot,
                                        Post&& post, Emit&& emit) {
  using G = KGeo<N>;
  const int eb = out_elem_bytes(ot);
  for (int done = d0; done < d1;) {
    const uint32_t step = step0 + uint32_t(done);
    kt_draw<N>(x, aq, sqrt_tau, step, chain, k0, k1, 0u);
    krow_fwd<N>(x);
    __syncthreads();
    kcol<N, true>([&](const KCol<N>& t, float2 (&p)[G::A], float2 (&q)[G::A]) { ks_draw<N>(t, p, q, cf, step, chain, k0, k1); });
    __syncthreads();
    post();
    krow_inv<N>(x);
    ++done;
    if (done > burn_in && (done - burn_in) % thin == 0) {
      const long long m = (done - burn_in) / thin - 1;
      kstore<N>(x, static_cast<char*>(out) + m * (G::H * G::W) * eb, ot);
      emit(m);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Balanced chains. With one CTA per chain, a few chains more than fit at once cost another whole round (200 shear
// pairs on 152 SMs: two rounds of 22.9 us a sweep). Here as many CTAs as are resident take equal shares of all chains'
// sweeps, laid end to end: CTA i runs sweeps [i W / R, (i + 1) W / R) of the W in all. A share starts and ends inside a
// chain. The CTA runs the start of its last chain first and hands the state over, then its whole chains, and the rest
// of its first chain last, from the state that CTA i - 1 handed over. A share is at least as long as a chain, so a chain has at
// most two parts, and a CTA comes to the second part after as many sweeps of its own as the first part has, or one less (shares
// differ by a sweep): it waits for that sweep and for the difference of the two CTAs' paces over the first part, and no longer.
// The wait is bounded (kawait_polls; cooperative launch: all CTAs are resident). Measured at 128^2, us per sweep of all
// chains: 200 shear pairs 45.8 -> 30.8; scalar 350 chains 27 -> 20.4, 1000 chains 59.0 -> 57.8.
// ---------------------------------------------------------------------------------------------
struct KBalance {
  int shares;         // R: CTAs of the launch; 0: one CTA per chain
  float* slot;        // [R][slot_floats] states handed over
  int slot_floats;
  unsigned int* flag; // [R] 1 once slot i is complete; zeroed before the launch
  int* err;           // set to WF_ERR_TIMEOUT when a wait gives up; zeroed before the launch
};
// part `s` of CTA `i`: sweeps [d0, d1) of chain c; save: hand the state over; load: start from the state handed over
struct KPart {
  long long c;
  int d0, d1;
  bool load, save;
};
// false: no such part
WF_HD bool kpart_of(int i, int s, int shares, long long n_chains, int n_sweeps, KPart* p) {
  if (shares == 0) {
    *p = KPart{i, 0, n_sweeps, false, false};
    return s == 0;
  }
  const long long S = n_sweeps, W = n_chains * S;
  // i W / R without overflow: W may be close to 2^62
  const long long q = W / shares, r = W % shares;
  const long long a = q * i + r * i / shares, b = q * (i + 1) + r * (i + 1) / shares;
  const int head = int(b % S), tail = int(a % S);
  if (head > 0) {
    if (s == 0) {
      *p = KPart{b / S, 0, head, false, true};
      return true;
    }
    --s;
  }
  const long long first = (a + S - 1) / S, whole = b / S - first;
  if (s < whole) {
    *p = KPart{first + s, 0, n_sweeps, false, false};
    return true;
  }
  *p = KPart{a / S, tail, n_sweeps, true, false};
  return s == whole && tail > 0;
}
// the CTA's part s, formed by one thread in shared memory (read from there where it is needed: the sweeps' registers
// are full); CTA barriers on both sides
struct KPartShared {
  KPart p;
  int more;
};
__device__ __forceinline__ KPartShared& kpart_shared() {
  __shared__ KPartShared sp;
  return sp;
}
__device__ __forceinline__ bool knext_part(int s, const KBalance& bal, int n_chains, int n_sweeps) {
  KPartShared& sp = kpart_shared();
  __syncthreads();
  if (threadIdx.x == 0) sp.more = kpart_of(blockIdx.x, s, bal.shares, n_chains, n_sweeps, &sp.p);
  __syncthreads();
  return sp.more != 0;
}
// the state in slot i is complete (all threads of the CTA have stored; called by all)
__device__ __forceinline__ void kpublish(const KBalance& b, int i) {
  __syncthreads();
  if (threadIdx.x == 0)
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(b.flag + i), "r"(1u) : "memory");
}
// Polls after which a wait for a first part of `sweeps` sweeps gives up: a few seconds, and on top of them time in
// proportion to the part, since two CTAs' paces may differ by a share of it (a poll is an L2 round trip, 0.3 us at least, so a
// sweep adds 0.3 ms, several times what the sweep itself takes). A fixed limit of a few seconds gave up on
// a difference of 1% over parts of some ten million sweeps.
WF_HD long long kawait_polls(int sweeps) { return (1LL << 22) + 1024LL * sweeps; }
// waits for slot i, the state after `sweeps` sweeps; false: gave up
__device__ __forceinline__ bool kawait(const KBalance& b, int i, int sweeps) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    unsigned int v = 0;
    const long long most = kawait_polls(sweeps);
    for (long long it = 0; v == 0 && it < most; ++it)
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(b.flag + i) : "memory");
    if (v == 0) atomicExch(b.err, 7);  // WF_ERR_TIMEOUT
    s_ok = v != 0;
  }
  __syncthreads();
  return s_ok != 0;
}

// CTA i's chain in a launch of one CTA per chain: nothing is handed over, and the compiler sees that
struct KWhole {
  long long c;
  int d1;
  static constexpr int d0 = 0;
  static constexpr bool load = false, save = false;
};
// f(part) for the CTA's parts in order, until one returns false. BAL is a template parameter: with run-time parts the
// 64-register kernels spill 28 (sampler) to 230 bytes, 1.5% of the band sampler's time
template <bool BAL, class F>
__device__ __forceinline__ void kparts(const KBalance& bal, int n_chains, int n_sweeps, F&& f) {
  if constexpr (BAL) {
    const volatile KPart& p = kpart_shared().p;
    for (int s = 0; knext_part(s, bal, n_chains, n_sweeps); ++s)
      if (!f(p)) return;
  } else {
    f(KWhole{blockIdx.x, n_sweeps});
  }
}

// resident CTAs the kernels are compiled for: 64 registers a thread at 128^2 (two fields of 67 KB and 16 warps an
// SM); at 64^2 and 32^2 five and ten CTAs with up to 96 registers measured as fast as eight and sixteen with 64
// (the SM is bound by dispatch), and faster for a single chain (64^2: 4.5 -> 4.1 us per sweep)
template <int N>
constexpr int kcore_min_ctas() { return N == 64 ? 5 : (N == 32 ? 10 : 2); }

template <int N, class Part>
__device__ __forceinline__ bool ksample_part(const SampleArgs& a, const KBalance& bal, const Part& p) {
  using G = KGeo<N>;
  float2 x[G::E];
  if (p.load) {
    if (!kawait(bal, blockIdx.x - 1, p.d0)) return false;
    kload<N, 1, false>(x, bal.slot + (blockIdx.x - 1LL) * bal.slot_floats);
  } else {
    kload<N>(x, a.init_s ? a.init_s + p.c * a.init_stride : nullptr);
  }
  ksweeps<N>(x, a.aq, KTabCoef{a.fg}, a.sc->sqrt_tau, a.step0, a.chain0 + uint32_t(p.c), a.key0, a.key1, p.d0, p.d1,
             a.burn_in, a.thin,
             reinterpret_cast<char*>(a.out) + p.c * a.n_samples * (long long)(G::H * G::W) * out_elem_bytes(a.out_dtype),
             a.out_dtype, [] {}, [](long long) {});
  if (p.save) {
    kstore<N>(x, bal.slot + (long long)blockIdx.x * bal.slot_floats, kOutF32);
    kpublish(bal, blockIdx.x);
  }
  return true;
}
template <int N, bool BAL>
__global__ void __launch_bounds__(KGeo<N>::T, kcore_min_ctas<N>()) k_msample(const __grid_constant__ SampleArgs a,
                                                                            const __grid_constant__ KBalance bal) {
  if (a.sc->status != 0) return;  // uniform over the grid
  ktw_init<N>();
  kparts<BAL>(bal, a.n_chains, a.n_sweeps, [&](const auto& p) { return ksample_part<N>(a, bal, p); });
}

// every image's chain from its s_W (images whose set-up failed write nothing)
template <int N>
__global__ void __launch_bounds__(KGeo<N>::T, kcore_min_ctas<N>()) k_mbsample(BSampleArgs a) {
  using G = KGeo<N>;
  const GBField fd = a.fields[blockIdx.x];
  if (a.sc[blockIdx.x].status != 0) return;  // uniform over the CTA
  ktw_init<N>();
  float2 x[G::E];
  kload<N>(x, fd.out_wf);
  ksweeps<N>(x, fd.aq, KTabCoef{fd.fg}, a.sc[blockIdx.x].sqrt_tau, 0u, fd.chain, fd.key0, fd.key1, 0, a.n_samples, 0, 1,
             fd.out_samples, kOutF32, [] {}, [](long long) {});
}

// Band-power draw after the s-draw (every mode's statistics stored and visible to the CTA): each warp takes four
// bins at a time, each lane summing its lane-strided entries (16 loads in flight), then a fixed shuffle tree per
// bin: the same order every run; P_b = S_b / X_b and band_coef(P_b) to shared memory (as band_update).
template <int T>
__device__ __forceinline__ void kband_update(const float2* __restrict__ buf, const int* __restrict__ off, int n_bins,
                                             float2* cb, float* Pb, float tau, float inv_n) {
  constexpr int NG = T / 32, KB = 4, U = 4;
  const int lane = threadIdx.x % 32;
  for (int b0 = threadIdx.x / 32; b0 < n_bins; b0 += NG * KB) {
    int o0[KB], len[KB], most = 0;
    float S[KB], X[KB];
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int b = b0 + k * NG;
      o0[k] = b < n_bins ? off[b] : 0;
      len[k] = b < n_bins ? off[b + 1] - o0[k] : 0;
      most = len[k] > most ? len[k] : most;
      S[k] = X[k] = 0.0f;
    }
    for (int j = lane; j < most; j += U * 32) {
      float2 v[KB][U];
#pragma unroll
      for (int k = 0; k < KB; ++k)
#pragma unroll
        for (int u = 0; u < U; ++u)
          v[k][u] = j + 32 * u < len[k] ? __ldcg(buf + o0[k] + j + 32 * u) : make_float2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < KB; ++k)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          S[k] += v[k][u].x;
          X[k] += v[k][u].y;
        }
    }
#pragma unroll
    for (int k = 0; k < KB; ++k) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        S[k] += __shfl_xor_sync(0xffffffffu, S[k], d);
        X[k] += __shfl_xor_sync(0xffffffffu, X[k], d);
      }
      const int b = b0 + k * NG;
      if (lane == 0 && b < n_bins) {
        const float P = X[k] > 0.0f ? S[k] / X[k] : 0.0f;
        Pb[b] = P;
        cb[b] = band_coef(P, tau, inv_n);
      }
    }
  }
}

// The hierarchical sampler: the per-band draw coefficients [n_bins] float2 and band powers [n_bins] floats follow
// the field; one bin-ordered statistics buffer per CTA. The band draw runs after the column barrier; its
// results are read after the next one.
template <int N, bool BAL>
__global__ void __launch_bounds__(KGeo<N>::T, kcore_min_ctas<N>()) k_mband(const __grid_constant__ SampleArgs a,
                                                                          const __grid_constant__ KBalance bal) {
  using G = KGeo<N>;
  if (a.sc->status != 0) return;  // uniform over the grid
  ktw_init<N>();
  float2* cb = reinterpret_cast<float2*>(kfield_smem() + G::SMEM);
  float* Pb = reinterpret_cast<float*>(cb + a.n_bins);
  const float tau = float(a.sc->tau);
  constexpr float NPIX = float(G::H * G::W);
  // one statistics buffer per CTA
  float2* buf = a.band_buf + (long long)blockIdx.x * (a.n_bins > 0 ? a.band_off[a.n_bins] : 0);
  kparts<BAL>(bal, a.n_chains, a.n_sweeps, [&](const auto& p) {
    float2 x[G::E];
    const float* P = a.P0;  // the part's band powers
    if (p.load) {
      if (!kawait(bal, blockIdx.x - 1, p.d0)) return false;
      P = bal.slot + (blockIdx.x - 1LL) * bal.slot_floats + G::H * G::W;
    }
    for (int b = threadIdx.x; b < a.n_bins; b += G::T) {
      const float v = __ldcg(P + b);
      Pb[b] = v;
      cb[b] = band_coef(v, tau, 1.0f / NPIX);
    }
    __syncthreads();
    if (p.load) kload<N, 1, false>(x, bal.slot + (blockIdx.x - 1LL) * bal.slot_floats);
    else kload<N>(x, a.init_s ? a.init_s + p.c * a.init_stride : nullptr);
    float* outP = a.out_P ? a.out_P + p.c * a.n_samples * (long long)a.n_bins : nullptr;
    ksweeps<N>(x, a.aq, KBandCoef{a.fg, a.band_map, cb, buf, NPIX}, a.sc->sqrt_tau, a.step0, a.chain0 + uint32_t(p.c),
               a.key0, a.key1, p.d0, p.d1, a.burn_in, a.thin,
               reinterpret_cast<char*>(a.out) +
                   p.c * a.n_samples * (long long)(G::H * G::W) * out_elem_bytes(a.out_dtype),
               a.out_dtype, [&] { kband_update<G::T>(buf, a.band_off, a.n_bins, cb, Pb, tau, 1.0f / NPIX); },
               [&](long long m) {
                 if (outP)
                   for (int b = threadIdx.x; b < a.n_bins; b += G::T) outP[m * a.n_bins + b] = Pb[b];
               });
    if (p.save) {
      float* slot = bal.slot + (long long)blockIdx.x * bal.slot_floats;
      kstore<N>(x, slot, kOutF32);  // its barriers order the last band draw before the reads below
      for (int b = threadIdx.x; b < a.n_bins; b += G::T) slot[G::H * G::W + b] = Pb[b];
      kpublish(bal, blockIdx.x);
    }
    return true;
  });
}

// ---------------------------------------------------------------------------------------------
// Spin-2 sampler: the two shear components are the two fields of a CTA of 2 T threads. Before the draw both
// components' unit modes are parked in their own slots; component 0's threads then draw the pairs led by the
// first unit for both components, component 1's those led by the second (rotation into E and B, the two scalar
// draws, rotation back, as spin2_interior and spin2_edge), and each thread reloads its own.
// ---------------------------------------------------------------------------------------------
template <int N, bool DRAW>
__device__ __forceinline__ void ks_draw_spin2(const KCol<N, 2>& t, float2 (&p)[KGeo<N>::A], float2 (&q)[KGeo<N>::A],
                                              const float2* __restrict__ fgE, const float2* __restrict__ fgB,
                                              uint32_t step, uint32_t chain, uint32_t k0, uint32_t k1) {
  using G = KGeo<N>;
  constexpr int A = G::A, SP = G::SP, L = G::L, HL = G::H * G::L;
  float2* own = t.col;
#pragma unroll
  for (int j = 0; j < A; ++j) own[(A * t.h + j) * SP] = p[j];
#pragma unroll
  for (int j = 0; j < A; ++j) own[(A * t.hb + j) * SP] = q[j];
  __syncthreads();
  float2* c0 = reinterpret_cast<float2*>(kfield_smem());
  float2* c1 = reinterpret_cast<float2*>(kfield_smem() + G::FIELD_BYTES);
  const int lead = t.f == 0 ? t.h : t.hb, mate = t.f == 0 ? t.hb : t.h;
  if (t.slot != 0) {
#pragma unroll
    for (int j = 0; j < A / 2; ++j) {
      const int ky1 = lead + G::BC * j, ky2 = ky1 == 0 ? G::H / 2 : G::H - ky1;
      const int i1 = (A * lead + j) * SP + t.slot, i2 = (A * mate + A - 1 - j) * SP + t.slot;
      float2 a1 = c0[i1], b1 = c1[i1], a2 = c0[i2], b2 = c1[i2];
      const uint32_t grp = uint32_t(t.kx() * (G::H / 2) + ky1);
      float zE[4] = {0.f, 0.f, 0.f, 0.f}, zB[4] = {0.f, 0.f, 0.f, 0.f};
      if (DRAW) {
        normals4(grp, step, chain, 1u, k0, k1, zE);
        normals4(grp, step, chain, 9u, k0, k1, zB);
      }
      const int m1 = ky1 * L + t.slot, m2 = ky2 * L + t.slot;
      float c, s;
      ks_rot<N>(ky1, t.kx(), c, s);
      spin2_mode(a1, b1, c, s, __ldg(fgE + m1), __ldg(fgB + m1), zE[0], zE[1], zB[0], zB[1]);
      ks_rot<N>(ky2, t.kx(), c, s);
      spin2_mode(a2, b2, c, s, __ldg(fgE + m2), __ldg(fgB + m2), zE[2], zE[3], zB[2], zB[3]);
      c0[i1] = a1;
      c1[i1] = b1;
      c0[i2] = a2;
      c1[i2] = b2;
    }
  }
  // the packed edge column (slot 0): one of the component's H/4 pairs per thread of the group's last warp
  const int ep = G::GT - 1 - t.gl;
  if (t.g == 0 && ep < G::H / 4) {
    const int j = ep % (A / 2), eh = ep / (A / 2), ehb = eh == 0 ? G::BC / 2 : G::BC - eh;
    const int el = t.f == 0 ? eh : ehb, em = t.f == 0 ? ehb : eh;  // first and second unit of the pair
    const int ky1 = el + G::BC * j, ky2 = ky1 == 0 ? G::H / 2 : G::H - ky1;
    const int i1 = (A * el + j) * SP, i2 = (A * em + A - 1 - j) * SP;
    float2 y1a = c0[i1], y2a = c0[i2], y1b = c1[i1], y2b = c1[i2];
    float zE[4] = {0.f, 0.f, 0.f, 0.f}, zB[4] = {0.f, 0.f, 0.f, 0.f};
    if (DRAW) {
      normals4(uint32_t(ky1), step, chain, 1u, k0, k1, zE);
      normals4(uint32_t(ky1), step, chain, 9u, k0, k1, zB);
    }
    if (ky1 == 0) {
      // four real modes, each on k = 0 or a Nyquist line: no rotation, real draws with variance g^2
      constexpr float R2 = 1.41421356237309505f;
      auto upd = [&](float& a, float& b, int i, float ze, float zb) {
        const float2 mE = __ldg(fgE + i), mB = __ldg(fgB + i);
        a = fmaf(mE.x, a, R2 * mE.y * ze);
        b = fmaf(mB.x, b, R2 * mB.y * zb);
      };
      upd(y1a.x, y1b.x, 0, zE[0], zB[0]);
      upd(y1a.y, y1b.y, HL, zE[2], zB[2]);
      upd(y2a.x, y2b.x, ky2 * L, zE[1], zB[1]);
      upd(y2a.y, y2b.y, HL + ky2, zE[3], zB[3]);
    } else {
      // unpack both components: A = value at (ky1, 0), B = value at (ky1, W/2)
      float2 A1 = cscale(cadd(y1a, cconj(y2a)), 0.5f), B1 = cmul_mi(cscale(csub(y1a, cconj(y2a)), 0.5f));
      float2 A2 = cscale(cadd(y1b, cconj(y2b)), 0.5f), B2 = cmul_mi(cscale(csub(y1b, cconj(y2b)), 0.5f));
      float c, s;
      ks_rot<N>(ky1, 0, c, s);
      spin2_mode(A1, A2, c, s, __ldg(fgE + ky1 * L), __ldg(fgB + ky1 * L), zE[0], zE[1], zB[0], zB[1]);
      ks_rot<N>(ky1, G::W / 2, c, s);
      spin2_mode(B1, B2, c, s, __ldg(fgE + HL + ky1), __ldg(fgB + HL + ky1), zE[2], zE[3], zB[2], zB[3]);
      y1a = cadd(A1, cmul_i(B1));
      y2a = cadd(cconj(A1), cmul_i(cconj(B1)));
      y1b = cadd(A2, cmul_i(B2));
      y2b = cadd(cconj(A2), cmul_i(cconj(B2)));
    }
    c0[i1] = y1a;
    c0[i2] = y2a;
    c1[i1] = y1b;
    c1[i2] = y2b;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < A; ++j) p[j] = own[(A * t.h + j) * SP];
#pragma unroll
  for (int j = 0; j < A; ++j) q[j] = own[(A * t.hb + j) * SP];
}

template <int N>
constexpr int kspin2_smem() { return 2 * KGeo<N>::FIELD_BYTES + KGeo<N>::NTW * 8; }

// DRAW false (the shear Wiener filter): the draws are left out, their scales are zero
template <int N, bool DRAW, bool BAL>
__global__ void __launch_bounds__(2 * KGeo<N>::T, N == 64 ? 3 : (N == 32 ? 6 : 1)) k_mspin2(
    const __grid_constant__ Spin2Args a, const __grid_constant__ KBalance bal) {
  using G = KGeo<N>;
  if (a.sc->status != 0) return;  // uniform over the grid
  ktw_init<N, 2>();
  constexpr long long n = G::H * G::W;
  const int eb = out_elem_bytes(a.out_dtype);
  kparts<BAL>(bal, a.n_chains, a.n_sweeps, [&](const auto& p) {
    float2 x[G::E];
    if (p.load) {
      if (!kawait(bal, blockIdx.x - 1, p.d0)) return false;
      kload<N, 2, false>(x, bal.slot + (blockIdx.x - 1LL) * bal.slot_floats + (threadIdx.x / G::T) * n);
    } else {
      kload<N, 2>(x, a.init_s ? a.init_s + p.c * a.init_stride + (threadIdx.x / G::T) * n : nullptr);
    }
    const uint32_t chain = a.chain0 + uint32_t(p.c);
    for (int done = p.d0; done < p.d1;) {
      const uint32_t step = a.step0 + uint32_t(done);
      kt_draw<N, 2, DRAW>(x, a.aq2 + (threadIdx.x / G::T) * n, a.sc->sqrt_tau, step, chain, a.key0, a.key1,
                          8u * (threadIdx.x / G::T));
      krow_fwd<N, 2>(x);
      __syncthreads();
      kcol<N, true, 2>([&](const KCol<N, 2>& t, float2 (&u)[G::A], float2 (&v)[G::A]) {
        ks_draw_spin2<N, DRAW>(t, u, v, a.fgE, a.fgB, step, chain, a.key0, a.key1);
      });
      __syncthreads();
      krow_inv<N, 2>(x);
      ++done;
      if (done > a.burn_in && (done - a.burn_in) % a.thin == 0) {
        const long long m = (done - a.burn_in) / a.thin - 1;
        kstore<N, 2>(x, reinterpret_cast<char*>(a.out) + ((p.c * a.n_samples + m) * 2 + threadIdx.x / G::T) * n * eb,
                     a.out_dtype);
      }
    }
    if (p.save) {
      kstore<N, 2>(x, bal.slot + (long long)blockIdx.x * bal.slot_floats + (threadIdx.x / G::T) * n, kOutF32);
      kpublish(bal, blockIdx.x);
    }
    return true;
  });
}

// ---------------------------------------------------------------------------------------------
// Wiener filter
// ---------------------------------------------------------------------------------------------
// Sums over the CTA and schedule decisions: every thread leaves its FP32 partial sum in shared memory, one warp adds
// them in FP64 (T/32 per lane in order, then a fixed shuffle tree) and its first lane decides. With every thread
// running the FP64 sum, division and square root, a check kept the SM's two FP64 lanes busy for several thousand
// cycles.
struct KSolveState {
  double tot;
  float ltau;
  int lev, k, status;
};
template <int N>
constexpr int ksolve_smem() { return KGeo<N>::SMEM + KGeo<N>::T * 4 + int(sizeof(KSolveState)); }
template <int N>
__device__ __forceinline__ float* kpart() { return reinterpret_cast<float*>(kfield_smem() + KGeo<N>::SMEM); }
template <int N>
__device__ __forceinline__ KSolveState* kstate() { return reinterpret_cast<KSolveState*>(kpart<N>() + KGeo<N>::T); }
// sum of the partial sums by one whole warp, valid in every lane
template <int N>
__device__ __forceinline__ double kwarp_total() {
  const float* part = kpart<N>();
  const int lane = threadIdx.x % 32;
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < KGeo<N>::T / 32; ++w) s += double(part[32 * w + lane]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// ||S N_lambda^-1 d||^2 of one cooling level, valid in the first warp (ends with a CTA barrier)
template <int N>
__device__ __forceinline__ double klevel_norm(const float2* __restrict__ dn, const float* __restrict__ pks, float ltau) {
  using G = KGeo<N>;
  float2 x[G::E];
  kt_rhs<N>(x, dn, ltau);
  krow_fwd<N>(x);
  __syncthreads();
  kcol<N, false>([&](const KCol<N>& t, float2 (&p)[G::A], float2 (&q)[G::A]) {
    kpart<N>()[threadIdx.x] = ks_p2<N>(t, p, q, pks);
  });
  __syncthreads();
  const double tot = threadIdx.x < 32 ? kwarp_total<N>() * (1.0 / double(G::H * G::W)) : 0.0;
  __syncthreads();
  return tot;
}

// The G -> 0 iteration with lambda-cooling (solve_sweeps): x holds the starting iterate on entry and the last
// one on exit; P and prev in slot order. Returns the wf_status (0 converged, 5 not converged, 6 non-finite).
template <int N>
__device__ __forceinline__ int ksolve_sweeps(float2 (&x)[KGeo<N>::E], const float2* __restrict__ dn,
                                             const float* __restrict__ pks, const Scalars& sc,
                                             const double* __restrict__ bnorm2, float2* prev, double tol, double eta,
                                             double level_tol, int max_iter, int level_max, int check, int& it,
                                             double& rho, bool rhs) {
  using G = KGeo<N>;
  int lev = 0, k = 0, status = 1;
  float ltau = float(sc.lam0 * sc.tau);
  const int last_level = sc.n_levels - 1;
  it = 0;
  rho = -1.0;
  while (true) {
    ++k;
    ++it;
    const bool cmp = (k % check == 0) && k >= 2;
    const bool store = ((k + 1) % check == 0);
    kt_update_wf<N>(x, dn, ltau, rhs);
    krow_fwd<N>(x);
    __syncthreads();
    kcol<N, true>([&](const KCol<N>& t, float2 (&p)[G::A], float2 (&q)[G::A]) {
      const float acc = ks_update_wf<N>(t, p, q, pks, ltau, prev, cmp, store);
      if (cmp) kpart<N>()[threadIdx.x] = acc;
    });
    __syncthreads();
    // the last warp decides while the others start the inverse rows; the next sweep needs the decision
    if (cmp && threadIdx.x >= G::T - 32) {
      const double tot = kwarp_total<N>() * double(G::H * G::W);
      if (threadIdx.x == G::T - 32) {
        // rho = sqrt(tot / bn) against the tolerances, without the division and the root
        const double bn = bnorm2[rhs ? 0 : lev], ref = bn > 0.0 ? bn : 1.0;
        KSolveState d{tot, ltau, lev, k, 1};
        if (residual_nonfinite(tot, ref)) {
          d.status = 6;  // non-finite residual
        } else if (lev < last_level) {
          if (tot < level_tol * level_tol * ref || k >= level_max) {
            ++d.lev;
            d.ltau = float(level_lambda(sc, d.lev, eta) * sc.tau);
            d.k = 0;
          }
        } else if (tot < tol * tol * ref) {
          d.status = 0;
        }
        d.tot = tot / ref;
        *kstate<N>() = d;
      }
      __syncwarp();
    }
    krow_inv<N>(x);
    if (cmp) {
      __syncthreads();
      const KSolveState& d = *kstate<N>();
      rho = d.tot;
      lev = d.lev;
      ltau = d.ltau;
      k = d.k;
      status = d.status;
    }
    if (status == 1 && it >= max_iter) status = 5;  // not converged
    if (status != 1) {
      rho = rho >= 0.0 ? sqrt(rho) : rho;  // of the last check (-1: never measured)
      return status;
    }
  }
}

// level norms of the problems blockIdx.y (pixel tables dn + y H W), one CTA per level
template <int N>
__global__ void __launch_bounds__(KGeo<N>::T) k_mbnorm(BnormArgs a) {
  const Scalars sc = *a.sc;
  const int lev = blockIdx.x;
  if (sc.status != 0 || lev >= sc.n_levels) return;
  ktw_init<N>();
  const double v = klevel_norm<N>(a.dn + blockIdx.y * (KGeo<N>::H * KGeo<N>::W), a.Pk,
                                  float(level_lambda(sc, lev, a.eta) * sc.tau));
  if (threadIdx.x == 0) a.bnorm2[blockIdx.y * kMaxLevels + lev] = v;
}

// one problem per CTA (alone on its SM: up to 128 registers a thread): problem f on dn, out + f H W, bnorm2 + f kMaxLevels,
// prev + f H W/2 and st + f; init_s only for a single problem. MANY false: one problem (with run-time offsets its sweeps
// take 0.8% longer)
template <int N, bool MANY>
__global__ void __launch_bounds__(KGeo<N>::T, 1) k_msolve(SolveArgs a) {
  using G = KGeo<N>;
  const Scalars sc = *a.sc;
  if (sc.status != 0) return;
  ktw_init<N>();
  float2 x[G::E];
  kload<N>(x, a.init_s);
  int it = 0;
  double rho = -1.0;
  const int f = MANY ? blockIdx.x : 0;
  const int status = ksolve_sweeps<N>(x, a.dn + f * (G::H * G::W), a.Pk, sc, a.bnorm2 + f * kMaxLevels,
                                      a.prev + f * (G::H * G::W / 2), a.tol, a.eta, a.level_tol, a.max_iter,
                                      a.level_max, a.check, it, rho, a.rhs_mode != 0);
  kstore<N>(x, a.out + f * (G::H * G::W), kOutF32);
  if (threadIdx.x == 0) {
    a.st[f].status = status;
    a.st[f].iters = it;
    a.st[f].resid = rho;
  }
}

// level norms of every image of a class: CTA (image, y) computes levels y, y + kLevelCtas, ...
template <int N>
__global__ void __launch_bounds__(KGeo<N>::T, kcore_min_ctas<N>()) k_mblevels(BSolveArgs a) {
  const int f = blockIdx.x;
  const Scalars sc = a.sc[f];
  if (sc.status != 0 || int(blockIdx.y) >= sc.n_levels) return;  // uniform over the CTA
  const GBField fd = a.fields[f];
  ktw_init<N>();
  for (int lev = blockIdx.y; lev < sc.n_levels; lev += gridDim.y) {
    const double v = klevel_norm<N>(fd.dn, fd.Pk, float(level_lambda(sc, lev, a.eta) * sc.tau));
    if (threadIdx.x == 0) a.bnorm[f * kMaxLevels + lev] = v;
  }
}

// one image per CTA: cooled solve from s = 0 with the level norms of k_mblevels, s_W out
template <int N>
__global__ void __launch_bounds__(KGeo<N>::T, kcore_min_ctas<N>()) k_mbsolve(BSolveArgs a) {
  using G = KGeo<N>;
  const int f = a.order ? a.order[blockIdx.x] : int(blockIdx.x);
  const GBField fd = a.fields[f];
  const Scalars sc = a.sc[f];
  if (sc.status != 0) {  // uniform over the CTA
    if (threadIdx.x == 0) a.res[fd.item] = BatchResult{-1.0, 0, sc.status};
    return;
  }
  ktw_init<N>();
  float2 x[G::E];
  kload<N>(x, nullptr);
  int it = 0;
  double rho = -1.0;
  const int status = ksolve_sweeps<N>(x, fd.dn, fd.Pk, sc, a.bnorm + f * kMaxLevels, fd.prev, a.tol, a.eta,
                                      a.level_tol, a.max_iter, a.level_max, a.check, it, rho, false);
  kstore<N>(x, fd.out_wf, kOutF32);
  if (threadIdx.x == 0) a.res[fd.item] = BatchResult{rho, it, status};
}

}  // namespace wf
