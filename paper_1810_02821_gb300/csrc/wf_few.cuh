// Few large fields with the least latency: every CTA holds one block of rows and one block of columns of one field for the
// whole launch. The transforms, draws and updates are those of the global-memory kernels (wf_global.cuh, natural table
// orders), and a sweep has the same two phases, but
//   - a CTA's pixel and mode tables (and the Wiener filter's previous iterate) stay in its shared memory;
//   - the normals of a phase depend on no state: they are drawn between arriving at the barrier before it and waiting;
//   - at up to 256^2 (XCluster) a field is one thread-block cluster and its half spectrum never leaves shared
//     memory: the last pass of a row transform stores each value into the CTA that owns its column, the last pass of a
//     column transform into the CTA that owns its row (runs of 8 columns, 64 bytes, at a time), so the next phase starts
//     with local loads, and a hardware cluster barrier takes the place of the counter in global memory;
//   - at 512^2 and 1024^2, and for 256^2 spin-2 pairs (XGrid), the half spectrum stays in global memory (L2)
//     and the barrier is the bounded one of the global-memory kernels: a cluster's 16 SMs would be too few.
// What bounds it: the instructions and latencies of two transforms, their exchanges and the draws at one or two warps a
// scheduler, and (XGrid) two L2 round trips and two barriers.
// Measured against the global-memory kernels, us per sweep: 128^2 one chain 6.5 -> 3.8, Wiener filter 6.9 -> 3.9; 256^2
// 7.1 -> 5.3 and 7.5 -> 5.3; 14 chains of 256^2 (two CTAs an SM) 10.2 -> 7.4; 512^2 8.8 -> 7.0 and 9.2 -> 7.7; 1024^2 13.1 ->
// 10.7 and 13.9 -> 11.3 (the Wiener filter's pixel table alone is 8 MB a sweep from L2); one spin-2 pair of 256^2 8.1 -> 6.0.
#pragma once

#include "wf_gspin2.cuh"

namespace wf {

__device__ __forceinline__ uint32_t x_addr(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }
// the address in CTA `rank` of the cluster that corresponds to this CTA's shared-memory address
__device__ __forceinline__ uint32_t x_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void x_store(uint32_t addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}

// How the CTAs of a field exchange the half spectrum: CTA b of a field owns rows RB b .. and columns CB b .. of each of
// its NC components. row(comp, yl) and col(comp): accessors as ZRow and ZCols; arrive(), wait(): a barrier of the field's
// CTAs (XGrid samplers: of the grid) in two parts, stores before the arrival visible after the wait, false after a timeout.
template <int N, int NC_>
struct XCluster {
  static constexpr int NC = NC_, RB = 16, C = N / RB, CB = N / 2 / C;
  static constexpr bool CLUSTER = true;
  // received columns [NC][H][CB] (components 4 float2 banks apart) and rows [NC][RB][RS] (the rows of one remote store in
  // different banks), float2
  static constexpr int RS = N / 2 + 8, CS = N * CB + 4, O_ROW = NC * CS, SIZE = O_ROW + NC * RB * RS;
  static_assert(C <= 16 && CB == 8, "geometry");
  float2* buf;
  int rank;
  struct Row {
    const float2* row;
    uint32_t col;  // of entry 0 of this row in a CTA's received columns
    __device__ __forceinline__ float2 ld(int kx) const { return row[kx]; }
    __device__ __forceinline__ void st(int kx, float2 v) const {
      x_store(x_map(col + uint32_t(kx % CB) * 8u, uint32_t(kx / CB)), v);
    }
  };
  struct Cols {
    const float2* p;
    uint32_t row;  // of this CTA's first column in row 0 of a CTA's received rows
    struct Col {
      const float2* p;
      uint32_t row;
      int y0;
      __device__ __forceinline__ float2 ld(int dy) const { return p[dy * CB]; }
      __device__ __forceinline__ void st(int dy, float2 v) const {
        const int y = y0 + dy;
        x_store(x_map(row + uint32_t(y % RB) * (RS * 8u), uint32_t(y / RB)), v);
      }
    };
    __device__ __forceinline__ Col at(int y0, int c) const { return Col{p + y0 * CB + c, row + uint32_t(c) * 8u, y0}; }
  };
  __device__ __forceinline__ Row row(int comp, int yl) const {
    return Row{buf + O_ROW + (comp * RB + yl) * RS, x_addr(buf + comp * CS + (rank * RB + yl) * CB)};
  }
  __device__ __forceinline__ Cols col(int comp) const {
    return Cols{buf + comp * CS, x_addr(buf + O_ROW + comp * RB * RS + rank * CB)};
  }
  __device__ __forceinline__ void arrive() const { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
  __device__ __forceinline__ bool wait() const {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    return true;
  }
};

template <int N, int NC_>
struct XGrid {
  static constexpr int NC = NC_, RB = 8 / NC, C = N / RB, CB = N / 2 / C;
  static constexpr bool CLUSTER = false;
  static constexpr int SIZE = 0;
  static_assert(CB == 4 / NC, "geometry");
  float2* Z;  // of the field: [NC][H][W/2]
  int rank;
  GridBar* bar;
  unsigned int count;  // CTAs that share the barrier
  unsigned int target;
  __device__ __forceinline__ ZRow row(int comp, int yl) const {
    return ZRow{Z + ((long long)comp * N + rank * RB + yl) * (N / 2)};
  }
  __device__ __forceinline__ ZCols<N> col(int comp) const {
    return ZCols<N>{Z + (long long)comp * N * (N / 2) + rank * CB};
  }
  __device__ __forceinline__ void arrive() {
    __syncthreads();
    target += count;
    if (threadIdx.x == 0) grid_arrive(bar);
  }
  __device__ __forceinline__ bool wait() const {
    __shared__ int s_ok;
    if (threadIdx.x == 0) s_ok = grid_wait(bar, target);
    __syncthreads();
    return s_ok != 0;
  }
};

template <int N, class X>
struct FewGeo {
  using G = GGeo<N, X::NC * X::RB>;
  static constexpr int T = G::T, H = N, W = N;
  // float2 offsets: the exchange buffers after the transforms' (spin-2: and the edge pairs of a second component), pixel
  // tables [NC][RB][W]; the sampler's mode tables [NC] x ([H][CB] and, in the first CTA, that of kx = W/2 [H]), or the
  // filter's previous iterate [H][CB], P [H][CB] and P at kx = W/2 (floats), and the CTAs' partial sums [2][16] (doubles)
  static constexpr int O_X = G::SMEM_F2 + (X::NC - 1) * H, O_PIX = O_X + X::SIZE, O_MODE = O_PIX + X::NC * X::RB * W;
  static constexpr int MS = H * X::CB + H, O_P = O_MODE + H * X::CB, O_PART = O_P + MS / 2;
  static constexpr int SMEM_SAMPLE = (O_MODE + X::NC * MS) * 8, SMEM_SOLVE = (O_PART + 32) * 8;
  static constexpr int MIN_CTAS = N == 1024 ? 1 : 512 / T;
  static_assert(X::NC * X::CB == G::CB && H / 2 <= 2 * T && O_X % 2 == 0 && O_PIX % 2 == 0, "geometry");
};

// scalar fields; a.mode 0 (chain blockIdx.x / C) or, with SOLVE, 1 (field blockIdx.x / C, each at its own pace)
template <int N, class X, bool SOLVE>
__global__ void __launch_bounds__(FewGeo<N, X>::T, FewGeo<N, X>::MIN_CTAS) k_few(const __grid_constant__ GlobalArgs a) {
  using K = FewGeo<N, X>;
  using G = typename K::G;
  constexpr int H = N, W = N, CB = X::CB, RB = X::RB, T = K::T, C = X::C, WH = W / 2 + 1, GR = X::NC * X::RB;
  const int rank = blockIdx.x % C, f = blockIdx.x / C;
  if (a.sc->status != 0) {  // uniform over the grid
    if (SOLVE && rank == 0 && threadIdx.x == 0) a.st[f].status = a.sc->status;
    return;
  }
  gtab_init<N, GR>();
  float2* s = gsmem();
  {
    const float4* src = reinterpret_cast<const float4*>(
        (SOLVE ? a.dn + (long long)f * H * W : a.aq) + rank * RB * W);
    for (int i = threadIdx.x; i < RB * W / 2; i += T) reinterpret_cast<float4*>(s + K::O_PIX)[i] = __ldg(src + i);
    float* P = reinterpret_cast<float*>(s + K::O_P);
    for (int i = threadIdx.x; i < H * CB; i += T) {
      const int at = (i / CB) * WH + rank * CB + i % CB;
      if (SOLVE) P[i] = __ldg(a.Pk + at);
      else s[K::O_MODE + i] = __ldg(a.fg + at);
    }
    if (rank == 0)
      for (int i = threadIdx.x; i < H; i += T) {
        if (SOLVE) P[H * CB + i] = __ldg(a.Pk + i * WH + W / 2);
        else s[K::O_MODE + H * CB + i] = __ldg(a.fg + i * WH + W / 2);
      }
  }
  X ex = [&] {
    if constexpr (X::CLUSTER) return X{s + K::O_X, rank};
    else return X{a.Z + (long long)f * H * (W / 2), rank, SOLVE ? a.bar + f : a.bar, SOLVE ? unsigned(C) : gridDim.x, 0u};
  }();
  __syncthreads();
  if constexpr (X::CLUSTER) {  // every CTA has started: its shared memory may be stored to
    ex.arrive();
    ex.wait();
  }
  const int yl = threadIdx.x / G::TR, y = rank * RB + yl;
  const auto zrow = ex.row(0, yl);
  const auto zcol = ex.col(0);
  const float4* pix = reinterpret_cast<const float4*>(s + K::O_PIX + yl * W);
  auto tab = [&](int e) { return pix[e]; };
  auto fg = [&](int ky, int kx) {
    const float2* m = s + K::O_MODE;
    return kx == W / 2 ? m[H * CB + ky] : m[ky * CB + kx % CB];
  };
  auto Pk = [&](int ky, int kx) {
    const float* P = reinterpret_cast<const float*>(s + K::O_P);
    return kx == W / 2 ? P[H * CB + ky] : P[ky * CB + kx % CB];
  };
  auto prev = [&](int ky, int kx) -> float2& { return s[K::O_MODE + ky * CB + kx % CB]; };

  if constexpr (!SOLVE) {
    constexpr int NG = G::E / 2, NE = (H / 2 + T - 1) / T;  // groups of four normals a thread needs in a phase; edge pairs
    const float sqrt_tau = a.sc->sqrt_tau;
    const uint32_t chain = a.chain0 + uint32_t(f);
    float z[NG][4], ze[NE][4];
    auto set = [](float (&v)[4], const float (&w)[4]) {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = w[j];
    };
    auto draw_pixels = [&](int done) {
#pragma unroll
      for (int i = 0; i < NG; ++i)
        normals4(pixel_group<N>(y, i), a.step0 + uint32_t(done), chain, 0u, a.key0, a.key1, z[i]);
    };
    auto draw_modes = [&](int done) {
      const int c = threadIdx.x % CB, h = threadIdx.x / CB, hb = h == 0 ? G::BC / 2 : G::BC - h;
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const int ky = i < NG / 2 ? h + G::BC * i : hb + G::BC * (i - NG / 2);
        normals4(uint32_t((rank * CB + c) * (H / 2) + ky), a.step0 + uint32_t(done), chain, 1u, a.key0, a.key1, z[i]);
      }
      if (rank == 0)
#pragma unroll
        for (int i = 0; i < NE; ++i)
          if (threadIdx.x + T * i < H / 2)
            normals4(threadIdx.x + T * i, a.step0 + uint32_t(done), chain, 1u, a.key0, a.key1, ze[i]);
    };
    float2 x[G::E];
    grow_load<N>(x, a.init_s ? a.init_s + f * a.init_stride + (long long)y * W : nullptr);
    draw_pixels(0);
    for (int done = 0;;) {
      pixel_update<N>(0, x, tab, [&](int i, float (&v)[4]) { set(v, z[i]); }, sqrt_tau, 0.f, 0, 0.f);
      grow_fwd<N, GR>(x, zrow);
      ex.arrive();
      draw_modes(done);
      if (!ex.wait()) return;
      gcol_update<N, GR>(
          0, zcol, rank * CB, fg, Pk, prev, [&](int i, uint32_t, float (&v)[4]) { set(v, z[i]); },
          [&](int ky, float (&v)[4]) {
            if constexpr (NE == 1) set(v, ze[0]);
            else set(v, ky < T ? ze[0] : ze[NE - 1]);
          },
          0.f, false, false);
      ex.arrive();
      ++done;
      if (done < a.n_sweeps) draw_pixels(done);
      if (!ex.wait()) return;
      grow_inv<N, GR>(zrow, x);
      if (done > a.burn_in && (done - a.burn_in) % a.thin == 0) {
        const long long ms = (done - a.burn_in) / a.thin - 1;
        grow_store<N>(x, a.out, ((long long)f * a.n_samples + ms) * H + y, a.out_dtype);
      }
      if (done == a.n_sweeps) return;  // no CTA stores to another after the last barrier
    }
  } else {
    // Wiener filter with lambda-cooling; every CTA follows the same schedule (k_global): decisions on the sum of the CTAs'
    // residual parts (XCluster: in rank order; XGrid: atomics)
    __shared__ double red[T];
    __shared__ GSolveState dec;
    double* part = reinterpret_cast<double*>(s + K::O_PART);
    const int last_level = a.sc->n_levels - 1;
    int lev = 0, it = 0, k = 0, status = 1, parity = 0;
    float ltau = float(a.sc->lam0 * a.sc->tau);
    double rho2 = -1.0;
    float2 x[G::E];
    grow_load<N>(x, nullptr);
    auto none = [](int, float (&)[4]) {};
    while (true) {
      pixel_update<N>(1, x, tab, none, 0.f, ltau, a.rhs_mode, 0.f);
      grow_fwd<N, GR>(x, zrow);
      ex.arrive();
      ++k;
      ++it;
      const bool cmp = (k % a.check == 0) && k >= 2;
      const bool store = ((k + 1) % a.check == 0);
      if (!ex.wait()) return;
      const float mine = gcol_update<N, GR>(
          1, zcol, rank * CB, fg, Pk, prev, [](int, uint32_t, float (&)[4]) {}, none, ltau, cmp, store);
      if (cmp) {
        const double v = gblock_sum<T>(double(mine), red);
        if constexpr (X::CLUSTER) {
          if (threadIdx.x < C)
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(x_map(x_addr(part + parity * C + rank), threadIdx.x)),
                         "d"(v)
                         : "memory");
        } else if (threadIdx.x == 0) {
          atomicAdd(a.acc + 2 * f + parity, v);
        }
      }
      ex.arrive();
      if (!ex.wait()) return;
      if (cmp) {
        if (threadIdx.x < 32) {
          double tot = 0.0;
          if constexpr (X::CLUSTER) {
            if (threadIdx.x < C) tot = part[parity * C + threadIdx.x];
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
          } else {
            tot = __ldcg(a.acc + 2 * f + parity);
            if (rank == 0 && threadIdx.x == 0) a.acc[2 * f + (parity ^ 1)] = 0.0;  // next check's accumulator
          }
          if (threadIdx.x == 0) {
            tot *= double(H) * W;
            const double bn = a.bnorm2[a.rhs_mode ? 0 : f * kMaxLevels + lev], ref = bn > 0.0 ? bn : 1.0;
            GSolveState d{tot, ltau, lev, k, 1};
            if (residual_nonfinite(tot, ref)) {
              d.status = 6;  // non-finite residual
            } else if (lev < last_level) {
              if (tot < a.level_tol * a.level_tol * ref || k >= a.level_max) {
                ++d.lev;
                d.ltau = float(level_lambda(*a.sc, d.lev, a.eta) * a.sc->tau);
                d.k = 0;
              }
            } else if (tot < a.tol * a.tol * ref) {
              d.status = 0;
            }
            if (rank == 0) d.rho2 = tot / ref;
            dec = d;
          }
        }
        __syncthreads();
        parity ^= 1;
        rho2 = dec.rho2;
        lev = dec.lev;
        ltau = dec.ltau;
        k = dec.k;
        status = dec.status;
      }
      if (status == 1 && it >= a.max_iter) status = 5;  // not converged
      grow_inv<N, GR>(zrow, x);
      if (status != 1) break;
    }
    grow_store<N>(x, a.out, (long long)f * H + y, kOutF32);
    if (rank == 0 && threadIdx.x == 0) {
      a.st[f].status = status;
      a.st[f].iters = it;
      a.st[f].resid = rho2 >= 0.0 ? sqrt(rho2) : rho2;
    }
  }
}

// Spin-2 pairs: both components of a pair in the same CTAs. Rows: the first half of a CTA holds component 0, the second
// component 1; columns: vector = component + 2 column, thread tid on vector tid % VH + VH (tid / (T / passes)) with VH = 8
// (XCluster: a half-warp holds 8 vectors and two units) or 4, so that the components are in neighbouring lanes.
// DRAW false (the shear Wiener filter): the draws are left out, their scales are zero.
template <int N, class X, bool DRAW>
__global__ void __launch_bounds__(FewGeo<N, X>::T, FewGeo<N, X>::MIN_CTAS) k_few2(const __grid_constant__ GSpin2Args ga) {
  using K = FewGeo<N, X>;
  using G = typename K::G;
  const Spin2Args& a = ga.s;
  constexpr int H = N, W = N, CB = X::CB, RB = X::RB, T = K::T, C = X::C, WH = W / 2 + 1, GR = X::NC * X::RB;
  constexpr long long n = (long long)H * W;
  static_assert(X::NC == 2, "spin-2");
  const int rank = blockIdx.x % C, f = blockIdx.x / C;
  if (a.sc->status != 0) return;  // uniform over the grid
  gtab_init<N, GR>();
  float2* s = gsmem();
  for (int i = threadIdx.x; i < RB * W; i += T)
    reinterpret_cast<float4*>(s + K::O_PIX)[i] =
        __ldg(reinterpret_cast<const float4*>(a.aq2 + (i / (RB * W / 2)) * n + rank * RB * W) + i % (RB * W / 2));
  for (int i = threadIdx.x; i < H * CB; i += T) {
    const int at = (i / CB) * WH + rank * CB + i % CB;
    s[K::O_MODE + i] = __ldg(a.fgE + at);
    s[K::O_MODE + K::MS + i] = __ldg(a.fgB + at);
  }
  if (rank == 0)
    for (int i = threadIdx.x; i < H; i += T) {
      s[K::O_MODE + H * CB + i] = __ldg(a.fgE + i * WH + W / 2);
      s[K::O_MODE + K::MS + H * CB + i] = __ldg(a.fgB + i * WH + W / 2);
    }
  X ex = [&] {
    if constexpr (X::CLUSTER) return X{s + K::O_X, rank};
    else return X{ga.Z + 2LL * f * H * (W / 2), rank, ga.bar, gridDim.x, 0u};
  }();
  __syncthreads();
  if constexpr (X::CLUSTER) {  // every CTA has started: its shared memory may be stored to
    ex.arrive();
    ex.wait();
  }
  // rows
  const int rc = threadIdx.x / (T / 2), yl = threadIdx.x % (T / 2) / G::TR, y = rank * RB + yl;
  const auto zrow = ex.row(rc, yl);
  const float4* pix = reinterpret_cast<const float4*>(s + K::O_PIX + (rc * RB + yl) * W);
  auto tab = [&](int e) { return pix[e]; };
  // columns
  constexpr int VH = G::CB < 8 ? G::CB : 8, TV = T / (G::CB / VH);
  const int vec = threadIdx.x % VH + VH * (threadIdx.x / TV), cc = vec & 1, cl = vec / 2, col = rank * CB + cl;
  const int h = threadIdx.x % TV / VH;
  const auto zcol = ex.col(cc);
  auto mode = [&](const float2* m, int ky, int kx) { return kx == W / 2 ? m[H * CB + ky] : m[ky * CB + kx % CB]; };

  constexpr int NG = G::E / 2;
  static_assert(NG == G::A && H / 2 <= T, "a phase needs as many groups of normals in rows and columns");
  const float sqrt_tau = a.sc->sqrt_tau;
  const uint32_t chain = a.chain0 + uint32_t(f);
  float z[NG][4] = {}, ze[2][4] = {};
  auto set = [](float (&v)[4], const float (&w)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = w[j];
  };
  auto draw_pixels = [&](int done) {
    if constexpr (DRAW) {
#pragma unroll
      for (int i = 0; i < NG; ++i)
        normals4(pixel_group<N>(y, i), a.step0 + uint32_t(done), chain, 8u * uint32_t(rc), a.key0, a.key1, z[i]);
    }
  };
  auto draw_modes = [&](int done) {
    if constexpr (DRAW) {
      const uint32_t step = a.step0 + uint32_t(done);
      const int lead = cc == 0 ? h : (h == 0 ? G::BC / 2 : G::BC - h);  // the unit whose pairs this lane draws
#pragma unroll
      for (int j = 0; j < NG / 2; ++j) {
        const uint32_t g = uint32_t(col * (H / 2) + lead + G::BC * j);
        normals4(g, step, chain, 1u, a.key0, a.key1, z[2 * j]);
        normals4(g, step, chain, 9u, a.key0, a.key1, z[2 * j + 1]);
      }
      if (rank == 0 && threadIdx.x < H / 2) {
        normals4(threadIdx.x, step, chain, 1u, a.key0, a.key1, ze[0]);
        normals4(threadIdx.x, step, chain, 9u, a.key0, a.key1, ze[1]);
      }
    }
  };
  float2 x[G::E];
  grow_load<N>(x, a.init_s ? a.init_s + f * a.init_stride + rc * n + (long long)y * W : nullptr);
  draw_pixels(0);
  for (int done = 0;;) {
    pixel_update<N>(DRAW ? 0 : 4, x, tab, [&](int i, float (&v)[4]) { set(v, z[i]); }, sqrt_tau, 0.f, 0, 0.f);
    grow_fwd<N, GR>(x, zrow);
    ex.arrive();
    draw_modes(done);
    if (!ex.wait()) return;
    gcol_spin2<N, GR, DRAW>(
        zcol.at((G::E / 8) * h, cl), s + vec * G::VCOL, s + G::O_EDGE, rank == 0, col, h,
        [&](int ky, int kx) { return mode(s + K::O_MODE, ky, kx); },
        [&](int ky, int kx) { return mode(s + K::O_MODE + K::MS, ky, kx); },
        [&](int j, uint32_t, float (&zE)[4], float (&zB)[4]) {
          set(zE, z[2 * j]);
          set(zB, z[2 * j + 1]);
        },
        [&](int, float (&zE)[4], float (&zB)[4]) {
          set(zE, ze[0]);
          set(zB, ze[1]);
        });
    ex.arrive();
    ++done;
    if (done < a.n_sweeps) draw_pixels(done);
    if (!ex.wait()) return;
    grow_inv<N, GR>(zrow, x);
    if (done > a.burn_in && (done - a.burn_in) % a.thin == 0) {
      const long long m = (done - a.burn_in) / a.thin - 1;
      grow_store<N>(x, a.out, ((f * a.n_samples + m) * 2 + rc) * H + y, a.out_dtype);
    }
    if (done == a.n_sweeps) return;  // no CTA stores to another after the last barrier
  }
}

}  // namespace wf
