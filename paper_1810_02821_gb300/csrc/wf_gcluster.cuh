// Few fields of 128^2 and 256^2 with the least latency: each field in one thread-block cluster of 8 or 16 CTAs. The
// transforms, draws and updates are those of the global-memory kernels (wf_global.cuh, 16 rows and 8 columns per CTA,
// natural table orders), and a sweep has the same two phases, but
//   - the half spectrum never leaves shared memory: the last pass of a row transform stores each value into the CTA that
//     owns its column, the last pass of a column transform into the CTA that owns its row (distributed shared memory;
//     runs of 8 columns, 64 bytes, at a time), so the next phase starts with local loads;
//   - a hardware cluster barrier takes the place of the counter in global memory;
//   - the normals of a phase depend on no state: they are drawn between arriving at the barrier before it and waiting;
//   - a CTA's pixel and mode tables (and the Wiener filter's previous iterate) stay in its shared memory.
// What bounds it: the instructions and latencies of two transforms, their exchanges and the draws at one (128^2) or two
// warps a scheduler. Measured against the fields in global memory, us per sweep: 128^2 one chain 6.3 -> 3.7, Wiener
// filter 6.8 -> 4.0; 256^2 one chain 7.0 -> 5.2, Wiener filter 7.5 -> 5.5; 14 chains of 256^2 (two CTAs an SM) 10.2 -> 7.4.
#pragma once

#include "wf_global.cuh"

namespace wf {

template <int N>
struct GCl {
  static constexpr int RB = 16, C = N / RB;  // rows per CTA, CTAs per cluster
  using G = GGeo<N, RB>;
  static constexpr int H = N, W = N, LR = N / 2, T = G::T, CB = G::CB, WH = W / 2 + 1;
  static constexpr int RS = LR + 8;  // stride of a received row: the rows of one remote store fall in different banks
  // float2 offsets: received columns [H][CB], received rows [RB][RS], pixel table [RB][W]; then the sampler's mode table
  // [H][CB] and, in the first CTA, that of kx = W/2 [H], or the filter's previous iterate [H][CB], P [H][CB] and P at
  // kx = W/2 (floats), and the CTAs' partial sums [2][C] of the residual (doubles)
  static constexpr int O_COL = G::SMEM_F2, O_ROW = O_COL + H * CB, O_PIX = O_ROW + RB * RS, O_MODE = O_PIX + RB * W;
  static constexpr int O_P = O_MODE + H * CB, O_PART = O_P + (H * CB + H) / 2;
  static constexpr int SMEM_SAMPLE = (O_MODE + H * CB + H) * 8, SMEM_SOLVE = (O_PART + 2 * C) * 8;
  static_assert(C <= 16 && C * CB == LR && H / 2 <= T && O_PIX % 2 == 0, "geometry");
};

__device__ __forceinline__ uint32_t gc_addr(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }
// the address in CTA `rank` of the cluster that corresponds to this CTA's shared-memory address
__device__ __forceinline__ uint32_t gc_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void gc_store(uint32_t addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
// all threads of the cluster: stores before the arrival, also remote ones, are visible after the wait
__device__ __forceinline__ void gc_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void gc_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// row y of the CTA: read from the received rows, stored to the columns' owners
template <int N>
struct GClRow {
  const float2* row;
  uint32_t col;  // of entry 0 of this row in a CTA's received columns
  __device__ __forceinline__ float2 ld(int kx) const { return row[kx]; }
  __device__ __forceinline__ void st(int kx, float2 v) const {
    gc_store(gc_map(col + uint32_t(kx % GCl<N>::CB) * 8u, uint32_t(kx / GCl<N>::CB)), v);
  }
};
// the CTA's columns: read from the received columns, stored to the rows' owners
template <int N>
struct GClCols {
  const float2* col;
  uint32_t row;  // of this CTA's first column in row 0 of a CTA's received rows
  struct Col {
    const float2* p;
    uint32_t row;
    int y0;
    __device__ __forceinline__ float2 ld(int dy) const { return p[dy * GCl<N>::CB]; }
    __device__ __forceinline__ void st(int dy, float2 v) const {
      using K = GCl<N>;
      const int y = y0 + dy;
      gc_store(gc_map(row + uint32_t(y % K::RB) * (K::RS * 8u), uint32_t(y / K::RB)), v);
    }
  };
  __device__ __forceinline__ Col at(int y0, int c) const {
    return Col{col + y0 * GCl<N>::CB + c, row + uint32_t(c) * 8u, y0};
  }
};

// the field (chain) of this cluster; a.mode 0 or (SOLVE) 1
template <int N, bool SOLVE>
__global__ void __launch_bounds__(GCl<N>::T, 512 / GCl<N>::T) k_gcluster(const __grid_constant__ GlobalArgs a) {
  using K = GCl<N>;
  using G = typename K::G;
  constexpr int H = K::H, W = K::W, CB = K::CB, RB = K::RB, T = K::T, C = K::C, WH = K::WH;
  const int rank = blockIdx.x % C, f = blockIdx.x / C;
  if (a.sc->status != 0) {  // uniform over the grid
    if (SOLVE && blockIdx.x == 0 && threadIdx.x == 0) a.st->status = a.sc->status;
    return;
  }
  gtab_init<N, RB>();
  float2* s = gsmem();
  {
    const float4* src = reinterpret_cast<const float4*>((SOLVE ? a.dn : a.aq) + rank * RB * W);
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
  // every CTA has started (its shared memory may be stored to) and has its tables
  gc_arrive();
  gc_wait();

  const int yl = threadIdx.x / G::TR, y = rank * RB + yl;
  const GClRow<N> zrow{s + K::O_ROW + yl * K::RS, gc_addr(s + K::O_COL + y * CB)};
  const GClCols<N> zcol{s + K::O_COL, gc_addr(s + K::O_ROW + rank * CB)};
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
    constexpr int NG = G::E / 2;  // groups of four normals a thread needs in a phase
    const float sqrt_tau = a.sc->sqrt_tau;
    const uint32_t chain = a.chain0 + uint32_t(f);
    float z[NG][4], ze[4];
    auto draw = [&](int i, float (&v)[4]) {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = z[i][j];
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
      if (rank == 0 && threadIdx.x < H / 2)
        normals4(threadIdx.x, a.step0 + uint32_t(done), chain, 1u, a.key0, a.key1, ze);
    };
    float2 x[G::E];
    grow_load<N>(x, a.init_s ? a.init_s + f * a.init_stride + (long long)y * W : nullptr);
    draw_pixels(0);
    for (int done = 0;;) {
      pixel_update<N>(0, x, tab, draw, sqrt_tau, 0.f, 0, 0.f);
      grow_fwd<N, RB>(x, zrow);
      gc_arrive();
      draw_modes(done);
      gc_wait();
      gcol_update<N, RB>(
          0, zcol, rank * CB, fg, Pk, prev, [&](int i, uint32_t, float (&v)[4]) { draw(i, v); },
          [&](int, float (&v)[4]) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = ze[j];
          },
          0.f, false, false);
      gc_arrive();
      ++done;
      if (done < a.n_sweeps) draw_pixels(done);
      gc_wait();
      grow_inv<N, RB>(zrow, x);
      if (done > a.burn_in && (done - a.burn_in) % a.thin == 0) {
        const long long ms = (done - a.burn_in) / a.thin - 1;
        grow_store<N>(x, a.out, ((long long)f * a.n_samples + ms) * H + y, a.out_dtype);
      }
      if (done == a.n_sweeps) return;  // no CTA stores to another after the last barrier
    }
  } else {
    // Wiener filter with lambda-cooling; every CTA follows the same schedule (k_global), its decisions on the sum of
    // the CTAs' residual parts in rank order
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
      grow_fwd<N, RB>(x, zrow);
      gc_arrive();
      ++k;
      ++it;
      const bool cmp = (k % a.check == 0) && k >= 2;
      const bool store = ((k + 1) % a.check == 0);
      gc_wait();
      const float mine = gcol_update<N, RB>(
          1, zcol, rank * CB, fg, Pk, prev, [](int, uint32_t, float (&)[4]) {}, none, ltau, cmp, store);
      if (cmp) {
        const double v = gblock_sum<T>(double(mine), red);
        if (threadIdx.x < C)
          asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(gc_map(gc_addr(part + parity * C + rank), threadIdx.x)),
                       "d"(v)
                       : "memory");
      }
      gc_arrive();
      gc_wait();
      if (cmp) {
        if (threadIdx.x < 32) {
          double tot = threadIdx.x < C ? part[parity * C + threadIdx.x] : 0.0;
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
          if (threadIdx.x == 0) {
            tot *= double(H * W);
            const double bn = a.bnorm2[a.rhs_mode ? 0 : lev], ref = bn > 0.0 ? bn : 1.0;
            GSolveState d{tot, ltau, lev, k, 1};
            if (!(tot == tot) || tot > 1e300 * ref) {
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
            if (blockIdx.x == 0) d.rho2 = tot / ref;
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
      grow_inv<N, RB>(zrow, x);
      if (status != 1) break;
    }
    grow_store<N>(x, a.out, y, kOutF32);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      a.st->status = status;
      a.st->iters = it;
      a.st->resid = rho2 >= 0.0 ? sqrt(rho2) : rho2;
    }
  }
}

}  // namespace wf
