// Batched form for images too large for one SM (N in {256, 512, 1024}): every image of a size class (or
// of a chunk of it) is one field of a single persistent cooperative launch.
//
// One launch of a single large image leaves most of the GPU idle (a 512 x 512 field has only 64 row and
// 64 column work items per phase) and pays two grid barriers per sweep for very little work. Here all
// fields advance together, sweep by sweep: a row phase over every (field, row block) and a column phase
// over every (field, column block), separated by the same bounded grid barrier as k_global. Each field
// runs its own schedule (Alg. 1 with A = I): the lambda-cooled Wiener solve of §2.2 from s = 0, then,
// from s_W, n_samples sweeps of the sampler; fields that finish early drop out of the work lists.
//
// Per-field schedule state is double-buffered by sweep parity: during the row phase of sweep s every CTA
// that owns a row block of field f reads state[s & 1][f] and the residual sums of the previous column
// phase, derives the same new state, and the owner of row block 0 stores it in state[(s + 1) & 1][f],
// which the column phase of sweep s reads after the barrier.
#pragma once

#include "wf_batch.cuh"
#include "wf_global.cuh"

namespace wf {

// one image of a large-image batch launch (device array, filled on the host)
struct GBField {
  const float2* aq;   // sampler pixel table (a, q), in the order of the size's kernels
  const float2* dn;   // Wiener-filter pixel table (d, 1/N_bar), likewise
  const float2* fg;   // [H][W/2+1] sampler mode table, likewise
  const float* Pk;    // [H][W/2+1], likewise
  float2* Z;          // [H][W/2] packed half spectrum (state)
  float2* prev;       // [H][W/2] previous Wiener iterate for the residual
  float* out_wf;      // [H][W] or null
  float* out_samples; // [n_samples][H][W] or null
  uint32_t chain, key0, key1;
  int item;           // index of the batch result
};

// per-field schedule (64 bytes, read with 16-byte L2 loads)
struct __align__(16) GBState {
  double tot, ref;  // residual sum of the last check (-1: none) and the level norm it is measured against
  float ltau;
  int phase;      // 0 Wiener solve, 1 sampling, 2 finished
  int lev, k, it; // cooling level, sweeps at this level, solve sweeps
  int parity;     // residual accumulator in use
  int status;     // solve status (1 while running)
  int cmp, store; // residual bookkeeping of this sweep's column phase
  int d;          // sampler step word of this sweep
};
static_assert(sizeof(GBState) == 64, "GBState layout");

struct GBArgs {
  const GBField* fields;
  const Scalars* sc;   // [F] per-field set-up
  GBState* state;      // [2][F]
  double* acc;         // [F][2] residual sums
  double* bnorm;       // [F][kMaxLevels] ||S N_lambda^-1 d||^2 per level
  BatchResult* res;    // indexed by GBField::item
  int* active;         // fields not finished (starts at F)
  GridBar* bar;
  int F;
  double tol, eta, level_tol;
  int max_iter, level_max, check, n_samples;
  int grid_pct;        // host side: percent of the co-resident grid
};

__device__ __forceinline__ GBState gb_load(const GBState* p) {
  GBState s;
  const int4* src = reinterpret_cast<const int4*>(p);
  int4* dst = reinterpret_cast<int4*>(&s);
#pragma unroll
  for (int i = 0; i < 4; ++i) dst[i] = __ldcg(src + i);
  return s;
}

template <int T>
__device__ __forceinline__ int block_max_levels(const Scalars* sc, int F, int* red) {
  int m = 0;
  for (int f = threadIdx.x; f < F; f += T) {
    const Scalars s = sc[f];
    if (s.status == 0 && s.n_levels > m) m = s.n_levels;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  int r = red[0];
#pragma unroll
  for (int w = 1; w < T / 32; ++w) r = max(r, red[w]);
  __syncthreads();
  return r;
}

template <int N>
__global__ void __launch_bounds__(GGeo<N>::T, GGeo<N>::MIN_CTAS) k_gbatch(const __grid_constant__ GBArgs a) {
  using G = GGeo<N>;
  __shared__ double red[G::T];
  __shared__ int ired[8];
  gtab_init<N>();
  constexpr double NPIX = double(G::H * G::W);
  const unsigned int nb = gridDim.x;
  const int F = a.F;
  unsigned int target = 0;  // of the grid barrier
  const int ty = threadIdx.x / G::TR;  // row of a row item
  const int row_items = G::ROW_ITEMS * F, col_items = G::COL_ITEMS * F;

  // 1. level norms, one cooling level at a time for all fields
  const int max_levels = block_max_levels<G::T>(a.sc, F, ired);
  for (int l = 0; l < max_levels; ++l) {
    for (int it = blockIdx.x; it < row_items; it += nb) {
      const int f = it / G::ROW_ITEMS, y0 = (it % G::ROW_ITEMS) * G::RB;
      const Scalars sc = a.sc[f];
      if (sc.status != 0 || l >= sc.n_levels) continue;
      const GBField fd = a.fields[f];
      float2 x[G::E];
      pixel_update<N>(2, x, y0 + ty, fd.aq, fd.dn, 0u, 0u, 0u, 0u, 0.f, 0.f, 0,
                      float(level_lambda(sc, l, a.eta) * sc.tau));
      grow_fwd<N>(x, ZRow{fd.Z + (long long)(y0 + ty) * G::LR});
    }
    if (!grid_barrier(a.bar, nb, target)) return;
    for (int it = blockIdx.x; it < col_items; it += nb) {
      const int f = it / G::COL_ITEMS;
      const Scalars sc = a.sc[f];
      if (sc.status != 0 || l >= sc.n_levels) continue;
      const GBField fd = a.fields[f];
      const double s = gblock_sum<G::T>(gcol_update<N>(2, fd.Z, (it % G::COL_ITEMS) * G::CB, fd.fg, fd.Pk, nullptr, 0u, 0u,
                                                       0u, 0u, 0.f, false, false), red);
      if (threadIdx.x == 0) atomicAdd(a.bnorm + f * kMaxLevels + l, s / NPIX);
    }
    if (!grid_barrier(a.bar, nb, target)) return;
  }

  // 2. sweeps: every field's Wiener solve, then its samples from s_W
  const long long max_sweeps = (long long)a.max_iter + a.n_samples + 4;
  for (long long sw = 0; sw < max_sweeps; ++sw) {
    const GBState* cur = a.state + (sw & 1) * F;
    GBState* nxt = a.state + ((sw + 1) & 1) * F;
    for (int it = blockIdx.x; it < row_items; it += nb) {
      const int f = it / G::ROW_ITEMS, rb = it % G::ROW_ITEMS, y0 = rb * G::RB;
      const bool owner = rb == 0 && threadIdx.x == 0;
      const Scalars sc = a.sc[f];
      const GBField fd = a.fields[f];
      GBState S;
      const bool fresh = sw == 0;
      if (fresh) {
        S.tot = -1.0;  // no check yet
        S.ref = 1.0;
        S.ltau = float(sc.lam0 * sc.tau);
        S.phase = 0;
        S.lev = S.k = S.it = S.parity = 0;
        S.status = 1;
        S.cmp = S.store = 0;
        S.d = 0;
        if (sc.status != 0) {  // set-up failed: no solve, no samples
          S.phase = 2;
          S.status = sc.status;
          if (owner) {
            a.res[fd.item] = BatchResult{-1.0, 0, sc.status};
            nxt[f] = S;
            atomicSub(a.active, 1);
          }
          continue;
        }
      } else {
        S = gb_load(cur + f);
        if (S.phase == 2) {
          if (owner) nxt[f] = S;
          continue;
        }
      }
      // decisions on the previous column phase (as in k_global's schedule)
      if (!fresh && S.phase == 0) {
        if (S.cmp) {
          const double tot = __ldcg(a.acc + 2 * f + S.parity) * NPIX;
          if (owner) a.acc[2 * f + (S.parity ^ 1)] = 0.0;  // the next check's accumulator
          S.parity ^= 1;
          const double bn = __ldcg(a.bnorm + f * kMaxLevels + S.lev);
          const double ref = bn > 0.0 ? bn : 1.0;  // rho = sqrt(tot / ref), compared without division and root
          S.tot = tot;
          S.ref = ref;
          if (residual_nonfinite(tot, ref)) {
            S.status = 6;
          } else if (S.lev < sc.n_levels - 1) {
            if (tot < a.level_tol * a.level_tol * ref || S.k >= a.level_max) {
              ++S.lev;
              S.ltau = float(level_lambda(sc, S.lev, a.eta) * sc.tau);
              S.k = 0;
            }
          } else if (tot < a.tol * a.tol * ref) {
            S.status = 0;
          }
        }
        if (S.status == 1 && S.it >= a.max_iter) S.status = 5;
      }
      const int y = y0 + ty;
      const ZRow z{fd.Z + (long long)y * G::LR};
      float2 x[G::E];
      if (fresh) grow_load<N>(x, nullptr);
      else grow_inv<N>(z, x);
      bool finished = false;
      if (S.phase == 0 && S.status != 1) {  // solve done: s_W out, then samples from it
        if (fd.out_wf) grow_store<N>(x, fd.out_wf, y, kOutF32);
        if (owner)
          a.res[fd.item] = BatchResult{S.tot >= 0.0 ? sqrt(S.tot / S.ref) : S.tot, S.it, S.status};
        if (a.n_samples > 0 && fd.out_samples) {
          S.phase = 1;
          S.d = 0;
        } else {
          finished = true;
        }
      } else if (S.phase == 1) {  // the sweep with step word d is complete: sample d
        grow_store<N>(x, fd.out_samples, (long long)S.d * G::H + y, kOutF32);
        ++S.d;
        finished = S.d >= a.n_samples;
      }
      if (finished) {
        S.phase = 2;
        if (owner) {
          nxt[f] = S;
          atomicSub(a.active, 1);
        }
        continue;
      }
      if (S.phase == 0) {
        ++S.k;
        ++S.it;
        S.cmp = (S.k % a.check == 0) && S.k >= 2;
        S.store = ((S.k + 1) % a.check == 0);
        pixel_update<N>(1, x, y, fd.aq, fd.dn, 0u, 0u, 0u, 0u, 0.f, S.ltau, 0, 0.f);
      } else {
        pixel_update<N>(0, x, y, fd.aq, fd.dn, uint32_t(S.d), fd.chain, fd.key0, fd.key1, sc.sqrt_tau, 0.f, 0, 0.f);
      }
      grow_fwd<N>(x, z);
      if (owner) nxt[f] = S;
    }
    if (!grid_barrier(a.bar, nb, target)) return;
    // no field changes state between here and the next barrier: every CTA sees the same count
    if (__ldcg(a.active) == 0) return;
    for (int it = blockIdx.x; it < col_items; it += nb) {
      const int f = it / G::COL_ITEMS;
      const GBState S = gb_load(nxt + f);
      if (S.phase == 2) continue;
      const GBField fd = a.fields[f];
      const int c0 = (it % G::COL_ITEMS) * G::CB;
      if (S.phase == 0) {
        const float mine = gcol_update<N>(1, fd.Z, c0, fd.fg, fd.Pk, fd.prev, 0u, 0u, 0u, 0u, S.ltau, S.cmp != 0,
                                           S.store != 0);
        if (S.cmp) {
          const double part = gblock_sum<G::T>(mine, red);
          if (threadIdx.x == 0) atomicAdd(a.acc + 2 * f + S.parity, part);
        }
      } else {
        gcol_update<N>(0, fd.Z, c0, fd.fg, fd.Pk, nullptr, uint32_t(S.d), fd.chain, fd.key0, fd.key1, 0.f, false,
                       false);
      }
    }
    if (!grid_barrier(a.bar, nb, target)) return;
  }
}

}  // namespace wf
