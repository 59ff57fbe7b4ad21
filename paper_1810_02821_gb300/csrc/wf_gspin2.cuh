// Spin-2 (shear) sweeps with the fields in global memory (256^2 and 512^2 beyond the pairs that k_few2 holds, 128^2 where
// it cannot run): both components of every chain as two
// fields of one persistent cooperative launch (the phases, transforms and barrier of wf_global.cuh).
//   row phase    (CTA = 8 rows of one component): as the scalar sampler, the t-draw from stream 0 or 8;
//   column phase (CTA = 2 columns of both components): thread tid holds component tid % 2 of column
//                c0 + tid % 4 / 2, so the two components of a mode pair are in neighbouring lanes, which exchange half
//                of their pairs by shuffles, rotate into E and B, draw both and rotate back (spin2_mode).
// With DRAW false (the shear Wiener filter) the draws are left out: their scales are zero there, and adding zero times
// a finite variate changes nothing.
// Measured against both components in one thread-block cluster (k_csample_spin2), us per sweep:
// one 256^2 pair 23.5 -> 8.4, one 512^2 pair 46.7 -> 11.4 (a phase is a few L2 round trips and a barrier; the cluster runs
// 32-point register transforms on 8 or 16 SMs), 36 pairs of 512^2 275 -> 168.
#pragma once

#include "wf_global.cuh"

namespace wf {

struct GSpin2Args {
  Spin2Args s;   // aq2 [2][H][W], fgE and fgB in natural order
  float2* Z;     // [n_chains][2][H][W/2]
  GridBar* bar;
};

// The thread's column `col` of component `comp` (its vector v): transform, draw, transform back. zc: rows of the
// column from NC h on (ZCols::at); e: 2 H float2 for the pairs of column 0, edge: whether the CTA holds it; fE(ky, kx),
// fB(ky, kx): the mode tables; draw(j, group, zE, zB): the normals of the thread's j-th pair, edraw(ky, zE, zB): those
// of a pair of column 0. Components in neighbouring lanes, comp = tid & 1.
template <int N, int RB, bool DRAW, class Z, class FE, class FB, class D, class X>
__device__ __forceinline__ void gcol_spin2(const Z& zc, float2* v, float2* e, bool edge, int col, int h, FE&& fE,
                                           FB&& fB, D&& draw, X&& edraw) {
  using G = GGeo<N, RB>;
  constexpr int H = G::H, BC = G::BC, E = G::E, A = G::A, NC = E / 8;
  const int comp = threadIdx.x & 1, hb = h == 0 ? BC / 2 : BC - h;
  const GTab t = gtab<N, false, RB>();
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
    if (edge) {  // the same in every thread of the CTA; e: component 0, then component 1 (H float2 each)
      if (col == 0) {
        float2* ec = e + comp * H;
#pragma unroll
        for (int j = 0; j < A / 2; ++j) {
          ec[2 * (h + BC * j)] = p[j];
          ec[2 * (h + BC * j) + 1] = q[A - 1 - j];
          ec[2 * (hb + BC * j)] = q[j];
          ec[2 * (hb + BC * j) + 1] = p[A - 1 - j];
        }
      }
      __syncthreads();
      for (int k = threadIdx.x; k < H / 2; k += G::T) {
        float2 y1a = e[2 * k], y2a = e[2 * k + 1], y1b = e[H + 2 * k], y2b = e[H + 2 * k + 1];
        float zE[4] = {0.f, 0.f, 0.f, 0.f}, zB[4] = {0.f, 0.f, 0.f, 0.f};
        if (DRAW) edraw(k, zE, zB);
        if (k == 0) {
          // four real modes, each on k = 0 or a Nyquist line: no rotation, real draws with variance g^2
          constexpr float R2 = 1.41421356237309505f;
          auto upd = [&](float& u, float& w, int ky, int kx, float ze, float zb) {
            const float2 mE = fE(ky, kx), mB = fB(ky, kx);
            u = fmaf(mE.x, u, R2 * mE.y * ze);
            w = fmaf(mB.x, w, R2 * mB.y * zb);
          };
          upd(y1a.x, y1b.x, 0, 0, zE[0], zB[0]);
          upd(y1a.y, y1b.y, 0, G::W / 2, zE[2], zB[2]);
          upd(y2a.x, y2b.x, H / 2, 0, zE[1], zB[1]);
          upd(y2a.y, y2b.y, H / 2, G::W / 2, zE[3], zB[3]);
        } else {
          float2 A1 = cscale(cadd(y1a, cconj(y2a)), 0.5f), B1 = cmul_mi(cscale(csub(y1a, cconj(y2a)), 0.5f));
          float2 A2 = cscale(cadd(y1b, cconj(y2b)), 0.5f), B2 = cmul_mi(cscale(csub(y1b, cconj(y2b)), 0.5f));
          float c, s;
          ks_rot<N>(k, 0, c, s);
          spin2_mode(A1, A2, c, s, fE(k, 0), fB(k, 0), zE[0], zE[1], zB[0], zB[1]);
          ks_rot<N>(k, G::W / 2, c, s);
          spin2_mode(B1, B2, c, s, fE(k, G::W / 2), fB(k, G::W / 2), zE[2], zE[3], zB[2], zB[3]);
          y1a = cadd(A1, cmul_i(B1));
          y2a = cadd(cconj(A1), cmul_i(cconj(B1)));
          y1b = cadd(A2, cmul_i(B2));
          y2b = cadd(cconj(A2), cmul_i(cconj(B2)));
        }
        e[2 * k] = y1a;
        e[2 * k + 1] = y2a;
        e[H + 2 * k] = y1b;
        e[H + 2 * k + 1] = y2b;
      }
    }
    // component 0's lane draws the pairs led by unit h, component 1's those led by unit hb, for both components
    auto swap1 = [](float2 u) {
      return make_float2(__shfl_xor_sync(0xffffffffu, u.x, 1), __shfl_xor_sync(0xffffffffu, u.y, 1));
    };
    const int lead = comp == 0 ? h : hb;
#pragma unroll
    for (int j = 0; j < A / 2; ++j) {
      // own: the pair this lane draws; give: the one its neighbour draws
      const float2 own1 = comp == 0 ? p[j] : q[j], own2 = comp == 0 ? q[A - 1 - j] : p[A - 1 - j];
      const float2 got1 = swap1(comp == 0 ? q[j] : p[j]), got2 = swap1(comp == 0 ? p[A - 1 - j] : q[A - 1 - j]);
      float2 a1 = comp == 0 ? own1 : got1, b1 = comp == 0 ? got1 : own1;
      float2 a2 = comp == 0 ? own2 : got2, b2 = comp == 0 ? got2 : own2;
      const int ky1 = lead + BC * j, ky2 = ky1 == 0 ? H / 2 : H - ky1;
      float zE[4] = {0.f, 0.f, 0.f, 0.f}, zB[4] = {0.f, 0.f, 0.f, 0.f};
      if (DRAW) draw(j, uint32_t(col * (H / 2) + ky1), zE, zB);
      float c, s;
      ks_rot<N>(ky1, col, c, s);
      spin2_mode(a1, b1, c, s, fE(ky1, col), fB(ky1, col), zE[0], zE[1], zB[0], zB[1]);
      ks_rot<N>(ky2, col, c, s);
      spin2_mode(a2, b2, c, s, fE(ky2, col), fB(ky2, col), zE[2], zE[3], zB[2], zB[3]);
      const float2 back1 = swap1(comp == 0 ? b1 : a1), back2 = swap1(comp == 0 ? b2 : a2);
      if (comp == 0) {
        p[j] = a1;
        q[A - 1 - j] = a2;
        q[j] = back1;
        p[A - 1 - j] = back2;
      } else {
        q[j] = b1;
        p[A - 1 - j] = b2;
        p[j] = back1;
        q[A - 1 - j] = back2;
      }
    }
    if (edge) {
      __syncthreads();
      if (col == 0) {
        const float2* ec = e + comp * H;
#pragma unroll
        for (int j = 0; j < A / 2; ++j) {
          p[j] = ec[2 * (h + BC * j)];
          q[A - 1 - j] = ec[2 * (h + BC * j) + 1];
          q[j] = ec[2 * (hb + BC * j)];
          p[A - 1 - j] = ec[2 * (hb + BC * j) + 1];
        }
      }
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

// two columns c0, c0 + 1 of both components of one chain in global memory
template <int N, bool DRAW>
__device__ __forceinline__ void gcols_spin2(const GSpin2Args& a, float2* Z, int c0, uint32_t step, uint32_t chain) {
  using G = GGeo<N>;
  constexpr int WH = G::WH;
  const int vec = threadIdx.x % 4, col = c0 + vec / 2, h = threadIdx.x / 4;
  const float2* __restrict__ fgE = a.s.fgE;
  const float2* __restrict__ fgB = a.s.fgB;
  auto draw = [&](uint32_t g, float (&zE)[4], float (&zB)[4]) {
    normals4(g, step, chain, 1u, a.s.key0, a.s.key1, zE);
    normals4(g, step, chain, 9u, a.s.key0, a.s.key1, zB);
  };
  gcol_spin2<N, 8, DRAW>(
      ZCols<N>{Z + (long long)(vec & 1) * G::H * G::LR}.at((G::E / 8) * h, col), gsmem() + vec * G::VCOL,
      gsmem() + G::O_EDGE, c0 == 0, col, h, [&](int ky, int kx) { return __ldg(fgE + ky * WH + kx); },
      [&](int ky, int kx) { return __ldg(fgB + ky * WH + kx); },
      [&](int, uint32_t g, float (&zE)[4], float (&zB)[4]) { draw(g, zE, zB); },
      [&](int ky, float (&zE)[4], float (&zB)[4]) { draw(uint32_t(ky), zE, zB); });
}

template <int N>
constexpr int gspin2_smem() { return GGeo<N>::SMEM + N * 8; }  // parked pairs of a second component

template <int N, bool DRAW>
__global__ void __launch_bounds__(GGeo<N>::T, GGeo<N>::MIN_CTAS) k_gspin2(const __grid_constant__ GSpin2Args a) {
  using G = GGeo<N>;
  if (a.s.sc->status != 0) return;
  gtab_init<N>();
  const unsigned int nb = gridDim.x;
  unsigned int target = 0;  // of the grid barrier
  const float sqrt_tau = a.s.sc->sqrt_tau;
  const int ty = threadIdx.x / G::TR;
  constexpr int COL = G::LR / 2;  // column items per chain
  const int row_items = 2 * G::ROW_ITEMS * a.s.n_chains, col_items = COL * a.s.n_chains;
  constexpr long long n = (long long)G::H * G::W, nz = (long long)G::H * G::LR;
  for (int done = 0;; ++done) {  // sweeps completed
    for (int it = blockIdx.x; it < row_items; it += nb) {
      const int f = it / G::ROW_ITEMS, comp = f & 1, ci = f / 2, y = (it % G::ROW_ITEMS) * G::RB + ty;
      const ZRow z{a.Z + f * nz + (long long)y * G::LR};
      float2 x[G::E];
      if (done == 0)
        grow_load<N>(x, a.s.init_s ? a.s.init_s + ci * a.s.init_stride + comp * n + (long long)y * G::W : nullptr);
      else
        grow_inv<N>(z, x);
      if (done > a.s.burn_in && (done - a.s.burn_in) % a.s.thin == 0) {
        const long long m = (done - a.s.burn_in) / a.s.thin - 1;
        grow_store<N>(x, a.s.out, ((ci * a.s.n_samples + m) * 2 + comp) * G::H + y, a.s.out_dtype);
      }
      if (done == a.s.n_sweeps) continue;
      pixel_update<N>(DRAW ? 0 : 4, x, y, a.s.aq2 + comp * n, nullptr, a.s.step0 + uint32_t(done),
                      a.s.chain0 + uint32_t(ci), a.s.key0, a.s.key1, sqrt_tau, 0.f, 0, 0.f, 8u * uint32_t(comp));
      grow_fwd<N>(x, z);
    }
    if (done == a.s.n_sweeps) return;
    if (!grid_barrier(a.bar, nb, target)) return;
    for (int it = blockIdx.x; it < col_items; it += nb) {
      const int ci = it / COL;
      gcols_spin2<N, DRAW>(a, a.Z + 2LL * ci * nz, (it % COL) * 2, a.s.step0 + uint32_t(done),
                          a.s.chain0 + uint32_t(ci));
    }
    if (!grid_barrier(a.bar, nb, target)) return;
  }
}

}  // namespace wf
