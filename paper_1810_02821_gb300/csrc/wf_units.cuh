// Pieces shared by the kernels that split a transform over several threads: the twiddle table, the unit pairs of
// a thread (units q and B - q of a length-B A transform, X[q + B j], which hold every mode pair (k, -k)) and the
// real-transform passes on such pairs.
#pragma once

#include "wf_math.cuh"

namespace wf {

// exp(-2 pi i j / 1024), rounded once from FP64, made at compile time
struct TwTable {
  float2 v[1024];
};
constexpr TwTable make_tw_table() {
  TwTable t{};
  for (int j = 0; j < 1024; ++j) {
    t.v[j].x = float(cos2pi(j, 1024));
    t.v[j].y = float(-sin2pi(j, 1024));
  }
  return t;
}
namespace {
__device__ const TwTable g_tw1024 = make_tw_table();
}

// the first thread's units 0 and B/2 hold their pairs (j, A - j) and (j, A - 1 - j) within each unit; swapping
// the upper halves (and rotating unit 0's) makes them pairs (p[j], q[A-1-j]), (q[j], p[A-1-j]), j < A/2, as in
// the other threads; the pair j = 0 of p is then (X[0], X[B A/2])
template <int A>
__device__ __forceinline__ void unit0_swap(float2 (&p)[A], float2 (&q)[A]) {
  float2 t[A / 2];
#pragma unroll
  for (int i = 0; i < A / 2; ++i) t[i] = p[A / 2 + i];
#pragma unroll
  for (int i = 0; i < A / 2; ++i) p[A / 2 + i] = q[A / 2 + i];
#pragma unroll
  for (int i = 0; i < A / 2; ++i) q[A / 2 + i] = t[(i + 1) % (A / 2)];
}
template <int A>
__device__ __forceinline__ void unit0_unswap(float2 (&p)[A], float2 (&q)[A]) {
  float2 t[A / 2];
#pragma unroll
  for (int i = 0; i < A / 2; ++i) t[(i + 1) % (A / 2)] = q[A / 2 + i];
#pragma unroll
  for (int i = 0; i < A / 2; ++i) q[A / 2 + i] = p[A / 2 + i];
#pragma unroll
  for (int i = 0; i < A / 2; ++i) p[A / 2 + i] = t[i];
}

// real-transform passes of the pair (K, L - K), w = exp(-2 pi i K / W): the packed-complex spectrum C to the
// half spectrum R, and back (unnormalised inverse)
__device__ __forceinline__ void k_post(float2& a, float2& b, float2 w) {
  const float2 E = cscale(cadd_conj(a, b), 0.5f);
  const float2 O = cmul_mi(cscale(csub_conj(a, b), 0.5f));
  const float2 WO = cmul(O, w);
  a = cadd(E, WO);
  b = cconj(csub(E, WO));
}
__device__ __forceinline__ void k_pre(float2& a, float2& b, float2 w) {
  const float2 E = cadd_conj(a, b);
  const float2 O = cmul(csub_conj(a, b), cconj(w));
  a = cadd(E, cmul_i(O));
  b = cadd(cconj(E), cmul_i(cconj(O)));
}

// c[k] *= w[k] (or its conjugate), k = 1 .. B-1, from a table row of B twiddles (16-byte aligned): two per load
template <int B, bool INV>
__device__ __forceinline__ void ktwiddle(float2 (&c)[B], const float2* w) {
#pragma unroll
  for (int k = 0; k < B; k += 2) {
    const float4 v = *reinterpret_cast<const float4*>(w + k);
    if (k > 0) c[k] = cmul(c[k], make_float2(v.x, INV ? -v.y : v.y));
    c[k + 1] = cmul(c[k + 1], make_float2(v.z, INV ? -v.w : v.w));
  }
}

}  // namespace wf
