// Size-specialised launchers of the fused kernels (one translation unit per image size).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "wf_gibbs.cuh"
#include "wf_global.cuh"
#include "wf_batch.cuh"
#include "wf_gbatch.cuh"
#include "wf_cluster.cuh"
#include "wf_cluster_ext.cuh"
#include "wf_bphase.cuh"
#include "wf_core.cuh"
#include "wf_gspin2.cuh"
#include "wf_few.cuh"

namespace wf {

// optional CUDA-event bracket around the main kernel of a launch
struct LaunchTimer {
  virtual void start() = 0;
  virtual void stop() = 0;
};

// fields (chains) per CTA of the one-thread-per-row kernels (16 x 16; the fused batch kernel's class count):
// 128 threads per CTA for every size
template <int N>
constexpr int fields_per_cta() { return N >= 128 ? 1 : 128 / N; }

// Samplers up to 128 x 128. *timeout (host, set to 0 by the caller) receives WF_ERR_TIMEOUT, once st has passed, when a
// wait of a balanced launch gave up; launch_sample with timeout null allocates nothing
template <int N>
cudaError_t launch_sample(const SampleArgs& a, cudaStream_t st, LaunchTimer* t, int* timeout);

// chains of one wave of the sampler with several threads per row (N in {32, 64, 128}) on the current device
template <int N>
cudaError_t sample_wave(int* chains);

template <int N>
cudaError_t launch_sample_band(const SampleArgs& a, cudaStream_t st, LaunchTimer* t, int* timeout);

template <int N>
cudaError_t launch_sample_spin2(const Spin2Args& a, cudaStream_t st, LaunchTimer* t, int* timeout);

template <int N>
cudaError_t launch_solve(const SolveArgs& a, const BnormArgs& b, cudaStream_t st, LaunchTimer* t);

// batched persistent form for N <= 128: grid = min(items, resident CTAs), per-CTA scratch slots
template <int N>
cudaError_t launch_batch(const BatchArgs& b, int* grid_out, cudaStream_t st);

// batched form for N <= 128 in phases (after the per-image set-up kernels): a few CTAs per image for the
// level norms, one CTA per image for the cooled solves, then the samplers with fpc images per CTA
template <int N>
cudaError_t launch_bsolve(const BSolveArgs& a, cudaStream_t st);
template <int N>
cudaError_t launch_bsample(const BSampleArgs& a, int fpc, cudaStream_t st);

// weighted spectral power of real fields (N <= 128, one CTA per field)
template <int N>
cudaError_t launch_wpower(const WpowerArgs& p, cudaStream_t st);
template <int N>
cudaError_t batch_grid(int n_items, int grid_pct, int* grid_out);

// large images (N >= 256): one cooperative launch of k_global<N> (all CTAs co-resident)
template <int N>
cudaError_t launch_global(const GlobalArgs& a, cudaStream_t st, LaunchTimer* t);

// the same sampler (mode 0) and, from 128, Wiener filter (mode 1) for few fields (wf_few.cuh; N in {64 .. 1024}; a.prev
// unused, a.Z, a.bar and a.acc up to 256 too). few_count: fields resident at once on the current device, 0 if it cannot run
template <int N>
cudaError_t launch_few(const GlobalArgs& a, cudaStream_t st, LaunchTimer* t);
template <int N>
cudaError_t few_count(bool solve, int* fields);
// the spin-2 sampler and filter in the same way (N in {128, 256, 512}), natural table orders
template <int N>
cudaError_t launch_few2(const GSpin2Args& a, cudaStream_t st, LaunchTimer* t);
template <int N>
cudaError_t few2_count(bool quiet, int* pairs);

// batched large images (N >= 256): one cooperative launch of k_gbatch<N> over all fields of a size class
template <int N>
cudaError_t launch_gbatch(const GBArgs& a, cudaStream_t st);

// spin-2 sampler with the fields in global memory (N in {256, 512}): one cooperative launch of k_gspin2<N>
template <int N>
cudaError_t launch_gspin2(const GSpin2Args& a, cudaStream_t st, LaunchTimer* t);

// cluster-resident sampler (N in {256, 512}): one cluster of N / MR CTAs of MR rows each per chain
// (MR = 64 at 256; 32 or 64 at 512). cudaErrorNotSupported when no cluster of that shape can be resident.
template <int N, int MR>
cudaError_t launch_csample(const SampleArgs& a, cudaStream_t st, LaunchTimer* t);
// clusters of k_csample<N, MR> that can be resident at once on the current device (0: none)
template <int N, int MR>
cudaError_t csample_clusters(int* clusters);
// whole pipeline (level norms, cooled solve, samples) of a batch of large images: one cluster per image
template <int N, int MR>
cudaError_t launch_cpipe(const CBArgs& a, cudaStream_t st, LaunchTimer* t);

// cluster-resident hierarchical sampler (a.band_clusters clusters of N / MR CTAs looping over the chains;
// a.fg and a.band_map in slot order) and
// spin-2 sampler (both components per cluster). cudaErrorNotSupported when no cluster of that shape
// can be resident.
template <int N, int MR>
cudaError_t launch_csample_band(const SampleArgs& a, cudaStream_t st, LaunchTimer* t);
// clusters of k_csample_band<N, MR> with n_bins bands that can be resident at once (0: none)
template <int N, int MR>
cudaError_t csample_band_clusters(int n_bins, int* clusters);
template <int N, int MR>
cudaError_t launch_csample_spin2(const Spin2Args& a, cudaStream_t st, LaunchTimer* t);

// definitions, included by the per-size translation units only
#if defined(WF_LAUNCH_DEFINE)
// one launch of a kernel with dynamic shared memory, timed when t is given
template <class Kern, class Args>
cudaError_t launch_smem(Kern kern, dim3 grid, int threads, int smem, const Args& a, cudaStream_t st, LaunchTimer* t) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  if (t) t->start();
  kern<<<grid, threads, smem, st>>>(a);
  if (t) t->stop();
  return cudaGetLastError();
}
// Whether equal shares (KBalance) are faster than one CTA per chain for n chains of N x N fields, `sweeps` sweeps each, on
// `sms` SMs with per_sm resident CTAs. In units of a full round's sweep: one CTA per chain takes its full rounds and, for
// the last one, the share of an SM's places that its fullest SM has taken, but not less than `lat` (a CTA alone on its SM: 0.27
// of a round at 32^2, 0.24 to 0.37 for shear pairs; 0.33 to 0.6 with the band statistics). Shares take n / R rounds, a few
// percent slower per sweep, and `fixed` sweeps a call more (allocation, flags, cooperative launch: 10 to 40 us, 50 to 120 with
// the band statistics). Measured, ms a call, one CTA per chain / shares: 128^2 100 sweeps 350 chains 2.94 / 2.36, 440 2.93 / 2.89,
// 607 3.79 / 3.87, 1000 6.34 / 6.17, 1500 8.93 / 9.11; 300 shear pairs 4.93 / 5.01; 32^2 1521 chains 0.95 / 0.87, 3000 1.35 / 1.44,
// 5000 2.07 / 2.20; 64^2 bands 20 sweeps 761 chains 0.91 / 0.83, 1500 1.20 / 1.39; 4 sweeps of 600 128^2 chains 0.42 / 0.45.
struct BalanceCost {
  double lat, fixed;
};
template <int N>
constexpr BalanceCost balance_cost(bool band) {
  return band ? BalanceCost{0.6, N == 32 ? 3.0 : 8.0} : BalanceCost{0.3, N == 32 ? 6.0 : 2.0};
}
WF_HD bool balance_pays(int N, const BalanceCost& c, long long n, int per_sm, int sms, long long sweeps) {
  const long long R = (long long)per_sm * sms;
  if (R <= 0 || n <= R || n % R == 0) return false;
  const double layers = double((n % R + sms - 1) / sms) / per_sm;
  const double whole = double(n / R) + (layers > c.lat ? layers : c.lat);
  const double shares = double(n) / double(R) * (N == 32 ? 1.08 : (N == 64 ? 1.06 : 1.03));
  return (whole - shares) * double(sweeps) > c.fixed;
}
// One CTA per chain, or a cooperative launch of equal shares where these are faster, whose scratch (slots, flags) comes
// from st's memory pool
template <int N, class Kern, class Args>
cudaError_t launch_chains(Kern whole, Kern balanced, const BalanceCost& cost, int n_chains, int threads, int smem, int slot_floats,
                          const Args& a, cudaStream_t st, LaunchTimer* t, int* timeout) {
  cudaError_t e = cudaFuncSetAttribute(balanced, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, balanced, threads, smem)) != cudaSuccess) return e;
  const int R = per_sm * sms;
  KBalance b{};
  void* base = nullptr;
  const size_t flags = (size_t(R) + 1) * sizeof(unsigned int), off = (flags + 255) / 256 * 256;
  bool bal = timeout && balance_pays(N, cost, n_chains, per_sm, sms, a.n_sweeps);
  if (bal) {
    e = cudaMallocAsync(&base, off + size_t(R) * size_t(slot_floats) * sizeof(float), st);
    if (e == cudaErrorMemoryAllocation) {  // no room for the states handed over: one CTA per chain needs none
      cudaGetLastError();
      bal = false;
    } else if (e != cudaSuccess) {
      return e;
    }
  }
  if (!bal) {
    if ((e = cudaFuncSetAttribute(whole, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
    if (t) t->start();
    whole<<<n_chains, threads, smem, st>>>(a, b);
    if (t) t->stop();
    return cudaGetLastError();
  }
  b.shares = R;
  b.slot_floats = slot_floats;
  b.flag = static_cast<unsigned int*>(base);
  b.err = reinterpret_cast<int*>(b.flag + R);
  b.slot = reinterpret_cast<float*>(static_cast<char*>(base) + off);
  e = cudaMemsetAsync(base, 0, flags, st);
  Args arg = a;
  void* args[] = {&arg, &b};
  if (t) t->start();
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(balanced), dim3(R), dim3(threads), args, smem, st);
  if (t) t->stop();
  if (e == cudaSuccess) e = cudaMemcpyAsync(timeout, b.err, sizeof(int), cudaMemcpyDeviceToHost, st);
  const cudaError_t e2 = cudaFreeAsync(base, st);
  return e != cudaSuccess ? e : e2;
}

template <int N>
cudaError_t sample_wave(int* chains) {
  *chains = 0;
  if constexpr (core_size(N)) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaFuncSetAttribute(k_msample<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, KGeo<N>::SMEM);
    if (e != cudaSuccess) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_msample<N, false>, KGeo<N>::T, KGeo<N>::SMEM);
    *chains = per_sm * sms;
    return e;
  }
  return cudaErrorInvalidValue;
}

template <int N>
cudaError_t launch_sample(const SampleArgs& a, cudaStream_t st, LaunchTimer* t, int* timeout) {
  if constexpr (core_size(N)) {
    if (a.cm != 0)
      return launch_chains<N>(k_msample<N, false>, k_msample<N, true>, balance_cost<N>(false), a.n_chains, KGeo<N>::T,
                              KGeo<N>::SMEM, N * N, a, st, t, timeout);
  }
  if constexpr (N == 16 || N == 64) {
    constexpr int FPC = fields_per_cta<N>();
    return launch_smem(k_sample<N, FPC>, (a.n_chains + FPC - 1) / FPC, N * FPC, FPC * Geo<N>::FIELD_BYTES, a, st, t);
  }
  return cudaErrorInvalidValue;
}

template <int N>
cudaError_t launch_sample_band(const SampleArgs& a, cudaStream_t st, LaunchTimer* t, int* timeout) {
  if constexpr (core_size(N)) {
    return launch_chains<N>(k_mband<N, false>, k_mband<N, true>, balance_cost<N>(true), a.n_chains, KGeo<N>::T,
                            KGeo<N>::SMEM + band_bytes(a.n_bins), N * N + (a.n_bins + 3) / 4 * 4, a, st, t, timeout);
  } else {
    constexpr int FPC = fields_per_cta<N>();
    return launch_smem(k_sample_band<N, FPC>, (a.n_chains + FPC - 1) / FPC, N * FPC,
                       FPC * (Geo<N>::FIELD_BYTES + band_bytes(a.n_bins)), a, st, t);
  }
}

template <int N>
cudaError_t launch_sample_spin2(const Spin2Args& a, cudaStream_t st, LaunchTimer* t, int* timeout) {
  if constexpr (core_size(N)) {
    // the filter (quiet) is one chain
    return launch_chains<N>(a.quiet ? k_mspin2<N, false, false> : k_mspin2<N, true, false>, k_mspin2<N, true, true>,
                            balance_cost<N>(false), a.n_chains, 2 * KGeo<N>::T, kspin2_smem<N>(), 2 * N * N, a, st, t, a.quiet ? nullptr : timeout);
  } else {
    constexpr int FPC = fields_per_cta<N>();  // images per CTA; two component fields each
    return launch_smem(k_sample_spin2<N, FPC>, (a.n_chains + FPC - 1) / FPC, 2 * N * FPC,
                       2 * FPC * Geo<N>::FIELD_BYTES, a, st, t);
  }
}

template <int N>
cudaError_t launch_solve(const SolveArgs& a, const BnormArgs& b, cudaStream_t st, LaunchTimer* t) {
  cudaError_t e = cudaSuccess;
  if constexpr (core_size(N)) {
    if (!a.rhs_mode)  // rhs mode: the level norms are supplied
      e = launch_smem(k_mbnorm<N>, dim3(kMaxLevels, unsigned(a.n_fields)), KGeo<N>::T, ksolve_smem<N>(), b, st, nullptr);
    if (e != cudaSuccess) return e;
    return launch_smem(a.n_fields > 1 ? k_msolve<N, true> : k_msolve<N, false>, unsigned(a.n_fields), KGeo<N>::T,
                       ksolve_smem<N>(), a, st, t);
  } else {
    if (a.n_fields != 1) return cudaErrorInvalidValue;
    const int smem = Geo<N>::FIELD_BYTES + 33 * 8;
    if (!a.rhs_mode) e = launch_smem(k_bnorm<N>, kMaxLevels, N, smem, b, st, nullptr);
    return e != cudaSuccess ? e : launch_smem(k_solve<N>, 1, N, smem, a, st, t);
  }
}

template <int N>
cudaError_t batch_grid(int n_items, int grid_pct, int* grid_out) {
  const int smem = batch_smem_bytes<N>();
  cudaError_t e = cudaFuncSetAttribute(k_batch<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch<N>, N, smem)) != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  int full = per_sm * sms;
  if (grid_pct > 0 && grid_pct < 100) full = (full * grid_pct + 99) / 100;
  *grid_out = n_items < full ? n_items : full;
  return cudaSuccess;
}

template <int N>
cudaError_t launch_batch(const BatchArgs& b, int* grid_out, cudaStream_t st) {
  int grid = 0;
  cudaError_t e = batch_grid<N>(b.n, b.grid_pct, &grid);
  if (e != cudaSuccess) return e;
  if (grid_out) *grid_out = grid;
  if (grid > 0) k_batch<N><<<grid, N, batch_smem_bytes<N>(), st>>>(b);
  return cudaGetLastError();
}

template <int N>
cudaError_t launch_bsolve(const BSolveArgs& a, cudaStream_t st) {
  if (a.F < 1) return cudaSuccess;
  if constexpr (core_size(N)) {
    const cudaError_t e = launch_smem(k_mblevels<N>, dim3(a.F, kLevelCtas), KGeo<N>::T, ksolve_smem<N>(), a, st, nullptr);
    return e != cudaSuccess ? e : launch_smem(k_mbsolve<N>, a.F, KGeo<N>::T, ksolve_smem<N>(), a, st, nullptr);
  } else {
    const int smem = bsolve_smem_bytes<N>();
    const cudaError_t e = launch_smem(k_blevels<N>, dim3(a.F, kLevelCtas), N, smem, a, st, nullptr);
    return e != cudaSuccess ? e : launch_smem(k_bsolve<N>, a.F, N, smem, a, st, nullptr);
  }
}

template <int N, int FPC>
cudaError_t launch_bsample_fpc(const BSampleArgs& a, cudaStream_t st) {
  if (a.F < 1 || a.n_samples < 1) return cudaSuccess;
  return launch_smem(k_bsample<N, FPC>, (a.F + FPC - 1) / FPC, N * FPC, FPC * Geo<N>::FIELD_BYTES, a, st, nullptr);
}

// fields (images) per CTA fpc in 1 .. 128 / N (0: fields_per_cta<N>()); the kernels with several threads per row
// always take one image per CTA
template <int N>
cudaError_t launch_bsample(const BSampleArgs& a, int fpc, cudaStream_t st) {
  if (fpc == 0) fpc = fields_per_cta<N>();
  if (fpc < 1 || fpc > fields_per_cta<N>()) return cudaErrorInvalidValue;
  if constexpr (core_size(N)) {
    if (a.F < 1 || a.n_samples < 1) return cudaSuccess;
    return launch_smem(k_mbsample<N>, a.F, KGeo<N>::T, KGeo<N>::SMEM, a, st, nullptr);
  } else {
    switch (fpc) {
      case 1: return launch_bsample_fpc<N, 1>(a, st);
      case 2: return launch_bsample_fpc<N, 2>(a, st);
      case 4: return launch_bsample_fpc<N, 4>(a, st);
      case 8: return launch_bsample_fpc<N, 8>(a, st);
    }
    return cudaErrorInvalidValue;
  }
}

template <int N>
cudaError_t launch_wpower(const WpowerArgs& p, cudaStream_t st) {
  const int smem = Geo<N>::FIELD_BYTES + 33 * 8;
  cudaError_t e = cudaFuncSetAttribute(k_wpower<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  if (p.n_fields > 0) k_wpower<N><<<p.n_fields, N, smem, st>>>(p);
  return cudaGetLastError();
}

#define WF_INSTANTIATE(N)                                                              \
  template cudaError_t launch_sample<N>(const SampleArgs&, cudaStream_t, LaunchTimer*, int*); \
  template cudaError_t sample_wave<N>(int*);                                             \
  template cudaError_t launch_sample_band<N>(const SampleArgs&, cudaStream_t, LaunchTimer*, int*); \
  template cudaError_t launch_sample_spin2<N>(const Spin2Args&, cudaStream_t, LaunchTimer*, int*); \
  template cudaError_t launch_solve<N>(const SolveArgs&, const BnormArgs&, cudaStream_t, LaunchTimer*); \
  template cudaError_t launch_batch<N>(const BatchArgs&, int*, cudaStream_t);                     \
  template cudaError_t batch_grid<N>(int, int, int*);                                                   \
  template cudaError_t launch_bsolve<N>(const BSolveArgs&, cudaStream_t);                                \
  template cudaError_t launch_bsample<N>(const BSampleArgs&, int, cudaStream_t);                         \
  template cudaError_t launch_wpower<N>(const WpowerArgs&, cudaStream_t);
#endif

#if defined(WF_LAUNCH_DEFINE_GLOBAL)
template <int N>
cudaError_t launch_global(const GlobalArgs& a, cudaStream_t st, LaunchTimer* t) {
  using G = GGeo<N>;
  cudaError_t e = cudaFuncSetAttribute(k_global<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_global<N>, G::T, G::SMEM)) != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const long long items = (long long)(G::ROW_ITEMS > G::COL_ITEMS ? G::ROW_ITEMS : G::COL_ITEMS) * a.n_fields;
  long long full = (long long)per_sm * sms;
  if (a.grid_pct > 0 && a.grid_pct < 100) full = (full * a.grid_pct + 99) / 100;
  const int grid = int(items < full ? items : full);
  GlobalArgs arg = a;
  void* args[] = {&arg};
  if (t) t->start();
  e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_global<N>), dim3(grid), dim3(G::T), args, G::SMEM, st);
  if (t) t->stop();
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}
template <int N>
cudaError_t launch_gbatch(const GBArgs& a, cudaStream_t st) {
  using G = GGeo<N>;
  cudaError_t e = cudaFuncSetAttribute(k_gbatch<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gbatch<N>, G::T, G::SMEM)) != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const long long items = (long long)(G::ROW_ITEMS > G::COL_ITEMS ? G::ROW_ITEMS : G::COL_ITEMS) * a.F;
  long long full = (long long)per_sm * sms;
  if (a.grid_pct > 0 && a.grid_pct < 100) full = (full * a.grid_pct + 99) / 100;
  const int grid = int(items < full ? items : full);
  GBArgs arg = a;
  void* args[] = {&arg};
  e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_gbatch<N>), dim3(grid), dim3(G::T), args, G::SMEM, st);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}
template <int N>
cudaError_t launch_gspin2(const GSpin2Args& a, cudaStream_t st, LaunchTimer* t) {
  using G = GGeo<N>;
  auto kern = a.s.quiet ? k_gspin2<N, false> : k_gspin2<N, true>;
  const int smem = gspin2_smem<N>();
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, G::T, smem)) != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const long long items = (long long)(G::LR / 2) * a.s.n_chains;  // column items (more than row items)
  const long long full = (long long)per_sm * sms;
  GSpin2Args arg = a;
  void* args[] = {&arg};
  if (t) t->start();
  e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(kern), dim3(unsigned(items < full ? items : full)),
                                  dim3(G::T), args, smem, st);
  if (t) t->stop();
  return e != cudaSuccess ? e : cudaGetLastError();
}
#define WF_INSTANTIATE_GSPIN2(N) template cudaError_t launch_gspin2<N>(const GSpin2Args&, cudaStream_t, LaunchTimer*);
#define WF_INSTANTIATE_GLOBAL_ONE(N) template cudaError_t launch_global<N>(const GlobalArgs&, cudaStream_t, LaunchTimer*);
#define WF_INSTANTIATE_GLOBAL(N)                                                               \
  WF_INSTANTIATE_GLOBAL_ONE(N)                                                                  \
  template cudaError_t launch_gbatch<N>(const GBArgs&, cudaStream_t);
#endif

#if defined(WF_LAUNCH_DEFINE_FEW)
// launches of k_few and k_few2: one cluster per field, or a cooperative grid
template <class X>
struct FewLaunch {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr{};
  template <class Kern>
  cudaError_t set(Kern kern, int T, int smem, int n_fields, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (X::CLUSTER) {
      if (X::C > 8 &&
          (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
        return e;
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = unsigned(X::C);
      attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    } else {
      attr.id = cudaLaunchAttributeCooperative;
      attr.val.cooperative = 1;
    }
    cfg.gridDim = dim3(unsigned(n_fields) * unsigned(X::C));
    cfg.blockDim = dim3(unsigned(T));
    cfg.dynamicSmemBytes = size_t(smem);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaSuccess;
  }
  template <class Kern>
  static cudaError_t count(Kern kern, int T, int smem, int* n) {
    FewLaunch l;
    cudaError_t e = l.set(kern, T, smem, 1, nullptr);
    if (e != cudaSuccess) return e;
    if (X::CLUSTER) return cudaOccupancyMaxActiveClusters(n, kern, &l.cfg);
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T, smem)) != cudaSuccess) return e;
    *n = per_sm * sms / X::C;
    return cudaSuccess;
  }
  template <class Kern, class Args>
  static cudaError_t run(Kern kern, int T, int smem, int n_fields, const Args& a, cudaStream_t st, LaunchTimer* t) {
    FewLaunch l;
    cudaError_t e = l.set(kern, T, smem, n_fields, st);
    if (e != cudaSuccess) return e;
    if (t) t->start();
    e = cudaLaunchKernelEx(&l.cfg, kern, a);
    if (t) t->stop();
    return e != cudaSuccess ? e : cudaGetLastError();
  }
};
template <int N>
using FewX = std::conditional_t<N <= 256, XCluster<N, 1>, XGrid<N, 1>>;
template <int N>
using FewX2 = std::conditional_t<N <= 128, XCluster<N, 2>, XGrid<N, 2>>;
template <int N>
cudaError_t few_count(bool solve, int* fields) {
  using X = FewX<N>;
  using K = FewGeo<N, X>;
  if constexpr (N >= 128)
    if (solve) return FewLaunch<X>::count(k_few<N, X, true>, K::T, K::SMEM_SOLVE, fields);
  return FewLaunch<X>::count(k_few<N, X, false>, K::T, K::SMEM_SAMPLE, fields);
}
template <int N>
cudaError_t launch_few(const GlobalArgs& a, cudaStream_t st, LaunchTimer* t) {
  using X = FewX<N>;
  using K = FewGeo<N, X>;
  if constexpr (N >= 128)
    if (a.mode == 1) return FewLaunch<X>::run(k_few<N, X, true>, K::T, K::SMEM_SOLVE, a.n_fields, a, st, t);
  return FewLaunch<X>::run(k_few<N, X, false>, K::T, K::SMEM_SAMPLE, a.n_fields, a, st, t);
}
template <int N>
cudaError_t few2_count(bool quiet, int* pairs) {
  using X = FewX2<N>;
  using K = FewGeo<N, X>;
  return FewLaunch<X>::count(quiet ? k_few2<N, X, false> : k_few2<N, X, true>, K::T, K::SMEM_SAMPLE, pairs);
}
template <int N>
cudaError_t launch_few2(const GSpin2Args& a, cudaStream_t st, LaunchTimer* t) {
  using X = FewX2<N>;
  using K = FewGeo<N, X>;
  return FewLaunch<X>::run(a.s.quiet ? k_few2<N, X, false> : k_few2<N, X, true>, K::T, K::SMEM_SAMPLE, a.s.n_chains, a,
                           st, t);
}
#define WF_INSTANTIATE_FEW(N)                       \
  template cudaError_t few_count<N>(bool, int*);     \
  template cudaError_t launch_few<N>(const GlobalArgs&, cudaStream_t, LaunchTimer*);
#define WF_INSTANTIATE_FEW2(N)                      \
  template cudaError_t few2_count<N>(bool, int*);    \
  template cudaError_t launch_few2<N>(const GSpin2Args&, cudaStream_t, LaunchTimer*);
#endif

#if defined(WF_LAUNCH_DEFINE_CLUSTER)
template <int N, int MR>
cudaError_t csample_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, int n_chains, cudaStream_t st) {
  using G = CGeo<N, MR>;
  cudaError_t e = cudaFuncSetAttribute(k_csample<N, MR>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_cpipe<N, MR>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
  if (e != cudaSuccess) return e;
  if (G::P > 8) {  // clusters above the portable size of 8
    e = cudaFuncSetAttribute(k_csample<N, MR>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_cpipe<N, MR>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = G::P;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(unsigned(n_chains) * G::P, 1, 1);
  cfg->blockDim = dim3(G::L, 1, 1);
  cfg->dynamicSmemBytes = G::SMEM;
  cfg->stream = st;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  return cudaSuccess;
}
template <int N, int MR>
cudaError_t csample_clusters(int* clusters) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e = csample_config<N, MR>(&cfg, attr, 1, nullptr);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveClusters(clusters, k_csample<N, MR>, &cfg);
}
template <int N, int MR>
cudaError_t launch_csample(const SampleArgs& a, cudaStream_t st, LaunchTimer* t) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e = csample_config<N, MR>(&cfg, attr, a.n_chains, st);
  if (e != cudaSuccess) return e;
  if (t) t->start();
  e = cudaLaunchKernelEx(&cfg, k_csample<N, MR>, a);
  if (t) t->stop();
  return e != cudaSuccess ? e : cudaGetLastError();
}
template <int N, int MR>
cudaError_t launch_cpipe(const CBArgs& a, cudaStream_t st, LaunchTimer* t) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e = csample_config<N, MR>(&cfg, attr, a.F, st);
  if (e != cudaSuccess) return e;
  if (t) t->start();
  e = cudaLaunchKernelEx(&cfg, k_cpipe<N, MR>, a);
  if (t) t->stop();
  return e != cudaSuccess ? e : cudaGetLastError();
}
#define WF_INSTANTIATE_CLUSTER(N, MR)                                                          \
  template cudaError_t launch_csample<N, MR>(const SampleArgs&, cudaStream_t, LaunchTimer*);   \
  template cudaError_t csample_clusters<N, MR>(int*);                                          \
  template cudaError_t launch_cpipe<N, MR>(const CBArgs&, cudaStream_t, LaunchTimer*);
#endif

#if defined(WF_LAUNCH_DEFINE_CLUSTER_EXT)
// launch configuration of `clusters` clusters of P CTAs of `threads` threads with `smem` dynamic shared
// bytes each; cudaErrorNotSupported when not one such cluster can be resident
template <class Kern>
cudaError_t cluster_launch_config(Kern kern, int P, int threads, int smem, int clusters, cudaStream_t st,
                                  cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  if (P > 8) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(P);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(unsigned(clusters) * unsigned(P), 1, 1);
  cfg->blockDim = dim3(unsigned(threads), 1, 1);
  cfg->dynamicSmemBytes = size_t(smem);
  cfg->stream = st;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  int resident = 0;
  e = cudaOccupancyMaxActiveClusters(&resident, kern, cfg);
  if (e != cudaSuccess) return e;
  return resident > 0 ? cudaSuccess : cudaErrorNotSupported;
}
template <int N, int MR>
cudaError_t csample_band_clusters(int n_bins, int* clusters) {
  using G = CGeo<N, MR>;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  *clusters = 0;
  cudaError_t e = cluster_launch_config(k_csample_band<N, MR>, G::P, G::L, cband_smem<N, MR>(n_bins), 1, nullptr,
                                        &cfg, attr);
  if (e == cudaErrorNotSupported) return cudaSuccess;
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveClusters(clusters, k_csample_band<N, MR>, &cfg);
}
template <int N, int MR>
cudaError_t launch_csample_band(const SampleArgs& a, cudaStream_t st, LaunchTimer* t) {
  using G = CGeo<N, MR>;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e = cluster_launch_config(k_csample_band<N, MR>, G::P, G::L, cband_smem<N, MR>(a.n_bins),
                                        a.band_clusters, st, &cfg, attr);
  if (e != cudaSuccess) return e;
  if (t) t->start();
  e = cudaLaunchKernelEx(&cfg, k_csample_band<N, MR>, a);
  if (t) t->stop();
  return e != cudaSuccess ? e : cudaGetLastError();
}
template <int N, int MR>
cudaError_t launch_csample_spin2(const Spin2Args& a, cudaStream_t st, LaunchTimer* t) {
  using G = CGeo<N, MR>;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e =
      cluster_launch_config(k_csample_spin2<N, MR>, G::P, cspin2_threads<N, MR>(), cspin2_smem<N, MR>(), a.n_chains,
                            st, &cfg, attr);
  if (e != cudaSuccess) return e;
  if (t) t->start();
  e = cudaLaunchKernelEx(&cfg, k_csample_spin2<N, MR>, a);
  if (t) t->stop();
  return e != cudaSuccess ? e : cudaGetLastError();
}
#define WF_INSTANTIATE_CLUSTER_BAND(N, MR)                                                      \
  template cudaError_t launch_csample_band<N, MR>(const SampleArgs&, cudaStream_t, LaunchTimer*); \
  template cudaError_t csample_band_clusters<N, MR>(int, int*);
#define WF_INSTANTIATE_CLUSTER_SPIN2(N, MR) \
  template cudaError_t launch_csample_spin2<N, MR>(const Spin2Args&, cudaStream_t, LaunchTimer*);
#endif

}  // namespace wf
