// Stand-alone eviction kernel: one CTA per (sample, kv-head) cache.  Used after a prefill block
// (candidates = cached pairs + the block's pairs) and by bm_evict (candidates = cached pairs).
#include <algorithm>

#include "evict.cuh"

namespace bm {
namespace {

constexpr int kEvictThreads = 512;

template <typename T, int D, bool FILL, int W>
__global__ void __launch_bounds__(kEvictThreads, W > 8 ? 1 : 2) evict_kernel(CacheView c, EvictArgs e) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t rank, count;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(count));
  const int unit = blockIdx.x / count;
  EvictShare share;
  share.rank = (int)rank;
  share.count = (int)count;
  pdl_wait();
  evict_body_impl<T, D, kEvictThreads, FILL, W>(c, unit, unit / c.Hkv, unit % c.Hkv, e, smem_raw, share);
}

template <typename T, int D, bool FILL, int W>
cudaError_t launch_w(const CacheView& c, const EvictArgs& e, int cluster, cudaStream_t st) {
  const size_t smem = evict_smem_bytes(c.n_old + e.I, e.target);
  static SmemConfigured configured;
  if (cudaError_t err = configured.ensure(evict_kernel<T, D, FILL, W>, smem); err != cudaSuccess) return err;
  ProfileScope prof(kEvict, st);
  const cudaError_t err = launch_dependent_cluster(evict_kernel<T, D, FILL, W>, dim3(c.nsamples * c.Hkv * cluster),
                                                   dim3(kEvictThreads), smem, cluster, st, c, e);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

// A call of few caches shares each among a cluster of 8, 4 or 2 CTAs, so that more SMs move rows, as long as all are
// resident at once and 256 KB and 64 KB for each CTA may move (a cluster's barrier costs about 1 us); its threads keep
// twice as many pieces in flight.  us per prefill call, all three kernels (cluster / one CTA per cache): 8 caches cut from
// 1536 to 1024 pairs of 512 bytes 40.0 / 41.2, 16 caches likewise 43.0 / 46.0 (4 CTAs), 32 caches from 1024 to 512 pairs 38.0
// / 40.0 and from 2012 to 1500 63.4 / 69.0, 64 caches from 768 to 512 37.0 / 38.2 (2) and from 1536 to 1024 70.0 / 73.0; less
// to move: 8 caches from 1024 to 512 32.0 / 31.5, 16 caches from 600 to 300 28.3 / 27.0.  Unordered caches move little and
// gained nothing (8 caches to 1024 pairs 40.2 / 39.4); as many pieces in flight without a cluster cost 1 to 4 us (128
// caches from 768 to 512 50.6 / 48.8).
// Up to two caches per SM in a layer the handle's caches decide, not the call's: sample ranges of such a batch may be in flight
// together, and clusters of one then take the SMs that the others' kernels need (16 samples, 16 blocks of 256 in a replayed graph,
// in 4 ranges on 4 streams 1.79 ms with clusters, 1.60 without, in 8 ranges 1.93 / 1.61, in one 1.59).  A range of a larger batch
// shares as a call of its own does (one sample of 64, 512 pairs more than the 1024 that stay 53.1 / 58.2 us per call).
template <typename T, int D>
cudaError_t launch_t(const CacheView& c, const EvictArgs& e, cudaStream_t st) {
  if (c.fill) return launch_w<T, D, true, 8>(c, e, 1, st);
  const int units = c.layer_units <= 2 * sm_count() ? c.layer_units : c.nsamples * c.Hkv;
  const int cluster = units <= 8 ? 8 : units <= 32 ? 4 : units <= 64 ? 2 : 1;
  const size_t bytes = (size_t)e.target * D * 2 * sizeof(T);   // that may move per cache
  if (cluster > 1 && cluster * units <= sm_count() && bytes >= std::max((size_t)256 << 10, (size_t)cluster << 16))
    return launch_w<T, D, false, 16>(c, e, cluster, st);
  return launch_w<T, D, false, 8>(c, e, 1, st);
}

}  // namespace

// Self-test of the checked build's row test: asks it about the first row index past the cache (nothing is accessed).
__global__ void row_check_selftest(CacheView c) { (void)row_ok(c, c.cap); }

cudaError_t launch_row_check_selftest(const CacheView& c, cudaStream_t st) {
  row_check_selftest<<<1, 1, 0, st>>>(c);
  count_launch();
  return cudaGetLastError();
}

size_t evict_smem_bytes(int n_cand, int target) { return evict_smem_layout(nullptr, n_cand, target, nullptr); }

cudaError_t launch_evict(int dtype, int d, const CacheView& c, const EvictArgs& e, cudaStream_t st) {
  if (dtype == 0 && d == 64) return launch_t<float, 64>(c, e, st);
  if (dtype == 0 && d == 128) return launch_t<float, 128>(c, e, st);
  if (dtype == 1 && d == 64) return launch_t<__nv_bfloat16, 64>(c, e, st);
  if (dtype == 1 && d == 128) return launch_t<__nv_bfloat16, 128>(c, e, st);
  return cudaErrorInvalidValue;
}

}  // namespace bm
