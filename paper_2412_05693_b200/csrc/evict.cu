// Stand-alone eviction kernel: one CTA per (sample, kv-head) cache.  Used after a prefill block
// (candidates = cached pairs + the block's pairs) and by bm_evict (candidates = cached pairs).
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

// A call of few caches shares each among a cluster, so that more SMs move rows -- at most 8 CTAs (64 bytes of a row
// each), only clusters that are all resident at once, and at least 96 KB of rows for each CTA (a cluster's barrier costs
// about 1 us).  Grids of at most one CTA per SM with more than a chunk of 64 KB to move keep twice as many pieces in
// flight (a chunk is one round trip to memory).  us per call, against one CTA per cache with 64 KB chunks: 8 caches cut
// from 1536 to 1024 pairs of 512 bytes 10.9 -> 8.6 (clusters of 8), 16 caches cut from 1024 to 512 pairs of 1 KB 12.2 ->
// 8.7 (4), 32 caches of 1024 to 512 pairs of 512 bytes 9.5 -> 8.3 (4), 128 caches of 768 to 512 pairs 10.5 -> 10.0.
template <typename T, int D, bool FILL>
cudaError_t launch_f(const CacheView& c, const EvictArgs& e, cudaStream_t st) {
  const int units = c.nsamples * c.Hkv, most = units <= 8 ? 8 : units <= 32 ? 4 : units <= 64 ? 2 : 1;
  const size_t bytes = (size_t)e.target * D * 2 * sizeof(T);   // that may move per cache
  int cluster = 1;
  while (cluster < most && bytes > (size_t)cluster * (96 << 10)) cluster *= 2;
  const bool wide = cluster * units <= sm_count() && bytes > (size_t)cluster * (64 << 10);
  return wide ? launch_w<T, D, FILL, 16>(c, e, cluster, st) : launch_w<T, D, FILL, 8>(c, e, 1, st);
}

template <typename T, int D>
cudaError_t launch_t(const CacheView& c, const EvictArgs& e, cudaStream_t st) {
  return c.fill ? launch_f<T, D, true>(c, e, st) : launch_f<T, D, false>(c, e, st);
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
