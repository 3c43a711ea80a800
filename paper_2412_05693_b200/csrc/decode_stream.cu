// bf16 decoding step (the token-generation step of Algorithm 1; Sec. 3.2 with I = 1) as a stream: the caches' rows pass
// through a ring of shared-memory tiles that one thread keeps filled by TMA, whatever the multiplying warps are doing,
// so that HBM is read at its rate while softmax, ranking and row moves of a cache go on.
//
// A cluster of C CTAs (C = 1, 2, 4 or 8) owns one cache at a time and takes further caches in turn (a persistent grid,
// one CTA per SM); each CTA holds a contiguous piece of the cache's rows, cut at tile borders.  Warps of a CTA:
//   0-7  consumers: logits = K-tile . q^T (m16n8k16 fragments by ldmatrix from the swizzled tile, heads padded to 8),
//        softmax, sum_weights update, ranking, out^T = V-tile^T . p^T (each warp owns 16 elements of the head dimension)
//   8    producer: K tiles, then V tiles of every cache the CTA has a piece of
//   9    V rows behind the pair that leaves: TMA stores straight from the ring, one row higher than they were read
//   10   K rows behind the pair that leaves, stored likewise: from the ring where it still holds them (one cache per CTA
//        and room for all of its piece), else read again out of L2, where the logits pass left them
// With C > 1 the CTAs exchange (maximum, sum), the ranking's minimum and the partial outputs through distributed
// shared memory, one mbarrier per exchange.  A thread waits for a barrier before the next phase of it can begin: the
// wait for the previous cache's moves is the publishing thread's alone (a form in which every thread waited behind
// the publication could fall two phases back and time out).
//
// What bounds it: HBM once there is a cache for every SM; below that the latency of one cache's chain (first tile ->
// softmax -> last tile -> moves), which is what splitting a cache over a cluster shortens.  One pair leaving per step,
// caches of 1024 pairs, d = 128, us per step against the kernel in decode_mma.cu: 8 caches (g = 4) 6.6 / 15.4 (10.1 with
// exchanges by plain remote stores and releasing arrivals, which wait for the sender's global stores; 8.2 with a loop
// over the peers' statistics and a releasing barrier at the end), 128
// caches 16.8 / 19.1, 1024 caches 95 / 112 (5.9 against 5.0 TB/s of algorithmic bytes), 3072 caches 267 / 304 (6.3 TB/s),
// 1024 caches without groups 88 / 104 (6.3 TB/s).  Since then per-row loops stay rolled, clusters have instances of their own and
// statistics are folded across lanes: 88 KB of code became 44 and 54, where an SM's instruction cache holds 32, and a
// replayed step on 8 caches went from 6.2 to 5.5 us, on 32 layers of 32 caches of 512 pairs from 8.0 to 7.1, on 1024 caches from 92
// to 91.  Not kept: tiles of 32 KB with two tiles' fragments in flight per warp
// (spills; 111 against 94 us at 1024 caches), the per-row loops four rows at a time (+2 to 8 %), sums and ids written by
// a warp of their own (+5 to 15 %: one warp's stores are on the chain to the next cache).
#include <algorithm>

#include "common.cuh"
#include "tc_common.cuh"

namespace bm {
namespace {

using namespace tc;

constexpr float kLog2e = 1.4426950408889634f;
constexpr int kConsumers = 256, kCWarps = 8;
constexpr int kThreads = kConsumers + 96;
constexpr int kTile = 16384;            // bytes of a ring tile
constexpr int kMaxCluster = 8;
constexpr int kMoveTiles = 2;           // staging tiles of the K move

struct StreamArgs {
  const void* q;
  const void* k;
  const void* v;
  void* out;
  int32_t pos;
  float scale;
  int32_t evict_one;   // 1: exactly one pair leaves (0: the step's pair is appended)
  int32_t units;       // caches of the call
  int32_t stages;      // ring tiles
  int32_t single;      // 1: every CTA works on one cache only
  int32_t keep_k;      // 1: ... and the ring holds all of its piece's tiles
  int32_t rows_cta;    // rows the per-row arrays have room for (a multiple of the tile's rows)
};
struct StreamMaps {
  CUtensorMap k_ld, v_ld;   // rows [0, n_old) of every cache, boxes of one tile x 64 elements
  CUtensorMap k_st, v_st;   // rows [0, n_old - 1), boxes of 8 rows x 64 elements
};

template <int D, int G>
struct StreamSmem {
  static constexpr int TR = kTile / (2 * D);     // rows per tile: 64 (d = 128) or 128 (d = 64)
  // barriers: ring full / empty (up to 16 stages each), K-move full, hole known, moves done, cluster exchanges [3], the piece before has been read (V, K)
  static constexpr int kMaxStages = 16;
  static constexpr int B_FULL = 0, B_EMPTY = kMaxStages, B_KM = 2 * kMaxStages, B_HOLE = B_KM + kMoveTiles, B_MOVED = B_HOLE + 1,
                       B_X = B_MOVED + 1, B_PREV = B_X + 3, B_COUNT = B_PREV + 2;
  static constexpr int kMisc = 4 * D + 16 * (kCWarps + kMaxCluster)              // first rows; minima
                               + 4 * (2 * kCWarps * G + kMaxCluster * 2 * G + G * D)   // maxima, sums, statistics, outputs
                               + 8 * B_COUNT + 8 + 4 * G + 64;                      // barriers, flags, slack
  __host__ __device__ static size_t row_bytes(int rows) {            // per-row arrays: p, pb, id [2], sw [2]
    return (size_t)rows * (4 * G + 16) + (size_t)G * (rows + 8) * 2;
  }
  __host__ __device__ static size_t total(int rows, int tiles) {     // tiles: of the ring and of the K move
    return 1024 + (size_t)tiles * kTile + row_bytes(rows) + kMisc;
  }
};

__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Stores into a peer's shared memory that count themselves on the peer's barrier `bar` (transaction bytes): the receiver
// waits for the bytes, and the sender needs no release fence, which would wait for its outstanding global stores.
__device__ __forceinline__ void st_peer(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
               ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_peer4(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}
__device__ __forceinline__ void arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// bounded like mbar_wait, with acquire semantics over the cluster
__device__ __forceinline__ void wait_cluster(uint64_t* b, uint32_t parity, volatile int* abort_flag, int* status) {
  const uint32_t addr = smem_u32(b);
  if (*abort_flag) return;
#pragma unroll 1
  for (int it = 0; it < kWaitLimit; ++it) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\nselp.b32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(addr), "r"(parity), "r"(kWaitSleepNs) : "memory");
    if (ok) return;
    if ((it & 255) == 255 && *abort_flag) return;
  }
  *abort_flag = 1;
  atomicExch(status, kErrTimeout);
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// one arrival of the warp, once all of its lanes are here
__device__ __forceinline__ void arrive_one(uint64_t* b, int lane) {
  __syncwarp();
  asm volatile("{\n.reg .pred p;\nsetp.eq.s32 p, %1, 0;\n@p mbarrier.arrive.shared::cta.b64 _, [%0];\n}\n" ::"r"(smem_u32(b)), "r"(lane) : "memory");
}
template <int G>
__device__ __forceinline__ void ld_heads(const float* p, float (&e)[G]) {
  if constexpr (G == 1) e[0] = p[0];
  else if constexpr (G == 2) { const float2 t = *reinterpret_cast<const float2*>(p); e[0] = t.x; e[1] = t.y; }
  else {
#pragma unroll
    for (int i = 0; i < G / 4; ++i) {
      const float4 t = reinterpret_cast<const float4*>(p)[i];
      e[4 * i] = t.x; e[4 * i + 1] = t.y; e[4 * i + 2] = t.z; e[4 * i + 3] = t.w;
    }
  }
}
template <int G>
__device__ __forceinline__ void st_heads(float* p, const float (&e)[G]) {
  if constexpr (G == 1) p[0] = e[0];
  else if constexpr (G == 2) *reinterpret_cast<float2*>(p) = make_float2(e[0], e[1]);
  else {
#pragma unroll
    for (int i = 0; i < G / 4; ++i)
      reinterpret_cast<float4*>(p)[i] = make_float4(e[4 * i], e[4 * i + 1], e[4 * i + 2], e[4 * i + 3]);
  }
}

// byte offset of the 16-byte piece pc (0 .. D/8 - 1) of tile row r
template <int D>
__device__ __forceinline__ uint32_t piece_offset(int r, int pc) {
  constexpr int TR = kTile / (2 * D);
  return (uint32_t)((pc >> 3) * (TR * 128) + r * 128 + (((pc & 7) ^ (r & 7)) << 4));
}

// One warp: rows [lo, hi) of the tile that starts at cache row g0 go one row up, from shared memory: up to the next
// multiple of 8 rows (the swizzle's period) by plain stores, the rest as TMA stores of 8 rows.  Rows that would land
// at n_old - 1 or above are clipped by the map.  The tile may be overwritten after moves_have_read().
template <int D>
__device__ __forceinline__ void move_rows_up(const CacheView& c, const unsigned char* tile, int g0, int lo, int hi,
                                             const CUtensorMap* map, int unit, __nv_bfloat16* slab, int lane) {
  constexpr int TR = kTile / (2 * D), PR = D / 8, CH = D / 64;
  const int lo8 = (lo + 7) & ~7, plain_end = min(lo8, hi);
#pragma unroll 1
  for (int x = lane; x < (plain_end - lo) * PR; x += 32) {
    const int row = lo + x / PR, pc = x % PR;
    if (row_ok(c, row - 1))
      st_global_16(slab + (size_t)(row - 1) * D + pc * 8, *reinterpret_cast<const uint4*>(tile + piece_offset<D>(row - g0, pc)));
  }
  const int ops = hi > lo8 ? (hi - lo8 + 7) / 8 * CH : 0;   // at most 16
  if (lane < ops) {
    const int grp = lane / CH, ch = lane % CH;
    tma_store_3d(map, tile + ch * (TR * 128) + (lo8 - g0 + 8 * grp) * 128, ch * 64, lo8 + 8 * grp - 1, unit);
  }
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// waits until at most n of the calls above still have to read their tile
template <int N>
__device__ __forceinline__ void moves_have_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
  __syncwarp();
}

// SHARED: clusters of 2, 4 or 8 CTAs own a cache together, and a CTA works on one cache only; instances of their own, so
// that neither kind carries the other's code
template <int D, int G, bool SHARED>
__global__ void __launch_bounds__(kThreads, 1)
decode_stream_kernel(const CacheView c, const StreamArgs a, const __grid_constant__ StreamMaps maps) {
  using T = __nv_bfloat16;
  using L = StreamSmem<D, G>;
  constexpr int TR = L::TR, PR = D / 8, CH = D / 64;
  constexpr int WPT = TR / 16;            // warps that share a K tile (16 rows each)
  constexpr int NG = kCWarps / WPT;       // K tiles are taken in turn by NG groups of warps
  constexpr int WS = D / 16;              // slices of the head dimension in the output product, one per warp
  constexpr int KH = kCWarps / WS;        // key groups that share a slice (2 at d = 64)
  extern __shared__ unsigned char smem_raw[];
  // (every CTA of a cluster has the same layout: peers address each other's arrays by offset)
  unsigned char* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int NS = a.stages, RC = a.rows_cta;
  unsigned char* ring = sm;
  // The K move's tiles pass through two tiles of their own -- or, when the CTA has no further cache to prefetch, through
  // the ring behind the V tiles (all of its tiles are then free for them), or they are still in the ring.
  unsigned char* kst = ring + NS * kTile;
  float* s_p = reinterpret_cast<float*>(kst + (SHARED || a.single ? 0 : kMoveTiles * kTile));   // [RC][G] logits, then exp2(logit - maximum of the CTA)
  float* s_sw2 = s_p + (size_t)RC * G;                // [2][RC] sum_weights of this cache and of the next one
  int* s_id2 = reinterpret_cast<int*>(s_sw2 + 2 * RC);   // [2][RC] kv_ids, likewise
  T* s_pb = reinterpret_cast<T*>(s_id2 + 2 * RC);     // [G][RC + 8] the exponentials as bf16
  const int PBS = RC + 8;                             // (row stride = 4 words modulo 32: the 8 heads' words do not collide)
  unsigned char* misc = reinterpret_cast<unsigned char*>(s_pb + (size_t)G * PBS);
  T* s_first = reinterpret_cast<T*>(misc);                                // [2][D]: first K / V row of the piece
  int4* s_best = reinterpret_cast<int4*>(misc + 4 * D);                   // [warps] (key, row, position)
  int4* s_xbest = s_best + kCWarps;                                       // [cluster], exchanged
  float* s_wmax = reinterpret_cast<float*>(s_xbest + kMaxCluster);        // [warps][G]
  float* s_wsum = s_wmax + kCWarps * G;                                   // [warps][G]
  float* s_xstat = s_wsum + kCWarps * G;                                  // [cluster][2][G], exchanged
  float* s_xout = s_xstat + kMaxCluster * 2 * G;                          // [cluster][G * D / C], exchanged
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_xout + G * D);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + L::B_COUNT);
  volatile int* s_hole = abort_flag + 1;
  float* s_enew = const_cast<float*>(reinterpret_cast<volatile float*>(s_hole + 1));   // [G] exponentials of the step's own pair

  uint32_t rank = 0, C = 1;
  if (SHARED) {
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  }
  const bool single = SHARED || a.single;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_old = c.n_old, n1 = n_old + 1;
  const int tiles = (n1 + TR - 1) / TR;
  const int t0 = (int)(rank * tiles / C), t1 = (int)((rank + 1) * tiles / C);   // this CTA's tiles
  const int kt = t1 - t0;
  const int r0 = t0 * TR, nr = min(n1, t1 * TR) - r0;                   // its rows (the step's own pair is row n_old)
  const int vt = min(t1, (n_old + TR - 1) / TR) - t0;                   // tiles that hold cached rows
  const bool has_new = r0 + nr == n1;
  const int cl0 = blockIdx.x / C, n_cl = gridDim.x / C;

  // a ring tile is given back by the consumers, the V-move warp and, where its own tiles follow in the ring, the K-move warp
  const bool k_in_ring = single && !a.keep_k;
  const int empty_count = kCWarps + 1 + (k_in_ring ? 1 : 0);
  if (tid == 0) {
    *abort_flag = 0;
#pragma unroll 1
    for (int s = 0; s < NS; ++s) { mbar_init(&bars[L::B_FULL + s], 1); mbar_init(&bars[L::B_EMPTY + s], empty_count); }
#pragma unroll 1
    for (int x = 0; x < kMoveTiles; ++x) mbar_init(&bars[L::B_KM + x], 1);
    mbar_init(&bars[L::B_HOLE], 1);
    mbar_init(&bars[L::B_MOVED], 2);
#pragma unroll 1
    for (int x = 0; x < 5; ++x) mbar_init(&bars[L::B_X + x], 1);
    mbar_fence_init();
  }
  if (tid == kConsumers) {
    const auto prefetch = [](const CUtensorMap* m) { asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory"); };
    prefetch(&maps.k_ld); prefetch(&maps.v_ld); prefetch(&maps.k_st); prefetch(&maps.v_st);
  }
  __syncthreads();
  if (SHARED) {   // the peers' barriers exist
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
  // programmatic dependent launch: nothing the predecessor may have written is touched before this point
  pdl_wait();
  pdl_release();
  const bool shift = a.evict_one && !c.fill;
  // (x = 0: V, 1: K) This CTA has read the rows of its piece: the next one may move its first row to the last of them.
  // The own first row goes there likewise, once the CTA before has said so.
  auto first_row_up = [&](int x, T* slab, int hole, const uint4& own) {
    __syncwarp();
    if (rank + 1 < C && lane == 0) arrive_cluster(mapa(smem_u32(&bars[L::B_PREV + x]), rank + 1));
    if (rank > 0) {
      wait_cluster(&bars[L::B_PREV + x], 0, abort_flag, c.status);
      if (shift && hole < r0 && lane < PR && row_ok(c, r0 - 1))   // (r0 may be the step's own pair)
        st_global_16(slab + (size_t)(r0 - 1) * D + lane * 8, r0 == n_old ? own : reinterpret_cast<const uint4*>(s_first + (x == 0 ? D : 0))[lane]);
    }
  };

  if (warp == kCWarps) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      int e = 0, slot = 0, ph = 0;
#pragma unroll 1
      for (int unit = cl0; unit < a.units; unit += n_cl)
#pragma unroll 1
        for (int x = 0; x < kt + vt; ++x, ++e) {
          if (e >= NS) mbar_wait(&bars[L::B_EMPTY + slot], ph ^ 1, abort_flag, c.status);
          const bool is_v = x >= kt;
          const int row = (t0 + (is_v ? x - kt : x)) * TR;
          mbar_expect_tx(&bars[L::B_FULL + slot], kTile);
#pragma unroll
          for (int ch = 0; ch < CH; ++ch)
            tma_load_3d(ring + slot * kTile + ch * (TR * 128), is_v ? &maps.v_ld : &maps.k_ld, ch * 64, row, unit,
                        &bars[L::B_FULL + slot]);
          if (++slot == NS) { slot = 0; ph ^= 1; }
        }
      if (k_in_ring && shift) {   // the K tiles behind the pair that leaves, once more
        mbar_wait(&bars[L::B_HOLE], 0, abort_flag, c.status);
#pragma unroll 1
        for (int x = max(0, (*s_hole + 1) / TR - t0); x < vt; ++x, ++e) {
          if (e >= NS) mbar_wait(&bars[L::B_EMPTY + slot], ph ^ 1, abort_flag, c.status);
          mbar_expect_tx(&bars[L::B_FULL + slot], kTile);
#pragma unroll
          for (int ch = 0; ch < CH; ++ch)
            tma_load_3d(ring + slot * kTile + ch * (TR * 128), &maps.k_ld, ch * 64, (t0 + x) * TR, cl0, &bars[L::B_FULL + slot]);
          if (++slot == NS) { slot = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp == kCWarps + 1) {
    // ---------------------------------------------------------------- V rows behind the pair that leaves; the step's V row
    int slot = 0, ph = 0, it = 0;
#pragma unroll 1
    for (int unit = cl0; unit < a.units; unit += n_cl, ++it) {
      T* vslab = reinterpret_cast<T*>(c.v_slab) + (size_t)unit * c.cap * D;
      uint4 own = make_uint4(0u, 0u, 0u, 0u);  // the step's own row
      if (lane < PR) own = ld_global_16(reinterpret_cast<const T*>(a.v) + (size_t)unit * D + lane * 8);
#pragma unroll 1
      for (int x = 0; x < kt; ++x) {          // (K tiles: the consumers')
        mbar_wait(&bars[L::B_FULL + slot], ph, abort_flag, c.status);
        arrive_one(&bars[L::B_EMPTY + slot], lane);
        if (++slot == NS) { slot = 0; ph ^= 1; }
      }
      mbar_wait(&bars[L::B_HOLE], it & 1, abort_flag, c.status);
      const int hole = *s_hole;
#pragma unroll 1
      for (int x = 0; x < vt; ++x) {
        mbar_wait(&bars[L::B_FULL + slot], ph, abort_flag, c.status);
        __syncwarp();
        const unsigned char* tile = ring + slot * kTile;
        const int g0 = (t0 + x) * TR;
        if (shift && g0 + TR > hole + 1) {
          int lo = max(g0, hole + 1);
          if (x == 0 && rank > 0 && lo == g0) {   // its place is still being read by another CTA: later
            if (lane < PR) reinterpret_cast<uint4*>(s_first + D)[lane] = *reinterpret_cast<const uint4*>(tile + piece_offset<D>(0, lane));
            ++lo;
          }
          move_rows_up<D>(c, tile, g0, lo, min(g0 + TR, n_old), &maps.v_st, unit, vslab, lane);
          moves_have_read<0>();
        }
        arrive_one(&bars[L::B_EMPTY + slot], lane);
        if (++slot == NS) { slot = 0; ph ^= 1; }
      }
      // every V row of the piece has been read: the step's own row takes its place
      const int dst = a.evict_one ? (c.fill ? hole : n_old - 1) : n_old;
      const bool mine = c.fill && a.evict_one ? (hole >= r0 && hole < r0 + nr) : (has_new && !(shift && r0 == n_old));
      if (hole != n_old && mine && lane < PR && row_ok(c, dst))
        st_global_16(vslab + (size_t)dst * D + lane * 8, own);
      if (SHARED) first_row_up(0, vslab, hole, own);
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[L::B_MOVED]);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  } else if (warp == kCWarps + 2) {
    // ---------------------------------------------------------------- K rows behind the pair that leaves; the step's K row
    int e = 0, it = 0;                        // K-move tiles so far: tile e sits in buffer e % kMoveTiles
#pragma unroll 1
    for (int unit = cl0; unit < a.units; unit += n_cl, ++it) {
      T* kslab = reinterpret_cast<T*>(c.k_slab) + (size_t)unit * c.cap * D;
      uint4 own = make_uint4(0u, 0u, 0u, 0u);
      if (lane < PR) own = ld_global_16(reinterpret_cast<const T*>(a.k) + (size_t)unit * D + lane * 8);
      if (k_in_ring)
#pragma unroll 1
        for (int f = 0; f < kt + vt; ++f) {
          mbar_wait(&bars[L::B_FULL + f % NS], (f / NS) & 1, abort_flag, c.status);
          arrive_one(&bars[L::B_EMPTY + f % NS], lane);
        }
      mbar_wait(&bars[L::B_HOLE], it & 1, abort_flag, c.status);
      const int hole = *s_hole;
      if (shift) {
        const int x0 = max(0, (hole + 1) / TR - t0);   // first tile of the piece with a row that moves
        auto fetch = [&](int x, int n) {
          const int b = n % kMoveTiles;
          if (lane == 0) {
            mbar_expect_tx(&bars[L::B_KM + b], kTile);
#pragma unroll
            for (int ch = 0; ch < CH; ++ch)
              tma_load_3d(kst + b * kTile + ch * (TR * 128), &maps.k_ld, ch * 64, (t0 + x) * TR, unit, &bars[L::B_KM + b]);
          }
        };
        auto move = [&](int x, const unsigned char* tile) {
          const int g0 = (t0 + x) * TR;
          int lo = max(g0, hole + 1);
          if (x == 0 && rank > 0 && lo == g0) {
            if (lane < PR) reinterpret_cast<uint4*>(s_first)[lane] = *reinterpret_cast<const uint4*>(tile + piece_offset<D>(0, lane));
            ++lo;
          }
          move_rows_up<D>(c, tile, g0, lo, min(g0 + TR, n_old), &maps.k_st, unit, kslab, lane);
        };
        if (single) {
#pragma unroll 1
          for (int x = x0; x < vt; ++x) {
            const int f = a.keep_k ? x : kt + vt + x - x0;   // the tile's place in the order of the ring
            mbar_wait(&bars[L::B_FULL + f % NS], (f / NS) & 1, abort_flag, c.status);
            move(x, ring + (f % NS) * kTile);
            if (k_in_ring && vt - x > NS) {                  // its place is needed once more: every arrival is this warp's
              moves_have_read<0>();
              if (lane == 0)
#pragma unroll 1
                for (int y = 0; y < empty_count; ++y) mbar_arrive(&bars[L::B_EMPTY + f % NS]);
            }
          }
        } else {
          // kMoveTiles - 1 tiles are on their way while one is being stored (their rows lie above everything stored so far)
          int ahead = x0;
          for (; ahead < min(vt, x0 + kMoveTiles - 1); ++ahead) fetch(ahead, e + ahead - x0);
#pragma unroll 1
          for (int x = x0; x < vt; ++x, ++e) {
            if (ahead < vt) {   // into the buffer of the tile before this one
              moves_have_read<0>();
              fetch(ahead, e + kMoveTiles - 1);
              ++ahead;
            }
            mbar_wait(&bars[L::B_KM + e % kMoveTiles], (e / kMoveTiles) & 1, abort_flag, c.status);
            move(x, kst + (e % kMoveTiles) * kTile);
          }
        }
        moves_have_read<0>();
      }
      const int dst = a.evict_one ? (c.fill ? hole : n_old - 1) : n_old;
      const bool mine = c.fill && a.evict_one ? (hole >= r0 && hole < r0 + nr) : (has_new && !(shift && r0 == n_old));
      if (hole != n_old && mine && lane < PR && row_ok(c, dst))
        st_global_16(kslab + (size_t)dst * D + lane * 8, own);
      if (SHARED) first_row_up(1, kslab, hole, own);
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[L::B_MOVED]);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  } else {
    // ---------------------------------------------------------------- consumers
    const int gid = lane >> 2, tq = lane & 3;
    const int ws = warp % WS, kg = warp / WS;              // slice of the head dimension, key group (output product)
    const int wg = warp / WPT, wr = (warp % WPT) * 16;     // tile group; first row of this warp in its tiles
    const float sc2 = a.scale * kLog2e;
    const bool avg = c.rule == 0 || c.rule == 4;
    uint32_t qf[D / 16][2];
    auto load_q = [&](int unit) {     // B fragments: elements 16 ks + 2 tq, +1 and + 8 of head gid
      const uint32_t* qp = reinterpret_cast<const uint32_t*>(reinterpret_cast<const T*>(a.q) + ((size_t)unit * G + gid) * D);
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        qf[ks][0] = gid < G ? qp[8 * ks + tq] : 0u;
        qf[ks][1] = gid < G ? qp[8 * ks + tq + 4] : 0u;
      }
    };
    // kv_ids and sum_weights of a cache's rows into buffer b; they arrive while the cache before it is worked on
    auto fetch_rows = [&](int unit, int b) {
      const size_t base = (size_t)unit * c.cap;
#pragma unroll 1
      for (int jl = tid; jl < nr; jl += kConsumers) {
        const int j = r0 + jl;
        if (j < n_old) {
          cp_async4(&s_id2[b * RC + jl], &c.kv_ids[base + j]);
          cp_async4(&s_sw2[b * RC + jl], &c.sum_weights[base + j]);
        } else {
          s_id2[b * RC + jl] = a.pos;
          s_sw2[b * RC + jl] = 0.f;
        }
      }
    };
    // the step's own key row (by the warp whose rows it joins) and the elements of its value row this warp adds up
    const int new_l = n_old - r0;
    const bool new_key_here = has_new && (new_l / TR) % NG == wg && (new_l % TR) / 16 * 16 == wr;
    uint4 k_new = make_uint4(0u, 0u, 0u, 0u);
    T v_next[2] = {};
    auto load_new_k = [&](int unit) {
      if (new_key_here && lane < PR) k_new = ld_global_16(reinterpret_cast<const T*>(a.k) + (size_t)unit * D + lane * 8);
    };
    auto load_new_v = [&](int unit) {
      if (has_new)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) v_next[hf] = reinterpret_cast<const T*>(a.v)[(size_t)unit * D + 16 * ws + gid + 8 * hf];
    };
    if (cl0 < a.units) {
      load_q(cl0);
      load_new_k(cl0);
      load_new_v(cl0);
      fetch_rows(cl0, 0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    int slot = 0, ph = 0, it = 0;
#pragma unroll 1
    for (int unit = cl0; unit < a.units; unit += n_cl, ++it) {
      const int smp = unit / c.Hkv, next = unit + n_cl;
      const size_t base = (size_t)unit * c.cap;
      const int pad = sample_left_pad(c, smp);
      const bool q_real = a.pos >= pad;
      int* s_id = s_id2 + (it & 1) * RC;
      float* s_sw = s_sw2 + (it & 1) * RC;
      if (next < a.units) fetch_rows(next, (it + 1) & 1);
      asm volatile("cp.async.commit_group;" ::: "memory");
      // ---- logits (log2 domain)
      float mx0 = -INFINITY, mx1 = -INFINITY;              // running maxima of heads 2 tq, 2 tq + 1
#pragma unroll 1
      for (int t = 0; t < kt; ++t) {
        mbar_wait(&bars[L::B_FULL + slot], ph, abort_flag, c.status);
        const int jl0 = t * TR + wr;                        // first row of this warp's 16, local
        if (t % NG == wg && jl0 < nr) {
          unsigned char* tile = ring + slot * kTile;
          if (new_key_here && t == new_l / TR) {
            if (lane < PR) *reinterpret_cast<uint4*>(tile + piece_offset<D>(new_l % TR, lane)) = k_new;
            fence_async_smem();                             // (the slot's next TMA write comes after it)
            __syncwarp();
          }
          float acc[2][4] = {};
          const int krow = wr + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            uint32_t a0, a1, a2, a3;
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3)
                         : "r"(smem_u32(tile) + piece_offset<D>(krow, 2 * ks + (lane >> 4))) : "memory");
            mma16816(acc[ks & 1], a0, a1, a2, a3, qf[ks][0], qf[ks][1]);
          }
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            const int jl = jl0 + gid + 8 * hf;
            const float x0 = (acc[0][2 * hf] + acc[1][2 * hf]) * sc2, x1 = (acc[0][2 * hf + 1] + acc[1][2 * hf + 1]) * sc2;
            if (jl < nr) {
              if constexpr (G == 1) { if (tq == 0) s_p[jl] = x0; }
              else if (2 * tq < G) *reinterpret_cast<float2*>(&s_p[jl * G + 2 * tq]) = make_float2(x0, x1);
              mx0 = fmaxf(mx0, x0);
              mx1 = fmaxf(mx1, x1);
            }
          }
        }
        arrive_one(&bars[L::B_EMPTY + slot], lane);
        if (++slot == NS) { slot = 0; ph ^= 1; }
      }
      const float v_new[2] = {__bfloat162float(v_next[0]), __bfloat162float(v_next[1])};
      if (next < a.units) {                                 // on their way for the next cache
        load_q(next);
        load_new_k(next);
        load_new_v(next);
      }
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) {
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, off));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, off));
      }
      if (gid == 0 && 2 * tq < G) {
        s_wmax[warp * G + 2 * tq] = mx0;
        if (G > 1) s_wmax[warp * G + 2 * tq + 1] = mx1;
      }
      asm volatile("cp.async.wait_group 1;" ::: "memory");  // this cache's ids and sums have arrived
      named_bar_sync(1, kConsumers);
      // [warps][G] folded into every thread: a lane takes one warp's value of one head (four heads at a time)
      auto all_warps = [&](const float* per_warp, float (&r)[G], auto op) {
        static_assert(kCWarps == 8, "");
#pragma unroll
        for (int q = 0; q < G; q += 4) {
          float t = per_warp[(lane & 7) * G + min(G - 1, q + (lane >> 3))];
#pragma unroll
          for (int off = 4; off > 0; off >>= 1) t = op(t, __shfl_xor_sync(0xffffffffu, t, off));
#pragma unroll
          for (int h = q; h < min(G, q + 4); ++h) r[h] = __shfl_sync(0xffffffffu, t, 8 * (h - q));
        }
      };
      float mc[G];
      all_warps(s_wmax, mc, [](float x, float y) { return fmaxf(x, y); });
      if (pad > 0 && q_real) {   // padding pairs are masked: the maxima again, over what is left
        float m2[G];
#pragma unroll
        for (int h = 0; h < G; ++h) m2[h] = -INFINITY;
#pragma unroll 1
        for (int jl = tid; jl < nr; jl += kConsumers) {
          float e[G];
          ld_heads<G>(&s_p[jl * G], e);
          const bool out_of_sight = s_id[jl] < pad;
#pragma unroll
          for (int h = 0; h < G; ++h) {
            if (out_of_sight) e[h] = -INFINITY;
            m2[h] = fmaxf(m2[h], e[h]);
          }
          st_heads<G>(&s_p[jl * G], e);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
          for (int h = 0; h < G; ++h) m2[h] = fmaxf(m2[h], __shfl_xor_sync(0xffffffffu, m2[h], off));
        named_bar_sync(1, kConsumers);                      // the first maxima have been read
        if (lane == 0)
#pragma unroll
          for (int h = 0; h < G; ++h) s_wmax[warp * G + h] = m2[h];
        named_bar_sync(1, kConsumers);
        all_warps(s_wmax, mc, [](float x, float y) { return fmaxf(x, y); });
      }
      // ---- exponentials relative to the CTA's maximum, and their sums
      {
        float t[G], ms[G];
#pragma unroll
        for (int h = 0; h < G; ++h) { t[h] = 0.f; ms[h] = mc[h] == -INFINITY ? 0.f : mc[h]; }   // (a piece of padding only)
#pragma unroll 1
        for (int jl = tid; jl < nr; jl += kConsumers) {
          float e[G];
          ld_heads<G>(&s_p[jl * G], e);
#pragma unroll
          for (int h = 0; h < G; ++h) { e[h] = ex2(e[h] - ms[h]); t[h] += e[h]; }
          st_heads<G>(&s_p[jl * G], e);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
          for (int h = 0; h < G; ++h) t[h] += __shfl_xor_sync(0xffffffffu, t[h], off);
        if (lane == 0)
#pragma unroll
          for (int h = 0; h < G; ++h) s_wsum[warp * G + h] = t[h];
      }
      named_bar_sync(1, kConsumers);
      float f[G];                                           // weight of a pair = its exponential * f
      if (!SHARED) {
        all_warps(s_wsum, f, [](float x, float y) { return x + y; });
#pragma unroll
        for (int h = 0; h < G; ++h) f[h] = q_real ? 1.f / f[h] : 0.f;
      } else {
        if (tid == 0) mbar_expect_tx(&bars[L::B_X], C * 2 * G * 4);
        if (warp == 0) {                                    // this CTA's statistics to every peer
          float t[G];
          all_warps(s_wsum, t, [](float x, float y) { return x + y; });
          if (lane < (int)C) {
            const uint32_t dst = mapa(smem_u32(s_xstat + rank * 2 * G), lane), bar = mapa(smem_u32(&bars[L::B_X]), lane);
            if constexpr (G % 4 == 0) {
#pragma unroll
              for (int h = 0; h < G; h += 4) {
                st_peer4(dst + 4 * h, __float_as_uint(mc[h]), __float_as_uint(mc[h + 1]), __float_as_uint(mc[h + 2]),
                         __float_as_uint(mc[h + 3]), bar);
                st_peer4(dst + 4 * (G + h), __float_as_uint(t[h]), __float_as_uint(t[h + 1]), __float_as_uint(t[h + 2]),
                         __float_as_uint(t[h + 3]), bar);
              }
            } else {
#pragma unroll
              for (int h = 0; h < G; ++h) {
                st_peer(dst + 4 * h, mc[h], bar);
                st_peer(dst + 4 * (G + h), t[h], bar);
              }
            }
          }
        }
        wait_cluster(&bars[L::B_X], it & 1, abort_flag, c.status);
        // a lane holds what one CTA said about one head (four heads at a time); the sum runs over the lanes in a fixed order
#pragma unroll
        for (int q = 0; q < G; q += 4) {
          const int p = lane & (kMaxCluster - 1), h = min(G - 1, q + (lane >> 3));
          const bool there = p < (int)C;
          const float m = there ? s_xstat[p * 2 * G + h] : -INFINITY, own = s_xstat[rank * 2 * G + h];
          float t = there ? s_xstat[p * 2 * G + G + h] : 0.f, top = m;
#pragma unroll
          for (int off = kMaxCluster / 2; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
          if (m != -INFINITY) t *= ex2(m - top);   // (-inf: a piece without weight, whose sum is 0, or NaN logits alone)
#pragma unroll
          for (int off = kMaxCluster / 2; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
          // (a piece without weight: 0; a cache whose logits are all -inf, or that holds a NaN: NaN)
          const float fh = q_real ? ex2(own - top) / t : 0.f;
#pragma unroll
          for (int y = q; y < min(G, q + 4); ++y) f[y] = __shfl_sync(0xffffffffu, fh, 8 * (y - q));
        }
      }
      // ---- sum_weights += attn_weights (heads added in a fixed order), candidate for eviction, bf16 exponentials
      // (the pair with the smallest ranking value leaves; ties: the higher position -- kv_ids, not rows: the rows of an
      // unordered cache are in no order.  Values are compared as ordered bit patterns, 0 = a padding pair.)
      uint32_t best_key = 0xffffffffu;
      int best_j = -1, best_id = -1;
      auto better = [&](uint32_t ok, int oj, int oi) {
        if (ok < best_key || (ok == best_key && oi > best_id)) { best_key = ok; best_j = oj; best_id = oi; }
      };
#pragma unroll 1
      for (int jl = nr + tid; jl < vt * TR; jl += kConsumers)   // rows of the last tile past the cache carry no weight
#pragma unroll
        for (int h = 0; h < G; ++h) s_pb[h * PBS + jl] = __float2bfloat16_rn(0.f);
#pragma unroll 1
      for (int jl = tid; jl < nr; jl += kConsumers) {
        const int j = r0 + jl, id = s_id[jl];
        float e[G];
        ld_heads<G>(&s_p[jl * G], e);
        float add = 0.f, add_sq = 0.f;
#pragma unroll
        for (int h = 0; h < G; ++h) {
          s_pb[h * PBS + jl] = __float2bfloat16_rn(e[h]);
          const float w = e[h] * f[h];
          add += w;
          add_sq = fmaf(w, w, add_sq);
        }
        if (j == n_old)
#pragma unroll
          for (int h = 0; h < G; ++h) s_enew[h] = e[h];
        const float sw = (rule_overwrites(c.rule) ? 0.f : s_sw[jl]) + add;   // rules 2, 3 keep this step's weights only
        if (c.sum_sq != nullptr) c.sum_sq[base + j] = (j < n_old ? c.sum_sq[base + j] : 0.f) + add_sq;   // rule 4
        if (a.evict_one) {
          s_sw[jl] = sw;
          float ave;   // ranking value: average attention (Sec. 3.2), or the raw weights with / without a recent window
          if (avg) ave = __fdividef(sw, (float)G * (float)(a.pos + 1 - id));
          else ave = (c.rule == 1 && j >= n1 - n_old / 2) ? INFINITY : sw;
          better(id < pad ? 0u : __float_as_uint(ave) + 1u, j, id);
        } else if (row_ok(c, j)) {
          c.sum_weights[base + j] = sw;
          if (j == n_old) c.kv_ids[base + j] = id;
        }
      }
      int hole = n1;   // no row leaves
      if (a.evict_one) {
        auto warp_best = [&]() {   // the smallest key of the warp's lanes, among equal ones the highest position
          const uint32_t key = __reduce_min_sync(0xffffffffu, best_key);
          const int id = __reduce_max_sync(0xffffffffu, best_key == key ? best_id : -1);
          const int src = __ffs(__ballot_sync(0xffffffffu, best_key == key && best_id == id)) - 1;
          best_j = __shfl_sync(0xffffffffu, best_j, src);
          best_key = key;
          best_id = id;
        };
        auto read_best = [&](const int4* from, int count) {
          const int4 b = from[min(lane, count - 1)];
          best_key = (uint32_t)b.x; best_j = b.y; best_id = b.z;
          warp_best();
        };
        warp_best();
        if (lane == 0) s_best[warp] = make_int4((int)best_key, best_j, best_id, 0);
        named_bar_sync(1, kConsumers);
        if (!SHARED || warp == 0) read_best(s_best, kCWarps);
        if (SHARED) {
          if (tid == 0) mbar_expect_tx(&bars[L::B_X + 1], C * 16);
          if (tid < (int)C)
            st_peer4(mapa(smem_u32(s_xbest + rank), tid), best_key, (uint32_t)best_j, (uint32_t)best_id, 0u,
                     mapa(smem_u32(&bars[L::B_X + 1]), tid));
          wait_cluster(&bars[L::B_X + 1], it & 1, abort_flag, c.status);
          read_best(s_xbest, (int)C);
        }
        hole = best_j;
      } else {
        named_bar_sync(1, kConsumers);                      // the bf16 exponentials are in place
      }
      if (tid == 0) {                                       // to the warps that move rows (done with the previous cache)
        if (it > 0) mbar_wait(&bars[L::B_MOVED], (it - 1) & 1, abort_flag, c.status);
        *s_hole = hole;
        mbar_arrive(&bars[L::B_HOLE]);
      }
      if (a.evict_one) {   // sum_weights and kv_ids in their final places
        if (c.moved != nullptr && tid == 0 && rank == 0) {
          if (c.fill) { if (hole < n_old) atomicAdd(&c.moved[unit & 15], 1ull); }
          else atomicAdd(&c.moved[unit & 15], (unsigned long long)(n1 - 1 - hole));
        }
#pragma unroll 1
        for (int jl = tid; jl < nr; jl += kConsumers) {
          const int j = r0 + jl;
          // rows behind the hole move up by one; in an unordered cache only the step's own pair moves, into the hole's row
          const int dst = c.fill ? (j == n_old ? hole : j) : (j > hole ? j - 1 : j);
          if (j == hole || dst >= n_old || !row_ok(c, dst)) continue;
          c.sum_weights[base + dst] = s_sw[jl];
          if (dst != j) c.kv_ids[base + dst] = s_id[jl];
        }
      }
      // ---- out^T = V^T p^T: warp = (16 elements of the head dimension, key group)
      float oacc[2][4] = {};
#pragma unroll 1
      for (int x = 0; x < vt; ++x) {
        constexpr int NK = TR / 16 / KH;                    // steps of 16 keys per tile and warp
        mbar_wait(&bars[L::B_FULL + slot], ph, abort_flag, c.status);
        const uint32_t tile = smem_u32(ring + slot * kTile);
        uint32_t fr[NK][4], b0[NK], b1[NK];
#pragma unroll
        for (int y = 0; y < NK; ++y) {
          // lane l addresses row l%8 of matrix l/8: keys 8 (l/16) + l%8, elements 16 ws + 8 ((l/8)%2) + [0, 8)
          const int krow = (y * KH + kg) * 16 + ((lane >> 4) << 3) + (lane & 7);
          asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                       : "=r"(fr[y][0]), "=r"(fr[y][1]), "=r"(fr[y][2]), "=r"(fr[y][3])
                       : "r"(tile + piece_offset<D>(krow, 2 * ws + ((lane >> 3) & 1))) : "memory");
        }
#pragma unroll
        for (int y = 0; y < NK; ++y) {
          b0[y] = b1[y] = 0u;
          if (gid < G) {
            const T* pp = s_pb + gid * PBS + x * TR + (y * KH + kg) * 16 + 2 * tq;
            b0[y] = *reinterpret_cast<const uint32_t*>(pp);
            b1[y] = *reinterpret_cast<const uint32_t*>(pp + 8);
          }
        }
#pragma unroll
        for (int y = 0; y < NK; ++y) mma16816(oacc[y & 1], fr[y][0], fr[y][1], fr[y][2], fr[y][3], b0[y], b1[y]);
        arrive_one(&bars[L::B_EMPTY + slot], lane);
        if (++slot == NS) { slot = 0; ph ^= 1; }
      }
      // oacc[.][0..1]: element 16 ws + gid of heads 2 tq, 2 tq + 1; [2..3]: element 16 ws + gid + 8
      float o[2][2];
#pragma unroll
      for (int hf = 0; hf < 2; ++hf)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) o[hf][hh] = oacc[0][2 * hf + hh] + oacc[1][2 * hf + hh];
      if (has_new && kg == 0) {                             // the step's own pair
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
          for (int hh = 0; hh < 2; ++hh)
            if (2 * tq + hh < G) o[hf][hh] = fmaf(s_enew[2 * tq + hh], v_new[hf], o[hf][hh]);
        }
      }
      if constexpr (KH > 1) {                               // key groups of a slice meet in a fixed order
        if (kg == 1) {                                      // (through the logits' place: no longer needed)
#pragma unroll
          for (int hf = 0; hf < 2; ++hf)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh)
              if (2 * tq + hh < G) s_p[(2 * tq + hh) * D + 16 * ws + gid + 8 * hf] = o[hf][hh];
        }
        named_bar_sync(1, kConsumers);
        if (kg == 0) {
#pragma unroll
          for (int hf = 0; hf < 2; ++hf)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh)
              if (2 * tq + hh < G) o[hf][hh] += s_p[(2 * tq + hh) * D + 16 * ws + gid + 8 * hf];
        }
      }
      T* op = reinterpret_cast<T*>(a.out) + (size_t)unit * G * D;
      if (!SHARED) {
        if (kg == 0)
#pragma unroll
          for (int hf = 0; hf < 2; ++hf)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              const int h = 2 * tq + hh;
              float fh = 0.f;
#pragma unroll
              for (int g = 0; g < G; ++g) fh = g == h ? f[g] : fh;
              if (h < G) op[h * D + 16 * ws + gid + 8 * hf] = __float2bfloat16_rn(o[hf][hh] * fh);
            }
      } else {
        const int lc = 31 - __clz((int)C), ldc = (D == 128 ? 7 : 6) - lc, dc = 1 << ldc;   // elements of every head that one CTA adds up
        if (tid == 0) mbar_expect_tx(&bars[L::B_X + 2], G * D * 4);
        if (kg == 0)
#pragma unroll
          for (int hf = 0; hf < 2; ++hf)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              const int h = 2 * tq + hh, d = 16 * ws + gid + 8 * hf;
              float fh = 0.f;
#pragma unroll
              for (int g = 0; g < G; ++g) fh = g == h ? f[g] : fh;
              if (h < G)
                st_peer(mapa(smem_u32(s_xout + (((int)rank * G + h) << ldc) + (d & (dc - 1))), d >> ldc), o[hf][hh] * fh,
                        mapa(smem_u32(&bars[L::B_X + 2]), d >> ldc));
            }
        wait_cluster(&bars[L::B_X + 2], it & 1, abort_flag, c.status);
#pragma unroll 1
        for (int x = tid; x < G * dc; x += kConsumers) {
          float part[kMaxCluster];
#pragma unroll
          for (int p = 0; p < kMaxCluster; ++p) part[p] = p < (int)C ? s_xout[(p * G << ldc) + x] : 0.f;
          float t = 0.f;
#pragma unroll
          for (int p = 0; p < kMaxCluster; ++p) t += part[p];   // fixed order
          op[(x >> ldc) * D + ((int)rank << ldc) + (x & (dc - 1))] = __float2bfloat16_rn(t);
        }
      }
      named_bar_sync(1, kConsumers);                        // the per-row arrays belong to the next cache
    }
  }
  // No CTA of a cluster leaves while a peer may still write into its shared memory.  It has waited for all that is sent
  // to it (B_X, B_PREV), so the barrier need not order memory (a releasing arrival waits for the global
  // stores); it is there for a CTA whose waits gave up.
  if (SHARED) {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
}


constexpr size_t kMaxDynamicSmem = 227 * 1024;

// How a call is laid out: cluster size, ring, shared memory.
struct Plan {
  int C = 0, grid = 0, stages = 0, single = 0, keep_k = 0, rows = 0;
  size_t smem = 0;
};

template <int D, int G>
bool plan_for(int C, int n1, int units, int sms, Plan* p) {
  using L = StreamSmem<D, G>;
  const int tiles = (n1 + L::TR - 1) / L::TR, piece = (tiles + C - 1) / C;
  if (tiles < C) return false;
  p->C = C;
  p->grid = std::min(units, sms) * C;
  p->rows = piece * L::TR;
  p->single = units <= sms;
  const int move = p->single ? 0 : kMoveTiles;
  const size_t fixed = L::total(p->rows, move);
  if (L::total(p->rows, kMoveTiles + 4) > kMaxDynamicSmem) return false;   // (whatever the call's share of the caches)
  p->stages = (int)std::min<size_t>((kMaxDynamicSmem - fixed) / kTile, L::kMaxStages);
  p->keep_k = p->single && p->stages >= 2 * piece;
  if (p->keep_k) p->stages = 2 * piece;
  p->smem = L::total(p->rows, p->stages + move);
  return true;
}

// Cluster size.  A cluster shortens the time a cache takes to pass through one SM and costs its exchanges.  us per step
// with 1, 2, 4 and 8 CTAs per cache, d = 128, g = 4: 8 caches of 200 pairs 5.5 / 5.6 / 5.4 / 6.2, of 700 pairs 9.4 / 8.4 /
// 6.6 / 6.3, of 1024 pairs 12.6 / 10.1 / 7.8 / 6.6; 32 caches of 200 pairs 6.2 / 6.4 / 6.7, of 1024 pairs 14.1 / 11.4 /
// 9.9; 64 caches of 384 pairs 8.3 / 8.3, of 1024 pairs 14.7 / 12.3; at d = 64 8 caches of 1024 pairs 9.1 / 8.1 / 6.6 /
// 6.0 -- the line through these is the estimate below.
// Only calls whose clusters are all resident at once are split (a GPC holds few clusters of 8: at 16 caches the second
// wave made the step 1.5 times as long as with clusters of 4), and the handle's caches of a layer decide, not the call's:
// sample ranges of one batch may be in flight together and must sum in the same order as the whole batch.
template <int D, int G>
Plan choose_plan(int n1, int units, int layer_units, int sms) {
  constexpr int kMostCaches[] = {0, kMostSharedCaches, 32, 8};   // for C = 2, 4, 8; measured on 148 SMs, and residency is tested besides
  Plan best;
  double best_us = 0;
  for (int x = 0, C = 1; C <= kMaxCluster; ++x, C *= 2) {
    Plan p;
    if (C > 1 && (layer_units > kMostCaches[x] || layer_units * C > sms)) continue;
    if (!plan_for<D, G>(C, n1, units, sms, &p)) continue;
    const double stream = n1 * (4.0 * D + 80) / C / 57e3;   // us: row bytes, and the work per row
    const double us = stream + (C == 1 ? 3.3 : 4.1 + 0.1 * C) + 1.9 * layer_units * C / sms;
    if (best.C == 0 || us < best_us) { best = p; best_us = us; }
  }
  return best;
}

template <int D, int G>
cudaError_t launch_stream(const CacheView& c, StreamArgs a, cudaStream_t st, bool* taken) {
  a.units = c.nsamples * c.Hkv;
  const Plan p = choose_plan<D, G>(c.n_old + 1, a.units, c.layer_units, sm_count());
  if (p.C == 0) return cudaSuccess;
  a.stages = p.stages; a.single = p.single; a.keep_k = p.keep_k; a.rows_cta = p.rows;
  StreamMaps m;
  constexpr int TR = StreamSmem<D, G>::TR;
  if (!encode_slab_rows_map(&m.k_ld, c.k_slab, D, c.n_old, c.cap, a.units, TR) ||
      !encode_slab_rows_map(&m.v_ld, c.v_slab, D, c.n_old, c.cap, a.units, TR) ||
      !encode_slab_rows_map(&m.k_st, c.k_slab, D, c.n_old - 1, c.cap, a.units, 8) ||
      !encode_slab_rows_map(&m.v_st, c.v_slab, D, c.n_old - 1, c.cap, a.units, 8))
    return cudaSuccess;
  *taken = true;
  ProfileScope prof(kDecode, st);
  g_last_decode_path = p.C > 1 ? 5 : 4;
  cudaError_t err;
  if (p.C > 1) {
    static SmemConfigured configured;
    if ((err = configured.ensure(decode_stream_kernel<D, G, true>, p.smem)) != cudaSuccess) return err;
    err = launch_dependent_cluster(decode_stream_kernel<D, G, true>, dim3(p.grid), dim3(kThreads), p.smem, p.C, st, c, a, m);
  } else {
    static SmemConfigured configured;
    if ((err = configured.ensure(decode_stream_kernel<D, G, false>, p.smem)) != cudaSuccess) return err;
    err = launch_dependent(decode_stream_kernel<D, G, false>, dim3(p.grid), dim3(kThreads), p.smem, st, c, a, m);
  }
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace

cudaError_t launch_decode_stream(int d, const CacheView& c, const void* q, const void* k, const void* v, void* out,
                                 int32_t pos, float scale, bool evict_one, cudaStream_t st, bool* taken) {
  StreamArgs a{};
  a.q = q; a.k = k; a.v = v; a.out = out; a.pos = pos; a.scale = scale; a.evict_one = evict_one ? 1 : 0;
  *taken = false;
  if (d == 64) {
    switch (c.g) {
      case 1: return launch_stream<64, 1>(c, a, st, taken);
      case 2: return launch_stream<64, 2>(c, a, st, taken);
      case 4: return launch_stream<64, 4>(c, a, st, taken);
      case 8: return launch_stream<64, 8>(c, a, st, taken);
    }
  } else if (d == 128) {
    switch (c.g) {
      case 1: return launch_stream<128, 1>(c, a, st, taken);
      case 2: return launch_stream<128, 2>(c, a, st, taken);
      case 4: return launch_stream<128, 4>(c, a, st, taken);
      case 8: return launch_stream<128, 8>(c, a, st, taken);
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace bm
