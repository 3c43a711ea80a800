// Average-attention eviction for one (sample, kv-head) cache, executed by one CTA (Sec. 3.2):
//   ave_weights = sum_weights / (g * (curr_id + 1 - kv_ids)),
// keep the `target` candidates ranking first under (ave_weights descending, kv_ids ascending),
// then compact rows, sum_weights and kv_ids to the front of the cache in ascending kv_ids order.
// (EvictArgs::recent selects the rule of the extreme decoding-only comparison instead, Algorithm 3:
// the `target` most recent candidates stay.)
// Candidates are the n_old cached pairs followed by I new pairs that still live in the caller's
// block buffers; both lists are ascending in kv_ids, so candidate index order is kv_ids order.
//
// What bounds it: with many caches the bytes of the rows that move; with few the chain of its phases (of 8.6 us for 8
// caches of 1536 candidates the select takes about half).  The ranking values are therefore formed while the candidates
// are read, a radix pass clears nothing and has two barriers, prefix sums cross the warps by one reduction, and the
// first row that changes falls out of the placement.  1024 caches cut from 1536 to 1024 pairs: 73.7 -> 69.6 us.
#pragma once
#include "common.cuh"

namespace bm {

struct EvictSmem {
  float* score;    // [n_cand]
  uint32_t* bits;  // [n_cand]   ranking value of every candidate as an ordered bit pattern (computed once)
  int32_t* id;     // [n_cand]
  int32_t* src;    // [target]   candidate index that lands in row r (fill mode: k-th candidate that has to move)
  int32_t* dst;    // [target]   fill mode: row the k-th moving candidate lands in
  uint32_t* hist;  // [4][256], one histogram per pass of a select
  int32_t* misc;   // [8]
  int32_t* wsum;   // [64]
};

__host__ __device__ inline size_t evict_smem_layout(unsigned char* base, int n_cand, int target, EvictSmem* s) {
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 15) & ~size_t(15); return o; };
  size_t o_score = take(sizeof(float) * n_cand), o_id = take(sizeof(int32_t) * n_cand);
  size_t o_bits = take(sizeof(uint32_t) * n_cand);
  size_t o_src = take(sizeof(int32_t) * (target > 0 ? target : 1)), o_dst = take(sizeof(int32_t) * (target > 0 ? target : 1));
  // (the histograms lie where src and dst will be: they are done with when those are written.  The 1 KB that is kept
  // behind these holds nothing: the size decides which calls are refused, and those stay the same.)
  const size_t o_tail = take(sizeof(uint32_t) * (target >= 512 ? 256 : 1024)), o_hist = target >= 512 ? o_src : o_tail;
  size_t o_misc = take(sizeof(int32_t) * 8), o_wsum = take(sizeof(int32_t) * 64);
  if (s != nullptr) {
    s->score = reinterpret_cast<float*>(base + o_score);
    s->bits = reinterpret_cast<uint32_t*>(base + o_bits);
    s->id = reinterpret_cast<int32_t*>(base + o_id);
    s->src = reinterpret_cast<int32_t*>(base + o_src);
    s->dst = reinterpret_cast<int32_t*>(base + o_dst);
    s->hist = reinterpret_cast<uint32_t*>(base + o_hist);
    s->misc = reinterpret_cast<int32_t*>(base + o_misc);
    s->wsum = reinterpret_cast<int32_t*>(base + o_wsum);
  }
  return off;
}

// Exclusive block scan of two counters (each below 2^16 in total); returns this thread's exclusive prefixes.  The
// warps' totals are summed by every warp for itself.
template <int NT>
__device__ inline void block_exclusive_scan2(int a, int b, int32_t* wsum /*[64]*/, int& ea, int& eb, int* total_a = nullptr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t own = ((uint32_t)a << 16) | (uint32_t)b;
  uint32_t incl = own;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += t;
  }
  if (lane == 31) wsum[warp] = (int32_t)incl;
  __syncthreads();
  const uint32_t w = lane < NT / 32 ? (uint32_t)wsum[lane] : 0u;
  const uint32_t excl = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + incl - own;
  if (total_a != nullptr) *total_a = (int)(__reduce_add_sync(0xffffffffu, w) >> 16);
  ea = (int)(excl >> 16);
  eb = (int)(excl & 0xffffu);
  __syncthreads();
}

// CTAs that share one cache with ordered rows (a cluster of `count`): every one of them ranks the candidates, each moves its own
// columns of the rows, and CTA 0 writes sum_weights and kv_ids once all have read them.
struct EvictShare {
  int rank = 0, count = 1;
  __device__ void have_read() const {            // once, when this CTA has read sum_weights, kv_ids and sum_sq
    if (count > 1) asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
  }
  __device__ void everyone_has_read() const {    // before any of them is written
    if (count > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
};

// W: 16-byte pieces a thread has in flight while rows move; 16 in clusters.
// FILL: the cache's rows are an unordered set (CacheView::fill); a template parameter, so that the instance for
// ordered rows carries none of that code (with both in one function the ordered instance ran 15 % slower).
template <typename T, int D, int NT, bool FILL, int W = 8>
__device__ inline void evict_body_impl(const CacheView& c, int unit, int smp, int kh, const EvictArgs& e,
                                  unsigned char* smem_raw, const EvictShare share = {}) {
  const int tid = threadIdx.x;
  const int n_old = c.n_old, n_c = c.n_old + e.I, target = e.target;
  const size_t base = (size_t)unit * c.cap;
  EvictSmem s;
  evict_smem_layout(smem_raw, n_c, target, &s);

  // What most calls rank by, the average, is formed while the candidates are read (one division each); the other
  // rules follow in a pass of their own.
  const int pad = sample_left_pad(c, smp);
  const bool plain = c.rule == 0 && pad == 0 && !e.recent && target < n_c;
#pragma unroll 1
  for (int t = tid; t < 1024; t += NT) s.hist[t] = 0;
#pragma unroll 4
  for (int j = tid; j < n_c; j += NT) {
    const bool old = j < n_old;
    const float w = old ? c.sum_weights[base + j] : e.new_sum[(size_t)unit * e.I + (j - n_old)];
    const int id = old ? c.kv_ids[base + j] : e.pos0 + (j - n_old);
    s.score[j] = w;
    s.id[j] = id;
    if (plain) s.bits[j] = __float_as_uint(w / ((float)c.g * (float)(e.curr_id + 1 - id)));   // average attention (Sec. 3.2)
  }
  __syncthreads();
  if (c.sum_sq == nullptr) share.have_read();
  const float gf = (float)c.g;
  int id_win = 0x7fffffff;   // unordered cache, rule 1: pairs at positions >= id_win form the window of recent pairs
  // rule 3 (Sec. 2, SnapKV): the min(window, target) most recent candidates always stay; every other score is replaced
  // by the maximum over the `pool` neighbours centred on it, the window left out
  const int pool_body = n_c - min(c.window, target), pool_half = c.pool / 2;
  auto ave_bits = [&](int j) -> uint32_t {
    const float cnt = (float)(e.curr_id + 1 - s.id[j]);
    uint32_t b;   // ranking value >= 0: the bit pattern orders like the value
    if (c.rule == 0 || c.rule == 4) b = __float_as_uint(s.score[j] / (gf * cnt));   // average attention (Sec. 3.2)
    else if (c.rule == 1 && (FILL ? s.id[j] >= id_win : j >= n_c - target / 2)) b = 0x7f800000u;   // recent window: always kept
    else if (c.rule == 3) {
      if (j >= pool_body) b = 0x7f800000u;
      else {
        float m = s.score[j];
#pragma unroll 1
        for (int x = max(0, j - pool_half); x < min(pool_body, j + pool_half + 1); ++x) m = fmaxf(m, s.score[x]);
        b = __float_as_uint(m);
      }
    }
    else b = __float_as_uint(s.score[j]);                                // raw (sum of / current) weights
    if (pad == 0) return b;
    return s.id[j] < pad ? 0u : max(b, 1u);   // padding pairs rank below every real pair (left-padded samples)
  };

  // Radix select over the candidates `key_of` admits: the key of the need-th largest, how many candidates equal to
  // that key belong to the `need` largest, and how many equal it.  Four passes of 8 bits, a histogram in shared memory
  // each (zero at entry and again at exit).
  auto radix_kth_largest = [&](auto key_of, int need, uint32_t& out_key, int& out_need_eq, int& out_eq) {
    uint32_t prefix = 0, mask = 0;
    int count = 0;
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      uint32_t* hist = s.hist + 256 * pass;
#pragma unroll 2
      for (int j = tid; j < n_c; j += NT) {
        uint32_t b;
        if (key_of(j, b) && (b & mask) == prefix) atomicAdd(&hist[(b >> shift) & 255u], 1u);
      }
      __syncthreads();
      if (tid < 32) {  // lane l owns digits 8l .. 8l+7; find the digit holding the need-th largest
        const uint4 h0 = reinterpret_cast<const uint4*>(hist)[2 * tid], h1 = reinterpret_cast<const uint4*>(hist)[2 * tid + 1];
        const int h[8] = {(int)h0.x, (int)h0.y, (int)h0.z, (int)h0.w, (int)h1.x, (int)h1.y, (int)h1.z, (int)h1.w};
        int loc = 0;
#pragma unroll
        for (int t = 0; t < 8; ++t) loc += h[t];
        int incl = loc;  // suffix sums over lanes above
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int t = __shfl_down_sync(0xffffffffu, incl, off);
          if (tid + off < 32) incl += t;
        }
        int cum = incl - loc;
#pragma unroll
        for (int t = 7; t >= 0; --t) {
          if (cum < need && need <= cum + h[t])
            *reinterpret_cast<int4*>(s.misc + 4) = make_int4(tid * 8 + t, need - cum, h[t], 0);
          cum += h[t];
        }
      }
      __syncthreads();
      const int4 found = *reinterpret_cast<const int4*>(s.misc + 4);   // (rewritten behind the next pass's first barrier)
      prefix |= (uint32_t)found.x << shift;
      need = found.y;
      count = found.z;
      mask |= 255u << shift;
    }
    out_key = prefix;
    out_need_eq = need;
    out_eq = count;
#pragma unroll 1
    for (int t = tid; t < 1024; t += NT) s.hist[t] = 0;   // (the next select's first barrier is behind other barriers)
  };

  // Unordered cache: nothing that stays moves.  The candidates that stay but sit outside the first `target` rows
  // (new pairs, and cached pairs beyond row `target`) fill the rows that are freed or still empty, in ascending
  // order on both sides.
  auto fill_rows = [&](auto stays) {
    const int chunk = (n_c + NT - 1) / NT;
    const int jb = min(tid * chunk, n_c), je = min(jb + chunk, n_c);
    int nfree = 0, nsrc = 0;
#pragma unroll 1
    for (int j = jb; j < je; ++j) {
      const bool k = stays(j);
      nfree += (j < target && (j >= n_old || !k));
      nsrc += (k && (j >= target || j >= n_old));
    }
    int fb, sb, nf;   // as many rows to fill as candidates to move
    block_exclusive_scan2<NT>(nfree, nsrc, s.wsum, fb, sb, &nf);
#pragma unroll 1
    for (int j = jb; j < je; ++j) {
      const bool k = stays(j);
      if (j < target && (j >= n_old || !k)) s.dst[fb++] = j;
      if (k && (j >= target || j >= n_old)) s.src[sb++] = j;
    }
    __syncthreads();
    if (c.moved != nullptr && tid == 0) atomicAdd(&c.moved[unit & 15], (unsigned long long)nf);
#pragma unroll 1
    for (int k = tid; k < nf; k += NT) {
      const int j = s.src[k], r = s.dst[k];
      if (!row_ok(c, r)) continue;
      c.sum_weights[base + r] = s.score[j];
      c.kv_ids[base + r] = s.id[j];
    }
    // sources lie outside the first `target` rows, destinations inside: no row is both read and written
    constexpr int PRF = D * (int)sizeof(T) / 16;
    T* kslab = reinterpret_cast<T*>(c.k_slab) + base * D;
    T* vslab = reinterpret_cast<T*>(c.v_slab) + base * D;
#pragma unroll 1
    for (int x0 = 0; x0 < nf * PRF; x0 += 4 * NT) {
      uint4 kb[4], vb[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int x = x0 + t * NT + tid;
        if (x < nf * PRF) {
          const int j = s.src[x / PRF], pc = x % PRF;
          if (j >= n_old) {
            const size_t off = ((size_t)(smp * e.I + (j - n_old)) * c.Hkv + kh) * D;
            kb[t] = ld_global_16(reinterpret_cast<const T*>(e.blk_k) + off + pc * (16 / sizeof(T)));
            vb[t] = ld_global_16(reinterpret_cast<const T*>(e.blk_v) + off + pc * (16 / sizeof(T)));
          } else {
            kb[t] = ld_global_16(kslab + (size_t)j * D + pc * (16 / sizeof(T)));
            vb[t] = ld_global_16(vslab + (size_t)j * D + pc * (16 / sizeof(T)));
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int x = x0 + t * NT + tid;
        if (x < nf * PRF) {
          const int r = s.dst[x / PRF], pc = x % PRF;
          if (!row_ok(c, r)) continue;
          st_global_16(kslab + (size_t)r * D + pc * (16 / sizeof(T)), kb[t]);
          st_global_16(vslab + (size_t)r * D + pc * (16 / sizeof(T)), vb[t]);
        }
      }
    }
  };

  int first_moved = n_old;   // rows before it keep their place and their contents
  if (target >= n_c) {
#pragma unroll 1
    for (int r = tid; r < n_c; r += NT) s.src[r] = r;
    __syncthreads();
  } else if (FILL && e.recent) {  // Algorithm 3's rule on an unordered cache: the `target` highest positions stay
    uint32_t key = 0;
    int unused, unused2;
    if (target > 0) radix_kth_largest([&](int j, uint32_t& k) { k = (uint32_t)s.id[j]; return true; }, target, key, unused, unused2);
    const int id_thr = target > 0 ? (int)key : 0x7fffffff;
    fill_rows([&](int j) { return s.id[j] >= id_thr; });
    return;
  } else if (e.recent) {  // Algorithm 3's rule: the most recent pairs stay, whatever their weights
#pragma unroll 1
    for (int r = tid; r < target; r += NT) s.src[r] = n_c - target + r;
    first_moved = 0;
    __syncthreads();
  } else {
    if (FILL && c.rule == 1 && target / 2 > 0) {   // the window's lowest position: the (target/2)-th highest
      uint32_t key;
      int unused, unused2;
      radix_kth_largest([&](int j, uint32_t& k) { k = (uint32_t)s.id[j]; return true; }, target / 2, key, unused, unused2);
      id_win = (int)key;
    }
    // ---- radix select: bit pattern `thr` of the target-th largest ave, and how many equal to it to keep
    uint32_t thr;
    int need_eq, eq_total;
    const int n_std = c.rule == 4 ? (int)(((long long)target * c.std_permille) / 1000) : 0;
    if (n_std > 0) {
      // rule 4 (Sec. 2 / Sec. 3.2, RoCo): the n_std candidates whose weights have the largest standard deviation,
      // sqrt(E[w^2] - E[w]^2) over the g * (curr_id + 1 - kv_ids) weights received, stay whatever their average
      // (ties: lower position first); they enter the ranking below as +inf, the others with their average
#pragma unroll 1
      for (int j = tid; j < n_c; j += NT) {
        const float cnt = gf * (float)(e.curr_id + 1 - s.id[j]);
        const float sq = j < n_old ? c.sum_sq[base + j] : e.new_sq[(size_t)unit * e.I + (j - n_old)];
        const float mean = s.score[j] / cnt;
        s.bits[j] = __float_as_uint(sqrtf(fmaxf(sq / cnt - mean * mean, 0.f)));
      }
      __syncthreads();
      uint32_t thr_s;
      int need_s, eq_s;
      radix_kth_largest([&](int j, uint32_t& key) { key = s.bits[j]; return true; }, n_std, thr_s, need_s, eq_s);
      const int chunk = (n_c + NT - 1) / NT;
      const int jb = min(tid * chunk, n_c), je = min(jb + chunk, n_c);
      int eq = 0;
#pragma unroll 1
      for (int j = jb; j < je; ++j) eq += (s.bits[j] == thr_s);
      int unused, eq_before;
      block_exclusive_scan2<NT>(0, eq, s.wsum, unused, eq_before);
#pragma unroll 1
      for (int j = jb; j < je; ++j) {       // every thread rewrites its own chunk only
        const uint32_t b = s.bits[j];
        const bool prot = b > thr_s || (b == thr_s && eq_before < need_s);
        eq_before += (b == thr_s);
        s.bits[j] = prot ? 0x7f800000u : ave_bits(j);
      }
    } else if (!plain) {
#pragma unroll 1
      for (int j = tid; j < n_c; j += NT) s.bits[j] = ave_bits(j);   // one division per candidate, not one per pass
    }
    if (!plain) __syncthreads();
    radix_kth_largest([&](int j, uint32_t& key) { key = s.bits[j]; return true; }, target, thr, need_eq, eq_total);
    if constexpr (FILL) {
      // ---- unordered cache: the rows of a cache are in no particular order, so (i) among the candidates equal to
      // the cut the need_eq lowest positions stay, found by a second select on kv_ids, and (ii) nothing that stays
      // moves: the candidates that stay but sit outside the first `target` rows (new pairs, and cached pairs beyond
      // row `target`) fill the rows that are freed or empty, in ascending order on both sides.
      int id_cut = 0x7fffffff;
      if (need_eq < eq_total) {
        __syncthreads();   // the histograms are zero again
        uint32_t key;
        int unused, unused2;
        radix_kth_largest([&](int j, uint32_t& k) { k = 0x7fffffffu - (uint32_t)s.id[j]; return s.bits[j] == thr; },
                          need_eq, key, unused, unused2);
        id_cut = (int)(0x7fffffffu - key);
      }
      fill_rows([&](int j) { const uint32_t b = s.bits[j]; return b > thr || (b == thr && s.id[j] <= id_cut); });
      return;
    }
    if (tid == 0) s.misc[2] = n_old;   // first row that changes: the first cached candidate that leaves, or the end
    // ---- stable destinations: candidates above thr, plus the first need_eq equal to thr (lower id first)
    const int chunk = (n_c + NT - 1) / NT;
    const int jb = min(tid * chunk, n_c), je = min(jb + chunk, n_c);
    int gt = 0, eq = 0;
#pragma unroll 1
    for (int j = jb; j < je; ++j) {
      const uint32_t b = s.bits[j];
      gt += (b > thr);
      eq += (b == thr);
    }
    int gt_before, eq_before, first_out = n_old;
    block_exclusive_scan2<NT>(gt, eq, s.wsum, gt_before, eq_before);
#pragma unroll 1
    for (int j = jb; j < je; ++j) {
      const uint32_t b = s.bits[j];
      const bool tie = b == thr, stays = b > thr || (tie && eq_before < need_eq);
      if (stays) s.src[gt_before + min(eq_before, need_eq)] = j;
      else if (first_out == n_old) first_out = min(j, n_old);
      gt_before += (b > thr);
      eq_before += tie;
    }
    if (first_out < n_old) atomicMin(&s.misc[2], first_out);
    __syncthreads();
    first_moved = min(s.misc[2], target);
  }

  if (c.sum_sq != nullptr) share.have_read();
  share.everyone_has_read();
  if (c.moved != nullptr && tid == 0 && share.rank == 0 && first_moved < target)   // stable compaction: every row from there on moves
    atomicAdd(&c.moved[unit & 15], (unsigned long long)(target - first_moved));

#pragma unroll 1
  for (int r = share.rank == 0 ? first_moved + tid : target; r < target; r += NT) {
    const int j = s.src[r];
    if (!row_ok(c, r) || j < 0 || j >= n_c) continue;
    c.sum_weights[base + r] = s.score[j];
    c.kv_ids[base + r] = s.id[j];
  }
  if (c.sum_sq != nullptr && share.rank == 0) {
    // rule 4: the sums of squares take the same places; they pass through shared memory (the ranking values are no
    // longer needed), so that every load has completed before the first store
#pragma unroll 1
    for (int j = tid; j < n_c; j += NT)
      s.bits[j] = __float_as_uint(j < n_old ? c.sum_sq[base + j] : e.new_sq[(size_t)unit * e.I + (j - n_old)]);
    __syncthreads();
#pragma unroll 1
    for (int r = first_moved + tid; r < target; r += NT)
      if (row_ok(c, r)) c.sum_sq[base + r] = __uint_as_float(s.bits[s.src[r]]);
  }

  // ---- rows: ascending chunks, every source row index >= its destination, loads of a chunk complete
  // (barrier) before its stores; later chunks only read rows above everything written so far.  The 2 PR pieces of a
  // row (key, then value) are dealt out to the CTAs of a cluster in contiguous shares.
  constexpr int PR = D * (int)sizeof(T) / 16;  // 16-byte pieces per row and tensor
  if constexpr (W > 8) {
    const int PC = 2 * PR / share.count;         // pieces per row of this CTA (a power of two)
    const int RC = NT * W / PC;                  // rows per chunk
    const int pc = share.rank * PC + (tid & (PC - 1)), rt = tid / PC;   // this thread's piece, its first row in a chunk
    T* slab = (pc < PR ? reinterpret_cast<T*>(c.k_slab) : reinterpret_cast<T*>(c.v_slab)) + base * D + (pc % PR) * (16 / sizeof(T));
    const T* blk = (pc < PR ? reinterpret_cast<const T*>(e.blk_k) : reinterpret_cast<const T*>(e.blk_v)) +
                   ((size_t)smp * e.I * c.Hkv + kh) * D + (pc % PR) * (16 / sizeof(T));
    const int RS = NT / PC;                      // rows between two pieces of a thread
#pragma unroll 1
    for (int r0 = first_moved; r0 < target; r0 += RC) {
      uint4 buf[W];
      bool mv[W];
#pragma unroll
      for (int t = 0; t < W; ++t) {
        const int r = r0 + t * RS + rt;
        mv[t] = false;
        if (r < target) {
          const int j = s.src[r];
          mv[t] = j != r || j >= n_old;
          if (mv[t]) buf[t] = ld_global_16(j >= n_old ? blk + (size_t)(j - n_old) * c.Hkv * D : slab + (size_t)j * D);
        }
      }
      __syncthreads();
#pragma unroll
      for (int t = 0; t < W; ++t) {
        const int r = r0 + t * RS + rt;
        if (mv[t] && row_ok(c, r)) st_global_16(slab + (size_t)r * D, buf[t]);
      }
    }
  } else {                 // a thread moves the same piece of a row's key and value
    constexpr int U = 4;                         // pieces per thread per tensor and chunk
    constexpr int RC = NT * U / PR;              // rows per chunk
    T* kslab = reinterpret_cast<T*>(c.k_slab) + base * D;
    T* vslab = reinterpret_cast<T*>(c.v_slab) + base * D;
#pragma unroll 1
    for (int r0 = first_moved; r0 < target; r0 += RC) {
      uint4 kb[U], vb[U];
      bool mv[U];
#pragma unroll
      for (int t = 0; t < U; ++t) {
        const int pidx = t * NT + tid, r = r0 + pidx / PR, pc = pidx % PR;
        mv[t] = false;
        if (r < target) {
          const int j = s.src[r];
          if (j >= n_old) {
            const size_t off = ((size_t)(smp * e.I + (j - n_old)) * c.Hkv + kh) * D;
            kb[t] = ld_global_16(reinterpret_cast<const T*>(e.blk_k) + off + pc * (16 / sizeof(T)));
            vb[t] = ld_global_16(reinterpret_cast<const T*>(e.blk_v) + off + pc * (16 / sizeof(T)));
            mv[t] = true;
          } else if (j != r) {
            kb[t] = ld_global_16(kslab + (size_t)j * D + pc * (16 / sizeof(T)));
            vb[t] = ld_global_16(vslab + (size_t)j * D + pc * (16 / sizeof(T)));
            mv[t] = true;
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int t = 0; t < U; ++t) {
        if (mv[t]) {
          const int pidx = t * NT + tid, r = r0 + pidx / PR, pc = pidx % PR;
          if (!row_ok(c, r)) continue;
          st_global_16(kslab + (size_t)r * D + pc * (16 / sizeof(T)), kb[t]);
          st_global_16(vslab + (size_t)r * D + pc * (16 / sizeof(T)), vb[t]);
        }
      }
    }
  }
}

template <typename T, int D, int NT>
__device__ inline void evict_body(const CacheView& c, int unit, int smp, int kh, const EvictArgs& e,
                                  unsigned char* smem_raw) {
  if (c.fill) evict_body_impl<T, D, NT, true>(c, unit, smp, kh, e, smem_raw);
  else evict_body_impl<T, D, NT, false>(c, unit, smp, kh, e, smem_raw);
}

}  // namespace bm
