// One decoding step (the token-generation step of Algorithm 1; Sec. 3.2 with I = 1) for every (sample, kv-head)
// cache of a range, in one bandwidth-bound pass per cache (one CTA):
//   append the step's pair -> logits (K streamed once for the g heads, 128-bit loads) -> softmax ->
//   sum_weights update -> choice of the pair to evict -> P.V (V streamed once) with the one-row
//   compaction of V fused into the same pass -> one-row compaction of K.
// With growth 1 (evict after every step) exactly one pair leaves, so the top-k select is an arg-min over
// ave_weights (ties: the higher position leaves) and the stable compaction is a one-row shift of the rows
// behind the hole.  Any other target falls back to the general select + compaction of evict_body.
#include "evict.cuh"

namespace bm {
namespace {

constexpr int kDecThreads = 512;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kUnroll = 4;   // rows in flight per thread and pass
constexpr float kLog2e = 1.4426950408889634f;

struct DecodeArgs {
  const void* q;  // [nsamples][Hq][d]
  const void* k;  // [nsamples][Hkv][d]
  const void* v;
  void* out;      // [nsamples][Hq][d]
  int32_t pos;
  float scale;
  int32_t target;  // < 0: no eviction
};

struct DecSmem {
  float* q;       // [G][D]
  float* p;       // [G][n1p]   logits, then probabilities
  float* score;   // [n1p]      updated sum_weights
  int32_t* id;    // [n1p]
  float* wred;    // [2][G][warps]
  float* best;    // [warps] + int [warps]
  float* ored;    // [warps][G][D]
};

__host__ __device__ inline size_t dec_smem_layout(unsigned char* base, int d, int g, int n1, DecSmem* s) {
  const size_t n1p = (size_t)((n1 + 3) & ~3);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 15) & ~size_t(15); return o; };
  const size_t oq = take(4 * (size_t)g * d), op = take(4 * (size_t)g * n1p), os = take(4 * n1p), oi = take(4 * n1p);
  const size_t ow = take(4 * 2 * (size_t)g * kDecWarps), ob = take(4 * 2 * kDecWarps);
  const size_t oo = take(4 * (size_t)kDecWarps * g * d);
  if (s != nullptr) {
    s->q = reinterpret_cast<float*>(base + oq);
    s->p = reinterpret_cast<float*>(base + op);
    s->score = reinterpret_cast<float*>(base + os);
    s->id = reinterpret_cast<int32_t*>(base + oi);
    s->wred = reinterpret_cast<float*>(base + ow);
    s->best = reinterpret_cast<float*>(base + ob);
    s->ored = reinterpret_cast<float*>(base + oo);
  }
  return off;
}

__device__ inline float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

template <typename T, int D, int G>
__global__ void __launch_bounds__(kDecThreads) decode_kernel(CacheView c, DecodeArgs a) {
  constexpr int V = Elem<T>::kVec;
  constexpr int LPR = D / V;                 // lanes that share one row (one 16-byte piece each)
  constexpr int SLOTS = kDecThreads / LPR;   // rows covered by one load per thread
  constexpr int RPI = SLOTS * kUnroll;       // rows per iteration of the CTA
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n1 = c.n_old + 1;
  const int n1p = (n1 + 3) & ~3;
  DecSmem s;
  dec_smem_layout(smem_raw, D, G, n1, &s);

  const int unit = blockIdx.x, smp = unit / c.Hkv, kh = unit % c.Hkv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t base = (size_t)unit * c.cap;
  T* kslab = reinterpret_cast<T*>(c.k_slab) + base * D;
  T* vslab = reinterpret_cast<T*>(c.v_slab) + base * D;
  // (an unordered cache takes the general path for every cut: there the new pair fills the freed row)
  const bool evict_one = (a.target == n1 - 1) && !c.fill && c.rule < 3;   // rules 3, 4 rank by more than one value per pair
  const bool evict_general = (a.target >= 0 && a.target < n1 && !evict_one);
  // left-padded sample: padding pairs are masked and leave first; a query at a padding position (not a real
  // decode step) gets a zero output and no weights
  const int pad = sample_left_pad(c, smp);
  const bool q_real = a.pos >= pad;

  // queries of the group -> smem (fp32); the step's pair -> row n_old of the cache
#pragma unroll 1
  for (int t = tid; t < G * D; t += kDecThreads) {
    const T* qp = reinterpret_cast<const T*>(a.q) + ((size_t)smp * c.Hq + kh * G) * D;
    s.q[t] = (float)qp[t];
  }
  if (tid < 2 * LPR) {
    const int pc = tid % LPR;
    const T* src = reinterpret_cast<const T*>(tid < LPR ? a.k : a.v) + ((size_t)smp * c.Hkv + kh) * D + pc * V;
    T* dst = (tid < LPR ? kslab : vslab) + (size_t)c.n_old * D + pc * V;
    if (row_ok(c, c.n_old)) st_global_16(dst, ld_global_16(src));
  }
#pragma unroll 1
  for (int j = tid; j < n1; j += kDecThreads) s.id[j] = (j < c.n_old) ? c.kv_ids[base + j] : a.pos;
  __syncthreads();

  const int slot = tid / LPR, lr = tid % LPR;
  const float sc2 = a.scale * kLog2e;
  const int n_iter = (n1 + RPI - 1) / RPI;  // same trip count for every thread
  {
    float qr[G][V];
#pragma unroll
    for (int h = 0; h < G; ++h)
#pragma unroll
      for (int e = 0; e < V; ++e) qr[h][e] = s.q[h * D + lr * V + e];
    // ---- logits (log2 domain): scale * log2(e) * <q_h, k_j>
#pragma unroll 1
    for (int it = 0; it < n_iter; ++it) {
      const int j0 = it * RPI + slot;
      uint4 raw[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int j = j0 + u * SLOTS;
        if (j < n1) raw[u] = ld_global_16(kslab + (size_t)j * D + lr * V);
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int j = j0 + u * SLOTS;
        float kf[V];
        if (j < n1) Elem<T>::unpack(raw[u], kf);
        else {
#pragma unroll
          for (int e = 0; e < V; ++e) kf[e] = 0.f;
        }
        float dot[G];
#pragma unroll
        for (int h = 0; h < G; ++h) {
          float acc = 0.f;
#pragma unroll
          for (int e = 0; e < V; ++e) acc = fmaf(qr[h][e], kf[e], acc);
          dot[h] = acc;
        }
#pragma unroll
        for (int off = LPR / 2; off > 0; off >>= 1)
#pragma unroll
          for (int h = 0; h < G; ++h) dot[h] += __shfl_xor_sync(0xffffffffu, dot[h], off);
        if (lr == 0 && j < n1) {
          const bool masked = q_real && s.id[j] < pad;
#pragma unroll
          for (int h = 0; h < G; ++h) s.p[h * n1p + j] = masked ? -INFINITY : dot[h] * sc2;
        }
      }
    }
  }
  __syncthreads();

  // ---- softmax over the n1 rows, all threads: row max, then exp2 and row sum, per head
  float mx[G], sm[G];
#pragma unroll
  for (int h = 0; h < G; ++h) {
    float m = -INFINITY;
#pragma unroll 1
    for (int j = tid; j < n1; j += kDecThreads) m = fmaxf(m, s.p[h * n1p + j]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if (lane == 0) s.wred[h * kDecWarps + warp] = m;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < G; ++h) {
    float m = -INFINITY;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) m = fmaxf(m, s.wred[h * kDecWarps + w]);
    mx[h] = m;
    float t = 0.f;
#pragma unroll 1
    for (int j = tid; j < n1; j += kDecThreads) {
      const float e = ex2f(s.p[h * n1p + j] - m);
      s.p[h * n1p + j] = e;
      t += e;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane == 0) s.wred[(G + h) * kDecWarps + warp] = t;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < G; ++h) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) t += s.wred[(G + h) * kDecWarps + w];  // fixed order
    sm[h] = q_real ? 1.f / t : 0.f;
  }
  (void)mx;

  // ---- normalise, sum_weights += attn_weights (group's heads added in a fixed order), eviction candidate
  float best_ave = INFINITY;
  int best_j = -1;
#pragma unroll 1
  for (int j = tid; j < n1; j += kDecThreads) {
    float add = 0.f;
#pragma unroll
    for (int h = 0; h < G; ++h) {
      const float p = s.p[h * n1p + j] * sm[h];
      s.p[h * n1p + j] = p;
      add += p;
    }
    // rules 2 and 3 (recent queries only) keep this step's weights only
    const float sw = ((j < c.n_old && !rule_overwrites(c.rule)) ? c.sum_weights[base + j] : 0.f) + add;
    if (c.sum_sq != nullptr) {                                       // rule 4: sum of squared weights as well
      float add_sq = 0.f;
#pragma unroll
      for (int h = 0; h < G; ++h) add_sq = fmaf(s.p[h * n1p + j], s.p[h * n1p + j], add_sq);
      c.sum_sq[base + j] = (j < c.n_old ? c.sum_sq[base + j] : 0.f) + add_sq;
    }
    s.score[j] = sw;
    if (evict_one) {
      float ave;   // ranking value: average attention (Sec. 3.2), or the raw weights with / without a recent window
      if (s.id[j] < pad) ave = -1.f;
      else if (c.rule == 0) ave = sw / ((float)G * (float)(a.pos + 1 - s.id[j]));
      else ave = (c.rule == 1 && j >= n1 - a.target / 2) ? INFINITY : sw;
      ave = fminf(ave, INFINITY);   // NaN (a NaN in the step's queries or keys) ranks like +inf: some row is always found
      if (ave <= best_ave) { best_ave = ave; best_j = j; }   // j ascends: ties move to the higher position
    } else if (row_ok(c, j)) {
      c.sum_weights[base + j] = sw;
    }
  }
  int hole = n1;  // no row leaves
  if (evict_one) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float oa = __shfl_xor_sync(0xffffffffu, best_ave, off);
      const int oj = __shfl_xor_sync(0xffffffffu, best_j, off);
      if (oa < best_ave || (oa == best_ave && oj > best_j)) { best_ave = oa; best_j = oj; }
    }
    if (lane == 0) { s.best[warp] = best_ave; reinterpret_cast<int*>(s.best)[kDecWarps + warp] = best_j; }
    __syncthreads();
    best_ave = s.best[0];
    best_j = reinterpret_cast<int*>(s.best)[kDecWarps];
#pragma unroll
    for (int w = 1; w < kDecWarps; ++w) {
      const float oa = s.best[w];
      const int oj = reinterpret_cast<int*>(s.best)[kDecWarps + w];
      if (oa < best_ave || (oa == best_ave && oj > best_j)) { best_ave = oa; best_j = oj; }
    }
    hole = best_j;
    if (c.moved != nullptr && tid == 0) atomicAdd(&c.moved[unit & 15], (unsigned long long)(n1 - 1 - hole));
    // sum_weights / kv_ids in their final places: rows behind the hole move up by one
#pragma unroll 1
    for (int j = tid; j < n1; j += kDecThreads) {
      if (j < hole) { if (j >= 0) c.sum_weights[base + j] = s.score[j]; }
      else if (j > hole) { c.sum_weights[base + j - 1] = s.score[j]; c.kv_ids[base + j - 1] = s.id[j]; }
    }
    if (hole >= c.n_old && tid == 0) { /* the new pair itself leaves: nothing to record */ }
  } else {
    if (tid == 0) c.kv_ids[base + c.n_old] = a.pos;
    __syncthreads();
  }

  // ---- out_h = sum_j p_h[j] v_j ; rows behind the hole are written back one row up while they are in registers
  float acc[G][V];
#pragma unroll
  for (int h = 0; h < G; ++h)
#pragma unroll
    for (int e = 0; e < V; ++e) acc[h][e] = 0.f;
#pragma unroll 1
  for (int it = 0; it < n_iter; ++it) {
    const int j0 = it * RPI + slot;
    uint4 raw[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int j = j0 + u * SLOTS;
      if (j < n1) raw[u] = ld_global_16(vslab + (size_t)j * D + lr * V);
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int j = j0 + u * SLOTS;
      if (j < n1) {
        float vf[V];
        Elem<T>::unpack(raw[u], vf);
#pragma unroll
        for (int h = 0; h < G; ++h) {
          const float p = s.p[h * n1p + j];
#pragma unroll
          for (int e = 0; e < V; ++e) acc[h][e] = fmaf(p, vf[e], acc[h][e]);
        }
      }
    }
    if (evict_one && (it + 1) * RPI > hole) {   // uniform over the CTA
      __syncthreads();                          // every load of rows < (it+1)*RPI has completed
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int j = j0 + u * SLOTS;
        if (j < n1 && j > hole && row_ok(c, j - 1)) st_global_16(vslab + (size_t)(j - 1) * D + lr * V, raw[u]);
      }
    }
  }
  // K rows behind the hole: same one-row shift (re-read, mostly from L2: the logits pass just streamed them)
  if (evict_one) {
#pragma unroll 1
    for (int it = hole / RPI; it < n_iter; ++it) {
      const int j0 = it * RPI + slot;
      uint4 raw[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int j = j0 + u * SLOTS;
        if (j < n1 && j > hole) raw[u] = ld_global_16(kslab + (size_t)j * D + lr * V);
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int j = j0 + u * SLOTS;
        if (j < n1 && j > hole && row_ok(c, j - 1)) st_global_16(kslab + (size_t)(j - 1) * D + lr * V, raw[u]);
      }
    }
  }

  // rows of one warp first (lanes lr, lr+LPR, ...), then across warps through smem, fixed order
#pragma unroll
  for (int off = 16; off >= LPR; off >>= 1)
#pragma unroll
    for (int h = 0; h < G; ++h)
#pragma unroll
      for (int e = 0; e < V; ++e) acc[h][e] += __shfl_xor_sync(0xffffffffu, acc[h][e], off);
  if (lane < LPR) {
#pragma unroll
    for (int h = 0; h < G; ++h)
#pragma unroll
      for (int e = 0; e < V; ++e) s.ored[(warp * G + h) * D + lr * V + e] = acc[h][e];
  }
  __syncthreads();
#pragma unroll 1
  for (int t = tid; t < G * D; t += kDecThreads) {
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) tot += s.ored[w * G * D + t];
    T* op = reinterpret_cast<T*>(a.out) + ((size_t)smp * c.Hq + kh * G) * D;
    op[t] = Elem<T>::to_out(tot);
  }

  // ---- any other target: general select + compaction over the cache (all candidates live in it now)
  if (evict_general) {
    __syncthreads();  // sum_weights / appended row visible to the whole CTA; smem reusable
    CacheView cv = c;
    cv.n_old = n1;
    EvictArgs e;
    e.blk_k = nullptr; e.blk_v = nullptr; e.new_sum = nullptr;
    e.I = 0; e.pos0 = 0; e.curr_id = a.pos; e.target = a.target;
    evict_body<T, D, kDecThreads>(cv, unit, smp, kh, e, smem_raw);
  }
}

// ------------------------------------------------------------------------------------------------
// The same step for few fp32 caches: a cluster of C CTAs shares one.  Each CTA keeps its rows (contiguous, the step's own pair is
// the last row of all) in shared memory, K and V, from one round of asynchronous copies; nothing of the cache is read after
// the first exchange, so that rows move straight from shared memory whatever the other CTAs do.  Two exchanges through
// distributed shared memory: every CTA's (maximum, sum) per head; its candidate for eviction and its partial outputs.
//
// What bounds it: one cache per CTA left 132 SMs idle at 16 caches, and the step took as long as one SM needs to pull a cache
// through its load units.  16 caches of 512 pairs, d = 128, g = 4: 22.7 -> 9.5 us per step, 8 caches of
// 900 without groups 54.1 -> 11.7, 8 caches of 128 at d = 64 7.0 -> 5.3.
constexpr int kShThreads = 256, kShWarps = kShThreads / 32, kShMaxCluster = 8;

template <int D, int G>
struct SharedDecSmem {
  static constexpr int LD = D + 4;                       // row stride of K: rows of a warp's reads lie in different banks
  static constexpr int RG = kShThreads / (D / 4);        // row groups of the output product
  static constexpr int kFixed = G * D + RG * G * D + G * D + 2 * kShMaxCluster * G + G + 2 * kShWarps + 2 * kShMaxCluster;
  static size_t bytes(int rows) { return 4 * ((size_t)rows * (LD + D + G + 2) + kFixed) + 64; }   // p, score and id per row besides
};

__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
// 2^n, exactly, for a whole n <= 0, or -inf; NaN stays NaN
__device__ __forceinline__ float pow2_whole(float n) {
  return n >= -126.f ? __int_as_float(((int)n + 127) << 23) : n < 0.f ? 0.f : n;
}
__device__ __forceinline__ void st_peer(const void* p, uint32_t rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_addr(p, rank)), "f"(v) : "memory");
}

template <int D, int G>
__global__ void __launch_bounds__(kShThreads) decode_shared_kernel(CacheView c, DecodeArgs a, int rows) {
  using L = SharedDecSmem<D, G>;
  constexpr int LD = L::LD, D4 = D / 4, RG = L::RG;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sK = reinterpret_cast<float*>(smem_raw);        // [rows][LD]
  float* sV = sK + (size_t)rows * LD;                    // [rows][D]
  float* sQ = sV + (size_t)rows * D;                     // [G][D]
  float* sRed = sQ + G * D;                              // [RG][G][D]
  float* sOut = sRed + RG * G * D;                       // [cluster][G D / C], exchanged
  float* sStat = sOut + G * D;           // [cluster][2][G], exchanged
  float* sF = sStat + 2 * kShMaxCluster * G;             // [G]
  float* sBest = sF + G;                                 // [warps][2], then [cluster][2] exchanged
  float* sP = sBest + 2 * kShWarps + 2 * kShMaxCluster;  // [G][rows]
  float* sScore = sP + (size_t)G * rows;                 // [rows]
  int* sId = reinterpret_cast<int*>(sScore + rows);      // [rows]
  float* sXBest = sBest + 2 * kShWarps;

  uint32_t rank, C;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // (waited for before a peer's memory is touched)
  const int n_old = c.n_old, n1 = n_old + 1;
  const int unit = blockIdx.x / C, smp = unit / c.Hkv, kh = unit % c.Hkv;
  const int r0 = (int)(rank * n1 / C), nr = (int)((rank + 1) * n1 / C) - r0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t base = (size_t)unit * c.cap;
  float* kslab = reinterpret_cast<float*>(c.k_slab) + base * D;
  float* vslab = reinterpret_cast<float*>(c.v_slab) + base * D;
  const float* k_new = reinterpret_cast<const float*>(a.k) + ((size_t)smp * c.Hkv + kh) * D;
  const float* v_new = reinterpret_cast<const float*>(a.v) + ((size_t)smp * c.Hkv + kh) * D;
  pdl_wait();
  pdl_release();

  auto copy_rows = [&](float* dst, int ld, const float* slab, const float* own) {
#pragma unroll 4
    for (int x = tid; x < nr * D4; x += kShThreads) {
      const int jl = x / D4, pc = x % D4, j = r0 + jl;
      const float* from = (j < n_old ? slab + (size_t)j * D : own) + 4 * pc;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + jl * ld + 4 * pc)), "l"(from) : "memory");
    }
  };
  copy_rows(sK, LD, kslab, k_new);
#pragma unroll 1
  for (int x = tid; x < G * D4; x += kShThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(sQ + 4 * x)),
                 "l"(reinterpret_cast<const float*>(a.q) + ((size_t)smp * c.Hq + kh * G) * D + 4 * x) : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
  copy_rows(sV, D, vslab, v_new);
  asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 1
  for (int jl = tid; jl < nr; jl += kShThreads) {
    const int j = r0 + jl;
    sId[jl] = j < n_old ? c.kv_ids[base + j] : a.pos;
    sScore[jl] = (j < n_old && !rule_overwrites(c.rule)) ? c.sum_weights[base + j] : 0.f;   // rules 2, 3 keep this step's weights only
  }
  const int pad = sample_left_pad(c, smp);
  const bool q_real = a.pos >= pad;
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();

  // ---- logits, unscaled: four threads per row, each every fourth 16-byte piece
#pragma unroll 1
  for (int j0 = 0; j0 < nr; j0 += kShThreads / 4) {
    const int jl = j0 + (tid >> 2), sub = tid & 3;
    const float* kr = sK + min(jl, nr - 1) * LD;
    // (four sums per head: one chain of 32 products made the weights' error against 64 bits a quarter larger)
    float4 acc[G];
#pragma unroll
    for (int h = 0; h < G; ++h) acc[h] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll (D == 128 ? 2 : 4)   // (16 caches of 512 pairs, g = 4: 11.0 us per step with four, 10.5 with two)
    for (int pc = sub; pc < D4; pc += 4) {
      const float4 k4 = *reinterpret_cast<const float4*>(kr + 4 * pc);
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const float4 q4 = *reinterpret_cast<const float4*>(sQ + h * D + 4 * pc);
        acc[h].x = fmaf(q4.x, k4.x, acc[h].x); acc[h].y = fmaf(q4.y, k4.y, acc[h].y);
        acc[h].z = fmaf(q4.z, k4.z, acc[h].z); acc[h].w = fmaf(q4.w, k4.w, acc[h].w);
      }
    }
    float dot[G];
#pragma unroll
    for (int h = 0; h < G; ++h) dot[h] = (acc[h].x + acc[h].y) + (acc[h].z + acc[h].w);
#pragma unroll
    for (int off = 1; off < 4; off <<= 1)
#pragma unroll
      for (int h = 0; h < G; ++h) dot[h] += __shfl_xor_sync(0xffffffffu, dot[h], off);
    if (sub == 0 && jl < nr) {
      const bool masked = q_real && sId[jl] < pad;       // padding pairs are masked
#pragma unroll
      for (int h = 0; h < G; ++h) sP[h * rows + jl] = masked ? -INFINITY : dot[h];
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");   // V too: after the first exchange nobody reads the cache
  __syncthreads();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  // ---- a warp per head: maximum, exponentials, their sum; to every peer.  The exponentials (log2 domain) are relative to the
  // maximum's next whole number, so that the factor between two CTAs' references is a power of two and a weight has the error of
  // one exponential, and a logit is scaled and its reference subtracted with one rounding.
  const float sc2 = a.scale * kLog2e;
  if (warp < G) {
    float* p = sP + warp * rows;
    float m = -INFINITY, t = 0.f;
#pragma unroll 1
    for (int jl = lane; jl < nr; jl += 32) m = fmaxf(m, p[jl]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    m = ceilf(m * sc2);
    const float ref = m == -INFINITY ? 0.f : m;          // (a piece of padding only)
#pragma unroll 1
    for (int jl = lane; jl < nr; jl += 32) { const float e = ex2f(fmaf(p[jl], sc2, -ref)); p[jl] = e; t += e; }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane < (int)C) {
      st_peer(sStat + (rank * 2) * G + warp, lane, m);
      st_peer(sStat + (rank * 2 + 1) * G + warp, lane, t);
    }
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp < G) {                                        // weight of a pair = its exponential * sF; a lane per CTA
    const int p = lane & (kShMaxCluster - 1);
    const bool there = p < (int)C;
    const float m = there ? sStat[p * 2 * G + warp] : -INFINITY;
    float t = there ? sStat[(p * 2 + 1) * G + warp] : 0.f, top = m;
#pragma unroll
    for (int off = kShMaxCluster / 2; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
    if (m != -INFINITY) t *= pow2_whole(m - top);        // (-inf: a piece without weight, whose sum is 0, or NaN logits alone)
#pragma unroll
    for (int off = kShMaxCluster / 2; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);   // fixed order
    // (a piece without weight: 0; a cache whose logits are all -inf, or that holds a NaN: NaN)
    if (lane == 0) sF[warp] = q_real ? pow2_whole(sStat[rank * 2 * G + warp] - top) / t : 0.f;
  }
  __syncthreads();

  // ---- weights, sum_weights += attn_weights (heads added in a fixed order), candidate for eviction
  const bool evict_one = a.target == n1 - 1;             // (other cuts follow as a launch of their own)
  float best_ave = INFINITY;
  int best_j = -1;
#pragma unroll 1
  for (int jl = tid; jl < nr; jl += kShThreads) {
    const int j = r0 + jl;
    float add = 0.f, add_sq = 0.f;
#pragma unroll
    for (int h = 0; h < G; ++h) {
      const float w = sP[h * rows + jl] * sF[h];
      sP[h * rows + jl] = w;
      add += w;
      add_sq = fmaf(w, w, add_sq);
    }
    const float sw = sScore[jl] + add;
    sScore[jl] = sw;
    if (c.sum_sq != nullptr && row_ok(c, j)) c.sum_sq[base + j] = (j < n_old ? c.sum_sq[base + j] : 0.f) + add_sq;   // rule 4
    if (evict_one) {
      float ave;   // ranking value: average attention (Sec. 3.2), or the raw weights with / without a recent window
      if (sId[jl] < pad) ave = -1.f;
      else if (c.rule == 0) ave = sw / ((float)G * (float)(a.pos + 1 - sId[jl]));
      else ave = (c.rule == 1 && j >= n1 - a.target / 2) ? INFINITY : sw;
      ave = fminf(ave, INFINITY);                        // NaN ranks like +inf: some row is always found
      if (ave <= best_ave) { best_ave = ave; best_j = j; }   // ties: the higher position leaves
    }
  }
  auto better = [&](float oa, int oj) { if (oa < best_ave || (oa == best_ave && oj > best_j)) { best_ave = oa; best_j = oj; } };
  if (evict_one) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float oa = __shfl_xor_sync(0xffffffffu, best_ave, off);
      const int oj = __shfl_xor_sync(0xffffffffu, best_j, off);
      better(oa, oj);
    }
    if (lane == 0) { sBest[2 * warp] = best_ave; sBest[2 * warp + 1] = __int_as_float(best_j); }
  }
  __syncthreads();                                       // weights and candidates are in place
  if (evict_one && tid < (int)C) {                       // this CTA's candidate to every peer
    for (int w = 0; w < kShWarps; ++w) better(sBest[2 * w], __float_as_int(sBest[2 * w + 1]));
    st_peer(sXBest + 2 * rank, tid, best_ave);
    st_peer(sXBest + 2 * rank + 1, tid, __int_as_float(best_j));
  }
  // ---- out_h = sum_j p_h[j] v_j: row groups, then their sums in a fixed order, every peer's share of the elements to it
  {
    const int d4 = tid % D4, rg = tid / D4;
    float4 acc[G];
#pragma unroll
    for (int h = 0; h < G; ++h) acc[h] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
    for (int jl = rg; jl < nr; jl += RG) {
      const float4 v4 = *reinterpret_cast<const float4*>(sV + jl * D + 4 * d4);
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const float w = sP[h * rows + jl];
        acc[h].x = fmaf(w, v4.x, acc[h].x); acc[h].y = fmaf(w, v4.y, acc[h].y);
        acc[h].z = fmaf(w, v4.z, acc[h].z); acc[h].w = fmaf(w, v4.w, acc[h].w);
      }
    }
#pragma unroll
    for (int h = 0; h < G; ++h) *reinterpret_cast<float4*>(sRed + (rg * G + h) * D + 4 * d4) = acc[h];
  }
  __syncthreads();
  const int share = G * D / (int)C;                      // elements that one CTA adds up
#pragma unroll 1
  for (int x = tid; x < G * D; x += kShThreads) {
    float t = 0.f;
#pragma unroll
    for (int g = 0; g < RG; ++g) t += sRed[g * G * D + x];
    st_peer(sOut + rank * share + x % share, x / share, t);
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // (the last that peers write here)
  float* op = reinterpret_cast<float*>(a.out) + ((size_t)smp * c.Hq + kh * G) * D;
#pragma unroll 1
  for (int x = tid; x < share; x += kShThreads) {
    float t = 0.f;
    for (uint32_t p = 0; p < C; ++p) t += sOut[p * share + x];
    op[rank * share + x] = t;
  }
  int hole = n1;                                         // no row leaves
  if (evict_one) {
    best_ave = sXBest[0];
    best_j = __float_as_int(sXBest[1]);
    for (uint32_t p = 1; p < C; ++p) better(sXBest[2 * p], __float_as_int(sXBest[2 * p + 1]));
    hole = best_j;
    if (c.moved != nullptr && tid == 0 && rank == 0) atomicAdd(&c.moved[unit & 15], (unsigned long long)(n1 - 1 - hole));
  }
  // ---- rows, sum_weights and kv_ids in their final places: rows behind the hole move up by one
#pragma unroll 1
  for (int jl = tid; jl < nr; jl += kShThreads) {
    const int j = r0 + jl, dst = j > hole ? j - 1 : j;
    if (j == hole || !row_ok(c, dst)) continue;
    c.sum_weights[base + dst] = sScore[jl];
    if (j > hole || j == n_old) c.kv_ids[base + dst] = sId[jl];
  }
  const int first = max(0, hole < n1 ? hole + 1 - r0 : n_old - r0);   // without an eviction the step's own row alone
#pragma unroll 4
  for (int x = first * D4 + tid; x < nr * D4; x += kShThreads) {
    const int jl = x / D4, pc = x % D4, dst = r0 + jl - (hole < n1 ? 1 : 0);
    if (!row_ok(c, dst)) continue;
    *reinterpret_cast<float4*>(kslab + (size_t)dst * D + 4 * pc) = *reinterpret_cast<const float4*>(sK + jl * LD + 4 * pc);
    *reinterpret_cast<float4*>(vslab + (size_t)dst * D + 4 * pc) = *reinterpret_cast<const float4*>(sV + jl * D + 4 * pc);
  }
}

constexpr size_t kMaxDynamicSmem = 227 * 1024;

// CTAs that share a cache, 1: none.  By the handle's caches of a layer and not the call's, since the sums are cut differently; a
// CTA keeps its rows in shared memory.  us per step, launched one by one, with 1, 2, 4 and 8 CTAs: 8 caches of 60 pairs 6.0 / -
// / 5.0 / 5.3, of 256 13.2 / 9.0 / 7.0 / 6.0, of 1500 (d = 64) 29.0 / - / 12.7 / 9.2; 16 of 700 29.0 / - / 12.3 / 10.9; 32 of 64 8.3 /
// 5.5 / 5.5 / 6.0; 64 of 300 17.6 / 12.0 / 11.6 / 17.9, of 700 (d = 64) 18.8 / - / 15.8 / 18.4; 128 of 300 18.4 / 21.4 / 20.9 / 26.6.
template <int D, int G>
int shared_cluster(const CacheView& c) {
  const int n1 = c.n_old + 1, caches = c.layer_units;
  if (n1 < 32 || caches > sm_count() / 2) return 1;
  for (int C = caches <= 8 && n1 >= 192 ? 8 : 4; C == 4 || (C == 8 && C * caches <= sm_count()); C *= 2)
    if (SharedDecSmem<D, G>::bytes((n1 + C - 1) / C) <= kMaxDynamicSmem) return C;
  return 1;
}

template <int D, int G>
cudaError_t launch_shared(const CacheView& c, DecodeArgs a, int C, cudaStream_t st) {
  const int n1 = c.n_old + 1, rows = (n1 + C - 1) / C, target = a.target;
  const bool cut = target >= 0 && target < n1, one = cut && target == n1 - 1 && !c.fill && c.rule < 3;   // rules 3, 4 rank by more than one value per pair
  if (!one) a.target = -1;
  const size_t smem = SharedDecSmem<D, G>::bytes(rows);
  static SmemConfigured configured;
  if (cudaError_t err = configured.ensure(decode_shared_kernel<D, G>, smem); err != cudaSuccess) return err;
  cudaError_t err;
  {
    ProfileScope prof(kDecode, st);
    g_last_decode_path = 1;
    err = launch_dependent_cluster(decode_shared_kernel<D, G>, dim3(c.nsamples * c.Hkv * C), dim3(kShThreads), smem, C, st, c, a, rows);
    count_launch();
  }
  if (err != cudaSuccess) return err;
  if (!cut || one) return cudaGetLastError();
  CacheView grown = c;
  grown.n_old = n1;
  EvictArgs e;
  e.blk_k = nullptr; e.blk_v = nullptr; e.new_sum = nullptr;
  e.I = 0; e.pos0 = 0; e.curr_id = a.pos; e.target = target;
  return launch_evict(0, D, grown, e, st);
}

template <typename T, int D, int G>
cudaError_t launch_t(const CacheView& c, const DecodeArgs& a, cudaStream_t st) {
  if constexpr (sizeof(T) == 4)
    if (const int C = shared_cluster<D, G>(c); C > 1) return launch_shared<D, G>(c, a, C, st);
  const size_t smem = decode_smem_bytes(D, G, c.n_old + 1, a.target);
  static SmemConfigured configured;
  if (cudaError_t err = configured.ensure(decode_kernel<T, D, G>, smem); err != cudaSuccess) return err;
  ProfileScope prof(kDecode, st);
  g_last_decode_path = 0;
  decode_kernel<T, D, G><<<c.nsamples * c.Hkv, kDecThreads, smem, st>>>(c, a);
  count_launch();
  return cudaGetLastError();
}

template <typename T, int D>
cudaError_t launch_g(const CacheView& c, const DecodeArgs& a, cudaStream_t st) {
  switch (c.g) {
    case 1: return launch_t<T, D, 1>(c, a, st);
    case 2: return launch_t<T, D, 2>(c, a, st);
    case 4: return launch_t<T, D, 4>(c, a, st);
    case 8: return launch_t<T, D, 8>(c, a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

size_t decode_smem_bytes(int d, int g, int n_rows, int target) {
  const size_t attn = dec_smem_layout(nullptr, d, g, n_rows, nullptr);
  const size_t ev = (target >= 0 && target < n_rows) ? evict_smem_bytes(n_rows, target) : 0;
  return attn > ev ? attn : ev;
}

cudaError_t launch_decode(int dtype, int d, const CacheView& c, const void* q, const void* k, const void* v,
                          void* out, int32_t pos, float scale, int32_t target, cudaStream_t st) {
  DecodeArgs a{q, k, v, out, pos, scale, target};
  if (dtype == 0 && d == 64) return launch_g<float, 64>(c, a, st);
  if (dtype == 0 && d == 128) return launch_g<float, 128>(c, a, st);
  if (dtype == 1 && d == 64) return launch_g<__nv_bfloat16, 64>(c, a, st);
  if (dtype == 1 && d == 128) return launch_g<__nv_bfloat16, 128>(c, a, st);
  return cudaErrorInvalidValue;
}

}  // namespace bm
