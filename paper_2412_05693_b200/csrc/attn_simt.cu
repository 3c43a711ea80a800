// fp32 SIMT forward pass over a block of inputs (Sec. 3.2): tiled attention with an online softmax
// (outputs + log-sum-exp), and the transposed score pass that turns the normalised weights into the
// column sums  sum_weights += sum_i attn_weights[i].  This is the production path for fp32 caches
// (fp32 accuracy rules out the bf16 tensor-core kernels) and the fallback shape coverage for bf16.
//
// What bounds it: the fp32 pipes once enough warps hide the latency of the shared-memory reads (with 8 warps on an SM the
// forward kernel issued in 41 % of the cycles and waited for fixed-latency results in most others).  A thread owns 4
// rows x 4 keys of a logit tile and 4 rows x D/16 outputs, reads its operands as 16-byte pieces, multiplies pairs with
// packed instructions and keeps an accumulator's two products of a step apart; 16 warps share an SM; K and V tiles
// arrive by asynchronous copies under the arithmetic that does not need them.  Measured with 4 samples, 16 heads in
// groups of 4, d = 128, a block of 256 against 1280 cached pairs: forward kernel 639 -> 407 us (29 TFLOP/s; fp32 pipes
// busy 56 % of the active cycles, 256 CTAs on 148 SMs: profiles/kernels_48_samples.md), score pass 324 -> 226 us, against 4 x 4 values per thread from
// scalar reads between barriers; 8 rows per thread on half the threads: 434 us.
#include "common.cuh"

namespace bm {
namespace {

constexpr int kTN = 64;       // keys per tile of the forward pass

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the float at the same place of CTA `rank` of the cluster
__device__ __forceinline__ float ld_peer(const float* p, uint32_t rank) {
  uint32_t at;
  float v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
  return v;
}

typedef unsigned long long f32x2;   // two floats side by side
__device__ __forceinline__ void fma_pair(f32x2& acc, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ f32x2 dup(float x) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ f32x2 mul_pair(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float lo_of(f32x2 x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float hi_of(f32x2 x) { return __uint_as_float((uint32_t)(x >> 32)); }

// Rows of D elements, widened to fp32, into shared memory with row stride LD; `row_ptr(r)` is the global address of row
// r or null for a row that does not exist (zeros).  fp32 rows are copied asynchronously (one commit group per call).
template <typename T, int D, int LD, int ROWS, int NT, typename F>
__device__ __forceinline__ void load_rows(float* dst, int tid, F row_ptr) {
  constexpr int V = Elem<T>::kVec, CH = D / V;   // elements per 16-byte piece, pieces per row
#pragma unroll 4
  for (int idx = tid; idx < ROWS * CH; idx += NT) {
    const int r = idx / CH, cv = idx % CH;
    const T* p = row_ptr(r);
    float* to = dst + r * LD + cv * V;
    if constexpr (sizeof(T) == 4) {
      const uint32_t s = (uint32_t)__cvta_generic_to_shared(to);
      if (p != nullptr) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(p + cv * V) : "memory");
      else *reinterpret_cast<float4*>(to) = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      float f[V];
#pragma unroll
      for (int e = 0; e < V; ++e) f[e] = 0.f;
      if (p != nullptr) Elem<T>::unpack(ld_global_16(p + cv * V), f);
#pragma unroll
      for (int e = 0; e < V; ++e) to[e] = f[e];
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void commit_nothing() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void wait_copies() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Dot products of rows ty + TY x of sA with rows tx + 16 y of sB (row stride LD = D + 4: the 16-byte pieces that a warp
// reads at one time lie in different banks).  Even and odd elements are added up apart and joined at the end.
template <int D, int LD, int TY, int RT, int KT>
__device__ __forceinline__ void dot_rows(const float* sA, const float* sB, int ty, int tx, float (&s)[RT][KT]) {
  f32x2 acc[RT][KT];
#pragma unroll
  for (int x = 0; x < RT; ++x)
#pragma unroll
    for (int y = 0; y < KT; ++y) acc[x][y] = 0;
  constexpr int kUnroll = RT * KT <= 8 ? 8 : 2;   // (few accumulators: more operand reads in flight)
#pragma unroll kUnroll
  for (int c = 0; c < D; c += 4) {
    ulonglong2 b[KT];
#pragma unroll
    for (int y = 0; y < KT; ++y) b[y] = *reinterpret_cast<const ulonglong2*>(sB + (tx + 16 * y) * LD + c);
    ulonglong2 a[RT];
#pragma unroll
    for (int x = 0; x < RT; ++x) a[x] = *reinterpret_cast<const ulonglong2*>(sA + (ty + TY * x) * LD + c);
#pragma unroll
    for (int x = 0; x < RT; ++x)   // (an accumulator's two products lie apart: the second waits for the first)
#pragma unroll
      for (int y = 0; y < KT; ++y) fma_pair(acc[x][y], a[x].x, b[y].x);
#pragma unroll
    for (int x = 0; x < RT; ++x)
#pragma unroll
      for (int y = 0; y < KT; ++y) fma_pair(acc[x][y], a[x].y, b[y].y);
  }
#pragma unroll
  for (int x = 0; x < RT; ++x)
#pragma unroll
    for (int y = 0; y < KT; ++y) s[x][y] = lo_of(acc[x][y]) + hi_of(acc[x][y]);
}

template <typename T, int D>
__device__ inline const T* key_row_ptr(const CacheView& c, const void* slab, const void* blk, int unit,
                                       int smp, int kh, int I, int j) {
  if (j < c.n_old) return reinterpret_cast<const T*>(slab) + ((size_t)unit * c.cap + j) * D;
  const int jj = j - c.n_old;
  if (jj < I) return reinterpret_cast<const T*>(blk) + ((size_t)(smp * I + jj) * c.Hkv + kh) * D;
  return nullptr;
}

template <typename T, int D>
__device__ inline const T* query_row_ptr(const CacheView& c, const BlockArgs& a, int smp, int kh, int row) {
  if (row >= a.I * c.g) return nullptr;
  const int i = row / c.g, h = row % c.g;
  return reinterpret_cast<const T*>(a.q) + ((size_t)(smp * a.I + i) * c.Hq + kh * c.g + h) * D;
}

// ------------------------------------------------------------------------------------------------
// Forward: out = softmax(scale * q k^T) v over the n_old cached pairs and the block's causal pairs.
// Grid: (row tiles of the unit's I*g query rows, units).  Row r of a unit = (input r / g, head r % g).  Thread (ty, tx)
// owns rows ty + TY x of the tile, keys tx + 16 y of a key tile and output elements 4 tx + 64 y + [0, 4).
template <int D, int RT, int NT>
struct FwdSmem {
  static constexpr int TY = NT / 16, TM = TY * RT, LD = D + 4, PLD = kTN / 2 + 4;
  static constexpr int kFloats = TM * LD + kTN * LD + kTN * D + TM * PLD;
  static constexpr size_t kBytes = sizeof(float) * kFloats + sizeof(int) * kTN;   // 108 KB at TM = 64, D = 128: two CTAs per SM
};

template <typename T, int D, int RT, int NT>
__global__ void __launch_bounds__(NT, 2) attn_fwd_simt(CacheView c, BlockArgs a) {
  using L = FwdSmem<D, RT, NT>;
  constexpr int TY = L::TY, TM = L::TM, LD = L::LD, PLD = L::PLD, CT = D / 64;
  extern __shared__ __align__(16) float sm[];
  float* sQ = sm;
  float* sK = sQ + TM * LD;
  float* sV = sK + kTN * LD;
  float* sP = sV + kTN * D;                         // [TM][PLD]: the probabilities of half a key tile
  int* sKp = reinterpret_cast<int*>(sP + TM * PLD);  // [kTN] 1 = the tile's key is a padding pair

  const int unit = blockIdx.y, smp = unit / c.Hkv, kh = unit % c.Hkv;
  const int pad = sample_left_pad(c, smp);
  // (row tiles are handed out last first: a later tile sees more of the block's own keys)
  const int R = a.I * c.g, row0 = (gridDim.x - 1 - blockIdx.x) * TM;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int last_row = min(R - 1, row0 + TM - 1);
  const int n_keys = c.n_old + last_row / c.g + 1;  // keys visible to the tile's last row

  auto load_k = [&](int j0) {
    load_rows<T, D, LD, kTN, NT>(sK, tid, [&](int r) { return key_row_ptr<T, D>(c, c.k_slab, a.k, unit, smp, kh, a.I, j0 + r); });
  };
  auto load_v = [&](int j0) {
    load_rows<T, D, D, kTN, NT>(sV, tid, [&](int r) { return key_row_ptr<T, D>(c, c.v_slab, a.v, unit, smp, kh, a.I, j0 + r); });
  };
  load_rows<T, D, LD, TM, NT>(sQ, tid, [&](int r) { return query_row_ptr<T, D>(c, a, smp, kh, row0 + r); });
  load_k(0);
  load_v(0);

  f32x2 o[RT][2 * CT];
  float m[RT], l[RT];                               // running maximum of a row; this thread's share of its sum
  int vis[RT];
  bool real[RT];
#pragma unroll
  for (int x = 0; x < RT; ++x) {
    const int row = row0 + ty + TY * x;
    m[x] = -INFINITY;
    l[x] = 0.f;
    vis[x] = row < R ? c.n_old + row / c.g + 1 : 1;
    // a real query does not see padding pairs; a padding query's row is computed over everything and dropped
    real[x] = row < R && a.pos0 + row / c.g >= pad;
#pragma unroll
    for (int y = 0; y < 2 * CT; ++y) o[x][y] = 0;
  }

  for (int j0 = 0; j0 < n_keys; j0 += kTN) {
    const bool more = j0 + kTN < n_keys;
    wait_copies<1>();                               // K has arrived (and Q)
    if (pad > 0 && tid < kTN) {
      const int j = j0 + tid;
      sKp[tid] = j < c.n_old + a.I && (j < c.n_old ? c.kv_ids[(size_t)unit * c.cap + j] : a.pos0 + (j - c.n_old)) < pad;
    }
    __syncthreads();
    float s[RT][4];
    dot_rows<D, LD, TY, RT, 4>(sQ, sK, ty, tx, s);
    int padded[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) padded[y] = pad > 0 ? sKp[tx + 16 * y] : 0;
    __syncthreads();                                // K's place is free
    if (more) load_k(j0 + kTN);
    else commit_nothing();
#pragma unroll
    for (int x = 0; x < RT; ++x) {
      float mt = -INFINITY;
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const bool ok = j0 + tx + 16 * y < vis[x] && !(real[x] && padded[y]);
        s[x][y] = ok ? s[x][y] * a.scale : -INFINITY;
        mt = fmaxf(mt, s[x][y]);
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, off));
      const float m_new = fmaxf(m[x], mt);
      const float alpha = m_new == -INFINITY ? 1.f : expf(m[x] - m_new);
      m[x] = m_new;
      float ps = 0.f;
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        s[x][y] = s[x][y] == -INFINITY ? 0.f : expf(s[x][y] - m_new);
        ps += s[x][y];
      }
      l[x] = l[x] * alpha + ps;
      const f32x2 al = dup(alpha);
#pragma unroll
      for (int y = 0; y < 2 * CT; ++y) o[x][y] = mul_pair(o[x][y], al);
    }
    wait_copies<1>();                               // V has arrived
    __syncthreads();
#pragma unroll
    for (int half = 0; half < 2; ++half) {          // rows of P are written and read by the same half warp
#pragma unroll
      for (int x = 0; x < RT; ++x) {
        sP[(ty + TY * x) * PLD + tx] = s[x][2 * half];
        sP[(ty + TY * x) * PLD + tx + 16] = s[x][2 * half + 1];
      }
      __syncwarp();
#pragma unroll (RT <= 2 ? 4 : 1)
      for (int k = 0; k < kTN / 2; k += 4) {
        float4 p[RT];
#pragma unroll
        for (int x = 0; x < RT; ++x) p[x] = *reinterpret_cast<const float4*>(sP + (ty + TY * x) * PLD + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          ulonglong2 v[CT];
#pragma unroll
          for (int y = 0; y < CT; ++y)
            v[y] = *reinterpret_cast<const ulonglong2*>(sV + (half * (kTN / 2) + k + kk) * D + 4 * tx + 64 * y);
#pragma unroll
          for (int x = 0; x < RT; ++x) {
            const f32x2 pp = dup(kk == 0 ? p[x].x : kk == 1 ? p[x].y : kk == 2 ? p[x].z : p[x].w);
#pragma unroll
            for (int y = 0; y < CT; ++y) {
              fma_pair(o[x][2 * y], pp, v[y].x);
              fma_pair(o[x][2 * y + 1], pp, v[y].y);
            }
          }
        }
      }
      __syncwarp();
    }
    __syncthreads();                                // V's place is free
    if (more) load_v(j0 + kTN);
    else commit_nothing();
  }
#pragma unroll
  for (int x = 0; x < RT; ++x) {
    const int row = row0 + ty + TY * x;
    float lt = l[x];
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) lt += __shfl_xor_sync(0xffffffffu, lt, off);
    if (row >= R) continue;
    const int i = row / c.g, h = row % c.g;
    const float inv = real[x] ? 1.f / lt : 0.f;     // a padding query: zero output, and +inf so that it has no weights
    T* op = reinterpret_cast<T*>(a.out) + ((size_t)(smp * a.I + i) * c.Hq + kh * c.g + h) * D;
#pragma unroll
    for (int y = 0; y < CT; ++y) {
      const float w[4] = {lo_of(o[x][2 * y]) * inv, hi_of(o[x][2 * y]) * inv, lo_of(o[x][2 * y + 1]) * inv,
                          hi_of(o[x][2 * y + 1]) * inv};
      T* to = op + 4 * tx + 64 * y;
      if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(to) = make_float4(w[0], w[1], w[2], w[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) to[e] = Elem<T>::to_out(w[e]);
      }
    }
    if (tx == 0) a.lse[(size_t)unit * R + row] = real[x] ? m[x] + logf(lt) : INFINITY;
  }
}

// ------------------------------------------------------------------------------------------------
// Score pass: for every candidate pair j (cached or new) the column sum over all query rows of the
// block of exp(scale * q.k_j - lse_row), i.e. sum_i attn_weights[i][j] added over the group's heads.
// Grid: (tiles of 16 KT keys, units); query tiles of TM rows, the next one on its way while one is multiplied.
// Sums are formed in a fixed order (deterministic, no float atomics).
template <int D, int KT, int RT, int NT>
struct ScoreSmemSimt {
  static constexpr int TY = NT / 16, TM = TY * RT, LD = D + 4, kKeys = 16 * KT;
  static constexpr size_t kBytes = sizeof(float) * (kKeys * LD + 2 * TM * LD + 2 * TM + TY * kKeys);
};

template <typename T, int D, int KT, int RT, int NT>
__global__ void __launch_bounds__(NT, 2) score_simt(CacheView c, BlockArgs a) {
  using L = ScoreSmemSimt<D, KT, RT, NT>;
  constexpr int TY = L::TY, TM = L::TM, LD = L::LD, NK = L::kKeys;
  extern __shared__ __align__(16) float sm[];
  float* sK = sm;
  float* sQ = sK + NK * LD;                         // [2] tiles
  float* sLse = sQ + 2 * TM * LD;                  // [2][TM]
  float* sRed = sLse + 2 * TM;                     // [TY][NK]

  const int unit = blockIdx.y, smp = unit / c.Hkv, kh = unit % c.Hkv;
  uint32_t rank, C;                                 // CTAs of a cluster share a key tile and take its query tiles in turn
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  const int R = a.I * c.g, j0 = blockIdx.x / C * NK, n_c = c.n_old + a.I;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int counted_from = rule_first_counted_row(c.rule, c.window, a.I, c.g);   // rules that look at the last queries only
  const int first_row = (j0 > c.n_old) ? (j0 - c.n_old) * c.g : 0;  // earlier rows cannot see this tile
  // query tile t is CTA t % C's whatever the first one is, so that key tiles of 16 and of 64 add up in the same order
  const int t0 = first_row / TM, first_tile = (t0 + (((int)rank - t0) & ((int)C - 1))) * TM, step = (int)C * TM;

  auto load_q = [&](int row0, int b) {
    load_rows<T, D, LD, TM, NT>(sQ + b * TM * LD, tid, [&](int r) { return query_row_ptr<T, D>(c, a, smp, kh, row0 + r); });
    if (tid < TM)
      sLse[b * TM + tid] = (row0 + tid < R && row0 + tid >= counted_from) ? a.lse[(size_t)unit * R + row0 + tid] : INFINITY;
  };
  load_rows<T, D, LD, NK, NT>(sK, tid, [&](int r) { return key_row_ptr<T, D>(c, c.k_slab, a.k, unit, smp, kh, a.I, j0 + r); });
  load_q(first_tile, 0);
  float col[KT], col_sq[KT];
#pragma unroll
  for (int y = 0; y < KT; ++y) col[y] = col_sq[y] = 0.f;
  int b = 0;
  for (int row0 = first_tile; row0 < R; row0 += step, b ^= 1) {
    if (row0 + step < R) load_q(row0 + step, b ^ 1);   // (its place was last read before the barrier that ended the previous tile)
    else commit_nothing();
    wait_copies<1>();
    __syncthreads();
    float s[RT][KT];
    dot_rows<D, LD, TY, RT, KT>(sQ + b * TM * LD, sK, ty, tx, s);
#pragma unroll
    for (int x = 0; x < RT; ++x) {
      const int row = row0 + ty + TY * x;
      const float lse = sLse[b * TM + ty + TY * x];
      const int vis = row < R ? c.n_old + row / c.g + 1 : 0;
#pragma unroll
      for (int y = 0; y < KT; ++y) {
        // (roundings spelled out: the instances with key tiles of 16 and of 64 agree bit by bit)
        const float w = j0 + tx + 16 * y < vis ? expf(fmaf(s[x][y], a.scale, -lse)) : 0.f;
        col[y] = __fadd_rn(col[y], w);
        col_sq[y] = fmaf(w, w, col_sq[y]);
      }
    }
    __syncthreads();
  }
  // sum of key tid over the TY groups of rows of every CTA of the cluster (CTA 0's copy is used), in a fixed order
  auto reduce = [&](const float (&v)[KT]) {
#pragma unroll
    for (int y = 0; y < KT; ++y) sRed[ty * NK + tx + 16 * y] = v[y];
    __syncthreads();
    float tot = 0.f;
    if (tid < NK)
#pragma unroll
      for (int t = 0; t < TY; ++t) tot += sRed[t * NK + tid];
    __syncthreads();
    if (C > 1) {
      if (tid < NK) sRed[tid] = tot;
      cluster_barrier();
      if (rank == 0 && tid < NK)
        for (uint32_t p = 1; p < C; ++p) tot += ld_peer(&sRed[tid], p);
      cluster_barrier();                             // nobody leaves, or writes again, before the sums have been read
    }
    return tot;
  };
  float tot = reduce(col);
  const int j = j0 + tid;
  const bool mine = rank == 0 && tid < NK && j < n_c;
  if (mine) {
    const int pad = sample_left_pad(c, smp);
    if (pad > 0 && (j < c.n_old ? c.kv_ids[(size_t)unit * c.cap + j] : a.pos0 + (j - c.n_old)) < pad)
      tot = 0.f;                                    // a padding pair is masked for every query
    if (j < c.n_old) {
      if (rule_overwrites(c.rule)) c.sum_weights[(size_t)unit * c.cap + j] = tot;   // nothing is carried over
      else c.sum_weights[(size_t)unit * c.cap + j] += tot;
    }
    else a.new_sum[(size_t)unit * a.I + (j - c.n_old)] = tot;
  }
  if (c.sum_sq != nullptr) {    // rule 4: the same reduction over the squares
    tot = reduce(col_sq);
    if (mine) {
      if (j < c.n_old) c.sum_sq[(size_t)unit * c.cap + j] += tot;
      else a.new_sq[(size_t)unit * a.I + (j - c.n_old)] = tot;
    }
  }
}

template <typename T, int D, int RT, int NT>
cudaError_t launch_attn_rt(const CacheView& c, const BlockArgs& a, cudaStream_t st) {
  using L = FwdSmem<D, RT, NT>;
  static SmemConfigured configured;
  if (cudaError_t e = configured.ensure(attn_fwd_simt<T, D, RT, NT>, L::kBytes); e != cudaSuccess) return e;
  dim3 grid((a.I * c.g + L::TM - 1) / L::TM, c.nsamples * c.Hkv);
  ProfileScope prof(kAttnFwd, st);
  attn_fwd_simt<T, D, RT, NT><<<grid, NT, L::kBytes, st>>>(c, a);
  count_launch();
  return cudaGetLastError();
}

// Rows per tile: as many as still give every SM a CTA (small tiles re-read K and V more often and multiply fewer rows per
// operand read, but leave no SM idle).  2 samples, 4 heads, d = 64, 64 inputs against 128 pairs: 45 us with tiles of 64
// rows (8 CTAs), 16 us with tiles of 8 (64 CTAs); 2 samples, 16 heads in groups of 4, 128 inputs against 512 pairs: 201
// us with 64 rows (64 CTAs), 82 us with 16 (256 CTAs).
template <typename T, int D>
cudaError_t launch_attn_t(const CacheView& c, const BlockArgs& a, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    const int rows = a.I * c.g, units = c.nsamples * c.Hkv;
    auto fills = [&](int tm) { return (rows + tm - 1) / tm * units >= sm_count(); };
    if (!fills(16)) return launch_attn_rt<T, D, 1, 128>(c, a, st);
    if (!fills(64)) return launch_attn_rt<T, D, 2, 128>(c, a, st);
  }
  return launch_attn_rt<T, D, 4, 256>(c, a, st);
}

template <typename T, int D, int KT, int RT, int NT>
cudaError_t launch_score_kt(const CacheView& c, const BlockArgs& a, int cluster, cudaStream_t st) {
  using L = ScoreSmemSimt<D, KT, RT, NT>;
  static SmemConfigured configured;
  if (cudaError_t e = configured.ensure(score_simt<T, D, KT, RT, NT>, L::kBytes); e != cudaSuccess) return e;
  const dim3 grid((c.n_old + a.I + L::kKeys - 1) / L::kKeys * cluster, c.nsamples * c.Hkv);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3(NT);
  lc.dynamicSmemBytes = L::kBytes;
  lc.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = cluster > 1 ? 1 : 0;
  ProfileScope prof(kScore, st);
  const cudaError_t e = cudaLaunchKernelEx(&lc, score_simt<T, D, KT, RT, NT>, c, a);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Key tiles of 64; a handle whose caches of a layer make fewer than four CTAs per SM shares each key tile among a cluster
// as long as there are query tiles to share (16 caches, 1024 query rows against 256 keys: 84 -> 45 us with clusters of 8;
// against 1536 keys 261 -> 226 us with clusters of 2, 287 with none below two CTAs per SM).  The cluster decides the
// order of the column sums, so the handle's caches decide it and not the call's.  Key tiles of 16, which add up in the
// same order, if SMs would still be idle.
template <typename T, int D>
cudaError_t launch_score_t(const CacheView& c, const BlockArgs& a, cudaStream_t st) {
  const int tiles = (c.n_old + a.I + 63) / 64, q_tiles = (a.I * c.g + 63) / 64;
  int cluster = 1;
  while (cluster < 8 && 2 * cluster <= q_tiles && (long long)tiles * c.layer_units * cluster < 4 * sm_count()) cluster *= 2;
  if constexpr (sizeof(T) == 4)
    if ((long long)tiles * c.nsamples * c.Hkv * cluster < sm_count()) return launch_score_kt<T, D, 1, 4, 256>(c, a, cluster, st);
  return launch_score_kt<T, D, 4, 4, 256>(c, a, cluster, st);
}

}  // namespace

cudaError_t launch_attn_simt(int dtype, int d, const CacheView& c, const BlockArgs& a, cudaStream_t st) {
  if (dtype == 0 && d == 64) return launch_attn_t<float, 64>(c, a, st);
  if (dtype == 0 && d == 128) return launch_attn_t<float, 128>(c, a, st);
  if (dtype == 1 && d == 64) return launch_attn_t<__nv_bfloat16, 64>(c, a, st);
  if (dtype == 1 && d == 128) return launch_attn_t<__nv_bfloat16, 128>(c, a, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_score_simt(int dtype, int d, const CacheView& c, const BlockArgs& a, cudaStream_t st) {
  if (dtype == 0 && d == 64) return launch_score_t<float, 64>(c, a, st);
  if (dtype == 0 && d == 128) return launch_score_t<float, 128>(c, a, st);
  if (dtype == 1 && d == 64) return launch_score_t<__nv_bfloat16, 64>(c, a, st);
  if (dtype == 1 && d == 128) return launch_score_t<__nv_bfloat16, 128>(c, a, st);
  return cudaErrorInvalidValue;
}

}  // namespace bm
