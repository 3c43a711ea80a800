// Forward pass, TWO tiles of 128 query rows of a cache per CTA, one CTA per SM (included by attn_tc.cu after TcMaps /
// TcArgs): the softmax of one tile runs under the MMAs of the other.
//
// Per tile the chain logits -> softmax -> P.V -> next logits is serial, because the bf16 probabilities take the place of
// the logits in tensor memory (S 128 + O 128 columns per tile: two tiles fill it).  That chain is what bounds the kernel
// (ncu, profiles/kernels_48_samples.md: tensor pipe busy 48 % of the cycles, special-function unit 37 %, issue slots 39 %,
// DRAM 14 %; most stalls are waits on tensor memory and barriers).  A thread holds all 128 logits of its row in registers:
// one read of tensor memory, no exchange of maxima.  Every fourth pair of exponentials is a polynomial of degree 5 on the
// FMA and integer pipes (all on the special-function unit: 7 % slower; an eighth: the same); a warp arrives once on a
// barrier, not lane by lane (9 % slower).
//
// Measured at 48 samples, 32 heads in groups of 4, d = 128, a block of 512 against 1024 pairs: 936 -> 963 TFLOP/s against
// the kernel with one tile per CTA and two CTAs per SM; 32 samples, 32 heads, a block of 1024: 930 -> 955; d = 64, 701
// pairs, groups of 8: 162 -> 156 us.  Not kept: one issuing thread for both tiles (936), issuers without turns (745: the
// tiles fall into step), publishing after 96 keys instead of 64 (882), exponentials relative to the running maximum with the tile's formed beside them (866), two
// threads per row (934), tile B started half a period later (936 to 955), polling softmax warps (952).
//
// Warps 0-3: rows of tile A, 4-7: rows of tile B, 8 and 9: MMA issue for A and B, 10: TMA producer.  Shared memory: Q_A |
// Q_B (reused to stage the outputs) | ring of two stages of a K and a V tile, shared by the two tiles.
#pragma once

template <int D>
struct PairSmem {
  static constexpr int kChunks = D / 64;
  static constexpr int kTileBytes = kChunks * 16384;     // 128 rows x D bf16
  static constexpr int kStages = 2;                      // ring: entry e = K_e | V_{e-1}, what one step of the chains needs
  static constexpr int kStageBytes = 2 * kTileBytes;
  static constexpr int kQ = 0;
  static constexpr int kKV = 2 * kTileBytes;
  static constexpr int kBars = kKV + kStages * kStageBytes;
  static constexpr int kTotal = kBars + 256 + 1024;      // + barriers + alignment slack
  static constexpr int kThreads = 384;
};

template <int D>
__global__ void __launch_bounds__(384, 1) attn_fwd_pair(const __grid_constant__ TcMaps maps, const TcArgs a) {
  using L = PairSmem<D>;
  constexpr int kMmaWarp = 8 /* tile A; 9: tile B */, kTmaWarp = 10, NS = L::kStages;
  constexpr int B_QFULL = 0 /* 2 tiles */, B_KVFULL = 2, B_KVEMPTY = B_KVFULL + NS, B_SFULL = B_KVEMPTY + NS, B_PHALF = B_SFULL + 2,
                B_PFULL = B_PHALF + 2, B_ODONE = B_PFULL + 2, B_TURN = B_ODONE + 2, B_COUNT = B_TURN + 2;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::kBars);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int unit = blockIdx.y, smp = unit / a.Hkv, kh = unit % a.Hkv;
  const int R = a.I * a.g;
  const int qpt = kTileM / a.g;                  // inputs (positions) covered by a row tile
  const int t_old = (a.n_old + kTileN - 1) / kTileN;
  // pairs of row tiles (or single ones: tile B has no rows) are handed out last first (a later tile sees more of the
  // block's own keys)
  const int rt0 = a.row_tiles * (gridDim.x - 1 - blockIdx.x);
  // key tiles a row tile sees: the cached ones and the block's up to its last input; no rows, no tiles
  auto n_tiles = [&](int x) {
    const int i0 = (rt0 + x) * qpt;
    return x >= a.row_tiles || i0 >= a.I ? 0 : t_old + min(a.I - 1, i0 + qpt - 1) / kTileN + 1;
  };
  const int T0 = n_tiles(0), T1 = n_tiles(1), T = max(T0, T1);   // T1 >= T0 unless tile B has no rows

  auto load_stage = [&](int e) {   // K_e (if there is one) and V_{e-1}
    unsigned char* dst = sm + L::kKV + (e % NS) * L::kStageBytes;
    uint64_t* bar = &bars[B_KVFULL + e % NS];
    mbar_expect_tx(bar, (e < T ? L::kTileBytes : 0) + (e > 0 ? L::kTileBytes : 0));
    for (int is_v = 0; is_v < 2; ++is_v) {
      const int j = e - is_v;
      if (j < 0 || j >= T) continue;
      for (int c = 0; c < L::kChunks; ++c) {
        unsigned char* to = dst + is_v * L::kTileBytes + c * 16384;
        if (j < t_old) tma_load_3d(to, is_v ? &maps.v_slab : &maps.k_slab, c * 64, j * kTileN, unit, bar);
        else tma_load_4d(to, is_v ? &maps.v_blk : &maps.k_blk, c * 64, kh, (j - t_old) * kTileN, smp, bar);
      }
    }
  };
  if (warp == kTmaWarp && lane == 0) {
    *abort_flag = 0;
    for (int x = 0; x < 2; ++x) {
      mbar_init(&bars[B_QFULL + x], 1);
      mbar_init(&bars[B_SFULL + x], 1);
      mbar_init(&bars[B_PHALF + x], 4);          // one arrival per warp
      mbar_init(&bars[B_PFULL + x], 4);
      mbar_init(&bars[B_ODONE + x], 1);
      mbar_init(&bars[B_TURN + x], 1);
    }
    for (int s = 0; s < NS; ++s) { mbar_init(&bars[B_KVFULL + s], 1); mbar_init(&bars[B_KVEMPTY + s], T1 > 0 ? 2 : 1); }
    mbar_fence_init();
    for (int x = 0; x < 2; ++x) {
      if (x == 1 && T1 == 0) break;
      mbar_expect_tx(&bars[B_QFULL + x], L::kTileBytes);
      for (int c = 0; c < L::kChunks; ++c)
        tma_load_5d(sm + L::kQ + x * L::kTileBytes + c * 16384, &maps.q, c * 64, 0, kh, (rt0 + x) * qpt, smp, &bars[B_QFULL + x]);
      if (x == 0) load_stage(0);
    }
    load_stage(1);
  }
  if (warp == kMmaWarp) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;              // S_A | S_B | O_A | O_B, 128 columns each

  if (warp >= kMmaWarp) {
    // 384 threads start with 168 registers each; the softmax threads take what these four warps leave
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp == kTmaWarp) {
      // ---------------------------------------------------------------- TMA producer
      if (lane == 0)
        for (int e = NS; e <= T; ++e) {
          mbar_wait(&bars[B_KVEMPTY + e % NS], (e / NS - 1) & 1, abort_flag, a.status);
          load_stage(e);
        }
    } else if (warp < kTmaWarp && lane == 0) {
      // ---------------------------------------------------------------- MMA issuer of tile x (one thread each: a
      // single one for both was 3 % slower)
      const int x = warp - kMmaWarp, Tx = x ? T1 : T0;
      const uint32_t idesc_qk = instr_desc(kTileM, kTileN, 0, 0);
      const uint32_t idesc_pv = instr_desc(kTileM, D, 0, 1);  // V is MN-major: d contiguous, keys along K
      const uint64_t dk_hi = smem_desc(0, 16, 1024) & 0xffffffff00000000ull;      // K-major operands (Q, K)
      const uint32_t dk_lo = (uint32_t)(smem_desc(0, 16, 1024) & 0xffffffffull);
      const uint64_t dv_hi = smem_desc(0, 16384, 1024) & 0xffffffff00000000ull;   // MN-major operand (V)
      const uint32_t dv_lo = (uint32_t)(smem_desc(0, 16384, 1024) & 0xffffffffull);
      const uint32_t q_lo = dk_lo + (smem_u32(sm + L::kQ + x * L::kTileBytes) >> 4), kv = smem_u32(sm + L::kKV) >> 4;
      const uint32_t tm_s = tmem + 128 * x, tm_o = tmem + 256 + 128 * x;
      auto issue_qk = [&](int e) {               // S = Q K_e^T; with it the ring entry is used up
        const uint32_t k_lo = dk_lo + kv + (uint32_t)(e % NS) * (L::kStageBytes >> 4);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t off = (ks >> 2) * 1024 + (ks & 3) * 2;   // (chunk * 16384 + kstep * 32) / 16
          mma_ss(tm_s, dk_hi | (q_lo + off), dk_hi | (k_lo + off), idesc_qk, ks > 0 ? 1u : 0u);
        }
        mma_commit(&bars[B_SFULL + x]);
      };
      auto wait = [&](int b, uint32_t parity) { mbar_poll(&bars[b], parity, abort_flag, a.status); };
      // The two issuers take turns, so that one tile's MMAs run behind each other and not between the other's: left to
      // themselves the tiles fell into step, both in their softmax and then both in their MMAs (745 against 963 TFLOP/s).
      auto my_turn = [&](int e) {                // A's e-th turn comes after B's e-1st, B's after A's e-th
        if (T1 > 0 && (x == 1 || e > 0)) wait(B_TURN + x, (uint32_t)(x ? e : e - 1) & 1);
      };
      auto pass_turn = [&]() { mbar_arrive(&bars[B_TURN + (x ^ 1)]); };
      if (Tx > 0) {
        mbar_wait(&bars[B_QFULL + x], 0, abort_flag, a.status);
        mbar_wait(&bars[B_KVFULL], 0, abort_flag, a.status);
        my_turn(0);
        tc_fence_after();
        issue_qk(0);
        pass_turn();
        mma_commit(&bars[B_KVEMPTY]);
        for (int e = 1; e <= T; ++e) {           // products of key tile e - 1, logits of key tile e
          mbar_wait(&bars[B_KVFULL + e % NS], (e / NS) & 1, abort_flag, a.status);
          if (e > Tx) {                          // (the other tile sees one key tile more)
            my_turn(e);                          // (a turn passed twice would leave the other tile's wait two phases behind)
            pass_turn();
            mbar_arrive(&bars[B_KVEMPTY + e % NS]);
            break;
          }
          const uint32_t v_lo = dv_lo + kv + ((uint32_t)(e % NS) * L::kStageBytes + L::kTileBytes >> 4);
          // O += P V, P read from tensor memory (over S), in two halves of 64 keys
#pragma unroll
          for (int ph = 0; ph < 2; ++ph) {
            if (ph == 1) my_turn(e);             // (usually long since passed on: not behind the wait below)
            wait((ph ? B_PFULL : B_PHALF) + x, (e - 1) & 1);
            tc_fence_after();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int ks = 4 * ph + q;
              mma_ts(tm_o, tm_s + ks * 8, dv_hi | (v_lo + ks * 128), idesc_pv, (e > 1 || ks > 0) ? 1u : 0u);
            }
          }
          if (e < Tx) issue_qk(e);
          else mma_commit(&bars[B_ODONE + x]);
          pass_turn();
          mma_commit(&bars[B_KVEMPTY + e % NS]);
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax + epilogue: a thread per row
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");   // 2 x 128 x 216 + 128 x 72 = 384 x 168
    const int x = warp >> 2, quad = warp & 3, Tx = x ? T1 : T0;
    const int r = quad * 32 + lane;               // row inside the tile == TMEM lane
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t tm_s = tmem + 128 * x + lane_addr, tm_o = tmem + 256 + 128 * x + lane_addr;
    const int i0 = (rt0 + x) * qpt, row = (rt0 + x) * kTileM + r;
    const int i_row = min(a.I - 1, i0 + r / a.g);  // rows past the block's end behave like its last input
    float m_used = -INFINITY, l = 0.f;
    for (int j = 0; j < Tx; ++j) {
      mbar_wait(&bars[B_SFULL + x], j & 1, abort_flag, a.status);
      tc_fence_after();
      uint32_t s[4][32];
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32(tm_s + 32 * c, s[c]);
      // visible columns of this key tile for this row: [0, nvis)
      const int nvis = (j < t_old) ? min(kTileN, a.n_old - j * kTileN)
                                   : max(0, min(kTileN, i_row - (j - t_old) * kTileN + 1));
      tmem_wait_ld();
      if (!__all_sync(0xffffffffu, nvis >= kTileN)) {   // hidden logits become -inf: probability 0
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int e = 0; e < 32; ++e) s[c][e] = 32 * c + e < nvis ? s[c][e] : 0xff800000u;
      }
      // A NaN or +inf among a row's visible logits makes the row NaN, through its maximum: the polynomial of every fourth
      // pair takes NaN for its lowest argument.
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int e = 0; e < 32; e += 2)
#pragma unroll
        for (int c = 0; c < 4; ++c) m4[c] = max3_nan(m4[c], __uint_as_float(s[c][e]), __uint_as_float(s[c][e + 1]));
      float mx2 = max3_nan(max3_nan(m4[0], m4[1], m4[2]), m4[3], -INFINITY) * a.scale_log2;
      if (mx2 == INFINITY) mx2 = __uint_as_float(0x7fffffffu);
      bool rescale = false;
      float alpha = 1.f;
      if (j == 0) m_used = mx2;
      else if (!(mx2 <= m_used + kRescaleThreshold)) { alpha = ex2(m_used - mx2); m_used = mx2; rescale = true; }
      // S(j) being complete implies the previous P.V into O has completed, so O may be touched here (rarely)
      if (__any_sync(0xffffffffu, rescale)) {
#pragma unroll 1
        for (int cc = 0; cc < D / 16; ++cc) {
          uint32_t raw[16];
          tmem_ld16(tm_o + cc * 16, raw);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) raw[e] = __float_as_uint(__uint_as_float(raw[e]) * alpha);
          tmem_st16(tm_o + cc * 16, raw);
        }
        l *= alpha;
      }
      const float neg_m = -m_used;
      float pa0 = 0.f, pa1 = 0.f, pb0 = 0.f, pb1 = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          float x0, x1, p0, p1;
          fma2(x0, x1, __uint_as_float(s[c][2 * e]), __uint_as_float(s[c][2 * e + 1]), a.scale_log2, neg_m);
          if (e % 4 == 3) ex2_poly2_deg5(x0, x1, p0, p1);
          else { p0 = ex2(x0); p1 = ex2(x1); }
          if (e & 1) add2(pb0, pb1, p0, p1);
          else add2(pa0, pa1, p0, p1);
          pk[e] = pack_bf16(p0, p1);
        }
        tmem_st16(tm_s + 16 * c, pk);             // over logits that are all in registers by now
        if (c & 1) {                              // the first 64 keys may enter P.V under the others' exponentials
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars[(c == 1 ? B_PHALF : B_PFULL) + x]);
        }
      }
      l += (pa0 + pb0) + (pa1 + pb1);
    }
    // epilogue: O / l -> bf16 -> swizzled tile in the (now idle) query buffer -> TMA store; log2-sum-exp
    if (Tx > 0) {
      mbar_wait(&bars[B_ODONE + x], 0, abort_flag, a.status);
      tc_fence_after();
      const float inv = 1.f / l;
      unsigned char* stage = sm + L::kQ + x * L::kTileBytes;
#pragma unroll 1
      for (int cc = 0; cc < D / 32; ++cc) {       // 32-column chunk of the output row
        uint32_t raw[32];
        tmem_ld32(tm_o + cc * 32, raw);
        tmem_wait_ld();
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          uint4 w;
          w.x = pack_bf16(__uint_as_float(raw[q4 * 8 + 0]) * inv, __uint_as_float(raw[q4 * 8 + 1]) * inv);
          w.y = pack_bf16(__uint_as_float(raw[q4 * 8 + 2]) * inv, __uint_as_float(raw[q4 * 8 + 3]) * inv);
          w.z = pack_bf16(__uint_as_float(raw[q4 * 8 + 4]) * inv, __uint_as_float(raw[q4 * 8 + 5]) * inv);
          w.w = pack_bf16(__uint_as_float(raw[q4 * 8 + 6]) * inv, __uint_as_float(raw[q4 * 8 + 7]) * inv);
          const int piece = cc * 4 + q4;          // 16-byte piece of the row: chunk = piece / 8
          *reinterpret_cast<uint4*>(stage + (piece >> 3) * 16384 + sw128_offset(r, piece & 7)) = w;
        }
      }
      if (row < R) a.lse2[(size_t)unit * R + row] = m_used + log2f(l);
      fence_async_smem();
      named_bar_sync(1 + x, 128);
      if (r == 0) {
        for (int c = 0; c < L::kChunks; ++c) tma_store_5d(&maps.o, stage + c * 16384, c * 64, 0, kh, i0, smp);
        tma_store_commit_and_wait();
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}
