// Forward pass, one persistent CTA per SM with two softmax groups, A and B (included by attn_tc.cu after TcMaps / TcArgs).
//
// Warps 0-3: softmax of A (a thread per query row), 4-7: of B, 8: issues every S = Q.K^T, 9 and 10: issue O += P.V of A and
// of B, 11: TMA producer, which also asks for the CTA's next work item.  A work item is
//   kPairs: two row tiles of a cache, one for each group (they share the K and V tiles), or
//   kAny: two row tiles of any caches, each with key tiles of its own, loaded in turn, or a single row tile (a row's arithmetic is
//   that of kPairs), or
//   kSplit: one row tile, whose key tiles the groups take in turn; their two partial outputs meet at the end.
//
// Tensor memory, 512 columns: O_A | O_B (D each) | P_A | P_B (64 each, bf16 pairs) | S (128 at D = 128, shared by the
// groups; two of 128 at D = 64).  A group reads its 128 logits of a row into registers at once and gives S back, so the
// next Q.K^T runs under the exponentials; P has columns of its own and P.V runs behind the softmax as well.
// What is left on a group's chain is its own softmax, and the two groups' chains are independent of each other.
//
// What bounds it: the two softmax warps that share a scheduler, about 2850 cycles per pair of tiles at d = 64 (their
// instructions alone take 2100 to 2250, the exponentials 1792 on the special-function unit, an eighth being polynomials),
// and at d = 128 the turns of the one logit buffer, 3150 (the tensor pipe needs 2048, and so do the exponentials: both busy
// 57 %).  Measured at 48 samples, 32 heads in groups of 4, d = 128, a block of 512 against 1024 pairs: 539 -> 479 us (1076
// TFLOP/s) against the kernel in which P takes the place of the logits and the next Q.K^T waits for P.V; 128 samples 1399
// -> 1254; 4 samples, 512 pairs 45.3 -> 40.3; d = 64, 701 pairs, groups of 8 161 -> 139.  What made the difference besides:
// code that fits the SM's 32 KB instruction cache with room for every role's loop (at 78 KB this kernel took 692 us at 48
// samples and 2.5 of every issue slot's waiting warps waited for instructions; at 54 KB 615), hence masks in a rolled loop,
// rolled waits, one copy per key tile; output through TMA (with plain stores 5 600 cycles per item, 4 100 now).  Not kept:
// a share of the exponentials as polynomials at d = 128 (a quarter: 513 against 492 us; an eighth 507; at d = 64 none 139,
// an eighth 135, a quarter 136), softmax warps that poll for their logits (527 against 513), 216 registers for them (530).
#pragma once

template <int D>
struct PairSmem {
  static constexpr int kChunks = D / 64;
  static constexpr int kTileBytes = kChunks * 16384;     // 128 rows x D bf16
  static constexpr int kStages = D == 128 ? 2 : 4;       // K tiles, and V tiles, in flight
  static constexpr int kQ = 0;                           // [2]
  static constexpr int kK = kQ + 2 * kTileBytes;
  static constexpr int kV = kK + kStages * kTileBytes;
  static constexpr int kOut = kV + kStages * kTileBytes;   // a softmax warp's 32 output rows, 64 elements at a time
  static constexpr int kBars = kOut + 8 * 4096;
  static constexpr int kTotal = kBars + 512 + 1024;      // + barriers + alignment slack
  static constexpr int kThreads = 384;
};

enum Items { kPairs, kAny, kSplit };   // what a work item is (above)

template <int D, bool PAD, Items ITEMS>
__global__ void __launch_bounds__(384, 1) attn_fwd_pair(const __grid_constant__ TcMaps maps, const TcArgs a) {
  using L = PairSmem<D>;
  constexpr bool SPLIT = ITEMS == kSplit, ANY = ITEMS == kAny;
  constexpr int kQkWarp = 8, kPvWarp = 9 /* A; 10: B */, kTmaWarp = 11, NS = L::kStages;
  constexpr int NSB = D == 128 ? 1 : 2;                  // logit buffers
  constexpr int B_QFULL = 0, B_QFREE = 2, B_KFULL = 4, B_KFREE = B_KFULL + NS, B_VFULL = B_KFREE + NS, B_VFREE = B_VFULL + NS,
                B_SFULL = B_VFREE + NS, B_SFREE = B_SFULL + 2, B_P = B_SFREE + 2 /* [half][group] */, B_PV = B_P + 4 /* likewise */,
                B_RESP = B_PV + 4, B_NEXT = B_RESP + 1, B_NEXTFREE = B_NEXT + 2, B_COUNT = B_NEXTFREE + 2;
  static_assert(8 * B_COUNT + 7 * 16 + 8 <= 512, "");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* resp = sm + L::kBars;                   // response to the request for a work item, 16 bytes
  int4* items = reinterpret_cast<int4*>(sm + L::kBars + 16);   // [2][2]: this work item and the next; [2]: kAny, the second group's caches
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::kBars + 112);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + B_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = a.I * a.g, qpt = kTileM / a.g;   // query rows of a cache; inputs (positions) covered by a row tile
  const int t_old = (a.n_old + kTileN - 1) / kTileN;

  struct Place { int unit, smp, kh; };           // cache, its sample, its head
  struct Item { int unit, smp, kh, rt0, rt1, n0, n1, T; };   // row tile and number of key tiles of either group; key tiles loaded
  // Written by the producer, m-th item into place m % 2 (T = 0: there is none).  Row tiles are handed out last first (a later
  // tile sees more of the block's own keys): within a cache, or (a.across, kAny) over all caches.
  auto write_item = [&](int m, bool there, int bx, int by) {
    Item it;
    const int row_tiles = ANY ? (R + kTileM - 1) / kTileM : 0, second = ANY ? a.any * bx + a.any - 1 : 0;
    it.unit = ANY ? a.any * bx % a.units : a.across ? bx : by;
    it.smp = it.unit / a.Hkv;
    it.kh = it.unit - it.smp * a.Hkv;
    const int grp = a.across ? (int)gridDim.y - 1 - by : (int)gridDim.x - 1 - bx;
    // key tiles a row tile sees: the cached ones and the block's up to its last input; no rows, no tiles
    auto n_tiles = [&](int rt) { return rt * qpt >= a.I ? 0 : t_old + min(a.I - 1, rt * qpt + qpt - 1) / kTileN + 1; };
    it.rt0 = ANY ? row_tiles - 1 - a.any * bx / a.units : SPLIT ? grp : 2 * grp;
    it.rt1 = ANY ? row_tiles - 1 - second / a.units : SPLIT ? grp : 2 * grp + 1;
    it.n0 = n_tiles(it.rt0);
    it.n1 = SPLIT ? it.n0 / 2 : ANY && (a.any < 2 || it.rt1 < 0) ? 0 : n_tiles(it.rt1);
    it.T = SPLIT ? it.n0 : ANY ? it.n0 + it.n1 : max(it.n0, it.n1);
    if (SPLIT) it.n0 -= it.n1;
    items[2 * (m & 1)] = make_int4(it.unit, it.smp, it.kh, there ? it.T : 0);
    items[2 * (m & 1) + 1] = make_int4(it.rt0, it.rt1, it.n0, it.n1);
    if (ANY) {
      const int unit = second % a.units, smp = unit / a.Hkv;
      items[4 + (m & 1)] = make_int4(unit, smp, unit - smp * a.Hkv, 0);
    }
  };
  auto place = [&](const Item& it, int m, int x) {   // of group x's row tile
    if (ANY && x == 1) { const int4 u = items[4 + (m & 1)]; return Place{u.x, u.y, u.z}; }
    return Place{it.unit, it.smp, it.kh};
  };
  auto read_item = [&](int m) {
    if (m > 0) mbar_wait(&bars[B_NEXT + (m & 1)], ((m - 1) >> 1) & 1, abort_flag, a.status);
    const int4 u = items[2 * (m & 1)], v = items[2 * (m & 1) + 1];
    Item it = {u.x, u.y, u.z, v.x, v.y, v.z, v.w, u.w};
    if (*abort_flag) it.T = 0;
    return it;
  };
  auto item_read = [&](int m) { mbar_arrive(&bars[B_NEXTFREE + (m & 1)]); };   // once per warp
  // kAny: the group whose key tile is the j-th that is loaded: in turn, then what the longer one has left
  auto owner = [&](const Item& it, int j) { return j < 2 * min(it.n0, it.n1) ? j & 1 : it.n0 > it.n1 ? 0 : 1; };
  auto takes = [&](const Item& it, int x, int j) {   // group x, j-th key tile
    return SPLIT ? (j & 1) == x : ANY ? owner(it, j) == x : j < (x ? it.n1 : it.n0);
  };
  if (warp == kTmaWarp && lane == 0) {
    *abort_flag = 0;
#pragma unroll 1
    for (int b = 0; b < B_COUNT; ++b)
      mbar_init(&bars[b], b >= B_NEXTFREE ? 11 : (b >= B_SFREE && b < B_PV) ? 4 /* a warp arrives once */ : (b >= B_VFREE && b < B_SFULL) ? 2 : 1);
    mbar_fence_init();
    write_item(0, true, blockIdx.x, blockIdx.y);
  }
  if (warp == kQkWarp) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tm_o0 = tmem, tm_p0 = tmem + 2 * D, tm_s0 = tmem + 2 * D + 128;   // group x: + D x, + 64 x, + 128 x (NSB = 2)
  auto wait = [&](int b, int n) { mbar_wait(&bars[b], (uint32_t)n & 1, abort_flag, a.status); };   // for the n-th completion
  auto poll = [&](int b, int n) { mbar_poll(&bars[b], (uint32_t)n & 1, abort_flag, a.status); };

  if (warp >= kQkWarp) {
    // 384 threads start with 168 registers each; the softmax threads take what these four warps leave
    asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    if (lane == 0) {
      const uint64_t dk_hi = smem_desc(0, 16, 1024) & 0xffffffff00000000ull;      // K-major operands (Q, K)
      const uint32_t dk_lo = (uint32_t)(smem_desc(0, 16, 1024) & 0xffffffffull);
      const uint64_t dv_hi = smem_desc(0, 16384, 1024) & 0xffffffff00000000ull;   // MN-major operand (V)
      const uint32_t dv_lo = (uint32_t)(smem_desc(0, 16384, 1024) & 0xffffffffull);
      if (warp == kTmaWarp) {
        // -------------------------------------------------------------- TMA producer
        int kc = 0, vc = 0, q0c = 0, q1c = 0, k = 0;   // tiles and items so far
        for (bool more = true; more; ++k) {
          const Item it = read_item(k);          // (its own)
          const bool two = !SPLIT && it.n1 > 0;  // query tiles
          const Place own[2] = {place(it, k, 0), place(it, k, 1)};
          // The second group's query tile follows the first keys, for which the first group waits: 48 caches of four row tiles, 512 pairs
          // 40.6 -> 39.1 us a call, serving batch 3262 -> 3245 per pass.  (At d = 64, half the bytes, unordered 2169 -> 2177: not there.)
          auto load_queries = [&](int x) {
            int& n = x ? q1c : q0c;
            if (n > 0) wait(B_QFREE + x, n - 1);
            ++n;
            mbar_expect_tx(&bars[B_QFULL + x], L::kTileBytes);
#pragma unroll 1
            for (int c = 0; c < L::kChunks; ++c)
              tma_load_5d(sm + L::kQ + x * L::kTileBytes + c * 16384, &maps.q, c * 64, 0, x ? own[1].kh : own[0].kh,
                          (x ? it.rt1 : it.rt0) * qpt, x ? own[1].smp : own[0].smp, &bars[B_QFULL + x]);
          };
#pragma unroll 1
          for (int e = 0; e <= it.T; ++e) {
            if (e == it.T - 1) {                 // (not earlier: a CTA that is ahead should find the item still there)
              // the next one: a CTA of the grid that has not started yet is taken off the launch queue
              mbar_expect_tx(&bars[B_RESP], 16);
              asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                           ::"r"(smem_u32(resp)), "r"(smem_u32(&bars[B_RESP])) : "memory");
            }
            if (e == 0)
#pragma unroll 1
              for (int x = 0; x <= (D == 64 && two ? 1 : 0); ++x) load_queries(x);
#pragma unroll 1
            for (int is_v = 0; is_v < 2; ++is_v) {   // K_e, V_{e-1}
              const int j = e - is_v;
              if (j < 0 || j >= it.T) continue;
              int& n = is_v ? vc : kc;
              const int s = n % NS;
              uint64_t* bar = &bars[(is_v ? B_VFULL : B_KFULL) + s];
              if (n >= NS) wait((is_v ? B_VFREE : B_KFREE) + s, n / NS - 1);
              ++n;
              mbar_expect_tx(bar, L::kTileBytes);
              const int both = ANY ? min(it.n0, it.n1) : 0;        // key tiles that the groups take in turn
              const int t = j < 2 * both ? j >> 1 : j - both;      // the tile's place in its cache
              const Place& of = ANY && owner(it, j) ? own[1] : own[0];
              const bool old = t < t_old;
              const CUtensorMap* m = old ? (is_v ? &maps.v_slab : &maps.k_slab) : (is_v ? &maps.v_blk : &maps.k_blk);
              tma_load_5d(sm + (is_v ? L::kV : L::kK) + s * L::kTileBytes, m, 0, old ? 0 : of.kh, (old ? t : t - t_old) * kTileN,
                          old ? of.unit : of.smp, 0, bar);
            }
            if (D == 128 && e == 0 && two) load_queries(1);
          }
          wait(B_RESP, k);
          uint32_t ok = 0, bx = 0, by = 0;
          asm volatile("{\n.reg .pred p;\n.reg .b128 r;\nld.shared.b128 r, [%3];\n"
                       "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\nselp.u32 %0, 1, 0, p;\n"
                       "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, %2, _, _}, r;\n}\n"
                       : "+r"(ok), "+r"(bx), "+r"(by) : "r"(smem_u32(resp)) : "memory");
          fence_async_smem();                    // (the next response comes into the same place)
          more = ok != 0 && !*abort_flag;
          const int m = k + 1;
          if (m >= 2) wait(B_NEXTFREE + (m & 1), (m >> 1) - 1);
          write_item(m, more, (int)bx, (int)by);
          mbar_arrive(&bars[B_NEXT + (m & 1)]);
        }
        if (*abort_flag) {                       // what is on its way into this CTA's shared memory arrives first
          auto drain = [&](int b, int n) {
#pragma unroll 1
            for (int i = 0; i < kWaitLimit && !mbar_test(smem_u32(&bars[b]), (uint32_t)n & 1); ++i) {}
          };
          for (int n = max(0, kc - NS); n < kc; ++n) drain(B_KFULL + n % NS, n / NS);
          for (int n = max(0, vc - NS); n < vc; ++n) drain(B_VFULL + n % NS, n / NS);
          drain(B_QFULL, q0c - 1);
          if (q1c > 0) drain(B_QFULL + 1, q1c - 1);
          drain(B_RESP, k - 1);
        }
      } else if (warp == kQkWarp) {
        // -------------------------------------------------------------- S = Q K^T of both groups, in turn
        const uint32_t idesc = instr_desc(kTileM, kTileN, 0, 0);
        const uint32_t q_lo = dk_lo + (smem_u32(sm + L::kQ) >> 4), k_base = dk_lo + (smem_u32(sm + L::kK) >> 4);
        int kc = 0, qc0 = 0, qc1 = 0, sc0 = 0, sc1 = 0, last = -1;
        for (int k = 0;; ++k) {
          const Item it = read_item(k);
          item_read(k);
          if (it.T == 0) break;
          wait(B_QFULL, qc0++);
          bool q1_there = false;
#pragma unroll 1
          for (int j = 0; j < it.T; ++j, ++kc) {
            wait(B_KFULL + kc % NS, kc / NS);
            const uint32_t k_lo = k_base + (uint32_t)(kc % NS) * (L::kTileBytes >> 4);
#pragma unroll 1
            for (int x = 0; x < 2; ++x) {
              if (!takes(it, x, j)) continue;
              if (x == 1 && !SPLIT && (ANY ? !q1_there : j == 0)) { wait(B_QFULL + 1, qc1++); q1_there = true; }
              // the logits that the buffer holds have been read
              const int before = NSB == 2 ? x : last, n = before == 0 ? sc0 : sc1;
              if (before >= 0 && n > 0) poll(B_SFREE + before, n - 1);
              last = x;
              if (x == 0) ++sc0; else ++sc1;
              tc_fence_after();
              const uint32_t q = q_lo + (SPLIT ? 0 : x) * (L::kTileBytes >> 4);
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks) {
                const uint32_t off = (ks >> 2) * 1024 + (ks & 3) * 2;   // (chunk * 16384 + kstep * 32) / 16
                mma_ss(tm_s0 + (NSB == 2 ? 128 * x : 0), dk_hi | (q + off), dk_hi | (k_lo + off), idesc, ks > 0 ? 1u : 0u);
              }
              mma_commit(&bars[B_SFULL + x]);
            }
            mma_commit(&bars[B_KFREE + kc % NS]);
          }
          mma_commit(&bars[B_QFREE]);
          if (!SPLIT && it.n1 > 0) mma_commit(&bars[B_QFREE + 1]);
        }
      } else {
        // -------------------------------------------------------------- O += P V of group x, in two halves of 64 keys
        const int x = warp - kPvWarp;
        const uint32_t idesc = instr_desc(kTileM, D, 0, 1);   // V is MN-major: d contiguous, keys along K
        const uint32_t v_base = dv_lo + (smem_u32(sm + L::kV) >> 4);
        const uint32_t tm_o = tm_o0 + D * x, tm_p = tm_p0 + 64 * x;
        int vc = 0, pc = 0;
        for (int k = 0;; ++k) {
          const Item it = read_item(k);
          item_read(k);
          if (it.T == 0) break;
          bool first = true;
#pragma unroll 1
          for (int j = 0; j < it.T; ++j, ++vc) {
            wait(B_VFULL + vc % NS, vc / NS);
            if (!takes(it, x, j)) { mbar_arrive(&bars[B_VFREE + vc % NS]); continue; }
            const uint32_t v_lo = v_base + (uint32_t)(vc % NS) * (L::kTileBytes >> 4);
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
              wait(B_P + 2 * h + x, pc);
              tc_fence_after();
#pragma unroll
              for (int q = 0; q < 4; ++q)
                mma_ts(tm_o, tm_p + (4 * h + q) * 8, dv_hi | (v_lo + (4 * h + q) * 128), idesc, (!first || h > 0 || q > 0) ? 1u : 0u);
              mma_commit(&bars[B_PV + 2 * h + x]);
            }
            mma_commit(&bars[B_VFREE + vc % NS]);
            first = false;
            ++pc;
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax + epilogue: a thread per row
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");   // 2 x 128 x 200 + 128 x 104 = 384 x 168
    const int x = warp >> 2, quad = warp & 3;
    const int r = quad * 32 + lane;               // row inside the tile == TMEM lane
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t tm_s = tm_s0 + (NSB == 2 ? 128 * x : 0) + lane_addr, tm_p = tm_p0 + 64 * x + lane_addr;
    const uint32_t tm_o = tm_o0 + D * x + lane_addr;
    unsigned char* stage = sm + L::kOut + warp * 4096;
    const int g_log = 31 - __clz(a.g);
    int n = 0;                                    // key tiles so far
    for (int k = 0;; ++k) {
      const Item it = read_item(k);
      const Place own = place(it, k, x);
      // Threads may see a wait give up at different times.  A SPLIT item has barriers of both groups: they enter it together or not at all.
      const bool go = SPLIT ? named_bar_all(1, 256, it.T > 0) : __all_sync(0xffffffffu, it.T > 0);
      if (lane == 0) item_read(k);
      if (!go) break;
      const int nx = x ? it.n1 : it.n0, rt = x ? it.rt1 : it.rt0, row = rt * kTileM + r;
      const int i_row = min(a.I - 1, row >> g_log);   // rows past the block's end behave like its last input
      // Left padding: a padding pair is masked for every real query.  Among the block's own keys padding is a prefix of
      // positions; among the cached pairs it is whatever kv_ids say (the rows of an unordered cache are in no order).
      const int pad = PAD ? a.left_pad[own.smp] : 0;
      const bool real_row = !PAD || a.pos0 + i_row >= pad;
      const int* ids = a.kv_ids + (size_t)own.unit * a.cap;
      int id4[4];
      auto fetch_ids = [&](int j) {               // of this warp's lanes, for the mask of a cached key tile
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int key = j * kTileN + 32 * c + lane;
          id4[c] = key < a.n_old ? ids[key] : 0x7fffffff;
        }
      };
      const int j_step = SPLIT ? 2 : 1, j_first = SPLIT ? x : 0;
      if (PAD && pad > 0 && j_first < t_old) fetch_ids(j_first);
      float m_used = -INFINITY, l = 0.f;
#pragma unroll 1
      for (int jj = 0, j = j_first; jj < nx; ++jj, j += j_step, ++n) {
        wait(B_SFULL + x, n);
        tc_fence_after();
        // visible columns of this key tile for this row: [0, nvis)
        const int nvis = (j < t_old) ? min(kTileN, a.n_old - j * kTileN)
                                     : max(0, min(kTileN, i_row - (j - t_old) * kTileN + 1));
        uint32_t pm[4] = {0u, 0u, 0u, 0u};        // padding among the columns
        if (PAD && pad > 0) {
          if (j < t_old) {
#pragma unroll
            for (int c = 0; c < 4; ++c) pm[c] = __ballot_sync(0xffffffffu, id4[c] < pad);
            if (j + j_step < t_old) fetch_ids(j + j_step);
          } else {
            const int nlo = max(0, min(kTileN, pad - a.pos0 - (j - t_old) * kTileN));
#pragma unroll
            for (int c = 0; c < 4; ++c) pm[c] = nlo >= 32 * c + 32 ? 0xffffffffu : nlo <= 32 * c ? 0u : (1u << (nlo - 32 * c)) - 1u;
          }
          if (!real_row)
#pragma unroll
            for (int c = 0; c < 4; ++c) pm[c] = 0u;
        }
        // Hidden logits become -inf (probability 0), in tensor memory and in a loop: these tiles are few, and the code of 128
        // selects beside the rest did not fit the instruction cache.
        const uint32_t padded = PAD ? pm[0] | pm[1] | pm[2] | pm[3] : 0u;
        if (!__all_sync(0xffffffffu, nvis >= kTileN && padded == 0u)) {
          const int from = padded != 0u ? 0 : nvis >> 4;
#pragma unroll 1
          for (int cc = __reduce_min_sync(0xffffffffu, from); cc < 8; ++cc) {
            uint32_t raw[16];
            tmem_ld16(tm_s + 16 * cc, raw);
            const uint32_t word = PAD ? (cc < 4 ? (cc < 2 ? pm[0] : pm[1]) : (cc < 6 ? pm[2] : pm[3])) >> (16 * (cc & 1)) : 0u;
            const uint32_t seen = ~word & ((1u << max(0, min(16, nvis - 16 * cc))) - 1u);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) raw[e] = (seen >> e) & 1 ? raw[e] : 0xff800000u;
            tmem_st16(tm_s + 16 * cc, raw);
          }
          tmem_wait_st();
        }
        uint32_t s[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(tm_s + 32 * c, s[c]);
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[B_SFREE + x]);
        // A NaN or +inf among a row's visible logits makes the row NaN, through its maximum (the polynomial takes NaN for its
        // lowest argument).
        float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int e = 0; e < 32; e += 2)
#pragma unroll
          for (int c = 0; c < 4; ++c) m4[c] = max3_nan(m4[c], __uint_as_float(s[c][e]), __uint_as_float(s[c][e + 1]));
        float mx2 = max3_nan(max3_nan(m4[0], m4[1], m4[2]), m4[3], -INFINITY) * a.scale_log2;
        if (mx2 == INFINITY) mx2 = __uint_as_float(0x7fffffffu);
        bool rescale = false;
        float alpha = 1.f;
        if (jj == 0) m_used = mx2;
        else if (!(mx2 <= m_used + kRescaleThreshold)) { alpha = ex2(m_used - mx2); m_used = mx2; rescale = true; }
        if (__any_sync(0xffffffffu, rescale)) {   // (rarely)
          wait(B_PV + 2 + x, n - 1);
          tc_fence_after();
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
        const float neg_m = m_used == -INFINITY ? 0.f : -m_used;   // (no visible key so far, or their logits are -inf)
        float pa0 = 0.f, pa1 = 0.f, pb0 = 0.f, pb1 = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            float x0, x1, p0, p1;
            fma2(x0, x1, __uint_as_float(s[c][2 * e]), __uint_as_float(s[c][2 * e + 1]), a.scale_log2, neg_m);
            if (D == 64 && e % 8 == 7) ex2_poly2_deg5(x0, x1, p0, p1);
            else { p0 = ex2(x0); p1 = ex2(x1); }
            if (e & 1) add2(pb0, pb1, p0, p1);
            else add2(pa0, pa1, p0, p1);
            pk[e] = pack_bf16(p0, p1);
          }
          if (!(c & 1) && n > 0) poll(B_PV + c + x, n - 1);   // the columns' probabilities of the tile before are used up
          tmem_st16(tm_p + 16 * c, pk);
          if (c & 1) {                            // 64 keys may enter P.V
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[B_P + c - 1 + x]);
          }
        }
        l += (pa0 + pb0) + (pa1 + pb1);
      }
      // ---- epilogue: O / l -> bf16 -> 32 rows of this warp in shared memory -> TMA store; log2-sum-exp
      // (the stores of the item before have long since read their rows)
      const int i_warp = rt * qpt + (quad * 32 >> g_log);   // input of the warp's first row
      auto store = [&](int chunk) {               // the staged 64 elements of every row
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (i_warp < a.I) tma_store_5d(&maps.o, stage, chunk * 64, 0, own.kh, i_warp, own.smp);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      };
      auto staged_has_been_read = [&]() {
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
      };
      if (!SPLIT) {
        if (nx > 0) {
          wait(B_PV + 2 + x, n - 1);
          tc_fence_after();
          if (m_used == -INFINITY) l = __uint_as_float(0x7fffffffu);   // every visible logit is -inf
          const float inv = real_row ? __frcp_rn(l) : 0.f;   // a padding query's output row is zero
#pragma unroll 1
          for (int cc = 0; cc < D / 64; ++cc) {
            uint32_t raw[64];
            tmem_ld32(tm_o + cc * 64, *reinterpret_cast<uint32_t(*)[32]>(raw));
            tmem_ld32(tm_o + cc * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(raw + 32));
            tmem_wait_ld();
            staged_has_been_read();
            uint32_t w[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) w[e] = pack_bf16(__uint_as_float(raw[2 * e]) * inv, __uint_as_float(raw[2 * e + 1]) * inv);
#pragma unroll
            for (int p = 0; p < 8; ++p)
              *reinterpret_cast<uint4*>(stage + sw128_offset(lane, p)) = make_uint4(w[4 * p], w[4 * p + 1], w[4 * p + 2], w[4 * p + 3]);
            store(cc);
          }
          if (row < R) a.lse2[(size_t)own.unit * R + row] = real_row ? m_used + log2f(l) : INFINITY;  // +inf: no weights
        }
      } else {
        // the groups exchange a row's (maximum, sum) through their P columns; either finishes half of the row's elements
        if (nx > 0) wait(B_PV + 2 + x, n - 1);
        tc_fence_after();
        tmem_st2(tm_p, __float_as_uint(m_used), __float_as_uint(l));
        staged_has_been_read();
        tmem_wait_st();
        tc_fence_before();
        named_bar_sync(1, 256);
        tc_fence_after();
        uint32_t om, ol;
        tmem_ld2(tm_p0 + 64 * (x ^ 1) + lane_addr, om, ol);
        tmem_wait_ld();
        const float m0 = x == 0 ? m_used : __uint_as_float(om), m1 = x == 0 ? __uint_as_float(om) : m_used;
        const float l0 = x == 0 ? l : __uint_as_float(ol), l1 = x == 0 ? __uint_as_float(ol) : l;
        const float m = max3_nan(m0, m1, -INFINITY);
        // a group that saw no key is left out; one whose weight is too small for fp32 is not, since its sums may be NaN
        const bool out0 = m0 == -INFINITY && m != -INFINITY, out1 = m1 == -INFINITY;
        const float w0 = out0 ? 0.f : ex2(m0 - m), w1 = out1 ? 0.f : ex2(m1 - m);
        const float lt = (out0 ? 0.f : l0 * w0) + (out1 ? 0.f : l1 * w1);
        const float inv = real_row ? 1.f / lt : 0.f;
        const float f0 = w0 * inv, f1 = w1 * inv;
        const int col0 = x * (D / 2);
        unsigned char* half = sm + L::kOut + (D == 128 ? warp : quad) * 4096;   // (at d = 64 a row's two halves meet in one tile)
#pragma unroll 1
        for (int cc = 0; cc < D / 64; ++cc) {
          uint32_t o0[32], o1[32];
          tmem_ld32(tm_o0 + lane_addr + col0 + 32 * cc, o0);
          tmem_ld32(tm_o0 + D + lane_addr + col0 + 32 * cc, o1);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e)   // (a group that is left out may hold anything)
            o0[e] = __float_as_uint((out0 ? 0.f : __uint_as_float(o0[e]) * f0) + (out1 ? 0.f : __uint_as_float(o1[e]) * f1));
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e] = pack_bf16(__uint_as_float(o0[8 * p + 2 * e]), __uint_as_float(o0[8 * p + 2 * e + 1]));
            *reinterpret_cast<uint4*>(half + sw128_offset(lane, (D == 128 ? 4 * cc : 4 * x) + p)) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
        tc_fence_before();
        if (D == 64) fence_async_smem();
        named_bar_sync(1, 256);                   // both outputs have been read: the next item may replace them
        if (D == 128 || x == 0) store(D == 128 ? x : 0);
        if (x == 0 && row < R) a.lse2[(size_t)own.unit * R + row] = real_row ? m + log2f(lt) : INFINITY;
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kQkWarp) tmem_dealloc(tmem, 512);
}
