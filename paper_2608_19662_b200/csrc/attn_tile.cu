// Tensor-core attention with ONE query tile to a work item (bf16, head_dim 128, Hq/G in {2,4,8}): encodes, packed
// prefills and later turns of few items a CTA.  (attn_tc.cu takes a pair; rule and figures at tc_item_tiles there.  Between
// two events, which add the launch's start to it, with a pair and with one: encoding one tool 21.1 and 16.9 us, one request's
// turn 25.0 and 19.1, later turns 39 and 33.)
//
// Persistent kernel, one CTA per SM; a work item = (sequence, KV group, query tile).
// A query tile is 128 rows = (128 / s) consecutive tokens x the s query heads of the group, so every K/V
// tile is shared by all heads of the group and the causal granularity is 128 / s tokens.
//
//   warps 0-3    softmax of every second K/V tile    warps 4-7    softmax of the others
//   warp  8      TMA producer         warp  9    issues S = Q K^T (+ tensor memory)
//   warp  10     scheduler: draws work items from a global counter (split launch: walks the CTA's range
//                of the K/V tiles) and publishes them through a two-slot ring in shared memory
//   warp  11     issues O += P V
//   warps 12-15  epilogue: O of a finished item goes from tensor memory to HBM
//   warps 16-19  rotate the next item's query tile in shared memory
//
// Tensor memory (512 columns): O | S0 | S1 | S2, 128 fp32 columns each.  K/V tile n of the CTA (counted on
// through its items) has S buffer n % 3 and softmax warpgroup n % 2.  S = Q K^T (both operands in
// 128B-swizzled shared memory, K-major); the softmax warps read S with tcgen05.ld, keep a running maximum
// with lazy rescaling of O, and write P = exp2(.) as bf16 over the first 64 columns of S; O += P V takes P
// from tensor memory and V (MN-major) from shared memory.
//
// Why one tile: a launch of few items leaves SMs idle or gives them one item, and its time is that item's.  Two
// warpgroups on alternate K/V tiles of the same rows go through it at 1.6k cycles a tile, where the
// two of a pair, each with rows of its own to walk alone, need 3.1k for each of its; half the items' work is in
// twice as many of them, over twice as many SMs.  And nothing stops at an item's end: its Q is double-buffered, loaded and
// rotated an item ahead, and S of the next item's first tiles is computed under this one's last.  The price, a
// K/V tile loaded for one query tile and not for two, is 41 B/clk of the 83 an SM gets from L2.  What bounds it: the
// chain P V of tile n -> Q K^T of tile n + 3 into its buffer -> softmax (4.6k cycles for three tiles); without any softmax a tile
// takes 1.1k (1024 of MMA), the softmax of two warps on a scheduler by themselves 1.12k (1024 of exponentials).
//
// Key tiles of an item: first the route's packed rows (all visible), then the
// causal rows of the sequence itself up to the tile's last token.  The
// query rows are rotated in shared memory after the TMA load (position = pos0 +
// token index) and rounded to bf16, so no rotated copy of Q ever touches HBM.
// Tiles are aligned to the sequence start, never to the batch: a resource, and a first turn,
// gives bit-identical outputs whatever else is in the launch, and the bits of attn_tc.cu: the same tiles in the
// same order, and a row's sum kept as two, over the even and the odd tiles.  (The items of a later turn may
// be split, see rc_plan_split; the cuts follow from the lengths of the whole launch.)
#include "tc_common.cuh"

using namespace rc_tc;

namespace {

constexpr int NTHREADS = 640;
// Registers per thread of the softmax warps and of warps 8-11, 12-15 and 16-19; they may sum up to what the
// launch hands out, 5 x 96.
constexpr int REGS_SOFTMAX = 168, REGS_ISSUE = 40, REGS_EPILOGUE = 56, REGS_ROTATE = 48;
static_assert(2 * REGS_SOFTMAX + REGS_ISSUE + REGS_EPILOGUE + REGS_ROTATE <= 5 * 96, "registers of the launch");

constexpr int NS = 3;                                // S buffers (Q, K and V are double-buffered)
constexpr int SM_Q = 0;                              // query tiles of this item and the next
constexpr int SM_K = SM_Q + 2 * TILE_BYTES;
constexpr int SM_V = SM_K + 2 * TILE_BYTES;
constexpr int SM_REF = SM_V + 2 * TILE_BYTES;        // [row] the row's reference, from one softmax warpgroup to the other
constexpr int SM_L = SM_REF + 128 * 4;               // [warpgroup][row] row sum, factor of the last tile
constexpr int SM_BAR = SM_L + 2 * 128 * 8;           // mbarriers

enum { B_IFULL = 0, B_IEMPTY = B_IFULL + 2, B_QFULL = B_IEMPTY + 2, B_QREADY = B_QFULL + 2, B_KFULL = B_QREADY + 2, B_VFULL = B_KFULL + 2,
       B_SFULL = B_VFULL + 2, B_PREADY = B_SFULL + NS, B_PVDONE = B_PREADY + NS, B_REF = B_PVDONE + NS, B_OFULL = B_REF + 8, B_OEMPTY,
       B_LFULL, B_LEMPTY = B_LFULL + 2, B_COUNT = B_LEMPTY + 2 };

constexpr int IT_WORDS = 16;                         // of a published work item
constexpr int SM_MISC = SM_BAR + B_COUNT * 8;        // tmem base, gave-up word
constexpr int SM_ITEM = (SM_MISC + 8 + 15) / 16 * 16;   // two published work items
constexpr int SM_TOTAL = SM_ITEM + 2 * IT_WORDS * 4;
constexpr int SM_ALLOC = SM_TOTAL + 1024;            // slack for 1024-byte alignment
static_assert(SM_ALLOC <= 227 * 1024, "shared memory of a CTA");

constexpr uint32_t COL_O = 0, COL_S = 128;           // + 128 * buffer

// Bounded wait: see rc_mbar_wait_small.
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, uint32_t gave_up) { rc_mbar_wait_small<WAIT_PROBES>(bar, parity, gave_up); }

// ---------------------------------------------------------------- kernel --
// Barriers, n counting the CTA's K/V tiles and j its items, all of them on through the launch; a phase of each is awaited before the
// one after it can end:
//   SFULL[n % 3]   S of tile n is there, its K stage (n % 2) free.  QREADY[j % 2]: Q of item j rotated.
//   PREADY[n % 3]  P of tile n is stored, O rescaled if it had to be.
//   PVDONE[n % 3]  tile n is in O; its S buffer and its V stage (n % 2) are free.
//   REF[n % 2][w]  the reference after tile n of rows 32 w .. + 31 is in shared memory.
//   LFULL / LEMPTY the row sums of a softmax warpgroup; OFULL / OEMPTY the item's O.
template <typename TO, bool SPLIT>
__global__ void __launch_bounds__(NTHREADS, 1) attn_tile_kernel(const __grid_constant__ CUtensorMap tm_q,
                                                                const __grid_constant__ CUtensorMap tm_ks,
                                                                const __grid_constant__ CUtensorMap tm_vs,
                                                                const __grid_constant__ CUtensorMap tm_kr,
                                                                const __grid_constant__ CUtensorMap tm_vr,
                                                                const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  const int s = p.s, TQ = 128 / s;
  const uint32_t sm = (smem_u32(smem_raw) + 1023u) & ~1023u, bars = sm + SM_BAR;
  uint8_t* smem = smem_raw + (sm - smem_u32(smem_raw));
  volatile int* gave_up = reinterpret_cast<volatile int*>(smem + SM_MISC + 4);
  const uint32_t gave_up_at = sm + SM_MISC + 4;
  auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
  auto wait = [&](int i, uint32_t parity) { mbar_wait(bar(i), parity, gave_up_at); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *gave_up = 0;
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      // producer, two issuers, eight softmax, four epilogue and four rotation warps
      mbar_init(bar(B_IFULL + i), 1); mbar_init(bar(B_IEMPTY + i), 19);
      mbar_init(bar(B_QFULL + i), 1); mbar_init(bar(B_QREADY + i), 4);
      mbar_init(bar(B_KFULL + i), 1); mbar_init(bar(B_VFULL + i), 1);
      mbar_init(bar(B_LFULL + i), 4); mbar_init(bar(B_LEMPTY + i), 4);
    }
#pragma unroll 1
    for (int i = 0; i < NS; ++i) { mbar_init(bar(B_SFULL + i), 1); mbar_init(bar(B_PREADY + i), 4); mbar_init(bar(B_PVDONE + i), 1); }
#pragma unroll 1
    for (int i = 0; i < 8; ++i) mbar_init(bar(B_REF + i), 1);
    mbar_init(bar(B_OFULL), 1); mbar_init(bar(B_OEMPTY), 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8 && lane == 0) {
    prefetch_tmap(&tm_q); prefetch_tmap(&tm_ks); prefetch_tmap(&tm_vs);
    if (p.route_cu || p.prefix_len > 0) { prefetch_tmap(&tm_kr); prefetch_tmap(&tm_vr); }
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm + SM_MISC), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + SM_MISC);
  // (everything above touches no global memory: it overlaps the end of the kernel before)
  rc_grid_wait();
  rc_grid_launch_next();

  // an arrival for the warp, after everything its lanes have done
  auto warp_arrive = [&](int i) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(i));
  };
  // Item j of this CTA lives in ring slot j & 1; every consumer copies what it needs to
  // registers and then releases the slot, a warp at a time (the producer is a single lane).
  auto fetch_item = [&](uint32_t j, Item& it, bool whole_warp) {
    const int sl = j & 1u;
    wait(B_IFULL + sl, (j >> 1) & 1u);
    const int4* r = reinterpret_cast<const int4*>(smem + SM_ITEM + sl * IT_WORDS * 4);   // (ordered by the wait above and the arrival below)
    const int4 a = r[0], b = r[1], c = r[2], d = r[3];
    it.n_tiles = a.x; it.g = a.y; it.seq0 = a.z; it.L = a.w;
    it.tok0 = b.x; it.kv_end = b.y; it.pos0 = b.z; it.rA0 = b.w;
    it.lenA = c.x; it.nA = c.y; it.H = c.z; it.part = SPLIT ? c.w : -1;
    it.base = (int64_t)(((uint64_t)(uint32_t)d.y << 32) | (uint32_t)d.x);
    if (*gave_up) it.n_tiles = -1;
    if (whole_warp) __syncwarp();
    if (!whole_warp || lane == 0) mbar_arrive(bar(B_IEMPTY + sl));
  };

  if (warp >= 16) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_ROTATE));
    // ===================== rotation warps =====================
    // Rotates the freshly loaded query tile in shared memory (swizzled 16-byte chunks; element i pairs with
    // i + 64 in the other box).  A thread takes one (token, chunk) pair at a time and goes through the
    // token's s heads, so that cos / sin are read once per token; the first pair's are read while Q is
    // still on its way.
    const int row = threadIdx.x & 127;
#pragma unroll 1
    for (uint32_t j = 0;; ++j) {
      Item it;
      fetch_item(j, it, true);
      if (it.n_tiles < 0) break;
      uint8_t* qt = smem + SM_Q + (j & 1u) * TILE_BYTES;
      bool landed = false;
#pragma unroll 1
      for (int u = row; u < TQ * 8; u += 128) {
        const int tok = u >> 3, c = u & 7;
        const int pos = it.pos0 + min(it.tok0 + tok, it.L - 1);
        if (pos < 0 || pos >= p.max_pos) rc_set_status(p.status, RECACHE_DEV_BAD_POS);
        const int64_t at = (int64_t)min(max(pos, 0), p.max_pos - 1) * 64 + c * 8;
        const float4 c0 = __ldg(reinterpret_cast<const float4*>(p.cos_tab + at)), c1 = __ldg(reinterpret_cast<const float4*>(p.cos_tab + at) + 1);
        const float4 s0 = __ldg(reinterpret_cast<const float4*>(p.sin_tab + at)), s1 = __ldg(reinterpret_cast<const float4*>(p.sin_tab + at) + 1);
        const float cs[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
        const float sn[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
        if (!landed) { wait(B_QFULL + (j & 1u), (j >> 1) & 1u); landed = true; }
#pragma unroll 1
        for (int h = 0; h < s; ++h) {
          const int r = tok * s + h;
          rotate_chunk(qt + r * 128 + ((c ^ (r & 7)) << 4), cs, sn);
        }
      }
      fence_async_smem();
      warp_arrive(B_QREADY + (j & 1u));
    }
  } else if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_EPILOGUE));
    // ===================== epilogue warps =====================
    // Warp 12 + q reads lanes 32 q .. 32 q + 31 of O.
    const int row = threadIdx.x & 127;
    const uint32_t t_o = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + COL_O;
    const float2* sums = reinterpret_cast<const float2*>(smem + SM_L) + row;
    uint32_t n = 0, had[2] = {0, 0};               // tiles of the items before; items each softmax warpgroup took part in
#pragma unroll 1
    for (uint32_t j = 0;; ++j) {
      Item it;
      fetch_item(j, it, true);
      if (it.n_tiles < 0) break;
      const int last = (n + it.n_tiles - 1) & 1;   // the warpgroup that has the item's last tile
      n += it.n_tiles;
      wait(B_LFULL + last, had[last]++ & 1u);
      const float2 lf = sums[last * 128];
      float l = lf.x;
      if (it.n_tiles > 1) {
        wait(B_LFULL + (last ^ 1), had[last ^ 1]++ & 1u);
        l = __fadd_rn(l, __fmul_rn(sums[(last ^ 1) * 128].x, lf.y));
        warp_arrive(B_LEMPTY + (last ^ 1));
      }
      warp_arrive(B_LEMPTY + last);
      const bool part = SPLIT && it.part >= 0;
      if (part) p.part_ml[(int64_t)it.part * 128 + row].y = l;
      const float inv = 1.f / l;
      const int t_row = it.tok0 + row / s;
      const bool row_valid = t_row < it.L;
      TO* orow = reinterpret_cast<TO*>(p.out) + ((int64_t)(it.seq0 + t_row) * p.Hq + it.g * s + row % s) * D;
      wait(B_OFULL, j & 1u);
      tc_fence_after();
#pragma unroll 1
      for (int ch = 0; ch < 4; ++ch) {
        uint32_t o[32];
        TMEM_LD32(t_o + 32 * ch, o, 0);
        tmem_wait_ld();
        if (ch == 3) {                             // the next item's first P V overwrites O
          tc_fence_before();
          warp_arrive(B_OEMPTY);
        }
        if (part) {
          float* prow = p.part_o + ((int64_t)it.part * 128 + row) * D + 32 * ch;
#pragma unroll
          for (int c = 0; c < 32; c += 8) st_global_v8(prow + c, o[c], o[c + 1], o[c + 2], o[c + 3], o[c + 4], o[c + 5], o[c + 6], o[c + 7]);
        } else if (row_valid) {
#pragma unroll
          for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * inv);
          if constexpr (sizeof(TO) == 4) {
            float* at = reinterpret_cast<float*>(orow) + 32 * ch;
#pragma unroll
            for (int c = 0; c < 32; c += 8) st_global_v8(at + c, o[c], o[c + 1], o[c + 2], o[c + 3], o[c + 4], o[c + 5], o[c + 6], o[c + 7]);
          } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) o[c] = pack2(__uint_as_float(o[2 * c]), __uint_as_float(o[2 * c + 1]));
            __nv_bfloat16* at = reinterpret_cast<__nv_bfloat16*>(orow) + 32 * ch;
#pragma unroll
            for (int c = 0; c < 16; c += 8) st_global_v8(at + 2 * c, o[c], o[c + 1], o[c + 2], o[c + 3], o[c + 4], o[c + 5], o[c + 6], o[c + 7]);
          }
        }
      }
    }
  } else if (warp >= 8) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_ISSUE));
  if (warp == 10) {
    // ===================== scheduler =====================
    if (lane == 0) {
      const int total = p.header[0] * p.G;   // (a CTA without work publishes "no more work" at once)
      bool first = true;
      const int n_split = SPLIT ? p.header[3] : 0;
      int2 cur = make_int2(0, 0), end = make_int2(0, 0);
      if ((int)blockIdx.x < n_split) { cur = p.start[blockIdx.x]; end = p.start[blockIdx.x + 1]; }
#pragma unroll 1
      for (uint32_t j = 0;; ++j) {
        const int sl = j & 1u;
        wait(B_IEMPTY + sl, ((j >> 1) & 1u) ^ 1u);
        Item it = {};
        it.part = -1;
#pragma unroll 1
        for (; n_split > 0;) {   // the CTA's range of the K/V tiles, one item after the other
          if (cur.x > end.x || (cur.x == end.x && cur.y >= end.y) || *gave_up) { it.n_tiles = -1; break; }
          const int w = cur.x, t0 = cur.y;
          cur = make_int2(w + 1, 0);
          if (!rc_load_item(p, w, it)) continue;
          const int t1 = w == end.x ? min(end.y, it.n_tiles) : it.n_tiles;
          if (t0 > 0 || t1 < it.n_tiles) it.part = 2 * (int)blockIdx.x + (t0 > 0 ? 0 : 1);
          else it.part = -1;
          // (counted from the part's first tile, everything below is the same as for a whole item)
          it.n_tiles = t1 - t0; it.nA -= t0; it.rA0 += t0 * TILE_N; it.lenA -= t0 * TILE_N;
          break;
        }
#pragma unroll 1
        for (; n_split == 0;) {   // CTA c starts with index c; every later index comes from the shared counter
          const int w = first ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(p.header + 1, 1);
          first = false;
          if (w >= total || *gave_up) { it.n_tiles = -1; break; }
          if (rc_load_item(p, p.header[2] ? p.order[w] : w, it)) break;
        }
        int4* r = reinterpret_cast<int4*>(smem + SM_ITEM + sl * IT_WORDS * 4);
        r[0] = make_int4(it.n_tiles, it.g, it.seq0, it.L);
        r[1] = make_int4(it.tok0, it.kv_end, it.pos0, it.rA0);
        r[2] = make_int4(it.lenA, it.nA, it.H, it.part);
        r[3] = make_int4((int)(uint32_t)(it.base & 0xffffffffll), (int)(uint32_t)((uint64_t)it.base >> 32), 0, 0);
        mbar_arrive(bar(B_IFULL + sl));
        if (it.n_tiles < 0) break;
      }
    }
    __syncwarp();
  } else if (warp == 8) {
    // ===================== TMA producer =====================
    if (lane == 0) {
      auto load_q = [&](const Item& it, uint32_t j) {
        mbar_expect_tx(bar(B_QFULL + (j & 1u)), TILE_BYTES);
        for (int kc = 0; kc < 2; ++kc)
          tma_load_3d(sm + SM_Q + (j & 1u) * TILE_BYTES + kc * BOX_BYTES, &tm_q, bar(B_QFULL + (j & 1u)), kc * 64, it.g * s, it.seq0 + it.tok0);
      };
      auto load = [&](uint32_t at, const CUtensorMap* map, int full, int row) {
        mbar_expect_tx(bar(full), TILE_BYTES);
        tma_load_2d(at, map, bar(full), 0, row);
        tma_load_2d(at + BOX_BYTES, map, bar(full), 64, row);
      };
      // V of a tile follows K of the next one, which is wanted first; v_route, v_row: the V to be loaded
      bool v_route = false;
      int v_row = 0;
      uint32_t n = 0, b = 0, ph = 0;               // tile, its S buffer, phase of that
      auto load_v = [&]() {                        // of tile n - 1, where that of tile n - 3 was
        if (n >= 3) wait(B_PVDONE + b, ph ^ 1u);
        const uint32_t st = (n - 1) & 1u;
        load(sm + SM_V + st * TILE_BYTES, v_route ? &tm_vr : &tm_vs, B_VFULL + st, v_row);
      };
      Item it, nx;
      fetch_item(0, it, false);
      if (it.n_tiles > 0) load_q(it, 0);
#pragma unroll 1
      for (uint32_t j = 0; it.n_tiles > 0; ++j) {
        // two steps at least: the next item's Q is loaded in the second, when S of the item before this one, whose
        // Q makes room for it, is complete
#pragma unroll 1
        for (int i = 0; i < max(it.n_tiles, 2); ++i) {
          const uint32_t b2 = b == NS - 1 ? 0 : b + 1, ph2 = b == NS - 1 ? ph : ph ^ 1u;   // of tile n - 2
          if (n >= 2) wait(B_SFULL + b2, ph2);
          const bool route = i < it.nA, tile = i < it.n_tiles;
          const int row = route ? it.rA0 + i * TILE_N
                                : (int)((int64_t)it.g * p.self_rows + it.base) + (i - it.nA) * TILE_N;
          if (tile) load(sm + SM_K + (n & 1u) * TILE_BYTES, route ? &tm_kr : &tm_ks, B_KFULL + (n & 1u), row);
          if (i == 1) {
            fetch_item(j + 1, nx, false);
            if (nx.n_tiles > 0) load_q(nx, j + 1);
          }
          if (!tile) break;
          if (n > 0) load_v();
          v_route = route; v_row = row;
          ++n;
          if (++b == NS) { b = 0; ph ^= 1u; }
        }
        it = nx;
      }
      if (n > 0) load_v();
    }
    __syncwarp();
  } else if (warp == 9) {
    // ===================== S = Q K^T =====================
    // The issuing lane is elected once: every MMA and every commit comes from that one thread
    // (a commit tracks the MMAs of the thread that executes it).
    const bool issuer = elect_one();
    const uint64_t d_q = smem_desc(0, 16, 1024) + ((sm + SM_Q) >> 4), d_k = smem_desc(0, 16, 1024) + ((sm + SM_K) >> 4);
    uint32_t n = 0, b = 0, ph = 0;
#pragma unroll 1
    for (uint32_t j = 0;; ++j) {
      Item it;
      fetch_item(j, it, true);
      if (it.n_tiles < 0) break;
      const int n_tiles = it.n_tiles, n_route = it.nA, len_route = it.lenA, kv_end = it.kv_end;
      const uint64_t qa = d_q + (j & 1u) * (TILE_BYTES >> 4);
      wait(B_QREADY + (j & 1u), (j >> 1) & 1u);
#pragma unroll 1
      for (int i = 0; i < n_tiles; ++i, ++n) {
        // keys that some row sees: at most 64 (the last tile of the route, or the causal one) are half a tile's work
        const uint32_t idesc = (i < n_route ? len_route - i * TILE_N : kv_end - (i - n_route) * TILE_N) > 64 ? IDESC_QK : IDESC_QK64;
        wait(B_KFULL + (n & 1u), (n >> 1) & 1u);
        wait(B_PVDONE + b, ph ^ 1u);
        tc_fence_after();
        if (issuer) {
          const uint64_t ka = d_k + (n & 1u) * (TILE_BYTES >> 4);
          const uint32_t dst = tmem + COL_S + 128 * b;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t off = ((k >> 2) * BOX_BYTES + (k & 3) * 32) >> 4;
            mma_ss(dst, qa + off, ka + off, idesc, k > 0);
          }
          tc_commit(bar(B_SFULL + b));
        }
        __syncwarp();
        if (++b == NS) { b = 0; ph ^= 1u; }
      }
    }
  } else {
    // ===================== O += P V =====================
    const bool issuer = elect_one();
    const uint64_t d_v = smem_desc(0, BOX_BYTES, 1024) + ((sm + SM_V) >> 4);
    uint32_t n = 0, b = 0, ph = 0;
#pragma unroll 1
    for (uint32_t j = 0;; ++j) {
      Item it;
      fetch_item(j, it, true);
      if (it.n_tiles < 0) break;
      const int n_tiles = it.n_tiles, nA = it.nA, lenA = it.lenA, L = it.H + it.L, kv_end = it.kv_end;
#pragma unroll 1
      for (int i = 0; i < n_tiles; ++i, ++n) {
        // rows of this tile that really belong to the segment; keys the query tile can see
        const int seg_rows = i < nA ? lenA - i * TILE_N : L - (i - nA) * TILE_N;
        const int vis_rows = i < nA ? seg_rows : kv_end - (i - nA) * TILE_N;
        const int ksteps = (min(vis_rows, TILE_N) + 15) >> 4;
        wait(B_VFULL + (n & 1u), (n >> 1) & 1u);
        if (seg_rows < ksteps * 16) {
          // rows past the segment hold whatever follows it in memory: zero them, 0 * NaN would poison O
          uint8_t* vb = smem + SM_V + (n & 1u) * TILE_BYTES;
          const int n_rows = ksteps * 16 - seg_rows;
#pragma unroll 1
          for (int e = lane; e < n_rows * 16; e += 32) {
            const int r = seg_rows + (e >> 4), c = e & 15;
            *reinterpret_cast<uint4*>(vb + (c >> 3) * BOX_BYTES + r * 128 + (c & 7) * 16) = make_uint4(0, 0, 0, 0);
          }
          fence_async_smem();
        }
        __syncwarp();
        if (i == 0) wait(B_OEMPTY, (j & 1u) ^ 1u);
        wait(B_PREADY + b, ph);
        tc_fence_after();
        if (issuer) {
          const uint64_t va = d_v + (n & 1u) * (TILE_BYTES >> 4);
          const uint32_t dst = tmem + COL_O, src = tmem + COL_S + 128 * b;
          // 16 keys each
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (k < ksteps) mma_ts(dst, src + 8 * k, va + k * (2048 >> 4), IDESC_PV, k > 0 ? 1u : (uint32_t)(i > 0));
          tc_commit(bar(B_PVDONE + b));
          if (i + 1 == n_tiles) tc_commit(bar(B_OFULL));
        }
        __syncwarp();
        if (++b == NS) { b = 0; ph ^= 1u; }
      }
    }
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX));
    // ===================== softmax warpgroups =====================
    const uint32_t x = warp >> 2, w = warp & 3;    // warpgroup: every tile n with n % 2 == x; rows 32 w .. + 31
    const int row = threadIdx.x & 127;             // row of the query tile = TMEM lane
    const uint32_t t_row0 = tmem + ((32u * w) << 16);
    const float c2 = p.scale_log2;
    const uint64_t c2c2 = pair2(c2, c2);
    volatile float* ref = reinterpret_cast<volatile float*>(smem + SM_REF) + row;
    uint32_t n = 0, had = 0;                       // tile; items this warpgroup took part in
#pragma unroll 1
    for (uint32_t j = 0;; ++j) {
      Item it;
      fetch_item(j, it, true);
      if (it.n_tiles < 0) break;
      const int n_tiles = it.n_tiles;
      // keys that the row sees, and that any row sees, in tile i: these less 128 i
      const int nA = it.nA, end_route = it.lenA;
      const int end_row = it.H + min(it.tok0 + row / s, it.L - 1) + 1 + nA * TILE_N, end_any = it.kv_end + nA * TILE_N;
      float m_ref = 0.f, l_sum = 0.f, f_last = 1.f;
      int i = (n ^ x) & 1u;
      const bool part_of = i < n_tiles;
      n += i;
#pragma unroll 1
      for (; i < n_tiles; i += 2, n += 2) {
        const uint32_t round = n / 3u, b = n - 3u * round;
        const uint32_t t_s = t_row0 + COL_S + 128 * b;
        const int lim = (i < nA ? end_route : end_row) - i * TILE_N;           // this row sees columns [0, lim)
        const bool upper = (i < nA ? end_route : end_any) - i * TILE_N > 64;   // some row sees one of the upper 64
        wait(B_SFULL + b, round & 1u);
        tc_fence_after();
        const int lim_warp = __reduce_min_sync(0xffffffffu, lim);
        if (lim_warp < TILE_N) {                   // masked where it lies, in a small loop
#pragma unroll 1
          for (int ch = max(lim_warp, 0) & ~15; ch < (upper ? 128 : 64); ch += 16) {
            uint32_t o[16];
            TMEM_LD16(t_s + ch, o);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 16; ++c) if (c >= lim - ch) o[c] = 0xff800000u;   // -inf
            TMEM_ST16(t_s + ch, o);
          }
          tmem_wait_st();
        }
        uint32_t sr[128];
        TMEM_LD32(t_s + 0, sr, 0); TMEM_LD32(t_s + 32, sr, 32);
        if (upper) { TMEM_LD32(t_s + 64, sr, 64); TMEM_LD32(t_s + 96, sr, 96); }
        tmem_wait_ld();
        float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};   // three-input max: 4 chains, 2 new values per step
#pragma unroll
        for (int c = 0; c < 64; c += 8) {
#pragma unroll
          for (int u = 0; u < 4; ++u) m[u] = fmax3(m[u], __uint_as_float(sr[c + 2 * u]), __uint_as_float(sr[c + 2 * u + 1]));
        }
        if (upper) {
#pragma unroll
          for (int c = 64; c < 128; c += 8) {
#pragma unroll
            for (int u = 0; u < 4; ++u) m[u] = fmax3(m[u], __uint_as_float(sr[c + 2 * u]), __uint_as_float(sr[c + 2 * u + 1]));
          }
        }
        const float mx = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
        // The reference after the tile before comes from the other warpgroup (the warp of the same rows).  Awaited for
        // an item's first tile too, so that neither group can pass the other by two tiles.
        if (n > 0) wait(B_REF + 4 * (x ^ 1u) + w, ((n - 1) >> 1) & 1u);
        // The reference moves only when a maximum leaves it behind by 2^8.
        const float m_prev = i > 0 ? *ref : mx, m_new = fmaxf(m_prev, mx);
        const bool need = (m_new - m_prev) * c2 > 8.f;
        if (i > 1 && m_ref != m_prev) l_sum = __fmul_rn(l_sum, ex2((m_ref - m_prev) * c2));
        m_ref = need ? m_new : m_prev;
        *ref = m_ref;
        f_last = 1.f;
        if (__any_sync(0xffffffffu, need)) {
          // O holds the tiles before this one once the last of them is in it; no later one can be
          const uint32_t before = (n - 1) / 3u;
          wait(B_PVDONE + (n - 1) - 3u * before, before & 1u);
          tc_fence_after();
          f_last = need ? ex2((m_prev - m_new) * c2) : 1.f;
#pragma unroll 1
          for (int ch = 0; ch < 128; ch += 16) {
            uint32_t o[16];
            TMEM_LD16(t_row0 + COL_O + ch, o);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 16; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * f_last);
            TMEM_ST16(t_row0 + COL_O + ch, o);
          }
          l_sum = __fmul_rn(l_sum, f_last);
        }
        const float neg_m = -m_ref * c2;
        const uint64_t neg2 = pair2(neg_m, neg_m);
        uint64_t acc0 = 0, acc1 = 0;
        auto exponents = [&](int q) {              // of 32 keys
          uint32_t pr[16];
#pragma unroll
          for (int c = 0; c < 16; c += 2) {
            const int at = 32 * q + 2 * c;
            float x0, x1, x2, x3;
            fma2(x0, x1, __uint_as_float(sr[at]), __uint_as_float(sr[at + 1]), c2c2, neg2);
            fma2(x2, x3, __uint_as_float(sr[at + 2]), __uint_as_float(sr[at + 3]), c2c2, neg2);
            const float p0 = ex2(x0), p1 = ex2(x1), p2 = ex2(x2), p3 = ex2(x3);
            add2(acc0, p0, p1);
            add2(acc1, p2, p3);
            pr[c] = pack2(p0, p1);
            pr[c + 1] = pack2(p2, p3);
          }
          TMEM_ST16(t_s + 16 * q, pr);
        };
        exponents(0); exponents(1);
        if (upper) exponents(2);
        warp_arrive(B_REF + 4 * x + w);
        if (upper) exponents(3);
        l_sum = __fadd_rn(l_sum, sum4(acc0, acc1));
        tmem_wait_st();
        tc_fence_before();
        warp_arrive(B_PREADY + b);
      }
      if (part_of) {
        wait(B_LEMPTY + x, (had++ & 1u) ^ 1u);
        reinterpret_cast<float2*>(smem + SM_L)[x * 128 + row] = make_float2(l_sum, f_last);
        if (SPLIT && it.part >= 0 && i == n_tiles + 1) p.part_ml[(int64_t)it.part * 128 + row].x = m_ref * c2;
        warp_arrive(B_LFULL + x);
      }
      n += n_tiles - i;                            // (i is one or none past the last tile)
    }
  }
  // ---- teardown: every thread is done with tensor memory before it is freed ----
  if (*gave_up) {                                  // a wait ran out: let what is in flight land first
    rc_set_status(p.status, RECACHE_DEV_TIMEOUT);
    rc_timeout_drain();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// Merges the parts of the items that a split launch cut: block (c - 1, q) looks at cut c and, if it is
// the first one inside its item, combines rows 64 q .. + 63 of the item's 128, a warp eight of them with
// the first two parts' loads all in flight, a lane four columns.  The parts are in slot 2a + 1 of the CTA
// a before the cut and slots 2j of those after it.  Bound by what an SM can read from L2: a whole item
// (256-512 KB) to a block took 16 us where this takes 8; merging inside the attention launch, by the
// last CTA of an item to end, 37 us.
constexpr int MERGE_THREADS = 256, MERGE_BATCH = 8, MERGE_SPLIT = 2;
static_assert(MERGE_SPLIT * MERGE_BATCH * MERGE_THREADS / 32 == 128, "rows of a query tile");
template <typename TO>
__global__ void __launch_bounds__(MERGE_THREADS) attn_merge_kernel(const __grid_constant__ TcParams p) {
  rc_grid_wait();
  rc_grid_launch_next();
  const int c = blockIdx.x + 1;
  const int n = p.header[3];
  const int4 m = p.merge[c];                             // (c < grid: there, if not written, in any case)
  if (c >= n || m.x == 0) return;
  const int last = c + m.x - 2, rows = m.z, lane = threadIdx.x & 31;
  const int r0 = (128 / MERGE_SPLIT) * blockIdx.y + MERGE_BATCH * (threadIdx.x >> 5);
  if (r0 < rows) {
    float2 ml[2][MERGE_BATCH];
    float4 v[2][MERGE_BATCH];
    auto load = [&](int h, int j) {
      const int64_t at = (int64_t)(j == c - 1 ? 2 * j + 1 : 2 * j) * 128 + r0;
#pragma unroll
      for (int k = 0; k < MERGE_BATCH; ++k) {
        ml[h][k] = p.part_ml[at + k];
        v[h][k] = *(reinterpret_cast<const float4*>(p.part_o + (at + k) * D) + lane);
      }
    };
    auto add = [&]() {                                   // part 1 into part 0
#pragma unroll
      for (int k = 0; k < MERGE_BATCH; ++k) {
        const float m = fmaxf(ml[0][k].x, ml[1][k].x), f0 = ex2(ml[0][k].x - m), f1 = ex2(ml[1][k].x - m);
        ml[0][k] = make_float2(m, ml[0][k].y * f0 + ml[1][k].y * f1);
        v[0][k].x = v[0][k].x * f0 + v[1][k].x * f1; v[0][k].y = v[0][k].y * f0 + v[1][k].y * f1;
        v[0][k].z = v[0][k].z * f0 + v[1][k].z * f1; v[0][k].w = v[0][k].w * f0 + v[1][k].w * f1;
      }
    };
    load(0, c - 1);
    for (int j = c; j <= last; ++j) { load(1, j); add(); }
#pragma unroll
    for (int k = 0; k < MERGE_BATCH; ++k) {
      const int r = r0 + k;                              // 128 rows are TQ tokens of s heads
      if (r >= rows) break;
      const float inv = 1.f / ml[0][k].y;
      TO* o = reinterpret_cast<TO*>(p.out) + ((int64_t)(m.y + r / p.s) * p.Hq + m.w * p.s + r % p.s) * D + 4 * lane;
      if constexpr (sizeof(TO) == 4) *reinterpret_cast<float4*>(o) = make_float4(v[0][k].x * inv, v[0][k].y * inv, v[0][k].z * inv, v[0][k].w * inv);
      else *reinterpret_cast<uint2*>(o) = make_uint2(pack2(v[0][k].x * inv, v[0][k].y * inv), pack2(v[0][k].z * inv, v[0][k].w * inv));
    }
  }
}

}  // namespace

cudaError_t rc_launch_attn_tile(const recache_ctx* ctx, const TcMaps& m, const TcParams& p, bool f32, bool split, unsigned grid, cudaStream_t st) {
  cudaError_t e;
  {
    RcLaunchScope scope(ctx, p.route_cu ? RC_K_PREFILL_ATTN : RC_K_ENCODE_ATTN, st);
    auto launch = [&](auto kernel) { return rc_launch_overlapped(kernel, grid, NTHREADS, SM_ALLOC, st, m.q, m.ks, m.vs, m.kr, m.vr, p); };
    if (split) e = f32 ? launch(attn_tile_kernel<float, true>) : launch(attn_tile_kernel<__nv_bfloat16, true>);
    else e = f32 ? launch(attn_tile_kernel<float, false>) : launch(attn_tile_kernel<__nv_bfloat16, false>);
  }
  if (e != cudaSuccess || !split) return e;
  RcLaunchScope scope(ctx, RC_K_PREFILL_MERGE, st);
  return f32 ? rc_launch_overlapped(attn_merge_kernel<float>, dim3(grid - 1, MERGE_SPLIT), MERGE_THREADS, 0, st, p)
             : rc_launch_overlapped(attn_merge_kernel<__nv_bfloat16>, dim3(grid - 1, MERGE_SPLIT), MERGE_THREADS, 0, st, p);
}
