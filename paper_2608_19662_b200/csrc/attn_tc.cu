// Tensor-core attention for encode and prefill (bf16, head_dim 128, Hq/G in {2,4,8}).
//
// Persistent kernel, one CTA per SM; a work item = (sequence, KV group, pair of
// query tiles).  A query tile is 128 rows = (128 / s) consecutive tokens x the s query heads of
// the group, so every K/V tile is shared by all heads of the group and the
// causal granularity is 128 / s tokens.  The two tiles of a CTA are consecutive
// and share each K/V tile, read once from L2/HBM by TMA.
//
//   warps 0-3    softmax of tile A    warps 4-7  softmax of tile B
//   warp  8      TMA producer         warp  9    tcgen05.mma issuer (+ TMEM alloc)
//   warp  10     scheduler: draws work items from a global counter and publishes them
//                through a two-slot ring in shared memory
//   warp  11     idle (completes the third warpgroup)
//   warps 12-15  epilogue: O of a finished tile goes from tensor memory to HBM
//                while the softmax warps already rotate the next item's Q; in
//                gather mode (route rows read from the resource cache through an
//                index list) the same 128 lanes also fill the route's K/V tiles
// setmaxnreg moves registers from warps 8-15 to the two softmax warpgroups,
// which hold 128 scores per thread.
//
// Tensor memory (512 columns): S_A | S_B | O_A | O_B, 128 fp32 columns each.
// S = Q K^T (both operands in 128B-swizzled shared memory, K-major); the softmax
// warps read S with tcgen05.ld, keep a running maximum with lazy rescaling of O,
// and write P = exp2(.) as bf16 over the first 64 columns of S; O += P V takes P
// from tensor memory and V (MN-major) from shared memory, the first 64 keys as
// soon as their half of P is stored.  While one tile's softmax runs, the tensor
// core works on the other tile.
//
// Key tiles of an item: first the route's packed rows (all visible), then the
// causal rows of the sequence itself up to the tile pair's last token.  The
// query rows are rotated in shared memory after the TMA load (position = pos0 +
// token index) and rounded to bf16, so no rotated copy of Q ever touches HBM.
// Tiles are aligned to the sequence start, never to the batch: a sequence gives
// bit-identical outputs whatever else is in the launch.
#include "tc_common.cuh"

using namespace rc_tc;

namespace {

constexpr int NSTAGE = 2;
constexpr int NTHREADS = 512;
// Registers per thread of the softmax warps and of the other eight; 256 * (softmax + aux) = 65536.  Epilogue
// warps that gather spill in 32 (8 zero-copy turns: 84.0 us with 32, 82.2 with 40); packed rows pay for 40 (one turn
// of 512 tokens: 34.8 us with 40, 34.3 with 32; an encode 1 %).
template <bool MORE_AUX> constexpr int REGS_SOFTMAX = MORE_AUX ? 216 : 224;
template <bool MORE_AUX> constexpr int REGS_AUX = MORE_AUX ? 40 : 32;

constexpr int SM_Q = 0;                              // 2 query tiles
constexpr int SM_K = SM_Q + 2 * TILE_BYTES;          // NSTAGE key tiles
constexpr int SM_V = SM_K + NSTAGE * TILE_BYTES;     // NSTAGE value tiles
constexpr int ROT_BYTES = 16384;                     // cos (and sin) rows of 64 positions, fp32
constexpr int SM_ROT = SM_V + NSTAGE * TILE_BYTES;   // cos | sin of the item's positions
constexpr int SM_BAR = SM_ROT + 2 * ROT_BYTES;       // mbarriers
constexpr int SM_MISC = SM_BAR + 32 * 8;             // tmem base, abort flag
constexpr int SM_ITEM = SM_MISC + 64;                // two published work items
constexpr int SM_INVL = SM_ITEM + 2 * 64;            // 1 / row sum of each query tile's rows, for the epilogue warps
constexpr int SM_TOTAL = SM_INVL + 2 * 128 * 4;
constexpr int SM_ALLOC = SM_TOTAL + 1024;            // slack for 1024-byte alignment

enum { B_QFULL = 0, B_QREADY, B_QEMPTY = B_QREADY + 2, B_KFULL, B_KEMPTY = B_KFULL + NSTAGE, B_VFULL = B_KEMPTY + NSTAGE,
       B_VEMPTY = B_VFULL + NSTAGE, B_SFULL = B_VEMPTY + NSTAGE, B_PREADY = B_SFULL + 2, B_ODONE = B_PREADY + 2,
       B_IFULL = B_ODONE + 2, B_IEMPTY = B_IFULL + 2, B_LREADY = B_IEMPTY + 2, B_ODRAIN = B_LREADY + 2,
       B_PHALF = B_ODRAIN + 2, B_COUNT = B_PHALF + 2 };
static_assert(B_COUNT <= 32, "barrier area");

constexpr uint32_t COL_S = 0, COL_O = 256;           // + 128 * tile

// Bounded wait: see rc_mbar_wait (no location word here).
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  rc_mbar_wait<WAIT_PROBES, 0>(bar, parity, abort_flag, status);
}


enum { IT_NTILES = 0, IT_G, IT_SEQ0, IT_L, IT_TOK0, IT_KVEND, IT_POS0, IT_RA0, IT_LENA, IT_NA, IT_BVALID, IT_BASE_LO,
       IT_BASE_HI, IT_H, IT_WORDS = 16 };

// ---------------------------------------------------------------- kernel --
// Persistent: a scheduler warp draws work indices from a global counter (the
// list is heavy-first inside each sequence, or heavy-first overall when the plan
// sorted it, so the tail of the launch is made of light items) and publishes
// items through a two-slot ring in shared memory.
// The next item's Q load, Q rotation and first K/V tiles overlap the current
// item's last tiles and its epilogue.  Barrier phases run on across items.
template <typename TO, bool ROT_SMEM, bool GATHER>
__global__ void __launch_bounds__(NTHREADS, 1) attn_tc_kernel(const __grid_constant__ CUtensorMap tm_q,
                                                              const __grid_constant__ CUtensorMap tm_ks,
                                                              const __grid_constant__ CUtensorMap tm_vs,
                                                              const __grid_constant__ CUtensorMap tm_kr,
                                                              const __grid_constant__ CUtensorMap tm_vr,
                                                              const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  const int s = p.s, TQ = 128 / s;

  const uint32_t sm = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* sm_gen = smem_raw + (sm - smem_u32(smem_raw));
  const uint32_t bars = sm + SM_BAR;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm_gen + SM_MISC + 4);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm_gen + SM_MISC);
  volatile int* item_ring = reinterpret_cast<volatile int*>(sm_gen + SM_ITEM);
  auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    mbar_init(bar(B_QFULL), 1);
    mbar_init(bar(B_QREADY + 0), 128); mbar_init(bar(B_QREADY + 1), 128);
    mbar_init(bar(B_QEMPTY), 1);
    for (int i = 0; i < NSTAGE; ++i) {   // gather mode: the 128 epilogue lanes and the TMA producer arrive on every stage
      mbar_init(bar(B_KFULL + i), GATHER ? 129 : 1); mbar_init(bar(B_KEMPTY + i), 1);
      mbar_init(bar(B_VFULL + i), GATHER ? 129 : 1); mbar_init(bar(B_VEMPTY + i), 1);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(bar(B_SFULL + x), 1); mbar_init(bar(B_PREADY + x), 128); mbar_init(bar(B_ODONE + x), 1);
      // producer + MMA + 256 softmax + 128 epilogue threads
      mbar_init(bar(B_IFULL + x), 1); mbar_init(bar(B_IEMPTY + x), 386);
      mbar_init(bar(B_LREADY + x), 128); mbar_init(bar(B_ODRAIN + x), 128); mbar_init(bar(B_PHALF + x), 128);
    }
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
  const uint32_t tmem = *tmem_slot;
  // (everything above touches no global memory: it overlaps the end of the kernel before)
  rc_grid_wait();
  rc_grid_launch_next();

  // Item n of this CTA lives in ring slot n & 1; every consumer copies it to
  // registers and then releases the slot.
  auto fetch_item = [&](uint32_t n, Item& it, bool release) {
    const int sl = n & 1u;
    mbar_wait(bar(B_IFULL + sl), (n >> 1) & 1u, abort_flag, p.status);
    const int* r = const_cast<const int*>(item_ring) + sl * IT_WORDS;   // (ordered by the barrier wait above and the arrive below)
    it.n_tiles = r[IT_NTILES]; it.g = r[IT_G]; it.seq0 = r[IT_SEQ0]; it.L = r[IT_L]; it.tok0 = r[IT_TOK0];
    it.kv_end = r[IT_KVEND]; it.pos0 = r[IT_POS0]; it.rA0 = r[IT_RA0]; it.lenA = r[IT_LENA]; it.nA = r[IT_NA];
    it.b_valid = r[IT_BVALID]; it.H = r[IT_H];
    it.base = (int64_t)(((uint64_t)(uint32_t)r[IT_BASE_HI] << 32) | (uint32_t)r[IT_BASE_LO]);
    if (*abort_flag) it.n_tiles = -1;
    if (release) mbar_arrive(bar(B_IEMPTY + sl));
  };

  if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_AUX<GATHER>));
    // ===================== epilogue warps =====================
    // O of a finished query tile leaves tensor memory here, so that the softmax warps can go
    // straight to the next item's Q.  Warp 12 + q reads lanes 32 q .. 32 q + 31.
    const int row = threadIdx.x & 127;
    const uint32_t lane_addr = ((uint32_t)(32 * (warp & 3)) << 16);
    const float* inv_l = reinterpret_cast<const float*>(sm_gen + SM_INVL);
    Item it, nx;
    uint32_t done[2] = {0, 0};
    fetch_item(0, it, true);
    uint32_t kv_n = 0;
    for (uint32_t item_n = 0; it.n_tiles > 0; ++item_n) {
      if (GATHER) {
        // Gather mode: these 128 lanes also fill the route tiles of the item.  Row n of the route is
        // row route_idx[n] of the resource cache: warp w takes rows 32 w .. 32 w + 31 of a tile, one
        // index per lane handed round by shuffles, 16 16-byte asynchronous copies per lane straight
        // to the swizzled positions of a TMA tile (zero-fill past the route's end).  A lane's arrival
        // fires when its copies have landed; the MMA warp puts a proxy fence before the reads.
        const int w = warp & 3, hi = lane >> 4, c = lane & 15;
        uint32_t sw[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) sw[m] = (uint32_t)(((c & 7) ^ ((2 * m + hi) & 7)) << 4);
        for (int i = 0; i < it.n_tiles; ++i) {
          const uint32_t n = kv_n + (uint32_t)i;
          const int st = n % NSTAGE;
          const uint32_t ph = (n / NSTAGE) & 1u;
          const bool route = i < it.nA;
          int idx = -1;
          if (route) {
            const int r = 32 * w + lane, cnt = min(TILE_N, it.lenA - i * TILE_N);
            if (r < cnt) {
              idx = p.route_idx[it.rA0 + i * TILE_N + r];
              if (idx < 0 || idx >= p.pool_tokens) { rc_set_status(p.status, RECACHE_DEV_BAD_SLOT); idx = -1; }
            }
          }
#pragma unroll
          for (int kv = 0; kv < 2; ++kv) {
            const int b_full = kv ? B_VFULL : B_KFULL, b_empty = kv ? B_VEMPTY : B_KEMPTY;
            mbar_wait(bar(b_empty + st), ph ^ 1u, abort_flag, p.status);
            if (route) {
              const uint8_t* src_l = (kv ? p.gather_v : p.gather_k) + (int64_t)it.g * p.pool_tokens * 256 + c * 16;
              const uint32_t dst_l = sm + (kv ? SM_V : SM_K) + st * TILE_BYTES + (c >> 3) * BOX_BYTES + (32 * w + hi) * 128;
#pragma unroll
              for (int kk = 0; kk < 16; ++kk) {
                const int ix = __shfl_sync(0xffffffffu, idx, 2 * kk + hi);
                cp_async16(dst_l + 2 * kk * 128 + sw[kk & 3], src_l + (int64_t)max(ix, 0) * 256, ix >= 0 ? 16u : 0u);
              }
              cp_async_arrive(bar(b_full + st));
            } else {
              mbar_arrive(bar(b_full + st));
            }
          }
        }
        kv_n += (uint32_t)it.n_tiles;
      }
      fetch_item(item_n + 1, nx, true);
      // The stores below and the rotation of the next item's Q go through the same load/store
      // path, and the rotation is the urgent one: a tile's O is written back once the same tile's
      // next Q has been rotated.  (O is not needed back before the next item's first P V, a whole
      // softmax later; tile B's rotation finishes after tile A's, so tile A is not held up by it.)
      // This wait is a matter of priority only, so it is taken only where the rotating warpgroup
      // cannot complete a second phase before it: tile A's warpgroup is active in every item and
      // stops at the end of the next item for this item's O-drained arrival, which comes after the
      // wait.  Tile B's warpgroup rotates Q even in items where its tile is empty and is held back by
      // nothing there, so with an empty tile B in this item or the next (short sequences) it could
      // pass two phases while tile A is being drained here, and a parity wait would then sleep
      // through the phase it wants.
      for (int x = 0; x < 2; ++x) {
        if (nx.n_tiles > 0 && (x == 0 || (it.b_valid && nx.b_valid)))
          mbar_wait(bar(B_QREADY + x), (item_n + 1u) & 1u, abort_flag, p.status);
        if (x == 1 && !it.b_valid) continue;
        mbar_wait(bar(B_LREADY + x), done[x] & 1u, abort_flag, p.status);
        mbar_wait(bar(B_ODONE + x), done[x] & 1u, abort_flag, p.status);
        ++done[x];
        tc_fence_after();
        const float inv = inv_l[x * 128 + row];
        const int t_row = it.tok0 + x * TQ + row / s;
        const bool row_valid = t_row < it.L;
        TO* orow = reinterpret_cast<TO*>(p.out) + ((int64_t)(it.seq0 + t_row) * p.Hq + it.g * s + row % s) * D;
        const uint32_t t_o = tmem + lane_addr + COL_O + 128 * x;
#pragma unroll 1
        for (int ch = 0; ch < 8; ++ch) {
          uint32_t orr[16];
          TMEM_LD16(t_o + 16 * ch, orr);
          tmem_wait_ld();
          if (row_valid) {
            if constexpr (sizeof(TO) == 4) {
#pragma unroll
              for (int c = 0; c < 16; c += 8)
                st_global_v8(reinterpret_cast<float*>(orow) + 16 * ch + c,
                             __float_as_uint(__uint_as_float(orr[c]) * inv), __float_as_uint(__uint_as_float(orr[c + 1]) * inv),
                             __float_as_uint(__uint_as_float(orr[c + 2]) * inv), __float_as_uint(__uint_as_float(orr[c + 3]) * inv),
                             __float_as_uint(__uint_as_float(orr[c + 4]) * inv), __float_as_uint(__uint_as_float(orr[c + 5]) * inv),
                             __float_as_uint(__uint_as_float(orr[c + 6]) * inv), __float_as_uint(__uint_as_float(orr[c + 7]) * inv));
            } else {
              st_global_v8(reinterpret_cast<__nv_bfloat16*>(orow) + 16 * ch,
                           pack2(__uint_as_float(orr[0]) * inv, __uint_as_float(orr[1]) * inv),
                           pack2(__uint_as_float(orr[2]) * inv, __uint_as_float(orr[3]) * inv),
                           pack2(__uint_as_float(orr[4]) * inv, __uint_as_float(orr[5]) * inv),
                           pack2(__uint_as_float(orr[6]) * inv, __uint_as_float(orr[7]) * inv),
                           pack2(__uint_as_float(orr[8]) * inv, __uint_as_float(orr[9]) * inv),
                           pack2(__uint_as_float(orr[10]) * inv, __uint_as_float(orr[11]) * inv),
                           pack2(__uint_as_float(orr[12]) * inv, __uint_as_float(orr[13]) * inv),
                           pack2(__uint_as_float(orr[14]) * inv, __uint_as_float(orr[15]) * inv));
            }
          }
        }
        // the next item's first P V overwrites O, its softmax overwrites 1 / l: both wait for this
        tc_fence_before();
        mbar_arrive(bar(B_ODRAIN + x));
      }
      it = nx;
    }
  } else if (warp >= 8) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_AUX<GATHER>));
  if (warp == 10) {
    // ===================== scheduler =====================
    if (lane == 0) {
      const int total = p.header[0] * p.G;   // (a CTA without work publishes "no more work" at once)
      bool first = true;
      for (uint32_t n = 0;; ++n) {
        const int sl = n & 1u;
        mbar_wait(bar(B_IEMPTY + sl), ((n >> 1) & 1u) ^ 1u, abort_flag, p.status);
        Item it;
        for (;;) {   // CTA c starts with index c; every later index comes from the shared counter
          const int w = first ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(p.header + 1, 1);
          first = false;
          if (w >= total || *abort_flag) { it.n_tiles = -1; break; }
          if (rc_load_item(p, p.header[2] ? p.order[w] : w, it)) break;
        }
        volatile int* r = item_ring + sl * IT_WORDS;
        r[IT_NTILES] = it.n_tiles;
        if (it.n_tiles > 0) {
          r[IT_G] = it.g; r[IT_SEQ0] = it.seq0; r[IT_L] = it.L; r[IT_TOK0] = it.tok0; r[IT_KVEND] = it.kv_end;
          r[IT_POS0] = it.pos0; r[IT_RA0] = it.rA0; r[IT_LENA] = it.lenA; r[IT_NA] = it.nA; r[IT_BVALID] = it.b_valid;
          r[IT_H] = it.H;
          r[IT_BASE_LO] = (int)(uint32_t)(it.base & 0xffffffffll); r[IT_BASE_HI] = (int)(uint32_t)((uint64_t)it.base >> 32);
        }
        mbar_arrive(bar(B_IFULL + sl));
        if (it.n_tiles < 0) break;
      }
    }
    __syncwarp();
  } else if (warp == 8) {
    // ===================== TMA producer =====================
    if (lane == 0) {
      Item it;
      uint32_t kv_n = 0;
      for (uint32_t item_n = 0;; ++item_n) {
        fetch_item(item_n, it, true);
        if (it.n_tiles < 0) break;
        // Q tiles: free once the previous item's last S = Q K^T has completed
        mbar_wait(bar(B_QEMPTY), (item_n & 1u) ^ 1u, abort_flag, p.status);
        uint32_t rot_bytes = 0;
        const int pos_start = it.pos0 + it.tok0;
        if (ROT_SMEM) {
          const int rows = min(2 * TQ, p.max_pos - pos_start);
          if (pos_start >= 0 && rows > 0) rot_bytes = (uint32_t)rows * 256u;
        }
        mbar_expect_tx(bar(B_QFULL), 2 * TILE_BYTES + 2 * rot_bytes);
        for (int x = 0; x < 2; ++x)
          for (int kc = 0; kc < 2; ++kc)
            tma_load_3d(sm + SM_Q + x * TILE_BYTES + kc * BOX_BYTES, &tm_q, bar(B_QFULL), kc * 64, it.g * s,
                        it.seq0 + it.tok0 + x * TQ);
        if (rot_bytes) {   // cos / sin rows of the item's positions (contiguous in the table)
          bulk_load(sm + SM_ROT, p.cos_tab + (int64_t)pos_start * 64, rot_bytes, bar(B_QFULL));
          bulk_load(sm + SM_ROT + ROT_BYTES, p.sin_tab + (int64_t)pos_start * 64, rot_bytes, bar(B_QFULL));
        }
        for (int i = 0; i < it.n_tiles; ++i, ++kv_n) {
          const int st = kv_n % NSTAGE;
          const uint32_t ph = (kv_n / NSTAGE) & 1u;
          const bool route = i < it.nA;
          const int row = route ? it.rA0 + i * TILE_N
                                : (int)((int64_t)it.g * p.self_rows + it.base) + (i - it.nA) * TILE_N;
          // (gather mode: a route tile is filled by the epilogue warps; every stage barrier expects
          // their 128 arrivals plus one from here, whoever brings the data)
          mbar_wait(bar(B_KEMPTY + st), ph ^ 1u, abort_flag, p.status);
          if (GATHER && route) {
            mbar_arrive(bar(B_KFULL + st));
          } else {
            mbar_expect_tx(bar(B_KFULL + st), TILE_BYTES);
            for (int kc = 0; kc < 2; ++kc)
              tma_load_2d(sm + SM_K + st * TILE_BYTES + kc * BOX_BYTES, route ? &tm_kr : &tm_ks, bar(B_KFULL + st), kc * 64, row);
          }
          mbar_wait(bar(B_VEMPTY + st), ph ^ 1u, abort_flag, p.status);
          if (GATHER && route) {
            mbar_arrive(bar(B_VFULL + st));
          } else {
            mbar_expect_tx(bar(B_VFULL + st), TILE_BYTES);
            for (int kc = 0; kc < 2; ++kc)
              tma_load_2d(sm + SM_V + st * TILE_BYTES + kc * BOX_BYTES, route ? &tm_vr : &tm_vs, bar(B_VFULL + st), kc * 64, row);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 9) {
    // ===================== MMA issuer =====================
    // descriptor words: low = (address >> 4) | (LBO >> 4) << 16, high = (SBO >> 4) | version | swizzle
    // The issuing lane is elected once: every MMA and every commit comes from that one thread
    // (a commit tracks the MMAs of the thread that executes it).
    const bool issuer = elect_one();
    const uint64_t d_q = smem_desc(0, 16, 1024) + ((sm + SM_Q) >> 4), d_k = smem_desc(0, 16, 1024) + ((sm + SM_K) >> 4);
    const uint64_t d_v = smem_desc(0, BOX_BYTES, 1024) + ((sm + SM_V) >> 4);
    auto issue_qk = [&](int x, int st) {
      const uint64_t qa = d_q + x * (TILE_BYTES >> 4), ka = d_k + st * (TILE_BYTES >> 4);
      const uint32_t dst = tmem + COL_S + 128 * x;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t off = ((j >> 2) * BOX_BYTES + (j & 3) * 32) >> 4;
        mma_ss(dst, qa + off, ka + off, IDESC_QK, j > 0);
      }
    };
    // K steps k0 .. ksteps-1 of O += P V (16 keys each); a full half (4 steps) is the common case
    auto issue_pv = [&](int x, int st, int k0, int ksteps, bool first) {
      const uint64_t va = d_v + st * (TILE_BYTES >> 4);
      const uint32_t dst = tmem + COL_O + 128 * x, src = tmem + COL_S + 128 * x;
      if (ksteps - k0 == 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          mma_ts(dst, src + 8 * (k0 + j), va + (k0 + j) * (2048 >> 4), IDESC_PV, (!first || j > 0) ? 1u : 0u);
      } else {
#pragma unroll 1
        for (int j = k0; j < ksteps; ++j)
          mma_ts(dst, src + 8 * j, va + j * (2048 >> 4), IDESC_PV, (!first || j > k0) ? 1u : 0u);
      }
    };
    Item it;
    uint32_t kv_n = 0, cnt[2] = {0, 0};   // K/V tiles, tiles per query tile so far
    uint32_t items_x[2] = {0, 0};         // items each query tile has taken part in
    for (uint32_t item_n = 0;; ++item_n) {
      fetch_item(item_n, it, false);
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_IEMPTY + (item_n & 1u)));
      if (it.n_tiles < 0) break;
      const int n_tiles = it.n_tiles, nA = it.nA, lenA = it.lenA, L = it.H + it.L, kv_end = it.kv_end;
      const bool b_valid = it.b_valid != 0;
      // each query tile starts as soon as its own half of Q has been rotated
      mbar_wait(bar(B_QREADY + 0), item_n & 1u, abort_flag, p.status);
      mbar_wait(bar(B_KFULL + kv_n % NSTAGE), (kv_n / NSTAGE) & 1u, abort_flag, p.status);
      if (GATHER) fence_async_smem();   // the tile may have been written by cp.async (generic proxy)
      tc_fence_after();
      const int st0 = kv_n % NSTAGE;
      if (issuer) { issue_qk(0, st0); tc_commit(bar(B_SFULL + 0)); }
      // (waited for even when the second tile is empty: its warps still rewrite that half of Q,
      // and the Q-empty commit below lets the next load overwrite it)
      mbar_wait(bar(B_QREADY + 1), item_n & 1u, abort_flag, p.status);
      tc_fence_after();
      if (issuer) {
        if (b_valid) { issue_qk(1, st0); tc_commit(bar(B_SFULL + 1)); }
        if (n_tiles == 1) tc_commit(bar(B_QEMPTY));
      }
      __syncwarp();
      for (int i = 0; i < n_tiles; ++i) {
        const uint32_t n = kv_n + (uint32_t)i;
        const int st = n % NSTAGE;
        const uint32_t ph = (n / NSTAGE) & 1u;
        // rows of this tile that really belong to the segment; keys the pair can see
        const int seg_rows = i < nA ? lenA - i * TILE_N : L - (i - nA) * TILE_N;
        const int vis_rows = i < nA ? seg_rows : kv_end - (i - nA) * TILE_N;
        const int ksteps = (min(vis_rows, TILE_N) + 15) >> 4;
        mbar_wait(bar(B_VFULL + st), ph, abort_flag, p.status);
        if (GATHER) fence_async_smem();
        if (seg_rows < ksteps * 16) {
          // rows past the segment hold whatever follows it in memory: zero them, 0 * NaN would poison O
          uint8_t* vb = sm_gen + SM_V + st * TILE_BYTES;
          const int n_rows = ksteps * 16 - seg_rows;
          for (int e = lane; e < n_rows * 16; e += 32) {
            const int r = seg_rows + (e >> 4), c = e & 15;
            *reinterpret_cast<uint4*>(vb + (c >> 3) * BOX_BYTES + r * 128 + (c & 7) * 16) = make_uint4(0, 0, 0, 0);
          }
          fence_async_smem();
        }
        __syncwarp();
        const int st1 = (n + 1) % NSTAGE;
        const uint32_t ph1 = ((n + 1) / NSTAGE) & 1u;
        const bool more = i + 1 < n_tiles;
        // P of keys 0..63 arrives first: half of P V runs while the softmax finishes the other half
        mbar_wait(bar(B_PHALF + 0), cnt[0] & 1u, abort_flag, p.status);
        if (i == 0 && items_x[0] > 0) mbar_wait(bar(B_ODRAIN + 0), (items_x[0] - 1u) & 1u, abort_flag, p.status);
        tc_fence_after();
        if (issuer) issue_pv(0, st, 0, min(ksteps, 4), i == 0);
        mbar_wait(bar(B_PREADY + 0), cnt[0]++ & 1u, abort_flag, p.status);
        tc_fence_after();
        if (issuer) { issue_pv(0, st, 4, ksteps, false); if (!more) tc_commit(bar(B_ODONE + 0)); }
        if (more) {
          mbar_wait(bar(B_KFULL + st1), ph1, abort_flag, p.status);
          if (GATHER) fence_async_smem();
          tc_fence_after();
          if (issuer) { issue_qk(0, st1); tc_commit(bar(B_SFULL + 0)); }
        }
        if (b_valid) {
          mbar_wait(bar(B_PHALF + 1), cnt[1] & 1u, abort_flag, p.status);
          if (i == 0 && items_x[1] > 0) mbar_wait(bar(B_ODRAIN + 1), (items_x[1] - 1u) & 1u, abort_flag, p.status);
          tc_fence_after();
          if (issuer) issue_pv(1, st, 0, min(ksteps, 4), i == 0);
          mbar_wait(bar(B_PREADY + 1), cnt[1]++ & 1u, abort_flag, p.status);
          tc_fence_after();
          if (issuer) { issue_pv(1, st, 4, ksteps, false); if (!more) tc_commit(bar(B_ODONE + 1)); }
        }
        if (issuer) {
          if (more) {
            if (b_valid) { issue_qk(1, st1); tc_commit(bar(B_SFULL + 1)); }
            if (i + 2 == n_tiles) tc_commit(bar(B_QEMPTY));   // the item's last S has been issued
          } else {
            tc_commit(bar(B_VEMPTY + st));                    // the item's last V tile (earlier ones: see the softmax side)
          }
        }
        __syncwarp();
      }
      kv_n += (uint32_t)n_tiles;
      ++items_x[0];
      if (b_valid) ++items_x[1];
    }
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX<GATHER>));
    // ===================== softmax warpgroups =====================
    const int x = warp >> 2;                       // tile A or B
    const int row = threadIdx.x & 127;             // row of the tile = TMEM lane
    const uint32_t lane_addr = ((uint32_t)(32 * (warp & 3)) << 16);
    const uint32_t t_s = tmem + lane_addr + COL_S + 128 * x;
    const uint32_t t_o = tmem + lane_addr + COL_O + 128 * x;
    const float c2 = p.scale_log2;
    const uint64_t c2c2 = pair2(c2, c2);
    uint32_t item_n = 0, cnt = 0;                  // items seen; tiles this query tile has gone through
    uint32_t kv_n = 0, done_n = 0;                 // K/V tiles of all items so far; items this query tile took part in

    // Rotates this query tile of the freshly loaded Q in shared memory (swizzled 16-byte chunks;
    // element i pairs with i + 64 in the other box).  A thread takes one (token, chunk) pair at a
    // time and goes through the token's s heads, so that cos / sin are read once per token, not
    // once per row; the 8 lanes of a token cover whole 128-byte rows of Q.
    auto rotate_q = [&](const Item& it, uint32_t n_item) {
      mbar_wait(bar(B_QFULL), n_item & 1u, abort_flag, p.status);
      uint8_t* qt = sm_gen + SM_Q + x * TILE_BYTES;
      for (int u = row; u < TQ * 8; u += 128) {
        const int tok = u >> 3, c = u & 7;
        const int t_eff = min(it.tok0 + x * TQ + tok, it.L - 1);
        const int pos = it.pos0 + t_eff;
        if (pos < 0 || pos >= p.max_pos) rc_set_status(p.status, RECACHE_DEV_BAD_POS);
        const float *cp, *sp;
        if (ROT_SMEM) {   // staged by the producer: row = token index inside the tile pair
          const int ri = min(max(t_eff - it.tok0, 0), 2 * TQ - 1);
          cp = reinterpret_cast<const float*>(sm_gen + SM_ROT + ri * 256) + c * 8;
          sp = reinterpret_cast<const float*>(sm_gen + SM_ROT + ROT_BYTES + ri * 256) + c * 8;
        } else {
          const int pc = min(max(pos, 0), p.max_pos - 1);
          cp = p.cos_tab + (int64_t)pc * 64 + c * 8;
          sp = p.sin_tab + (int64_t)pc * 64 + c * 8;
        }
        // lanes c and c + 4 would hit the same banks: they take the two halves in opposite order
        const int first = (c & 4) ? 4 : 0;
        const float4 ca = *reinterpret_cast<const float4*>(cp + first), cb = *reinterpret_cast<const float4*>(cp + 4 - first);
        const float4 sa = *reinterpret_cast<const float4*>(sp + first), sb = *reinterpret_cast<const float4*>(sp + 4 - first);
        const float4 c0 = first ? cb : ca, c1 = first ? ca : cb, s0 = first ? sb : sa, s1 = first ? sa : sb;
        const float cs[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
        const float sn[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll 2
        for (int h = 0; h < s; ++h) {
          const int r = tok * s + h;
          uint8_t* qb = qt + r * 128 + ((c ^ (r & 7)) << 4);
          rotate_chunk(qb, cs, sn);
        }
      }
      fence_async_smem();
      mbar_arrive(bar(B_QREADY + x));
    };

    Item it, nx;
    fetch_item(0, it, true);
    if (it.n_tiles > 0) rotate_q(it, 0);
    while (it.n_tiles > 0) {
      const bool active = x == 0 || it.b_valid;
      const bool releaser = row == 0 && x == (it.b_valid ? 1 : 0);   // the tile whose S = Q K^T is issued last
      const int t_row = it.tok0 + x * TQ + row / s;     // token (local index)
      const int t_eff = min(t_row, it.L - 1);
      const int n_tiles = it.n_tiles, nA = it.nA, lenA = it.lenA, H = it.H;
      float m_ref = -INFINITY, l_sum = 0.f, l_other = 0.f;   // sums over every second tile, swapped after each (as attn_tile.cu adds them)
      if (active) {
        for (int i = 0; i < n_tiles; ++i, ++cnt) {
          mbar_wait(bar(B_SFULL + x), cnt & 1u, abort_flag, p.status);
          tc_fence_after();
          if (releaser) {
            // S of tile i is complete: so is every earlier MMA, i.e. the last reader of K tile i
            // and of V tile i - 1.  Hand both stages back to the producer.
            mbar_arrive(bar(B_KEMPTY + (kv_n + i) % NSTAGE));
            if (i > 0) mbar_arrive(bar(B_VEMPTY + (kv_n + i - 1) % NSTAGE));
          }
          uint32_t sr[128];
          TMEM_LD32(t_s + 0, sr, 0); TMEM_LD32(t_s + 32, sr, 32); TMEM_LD32(t_s + 64, sr, 64); TMEM_LD32(t_s + 96, sr, 96);
          tmem_wait_ld();
          // keys this row may see in this tile: columns [0, lim)
          const int lim = i < nA ? lenA - i * TILE_N : H + t_eff - (i - nA) * TILE_N + 1;
          if (lim < TILE_N) {
#pragma unroll
            for (int c = 0; c < 128; ++c) if (c >= lim) sr[c] = 0xff800000u;   // -inf
          }
          float mx4[4] = {__uint_as_float(sr[0]), __uint_as_float(sr[1]), __uint_as_float(sr[2]), __uint_as_float(sr[3])};
#pragma unroll
          for (int c = 4; c < 124; c += 8) {     // three-input max: 4 chains, 2 new values per step
#pragma unroll
            for (int u = 0; u < 4; ++u) mx4[u] = fmax3(mx4[u], __uint_as_float(sr[c + 2 * u]), __uint_as_float(sr[c + 2 * u + 1]));
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) mx4[u] = fmaxf(mx4[u], __uint_as_float(sr[124 + u]));
          const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
          const float m_new = fmaxf(m_ref, mx);
          bool need = false;
          if (i == 0) m_ref = m_new;                       // O is overwritten by the first P V
          else need = (m_new - m_ref) * c2 > 8.f;          // lazy: P stays below 2^8 otherwise
          if (__any_sync(0xffffffffu, need)) {
            // the previous P V of this tile was issued before this S, so it is complete as well
            const float f = need ? ex2((m_ref - m_new) * c2) : 1.f;
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              uint32_t orr[32];
              TMEM_LD32(t_o + 32 * ch, orr, 0);
              tmem_wait_ld();
#pragma unroll
              for (int c = 0; c < 32; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * f);
              TMEM_ST32(t_o + 32 * ch, orr, 0);
            }
            tmem_wait_st();
            if (need) { l_sum = __fmul_rn(l_sum, f); l_other = __fmul_rn(l_other, f); m_ref = m_new; }
          }
          const float neg_m = -m_ref * c2;
          uint32_t pr[64];
          const uint64_t neg2 = pair2(neg_m, neg_m);
          uint64_t acc0 = 0, acc1 = 0;
#pragma unroll
          for (int c = 0; c < 64; c += 2) {
            float x0, x1, x2, x3;
            fma2(x0, x1, __uint_as_float(sr[2 * c]), __uint_as_float(sr[2 * c + 1]), c2c2, neg2);
            fma2(x2, x3, __uint_as_float(sr[2 * c + 2]), __uint_as_float(sr[2 * c + 3]), c2c2, neg2);
            const float p0 = ex2(x0), p1 = ex2(x1), p2 = ex2(x2), p3 = ex2(x3);
            add2(acc0, p0, p1);
            add2(acc1, p2, p3);
            pr[c] = pack2(p0, p1);
            pr[c + 1] = pack2(p2, p3);
            if (c == 30) {   // first half of P goes out, and into P V, while the second is computed
              TMEM_ST32(t_s + 0, pr, 0);
              tmem_wait_st();
              tc_fence_before();
              mbar_arrive(bar(B_PHALF + x));
            }
          }
          const float l_new = __fadd_rn(l_sum, sum4(acc0, acc1));
          l_sum = l_other; l_other = l_new;
          TMEM_ST32(t_s + 32, pr, 32);
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(bar(B_PREADY + x));
        }
      }
      // ---- hand the finished tile to the epilogue warps (they wait for its last P V themselves) ----
      if (active) {
        if (done_n > 0) mbar_wait(bar(B_ODRAIN + x), (done_n - 1u) & 1u, abort_flag, p.status);   // 1 / l of the item before was read
        reinterpret_cast<float*>(sm_gen + SM_INVL)[x * 128 + row] = 1.f / (l_sum + l_other);
        mbar_arrive(bar(B_LREADY + x));
        ++done_n;
      }
      kv_n += (uint32_t)n_tiles;
      // ---- next item's Q (its load was issued a tile ago) ----
      fetch_item(item_n + 1, nx, true);
      if (nx.n_tiles > 0) rotate_q(nx, item_n + 1);
      it = nx; ++item_n;
    }
  }
  // ---- teardown: every thread is done with tensor memory before it is freed ----
  if (*abort_flag) rc_timeout_drain();   // a wait ran out: let what is in flight land first
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// ------------------------------------------------------------------ host --
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)ptr;
  }
  return fn;
}

// rows x 128 bf16, row-major; box = 128 rows x 64 columns
bool map_rows(CUtensorMap* m, const void* base, uint64_t rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  if (rows == 0) rows = 1;
  cuuint64_t dims[2] = {128, rows};
  cuuint64_t strides[1] = {256};
  cuuint32_t box[2] = {64, 128};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// q [tokens][Hq][128]; box = (128/s tokens) x (s heads) x 64 columns -> 128 rows ordered (token, head)
bool map_q(CUtensorMap* m, const void* base, uint64_t tokens, int Hq, int s) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {128, (cuuint64_t)Hq, tokens};
  cuuint64_t strides[2] = {256, (cuuint64_t)Hq * 256};
  cuuint32_t box[3] = {64, (cuuint32_t)s, (cuuint32_t)(128 / s)};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int64_t align256(int64_t x) { return (x + 255) & ~(int64_t)255; }

}  // namespace

bool rc_tc_supported(const recache_ctx* ctx) {
  const int s = ctx->desc.n_q_heads / ctx->desc.n_kv_heads;
  return ctx->desc.dtype == RECACHE_BF16 && ctx->desc.head_dim == 128 && (s == 2 || s == 4 || s == 8);
}

static int tc_tok_per_item(const recache_ctx* ctx, int item_tiles) { return item_tiles * 128 / (ctx->desc.n_q_heads / ctx->desc.n_kv_heads); }
static int64_t tc_max_items(const recache_ctx* ctx, int n_seq, int total, int item_tiles) {
  return (int64_t)total / tc_tok_per_item(ctx, item_tiles) + n_seq;
}
// Work items of a sequence up to which its length is taken for what max_len says: whole pairs of tiles in both kernels, so that
// a call is not refused by one of them that the other takes.
static int tc_levels(const recache_ctx* ctx, int max_len, int item_tiles) {
  const int t = tc_tok_per_item(ctx, 2);
  return ((max_len + t - 1) / t + 1) * (2 / item_tiles);
}

static int tc_ctas(const recache_ctx* ctx) { return ctx->sm_count > 0 ? ctx->sm_count : 148; }
// A later turn of at most this many rounds of CTAs, in items of one query tile, may be split (see rc_plan_split).
// Of 61 turns of 3-4 rounds none was more than 1 % faster split than whole by the better of the two kernels; of 391 with
// fewer items 100 are 5-58 % faster split than whole.
constexpr int64_t SPLIT_ROUNDS = 3;
static bool tc_may_split(const recache_ctx* ctx, int64_t max_items) {
  const int64_t n = max_items * ctx->desc.n_kv_heads;
  return n <= SPLIT_ROUNDS * tc_ctas(ctx) && n <= RC_SORT_MAX;
}

// Query tiles of a work item: one (attn_tile.cu), or a pair that shares its K/V tiles (attn_tc_kernel).  The
// results are the same bits.  One is better where the launch has few items a CTA, a pair where it has many (a
// K/V tile is then loaded, and its MMAs are issued, for two), us with one and with a pair:
//   encode, 4 query heads a group: 1 x 500 tokens (128 items) 18.4 / 20.1, 8 x 500 (1000) 44.6 / 45.1, 12 x 500 (1500) 69.6 / 65.3;
//     2 x 1500 (750) 59.1 / 61.5, 3 x 1500 (1125) 89.0 / 85.3
//   first turns: 1 x 512 tokens 32.1 / 40.3, 4 x 1024 (1024 items) 97.1 / 98.9, 16 x 256 (1024) 80.3 / 86.7, 16 x 512 (2048) 157 / 152
// Where a route has room for more than 64 K/V tiles, an item is long, and the pair's fewer loads count for more (the
// room is all the host knows of it; only the time depends on it): 2048 tokens over 64 long tools (512 items) 300 / 290.
// Behind a shared prefix an encode's items are as long as the prefix, which is known here:
//   500 rows, 6 x 1000 tokens, 2 heads a group (792 items) 75.9 / 75.8; 2000 rows, 1 x 1500, 4 heads (376) 77.9 / 92.2,
//   4 x 500 (528) 89.3 / 81.4; 8000 rows, 1 x 500 (128) 71.3 / 118, 2 x 500 (264) 145 / 124, 4 x 500, 2 heads (280) 150 / 127
// A gather's copies are bound by the rate at which a CTA issues them, so it always takes pairs.
// A later turn is split, if at all, in items of one tile (tc_may_split), so up to SPLIT_ROUNDS rounds of CTAs it has one;
// so it has where no request has a second tile to pair (32 x 16 tokens over 4000 rows, 2 heads a group 118 / 141).  Beyond,
// never split, it goes by the room for its keys, 24 K/V tiles an item, up to eight rounds, and takes pairs from there:
//   2 heads, 16 x 256 tokens (640 items) over 300 rows 62.3 / 62.2, over 4000 219 / 189
//   4 heads, 8 x 256 (576) over 300 56.8 / 54.6, over 4000 201 / 179; 16 x 512 (2176) over 300 212 / 196
//   187 turns in a grid and at random: those of 3-8 rounds take 0.98 of the pair's time with up to 24 tiles an item
//   (0.79-1.07), 1.05 with more (0.96-1.16), those of more rounds 1.04 (0.94-1.15)
static int tc_item_tiles(const recache_ctx* ctx, const TcAttnArgs& a) {
  if (a.route_idx) return 2;
  const int64_t G = ctx->desc.n_kv_heads, ctas = tc_ctas(ctx), items = tc_max_items(ctx, a.n_seq, a.total, 1) * G;
  if (a.hist) {
    if (items <= SPLIT_ROUNDS * ctas || a.max_len <= tc_tok_per_item(ctx, 1)) return 1;
    return items <= 8 * ctas && a.route_rows / G + a.self_rows <= (int64_t)24 * TILE_N * a.n_seq ? 1 : 2;
  }
  int rounds;
  if (a.route_cu) rounds = a.route_rows > 64 * TILE_N * G * a.n_seq ? 2 : 8;
  else rounds = a.prefix_len <= 8 * TILE_N ? 6 : a.prefix_len <= 32 * TILE_N ? 3 : 1;
  return items <= rounds * ctas ? 1 : 2;
}

constexpr int64_t PART_ROWS = 2 * 128;       // per CTA: two slots

int64_t rc_tc_workspace_bytes(const recache_ctx* ctx, int n_seq, int total, int max_len) {
  return 256 + align256(tc_max_items(ctx, n_seq, total, 1) * 8) + align256(2 * RC_SORT_MAX * 4);
}
// What a split takes on top, whatever the call's size: cuts, unit prefix, and two partial results per CTA.
int64_t rc_tc_split_bytes(const recache_ctx* ctx) {
  const int64_t n = tc_ctas(ctx);
  return align256((n + 1) * 8) + align256((n + 1) * 16) + align256(RC_SORT_MAX * 4) + align256(n * PART_ROWS * 8) + n * PART_ROWS * D * 4;
}

// Whether a launch is made splittable, which costs the merge launch behind it (2 us) even when the device
// then decides against it.  Only a later turn is: its keys are the history's, thousands for a few new tokens.
// A first turn's result must be the same bits whether its rows are packed or gathered, and both must be free
// to come in buffers of any size, of which the host cannot tell how much is filled.
// Nothing here may depend on capacities, except to leave the merge launch out where rc_plan_split cannot say yes
// whatever they hold: ranges have more than four units, and whole items take, in one round, RC_ITEM_UNITS more than the
// longest has tiles, in more at most 0.8 of its tiles more than a range.
static bool tc_splits(const recache_ctx* ctx, const TcAttnArgs& a, int64_t max_items) {
  if (!a.hist || !tc_may_split(ctx, max_items) || tc_ctas(ctx) < 2) return false;
  if (a.workspace_bytes < rc_tc_workspace_bytes(ctx, a.n_seq, a.total, a.max_len) + rc_tc_split_bytes(ctx)) return false;
  const int64_t most = a.route_rows / TILE_N + a.self_rows / TILE_N + 2;     // tiles of an item that had every row there is
  return most > 4 + RC_MERGE_UNITS;
}

cudaError_t rc_launch_attn_tc(const recache_ctx* ctx, const RopeStoreArgs& rope, const TcAttnArgs& a, cudaStream_t st) {
  const int G = ctx->desc.n_kv_heads, Hq = ctx->desc.n_q_heads, s = Hq / G;
  if (a.total == 0 || a.n_seq == 0) return cudaSuccess;
  const bool gather = a.route_idx != nullptr;
  const int item_tiles = tc_item_tiles(ctx, a);
  const int64_t max_items = tc_max_items(ctx, a.n_seq, a.total, item_tiles);
  uint8_t* ws = (uint8_t*)a.workspace;

  TcMaps m;
  const uint64_t self_total = (uint64_t)G * (uint64_t)a.self_rows;
  // TMA coordinates are 32-bit row indices
  if (self_total + TILE_N > 0x7fffffffull || (uint64_t)a.route_rows + TILE_N > 0x7fffffffull) return cudaErrorInvalidValue;
  if (!map_q(&m.q, a.q, (uint64_t)a.total, Hq, s) || !map_rows(&m.ks, a.k_self, self_total) ||
      !map_rows(&m.vs, a.v_self, self_total))
    return cudaErrorInvalidValue;
  const bool has_route = (a.route_cu != nullptr || a.prefix_len > 0) && a.route_rows > 0 && !gather;
  if (!has_route) { m.kr = m.ks; m.vr = m.vs; }   // unused
  else if (!map_rows(&m.kr, a.k_route, (uint64_t)a.route_rows) || !map_rows(&m.vr, a.v_route, (uint64_t)a.route_rows))
    return cudaErrorInvalidValue;

  TcParams p;
  p.header = (int32_t*)ws; p.items = (int2*)(ws + 256); p.order = (int32_t*)(ws + 256 + align256(max_items * 8));
  const bool may_split = item_tiles == 1 && tc_splits(ctx, a, max_items);
  const int sms = tc_ctas(ctx);
  const unsigned grid = (unsigned)(may_split || max_items * G > sms ? sms : max_items * G);
  p.start = nullptr; p.merge = nullptr; p.unit_cu = nullptr; p.part_o = nullptr; p.part_ml = nullptr; p.n_cta = (int)grid;
  if (may_split) {
    uint8_t* at = ws + rc_tc_workspace_bytes(ctx, a.n_seq, a.total, a.max_len);
    p.start = (int2*)at; at += align256((int64_t)(sms + 1) * 8);
    p.merge = (int4*)at; at += align256((int64_t)(sms + 1) * 16);
    p.unit_cu = (int32_t*)at; at += align256(RC_SORT_MAX * 4);
    p.part_ml = (float2*)at; at += align256(sms * PART_ROWS * 8);
    p.part_o = (float*)at;
  }
  p.cu = a.cu; p.pos0 = a.pos0; p.slot = a.slot; p.route_cu = a.route_cu; p.hist = a.hist;
  p.n_seq = a.n_seq; p.G = G; p.Hq = Hq; p.s = s; p.self_rows = a.self_rows; p.route_rows = a.route_rows;
  p.prefix_len = a.route_cu ? 0 : a.prefix_len;
  p.item_tiles = item_tiles; p.n_levels = tc_levels(ctx, a.max_len, item_tiles); p.max_items = (int)max_items;
  p.status = ctx->status;
  p.out = a.o;
  p.cos_tab = ctx->cos_tab; p.sin_tab = ctx->sin_tab; p.max_pos = ctx->desc.max_pos;
  p.scale_log2 = (float)(1.4426950408889634 / sqrt((double)ctx->desc.head_dim));
  p.gather_k = (const uint8_t*)a.k_cache; p.gather_v = (const uint8_t*)a.v_cache; p.route_idx = a.route_idx;
  p.pool_tokens = a.pool_tokens;
  cudaError_t e = rc_launch_rope_store(ctx, rope, &p, st);   // builds the work list on the side
  if (e != cudaSuccess) return e;
  const bool f32 = a.out_dtype == RECACHE_F32, rot = s >= 4;   // 2 * 128 / s <= 64 positions fit the staging area
  if (item_tiles == 1) return rc_launch_attn_tile(ctx, m, p, f32, may_split, grid, st);
  RcLaunchScope scope(ctx, a.route_cu ? RC_K_PREFILL_ATTN : RC_K_ENCODE_ATTN, st);
  auto launch = [&](auto kernel) { return rc_launch_overlapped(kernel, grid, NTHREADS, SM_ALLOC, st, m.q, m.ks, m.vs, m.kr, m.vr, p); };
  auto pick = [&](auto type) {
    using TO = decltype(type);
    if (gather) return rot ? launch(attn_tc_kernel<TO, true, true>) : launch(attn_tc_kernel<TO, false, true>);
    return rot ? launch(attn_tc_kernel<TO, true, false>) : launch(attn_tc_kernel<TO, false, false>);
  };
  return f32 ? pick(float()) : pick(__nv_bfloat16());
}
