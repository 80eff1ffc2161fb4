// Routed split-KV decode for bf16, head_dim 128, 64-token pages: memory-bound.
//
// Persistent kernel, one CTA per SM.  The pages of all items (item = sequence x KV group; its
// resource pages first, then its history pages) form one list, and CTA c of n takes pages
// T c / n .. T (c+1) / n - 1 of the T there are, across item boundaries: every CTA streams the same
// number of bytes whatever the lengths are.  (The list is never stored: each CTA sums the items'
// page counts itself, 512 items in about half a microsecond.  A fixed number of splits per item
// instead made the launch as long as the longest histories' units: 16 sequences with 300 .. 4000
// history rows took 70 us for 203 MB that way and take 46 us now; 64 equal ones 128 us and 116 us
// for 727 MB, 6.3 TB/s.)  Where there are few items, each gets CTAs of its own instead, as long as the
// longest item's share then costs no more than a second beginning: a CTA whose range crosses into
// another item takes 2-3 us longer, as much as three pages (one sequence, 430 pages: all but 7 of the
// CTAs had ended after 3.5 us, those after 6.8).  Inside a CTA
//   warp 3     : TMA producer.  Walks the CTA's pages in order and keeps a ring
//                of NSTAGE (K page + V page) buffers full; it runs ahead across
//                item boundaries, so the HBM stream never drains.
//   warps 0-2  : consumers.  The page at ring position n belongs to warp n % 3
//                and stage n % 6, so a stage is always consumed by the same warp
//                and that warp sees every phase of its stages' barriers in
//                order (a parity wait is only valid one phase ahead).  The s
//                query heads of the group are the first s rows of a 16-row
//                mma.sync tile, so each K/V byte is read once for all heads.
//                Scores: m16n8k16 over ldmatrix fragments of the swizzled K page;
//                online softmax in registers (quad shuffles); O += P V with
//                transposed ldmatrix fragments of the V page.
// The current token's key and value (k_new / v_new) are appended by the warp that consumes the
// item's last history page: into the page in HBM, and into the copy in shared memory, which was
// loaded before the row existed.  (With many items to a CTA by a launch of its own, see the launch.)
// The consumer warps' partial (max, sum, O) are merged through shared memory.  An item that lies
// inside one CTA's range is written out there; the parts of one that spans several go to the
// workspace (at most two per CTA: one for an item that began in an earlier CTA, one for an item
// that goes on in a later one) and a second small kernel merges them.
// Every K/V byte crosses HBM once; the roofline is bytes / HBM bandwidth.
#include <cuda.h>

#include <atomic>
#include <type_traits>

#include "common.cuh"

namespace {

constexpr int D = 128;
constexpr int PT = 64;                 // tokens per page
constexpr int NSTAGE = 6;
constexpr int PAGE_BYTES = PT * D * 2; // 16 KB
constexpr int BOX_BYTES = 8192;        // [64 tokens][64 bf16], 128-byte swizzle
constexpr int STAGE_BYTES = 2 * PAGE_BYTES;
// Gather variant: the resource rows of a chunk come straight from the cache with 16-byte cp.async
// copies (half a warp per 256-byte row) written at the swizzled positions a TMA page load would use,
// so the consumers see one layout.  Four producer warps share a chunk (16 rows each): one warp alone
// cannot issue the 2048 copies of a chunk fast enough.  (TMA's four-row gather, 64 instructions a
// chunk from one warp, is slower still: 89 us against 46 us for 16 sequences with 203 MB to read.)  A full barrier then
// takes 128 arrivals: every producer lane's copies (gathered chunk), or the expect-tx arrival plus 127
// plain ones (TMA page).
constexpr int NCW = 3;                 // consumer warps; NSTAGE % NCW == 0
constexpr int NPW_GATHER = 4;          // producer warps of the gather variant (the paged variant has one)
static_assert(NSTAGE % NCW == 0, "a stage must always be consumed by the same warp");
template <bool GATHER> constexpr int THREADS = (NCW + (GATHER ? NPW_GATHER : 1)) * 32;
constexpr int SM_BAR = NSTAGE * STAGE_BYTES;                          // full[NSTAGE], empty[NSTAGE]
constexpr int SM_Q = SM_BAR + 2 * NSTAGE * 8 + 32;                    // per-warp rotated q: NCW x 8 x 128 bf16
constexpr int SM_MERGE = SM_Q + NCW * 8 * D * 2;                      // NCW x 8 x (2 + 128) floats
constexpr int SM_MISC = SM_MERGE + NCW * 8 * 130 * 4;                 // abort flag, the CTA's page range, scan sums
constexpr int SM_TOTAL = SM_MISC + 128;
constexpr int SM_ALLOC = SM_TOTAL + 1024;
static_assert(SM_ALLOC <= 232448, "shared memory");
constexpr uint32_t WAIT_PROBES = 1u << 21;   // ~2.8 s

struct DecParams {
  const __nv_bfloat16* q; const int32_t* q_pos;
  const __nv_bfloat16* k_new; const __nv_bfloat16* v_new;   // current token's key / value, or null
  __nv_bfloat16* k_pages; __nv_bfloat16* v_pages;
  const int32_t* res_pt; int max_res_pages; const int32_t* res_len;
  const int32_t* hist_pt; int max_hist_pages; const int32_t* hist_len;
  int n_items, G, Hq, s;
  int per_item;     // > 0: one sequence, every item has this many CTAs (its items differ by their routes only)
  int64_t n_pages;
  // partials: [slot][s][128], [slot][s][2]; part_cta[item] = first and last CTA of the item
  void* out; float* part_o; float* part_ml; int2* part_cta;
  const float* cos_tab; const float* sin_tab; int max_pos;
  float scale_log2;
  int32_t* status;
  // gather variant: the resource part of item `it` is rows route_idx[route_cu[it] .. route_cu[it+1]) of the cache
  const __nv_bfloat16* k_cache; const __nv_bfloat16* v_cache; int64_t pool_tokens;
  const int32_t* route_idx; const int32_t* route_cu; int64_t route_rows;   // entries of route_idx
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait: see rc_mbar_wait; this kernel also records where a wait ran out.
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  rc_mbar_wait<WAIT_PROBES, RC_WHERE_DECODE_SPLIT>(bar, parity, abort_flag, status);
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)) : "memory");
}
// the barrier gets one (pre-counted) arrival when all earlier cp.async of this thread have landed
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&p);
}
__device__ __forceinline__ void bar_consumers() { asm volatile("bar.sync 1, %0;" ::"n"(NCW * 32) : "memory"); }

// Pages of item `it`.  An item without a readable row still counts one page, so that its (zero)
// output is written by somebody.  (A gathered page keeps its CTA longer than one that TMA brings, but
// both variants deal alike: with the same max_res_pages, which bounds the number of CTAs, the same rows give
// the same bits whichever way they come.)
struct ItemPages { int n_res, n_hist, total, res_len, hist_len, r0; };
template <bool GATHER>
__device__ __forceinline__ ItemPages item_pages(const DecParams& p, int it) {
  ItemPages u;
  u.r0 = 0;
  if (GATHER) {
    // the item's slice of the index list must lie inside it; otherwise the route is treated as empty
    const int r0 = p.route_cu[it], r1 = p.route_cu[it + 1];
    const bool ok = r0 >= 0 && r1 >= r0 && (int64_t)r1 <= p.route_rows;
    if (!ok) rc_set_status(p.status, RECACHE_DEV_OVERFLOW);
    u.r0 = ok ? r0 : 0;
    u.res_len = ok ? r1 - r0 : 0;
  } else {
    u.res_len = max(p.res_len[it], 0);
  }
  u.hist_len = max(p.hist_len[it], 0);
  u.n_res = GATHER ? (u.res_len + PT - 1) / PT : min((u.res_len + PT - 1) / PT, p.max_res_pages);
  u.n_hist = min((u.hist_len + PT - 1) / PT, p.max_hist_pages);
  u.total = max(u.n_res + u.n_hist, 1);
  return u;
}
// CTA of n whose range of the T pages holds page x
__device__ __forceinline__ int cta_of_page(int64_t x, int64_t T, int n) { return (int)(((x + 1) * n - 1) / T); }

// A CTA's share: pages [lo, hi) of the T of all items (the item that holds `lo` begins at page `start`),
// or, with per_item > 0, a share of one item.
struct Share { int T, n_cta, lo, hi, item, start, per_item; };
// The pages [p0, p1) of item `it` that are the CTA's, and the last CTA that has any of the item.
__device__ __forceinline__ void own_pages(const Share& sh, const ItemPages& u, int start, int& p0, int& p1, int& last) {
  if (sh.per_item > 0) {
    const int k = min(sh.per_item, u.total), j = (int)blockIdx.x % sh.per_item;
    p0 = min(u.total, u.total * j / k); p1 = min(u.total, u.total * (j + 1) / k);
    last = (int)blockIdx.x - j + k - 1;
  } else {
    p0 = max(sh.lo - start, 0); p1 = min(sh.hi - start, u.total);
    last = cta_of_page((int64_t)start + u.total - 1, sh.T, sh.n_cta);
  }
}

template <typename TO, bool GATHER>
__global__ void __launch_bounds__(THREADS<GATHER>, 1) decode_split_kernel(const __grid_constant__ CUtensorMap tm_k,
                                                                   const __grid_constant__ CUtensorMap tm_v,
                                                                   const DecParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t sm = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* sm_gen = smem_raw + (sm - smem_u32(smem_raw));
  const uint32_t bars = sm + SM_BAR;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm_gen + SM_MISC);
  volatile int* range_sm = reinterpret_cast<volatile int*>(sm_gen + SM_MISC + 8);    // first item, its first page
  volatile int* sums_sm = reinterpret_cast<volatile int*>(sm_gen + SM_MISC + 32);    // per warp: pages, the longest item's
  auto full = [&](int i) { return bars + 8u * (uint32_t)i; };
  auto empty = [&](int i) { return bars + 8u * (uint32_t)(NSTAGE + i); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int i = 0; i < NSTAGE; ++i) { mbar_init(full(i), GATHER ? 32 * NPW_GATHER : 1); mbar_init(empty(i), 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == NCW && lane == 0) { prefetch_tmap(&tm_k); prefetch_tmap(&tm_v); }
  __syncthreads();         // no warp touches a barrier or the abort flag before they are set, on either way to the roles
  rc_grid_wait();
  rc_grid_launch_next();   // (the merge waits for this grid's end; it only comes up early)

  Share sh;
  sh.T = 0; sh.n_cta = gridDim.x; sh.lo = 0; sh.hi = 1; sh.start = 0; sh.per_item = p.per_item;
  if (p.per_item == 0) {
    // ---- this CTA's share of the page list: every thread sums a run of items, then one block scan ----
    constexpr int NTHREADS = THREADS<GATHER>;
    const int per = (p.n_items + NTHREADS - 1) / NTHREADS;
    const int i0 = min(p.n_items, (int)threadIdx.x * per), i1 = min(p.n_items, i0 + per);
    int sum = 0, most = 0;
#pragma unroll 4
    for (int i = i0; i < i1; ++i) {
      const ItemPages u = item_pages<GATHER>(p, i);
      sum += u.total;
      most = max(most, u.total);
    }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 31) { sums_sm[2 * warp] = incl; sums_sm[2 * warp + 1] = most; }
    __syncthreads();
    int before = 0;
#pragma unroll
    for (int w = 0; w < NTHREADS / 32; ++w) {
      if (w < warp) before += sums_sm[2 * w];
      sh.T += sums_sm[2 * w];
      most = max(most, sums_sm[2 * w + 1]);
    }
    sh.n_cta = min((int)gridDim.x, sh.T);          // every one of them has a page
    const int k = gridDim.x / p.n_items;
    if (k >= 2 && most / k <= sh.T / sh.n_cta + 3) {
      sh.per_item = k;
    } else {
      if ((int)blockIdx.x >= sh.n_cta) return;
      sh.lo = (int)((int64_t)sh.T * blockIdx.x / sh.n_cta); sh.hi = (int)((int64_t)sh.T * (blockIdx.x + 1) / sh.n_cta);
      before += incl - sum;
      if (sh.lo >= before && sh.lo < before + sum) {
        int i = i0, acc = before;
        for (;; ++i) {
          const int m = item_pages<GATHER>(p, i).total;
          if (sh.lo < acc + m) break;
          acc += m;
        }
        range_sm[0] = i; range_sm[1] = acc;
      }
      __syncthreads();
      sh.item = range_sm[0]; sh.start = range_sm[1];
    }
  }
  if (sh.per_item > 0) {
    sh.item = blockIdx.x / sh.per_item;
    if (sh.item >= p.n_items) return;
  }

  if (warp >= NCW) {
    // ===================== producer(s) =====================
    const int pw = warp - NCW;                         // producer warp index (0 in the paged variant)
    uint32_t n = 0;   // pages issued so far (ring position)
    for (int it = sh.item, start = sh.start; start < sh.hi; ++it) {
      const ItemPages u = item_pages<GATHER>(p, it);
      int p0, p1, last;
      own_pages(sh, u, start, p0, p1, last);
      start += u.total;
      // gather variant: cache row of chunk row pw * 16 + lane % 16, fetched one chunk ahead inside an item
      constexpr int RPW = PT / NPW_GATHER;             // rows of a chunk per producer warp (16)
      auto load_idx = [&](int chunk) {
        const int r = chunk * PT + pw * RPW + (lane & (RPW - 1));
        return r < u.res_len ? p.route_idx[u.r0 + r] : 0;
      };
      int idx_next = GATHER && p0 < p1 && p0 < u.n_res ? load_idx(p0) : 0;
      const int64_t group_off = (int64_t)(it % p.G) * p.pool_tokens * D;
      for (int lp = p0; lp < p1; ++lp, ++n) {
        const int st = n % NSTAGE;
        const uint32_t dst = sm + st * STAGE_BYTES;
        if (GATHER && lp < u.n_res) {
          // 64 route rows straight from the cache: half a warp copies one 256-byte row, 16 bytes per lane
          const int valid = min(PT, u.res_len - lp * PT);
          int idx_l = idx_next;
          if (lp + 1 < p1 && lp + 1 < u.n_res) idx_next = load_idx(lp + 1);
          if (idx_l < 0 || idx_l >= p.pool_tokens) {
            rc_set_status(p.status, RECACHE_DEV_BAD_SLOT);
            idx_l = (int)min(max((int64_t)idx_l, (int64_t)0), p.pool_tokens - 1);
          }
          if (lane == 0) mbar_wait(empty(st), ((n / NSTAGE) & 1u) ^ 1u, abort_flag, p.status);
          __syncwarp();
          const int c = lane & 15;
#pragma unroll
          for (int rr = 0; rr < RPW; rr += 2) {
            const int lrow = rr + (lane >> 4);
            const int row = pw * RPW + lrow;
            const int idx = __shfl_sync(0xffffffffu, idx_l, lrow);
            if (row < valid) {
              const int64_t src = group_off + (int64_t)idx * D + c * 8;
              const uint32_t d0 = dst + (c >> 3) * BOX_BYTES + row * 128 + (((c & 7) ^ (row & 7)) << 4);
              cp_async16(d0, p.k_cache + src);
              cp_async16(d0 + PAGE_BYTES, p.v_cache + src);
            }
          }
          cp_async_arrive(full(st));
        } else {
          if (lane == 0 && pw == 0) {
            int pg = (!GATHER && lp < u.n_res) ? p.res_pt[(int64_t)it * p.max_res_pages + lp]
                                               : p.hist_pt[(int64_t)it * p.max_hist_pages + (lp - u.n_res)];
            if (pg < 0 || pg >= p.n_pages) { rc_set_status(p.status, RECACHE_DEV_BAD_PAGE); pg = 0; }
            mbar_wait(empty(st), ((n / NSTAGE) & 1u) ^ 1u, abort_flag, p.status);
            mbar_expect_tx(full(st), STAGE_BYTES);
            tma_load_2d(dst, &tm_k, full(st), 0, pg * PT);
            tma_load_2d(dst + BOX_BYTES, &tm_k, full(st), 64, pg * PT);
            tma_load_2d(dst + PAGE_BYTES, &tm_v, full(st), 0, pg * PT);
            tma_load_2d(dst + PAGE_BYTES + BOX_BYTES, &tm_v, full(st), 64, pg * PT);
          }
          if (GATHER) {           // the other 127 of the 128 arrivals a full barrier takes in this variant
            if (lane == 0 && pw != 0) mbar_wait(empty(st), ((n / NSTAGE) & 1u) ^ 1u, abort_flag, p.status);
            __syncwarp();         // (not before this warp has seen the stage released)
            if (lane != 0 || pw != 0) mbar_arrive(full(st));
          }
        }
        __syncwarp();
      }
    }
  } else {
    // ===================== consumers =====================
    const int gq = lane >> 2, tq = lane & 3;           // fragment row (query head) and column pair
    const int s = p.s;
    uint32_t n_base = 0;                                // ring position of the item's first page here
    __nv_bfloat16* q_sm = reinterpret_cast<__nv_bfloat16*>(sm_gen + SM_Q) + warp * 8 * D;
    float* mrg = reinterpret_cast<float*>(sm_gen + SM_MERGE);
    for (int it = sh.item, start = sh.start; start < sh.hi; ++it) {
      const int b = it / p.G, g = it % p.G;
      const int pos_q = p.q_pos[b];
      const ItemPages u = item_pages<GATHER>(p, it);
      int p0, p1, last;
      own_pages(sh, u, start, p0, p1, last);
      start += u.total;
      if (p0 == p1) continue;
      const bool whole = p0 == 0 && p1 == u.total;
      if (p0 == 0 && lane == 0 && warp == 0) {
        p.part_cta[it] = make_int2(blockIdx.x, whole ? (int)blockIdx.x : last);
        if (u.hist_len < 1 || (!GATHER && (u.res_len + PT - 1) / PT > p.max_res_pages) ||
            (u.hist_len + PT - 1) / PT > p.max_hist_pages)
          rc_set_status(p.status, RECACHE_DEV_BAD_PAGE);
      }
      const bool pos_ok = pos_q >= 0 && pos_q < p.max_pos;
      const int64_t tab = (int64_t)min(max(pos_q, 0), p.max_pos - 1) * 64;   // cos / sin row
      if (!pos_ok) rc_set_status(p.status, RECACHE_DEV_BAD_POS);
      // ---- rotated query heads of the group -> A fragments (rows >= s are zero) ----
      {
        const __nv_bfloat16* qg = p.q + ((int64_t)b * p.Hq + g * s) * D;
        // lane -> the rotation pairs 2 lane, 2 lane + 1 of every head
        const float2 c = *reinterpret_cast<const float2*>(p.cos_tab + tab + 2 * lane);
        const float2 sn = *reinterpret_cast<const float2*>(p.sin_tab + tab + 2 * lane);
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          uint32_t wl = 0, wh = 0;
          if (h < s) {
            wl = *reinterpret_cast<const uint32_t*>(qg + h * D + 2 * lane);
            wh = *reinterpret_cast<const uint32_t*>(qg + h * D + 64 + 2 * lane);
          }
          const float l0 = __uint_as_float(wl << 16), l1 = __uint_as_float(wl & 0xffff0000u);
          const float h0 = __uint_as_float(wh << 16), h1 = __uint_as_float(wh & 0xffff0000u);
          *reinterpret_cast<uint32_t*>(q_sm + h * D + 2 * lane) =
              pack2(__fmaf_rn(l0, c.x, -__fmul_rn(h0, sn.x)), __fmaf_rn(l1, c.y, -__fmul_rn(h1, sn.y)));
          *reinterpret_cast<uint32_t*>(q_sm + h * D + 64 + 2 * lane) =
              pack2(__fmaf_rn(h0, c.x, __fmul_rn(l0, sn.x)), __fmaf_rn(h1, c.y, __fmul_rn(l1, sn.y)));
        }
        __syncwarp();
      }
      uint32_t qa[8][2];   // per k-step: a0 (cols 2tq,+1) and a2 (cols 8+2tq,+1) of row gq; rows 8..15 are zero
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        qa[kk][0] = *reinterpret_cast<const uint32_t*>(q_sm + gq * D + kk * 16 + tq * 2);
        qa[kk][1] = *reinterpret_cast<const uint32_t*>(q_sm + gq * D + kk * 16 + 8 + tq * 2);
      }
      __syncwarp();

      float o[16][4];
#pragma unroll
      for (int nt = 0; nt < 16; ++nt) { o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f; }
      float m_run = -INFINITY, l_run = 0.f;      // row gq (replicated over the quad), log2 domain

      // first page of the range whose ring position belongs to this warp
      const int first = (int)(((uint32_t)warp + NCW - n_base % NCW) % NCW);
      for (int lp = p0 + first; lp < p1; lp += NCW) {
        const uint32_t n = n_base + (uint32_t)(lp - p0);
        const int st = n % NSTAGE;
        // tokens of this page that exist
        int valid = PT;
        if (lp < u.n_res) valid = min(PT, u.res_len - lp * PT);
        else valid = min(PT, u.hist_len - (lp - u.n_res) * PT);
        mbar_wait(full(st), (n / NSTAGE) & 1u, abort_flag, p.status);
        const uint32_t kb = sm + st * STAGE_BYTES, vb = kb + PAGE_BYTES;
        const int hn = u.hist_len - 1;                   // the current token's history row
        const bool appends = p.k_new && hn >= 0 && pos_ok && lp >= u.n_res && hn / PT == lp - u.n_res;
        if (valid < PT) {
          // slots past the end of the part were never written: clear their values (0 * NaN would poison O)
          uint8_t* vg = sm_gen + st * STAGE_BYTES + PAGE_BYTES;
          const int v0 = max(valid, 0);
          for (int e = lane; e < (PT - v0) * 16; e += 32) {
            const int r = v0 + (e >> 4), c = e & 15;
            *reinterpret_cast<uint4*>(vg + (c >> 3) * BOX_BYTES + r * 128 + (c & 7) * 16) = make_uint4(0, 0, 0, 0);
          }
        }
        if (appends) {
          const int pg = p.hist_pt[(int64_t)it * p.max_hist_pages + hn / PT], r = hn % PT;
          const __nv_bfloat16* ks = p.k_new + (int64_t)it * D;
          const __nv_bfloat16* vs = p.v_new + (int64_t)it * D;
          if (pg >= 0 && pg < p.n_pages) {
            uint8_t* kg = sm_gen + st * STAGE_BYTES + r * 128;
            const int64_t row = ((int64_t)pg * PT + r) * D;
#pragma unroll
            for (int x = 0; x < 2; ++x) {                // element i of the low half, i + 64 of the high half (next box)
              const int i = lane + 32 * x;
              const float l = __bfloat162float(ks[i]), h = __bfloat162float(ks[i + 64]);
              const float c = p.cos_tab[tab + i], sn = p.sin_tab[tab + i];
              const __nv_bfloat16 kl = __float2bfloat16_rn(__fmaf_rn(l, c, -__fmul_rn(h, sn)));
              const __nv_bfloat16 kh = __float2bfloat16_rn(__fmaf_rn(h, c, __fmul_rn(l, sn)));
              const __nv_bfloat16 vl = vs[i], vh = vs[i + 64];
              uint8_t* e = kg + (((i >> 3) ^ (r & 7)) << 4) + (i & 7) * 2;
              *reinterpret_cast<__nv_bfloat16*>(e) = kl;
              *reinterpret_cast<__nv_bfloat16*>(e + BOX_BYTES) = kh;
              *reinterpret_cast<__nv_bfloat16*>(e + PAGE_BYTES) = vl;
              *reinterpret_cast<__nv_bfloat16*>(e + PAGE_BYTES + BOX_BYTES) = vh;
              p.k_pages[row + i] = kl; p.k_pages[row + i + 64] = kh;
              p.v_pages[row + i] = vl; p.v_pages[row + i + 64] = vh;
            }
          }
        }
        if (valid < PT || appends) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // a later TMA load overwrites these bytes
          __syncwarp();
        }
        // ---- S = q K^T : 8 token tiles x 8 k-steps ----
        float sc[8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
          const int tok = nt * 8 + (lane & 7);
#pragma unroll
          for (int kq = 0; kq < 4; ++kq) {
            const int c = 4 * kq + (lane >> 3);
            const uint32_t addr = kb + (c >> 3) * BOX_BYTES + tok * 128 + (((c & 7) ^ (tok & 7)) << 4);
            uint32_t b0, b1, b2, b3;
            ldsm_x4(addr, b0, b1, b2, b3);
            mma_bf16(sc[nt], qa[2 * kq][0], 0u, qa[2 * kq][1], 0u, b0, b1);
            mma_bf16(sc[nt], qa[2 * kq + 1][0], 0u, qa[2 * kq + 1][1], 0u, b2, b3);
          }
        }
        // ---- online softmax of row gq (columns nt*8 + 2tq, +1) ----
        float mx = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const int c0 = nt * 8 + tq * 2;
          sc[nt][0] = c0 < valid ? sc[nt][0] * p.scale_log2 : -INFINITY;
          sc[nt][1] = c0 + 1 < valid ? sc[nt][1] * p.scale_log2 : -INFINITY;
          mx = fmaxf(mx, fmaxf(sc[nt][0], sc[nt][1]));
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run, mx);
        const float m_use = m_new == -INFINITY ? 0.f : m_new;    // a page with no valid token
        const float corr = ex2(m_run - m_use);                   // 0 on the first page
        float ps = 0.f;
        uint32_t pa[4][2];   // P as A fragments: per 16-token k-step, a0 / a2 of row gq
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const float p0 = ex2(sc[nt][0] - m_use), p1 = ex2(sc[nt][1] - m_use);
          ps += p0 + p1;
          pa[nt >> 1][nt & 1] = pack2(p0, p1);
        }
        ps += __shfl_xor_sync(0xffffffffu, ps, 1);
        ps += __shfl_xor_sync(0xffffffffu, ps, 2);
        l_run = l_run * corr + ps;
        m_run = m_new;
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) { o[nt][0] *= corr; o[nt][1] *= corr; }
        // ---- O += P V : 4 k-steps (16 tokens) x 16 d tiles ----
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const int tok = kk * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
          for (int np = 0; np < 8; ++np) {
            const int c = 2 * np + (lane >> 4);
            const uint32_t addr = vb + (c >> 3) * BOX_BYTES + tok * 128 + (((c & 7) ^ (tok & 7)) << 4);
            uint32_t b0, b1, b2, b3;
            ldsm_x4_t(addr, b0, b1, b2, b3);
            mma_bf16(o[2 * np], pa[kk][0], 0u, pa[kk][1], 0u, b0, b1);
            mma_bf16(o[2 * np + 1], pa[kk][0], 0u, pa[kk][1], 0u, b2, b3);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(st));
      }
      n_base += (uint32_t)(p1 - p0);

      // ---- merge the consumer warps' partials (rows gq < s) ----
      if (gq < s) {
        float* mine = mrg + (warp * 8 + gq) * 130;
        if (tq == 0) { mine[0] = m_run; mine[1] = l_run; }
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) {
          mine[2 + nt * 8 + tq * 2] = o[nt][0];
          mine[2 + nt * 8 + tq * 2 + 1] = o[nt][1];
        }
      }
      bar_consumers();
      {
        const int t = threadIdx.x;               // head t/32 (+NCW ...), dims (t%32)*4..+3
        for (int h = t >> 5; h < s; h += NCW) {
          float mw[NCW], M = -INFINITY;
#pragma unroll
          for (int w = 0; w < NCW; ++w) { mw[w] = mrg[(w * 8 + h) * 130]; M = fmaxf(M, mw[w]); }
          float Lsum = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int w = 0; w < NCW; ++w) {
            const float f = mw[w] == -INFINITY ? 0.f : ex2(mw[w] - M);
            Lsum += mrg[(w * 8 + h) * 130 + 1] * f;
            const float* ow = mrg + (w * 8 + h) * 130 + 2 + (t & 31) * 4;
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c] += ow[c] * f;
          }
          if (whole) {
            const float inv = Lsum > 0.f ? 1.f / Lsum : 0.f;
            TO* orow = reinterpret_cast<TO*>(p.out) + ((int64_t)b * p.Hq + g * s + h) * D + (t & 31) * 4;
            if constexpr (sizeof(TO) == 4) {
              *reinterpret_cast<float4*>(orow) = make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv);
            } else {
              *reinterpret_cast<uint2*>(orow) = make_uint2(pack2(acc[0] * inv, acc[1] * inv), pack2(acc[2] * inv, acc[3] * inv));
            }
          } else {
            const int row = (2 * (int)blockIdx.x + (p0 == 0 ? 1 : 0)) * s + h;     // the CTA's slot for this part
            *reinterpret_cast<float4*>(p.part_o + (int64_t)row * D + (t & 31) * 4) = make_float4(acc[0], acc[1], acc[2], acc[3]);
            if ((t & 31) == 0) *reinterpret_cast<float2*>(p.part_ml + row * 2) = make_float2(M, Lsum);
          }
        }
      }
      bar_consumers();
    }
  }
  if (*abort_flag) rc_timeout_drain();   // a wait ran out: let the loads in flight land before the CTA ends
}

// Combines the parts of the items that span several CTAs: one warp per output row (32 lanes x 4
// dims), MERGE_ROWS rows per CTA.  The parts of item it lie in slot 2a + 1 of its first CTA a and
// slots 2c of the later ones up to b.  A round takes 24 parts: their (max, sum) pairs, a lane each, and
// their rows of O are all asked for at once, so that the launch is one or two loads deep.  With one
// sequence a and b follow from the lengths, which are read while the attention kernel still runs (its
// blocks have all seen the end of the kernels before it by then).
constexpr int MERGE_ROWS = 4, MERGE_PARTS = 24;
template <typename TO, bool GATHER>
__global__ void __launch_bounds__(32 * MERGE_ROWS) decode_merge_kernel(const __grid_constant__ DecParams p, int n_rows) {
  const int row = blockIdx.x * MERGE_ROWS + (threadIdx.x >> 5);   // b * Hq + head
  const int Hq = p.Hq, s = p.s, head = row % Hq, it = row / Hq * p.G + head / s, h = head % s;
  const int t = threadIdx.x & 31;
  int2 ab = make_int2(0, 0);
  if (p.per_item > 0 && row < n_rows) {
    ab.x = it * p.per_item;
    ab.y = ab.x + min(p.per_item, item_pages<GATHER>(p, it).total) - 1;
  }
  rc_grid_wait();
  rc_grid_launch_next();
  if (row >= n_rows) return;
  if (p.per_item == 0) ab = p.part_cta[it];
  if (ab.x == ab.y) return;                                        // written by the CTA that had all of it
  const int n = ab.y - ab.x + 1;
  auto slot_row = [&](int i) { return (i == 0 ? 2 * ab.x + 1 : 2 * (ab.x + i)) * s + h; };
  float M = -INFINITY, L = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int i0 = 0; i0 < n; i0 += MERGE_PARTS) {
    const int cnt = min(MERGE_PARTS, n - i0);
    float2 ml = make_float2(-INFINITY, 0.f);
    if (t < cnt) ml = *reinterpret_cast<const float2*>(p.part_ml + slot_row(i0 + t) * 2);
    float4 v[MERGE_PARTS];
#pragma unroll
    for (int j = 0; j < MERGE_PARTS; ++j)
      if (j < cnt) v[j] = *reinterpret_cast<const float4*>(p.part_o + (int64_t)slot_row(i0 + j) * D + t * 4);
    float m_new = fmaxf(M, ml.x);
#pragma unroll
    for (int off = 16; off; off >>= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xffffffffu, m_new, off));
    const float m_use = m_new == -INFINITY ? 0.f : m_new;
    const float corr = ex2(M - m_use), f = ex2(ml.x - m_use);      // 0 where nothing was seen yet / in that part
    M = m_new;
    float l = ml.y * f;
#pragma unroll
    for (int off = 16; off; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    L = L * corr + l;
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] *= corr;
#pragma unroll
    for (int j = 0; j < MERGE_PARTS; ++j) {
      const float fj = __shfl_sync(0xffffffffu, f, j);
      if (j < cnt) { acc[0] += v[j].x * fj; acc[1] += v[j].y * fj; acc[2] += v[j].z * fj; acc[3] += v[j].w * fj; }
    }
  }
  const float inv = L > 0.f ? 1.f / L : 0.f;
  TO* orow = reinterpret_cast<TO*>(p.out) + (int64_t)row * D + t * 4;
  if constexpr (sizeof(TO) == 4) {
    *reinterpret_cast<float4*>(orow) = make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv);
  } else {
    *reinterpret_cast<uint2*>(orow) = make_uint2(pack2(acc[0] * inv, acc[1] * inv), pack2(acc[2] * inv, acc[3] * inv));
  }
}

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
// page pool viewed as [n_pages * 64 rows][128 bf16]; box = one page x 64 columns
bool map_pages(CUtensorMap* m, const void* base, uint64_t n_pages) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {128, n_pages * PT};
  cuuint64_t strides[1] = {256};
  cuuint32_t box[2] = {64, PT};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int64_t align256(int64_t x) { return (x + 255) & ~(int64_t)255; }

}  // namespace

bool rc_decode_split_supported(const recache_ctx* ctx) {
  const int s = ctx->desc.n_q_heads / ctx->desc.n_kv_heads;
  return ctx->desc.dtype == RECACHE_BF16 && ctx->desc.head_dim == 128 && ctx->desc.page_tokens == PT && s <= 8;
}

static int grid_ctas(const recache_ctx* ctx) { return ctx->sm_count > 0 ? ctx->sm_count : 148; }

int64_t rc_decode_split_workspace_bytes(const recache_ctx* ctx, int batch, int max_res_pages, int max_hist_pages) {
  const int s = ctx->desc.n_q_heads / ctx->desc.n_kv_heads;
  const int64_t slots = 2 * (int64_t)grid_ctas(ctx);
  return align256(slots * s * D * 4) + align256(slots * s * 2 * 4) + align256((int64_t)batch * ctx->desc.n_kv_heads * 8);
}

cudaError_t rc_launch_decode_split(const recache_ctx* ctx, const DecodeArgs& a, cudaStream_t st) {
  const int G = ctx->desc.n_kv_heads, Hq = ctx->desc.n_q_heads, s = Hq / G;
  if ((uint64_t)a.n_pages * PT > 0x7fffffffull) return cudaErrorInvalidValue;   // TMA coordinates are 32-bit row indices
  const bool f32 = a.out_dtype == RECACHE_F32, gather = a.route_idx != nullptr;
  CUtensorMap tk, tv;
  if (!map_pages(&tk, a.k_pages, (uint64_t)a.n_pages) || !map_pages(&tv, a.v_pages, (uint64_t)a.n_pages))
    return cudaErrorInvalidValue;
  const int64_t slots = 2 * (int64_t)grid_ctas(ctx);
  DecParams p;
  p.q = (const __nv_bfloat16*)a.q; p.q_pos = a.q_pos;
  p.k_new = (const __nv_bfloat16*)a.k_new; p.v_new = (const __nv_bfloat16*)a.v_new;
  p.k_pages = (__nv_bfloat16*)a.k_pages; p.v_pages = (__nv_bfloat16*)a.v_pages;
  p.res_pt = a.res_pt; p.max_res_pages = a.max_res_pages; p.res_len = a.res_len;
  p.hist_pt = a.hist_pt; p.max_hist_pages = a.max_hist_pages; p.hist_len = a.hist_len;
  p.n_items = a.batch * G; p.G = G; p.per_item = 0; p.Hq = Hq; p.s = s; p.n_pages = a.n_pages;
  p.out = a.o;
  uint8_t* ws = (uint8_t*)a.workspace;
  p.part_o = (float*)ws; ws += align256(slots * s * D * 4);
  p.part_ml = (float*)ws; ws += align256(slots * s * 2 * 4);
  p.part_cta = (int2*)ws;
  p.cos_tab = ctx->cos_tab; p.sin_tab = ctx->sin_tab; p.max_pos = ctx->desc.max_pos;
  p.scale_log2 = (float)(1.4426950408889634 / sqrt((double)D));
  p.status = ctx->status;
  p.k_cache = (const __nv_bfloat16*)a.k_cache; p.v_cache = (const __nv_bfloat16*)a.v_cache;
  p.pool_tokens = a.pool_tokens; p.route_idx = a.route_idx; p.route_cu = a.route_cu; p.route_rows = a.route_rows;
  // no more CTAs than pages there can be; the paged kernel's lengths live on the device, the tables' widths here
  const int64_t most = (int64_t)p.n_items * (a.max_res_pages + (int64_t)a.max_hist_pages);
  unsigned grid = (unsigned)(most > grid_ctas(ctx) ? grid_ctas(ctx) : (most > 0 ? most : 1));
  // One sequence: its items have the history in common, so equal shares need no look at the lengths
  // (0.8 us of a step of 7).
  if (a.batch == 1 && (unsigned)G <= grid) { p.per_item = (int)grid / G; grid = (unsigned)(p.per_item * G); }
  // Appending holds an item's consumers up by about a microsecond, a launch that appends for all takes 4-8 us:
  // 512 items (64 sequences of 200 rows, 8 groups) 2.0 us here and 8.0 there, 1024 items 6.8 and 4.1, 8192 items
  // 41 and 9; so up to four items a CTA.
  if (a.k_new && p.n_items > 4 * grid_ctas(ctx)) {
    const cudaError_t e = rc_launch_decode_append(ctx, a, st);
    if (e != cudaSuccess) return e;
    p.k_new = p.v_new = nullptr;
  }
  auto run = [&](auto type, auto gathers) {
    using TO = decltype(type);
    constexpr bool GATHER = decltype(gathers)::value;
    {
      RcLaunchScope scope(ctx, RC_K_DECODE_ATTN, st);
      const cudaError_t e = rc_launch_overlapped(decode_split_kernel<TO, GATHER>, grid, THREADS<GATHER>, SM_ALLOC, st, tk, tv, p);
      if (e != cudaSuccess) return e;
    }
    RcLaunchScope scope(ctx, RC_K_DECODE_MERGE, st);
    const int n_rows = a.batch * Hq, blocks = (n_rows + MERGE_ROWS - 1) / MERGE_ROWS;
    return rc_launch_overlapped(decode_merge_kernel<TO, GATHER>, blocks, 32 * MERGE_ROWS, 0, st, p, n_rows);
  };
  if (gather) return f32 ? run(float(), std::true_type()) : run(__nv_bfloat16(), std::true_type());
  return f32 ? run(float(), std::false_type()) : run(__nv_bfloat16(), std::false_type());
}

// ---------------------------------------------------------------------------
// Allocation-free decode.
//
// recache_attend_decode needs a scratch buffer for the split partials, which the
// caller normally gets from its allocator.  Some callers cannot allocate at the
// point where they decode: code running inside a region where the CUDA allocator
// must not be touched (a serving loop that has pinned down its memory plan, a
// plugin loaded into a host process that owns all device memory, a signal-safe
// or real-time path).  For them the scratch lives in this file-scope device
// array, reserved by every GPU that loads the library until the process exits.
// ---------------------------------------------------------------------------
namespace {

constexpr int64_t NOALLOC_SCRATCH_BYTES = 4ll << 20;   // 4 MiB per device
static __device__ __align__(256) unsigned char g_decode_scratch[NOALLOC_SCRATCH_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
// Device address of g_decode_scratch, per device.  Host threads may make the first call on a
// device at the same time: each looks the address up and stores the same value, through an atomic
// so that the concurrent store and load are well defined.
std::atomic<void*> g_scratch_addr[NOALLOC_MAX_DEVICES];

}  // namespace

extern "C" RECACHE_API recache_status recache_attend_decode_noalloc(
    recache_ctx* ctx, const void* q, const int32_t* q_pos, int32_t batch, const void* k_new, const void* v_new,
    void* k_pages, void* v_pages, int64_t n_pages, const int32_t* res_page_table, int32_t max_res_pages,
    const int32_t* res_len, const int32_t* hist_page_table, int32_t max_hist_pages, const int32_t* hist_len,
    void* out_o, int32_t out_dtype, void* stream) {
  if (!ctx) return RECACHE_EINVAL;
  auto fail = [&](recache_status st, const char* msg) { ctx->err = msg; return st; };
  if (batch < 0 || n_pages < 0 || max_res_pages < 0 || max_hist_pages <= 0)
    return fail(RECACHE_EINVAL, "decode_noalloc: bad size");
  if (out_dtype != RECACHE_F32 && out_dtype != ctx->desc.dtype)
    return fail(RECACHE_EINVAL, "decode_noalloc: out_dtype must be f32 or the context dtype");
  if (batch == 0) return RECACHE_OK;
  if (!q || !q_pos || !k_pages || !v_pages || !res_len || !hist_page_table || !hist_len || !out_o ||
      (max_res_pages > 0 && !res_page_table) || ((k_new == nullptr) != (v_new == nullptr)))
    return fail(RECACHE_EINVAL, "decode_noalloc: null pointer");
  if (((uintptr_t)q | (uintptr_t)k_pages | (uintptr_t)v_pages | (uintptr_t)out_o) & 15)
    return fail(RECACHE_EINVAL, "decode_noalloc: tensors must be 16-byte aligned");
  if (!rc_decode_split_supported(ctx))
    return fail(RECACHE_EUNSUPPORTED, "decode_noalloc: needs a bf16 context with head_dim 128 and 64-token pages");
  if (ctx->timer_on)
    return fail(RECACHE_EINVAL, "decode_noalloc: the kernel timer creates event objects; disable it first");
  // the contract's bound is one unsplit partial per (sequence, query head); what a call really needs is below it
  const int64_t need = rc_decode_split_workspace_bytes(ctx, batch, max_res_pages, max_hist_pages);
  if (need > NOALLOC_SCRATCH_BYTES || (int64_t)batch * ctx->desc.n_q_heads * (D + 2) * 4 > NOALLOC_SCRATCH_BYTES)
    return fail(RECACHE_ENOMEM, "decode_noalloc: batch x query heads x 520 bytes exceeds the 4 MiB built-in scratch; "
                                "use recache_attend_decode with a caller workspace");
  if (ctx->device < 0 || ctx->device >= NOALLOC_MAX_DEVICES)
    return fail(RECACHE_EUNSUPPORTED, "decode_noalloc: device index out of range");
  if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(RECACHE_ECUDA, "decode_noalloc: set device");
  // In host code the array's name is only a handle; the kernel needs its device
  // address, looked up once per device with that device current.
  void* scratch = g_scratch_addr[ctx->device].load(std::memory_order_relaxed);
  if (!scratch) {
    cudaError_t e = cudaGetSymbolAddress(&scratch, g_decode_scratch);
    if (e != cudaSuccess || !scratch) {
      ctx->err = std::string("decode_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e);
      return RECACHE_ECUDA;
    }
    g_scratch_addr[ctx->device].store(scratch, std::memory_order_relaxed);
  }
  cudaStream_t st = (cudaStream_t)stream;
  DecodeArgs a{q, q_pos, batch, k_new, v_new, k_pages, v_pages, n_pages, res_page_table, max_res_pages, res_len,
               hist_page_table, max_hist_pages, hist_len, out_o, out_dtype, scratch, NOALLOC_SCRATCH_BYTES};
  const cudaError_t e = rc_launch_decode_split(ctx, a, st);
  if (e != cudaSuccess) {
    ctx->err = std::string("decode_noalloc: launch: ") + cudaGetErrorString(e);
    return RECACHE_ECUDA;
  }
  return RECACHE_OK;
}
