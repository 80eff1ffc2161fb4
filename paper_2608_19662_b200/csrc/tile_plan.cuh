// Work list of the tensor-core attention.  Built by one block of the rotate-and-store kernel that
// precedes the attention launch (it only depends on the call's index arrays), read by the attention
// kernel's scheduler warps.  As a launch of its own, on a side stream between two events, it took 6-9 us
// of the smallest calls (encoding one resource of 500 tokens: 26.6 us with it, 20.6 us now).
#pragma once
#include "common.cuh"

constexpr int RC_TILE_N = 128;       // keys of a K/V tile
constexpr int RC_SORT_MAX = 4096;    // work items up to which the plan sorts a prefill by weight (encode: a quarter)
constexpr int RC_ITEM_UNITS = 2;     // what beginning an item costs, in K/V tiles of about 0.95 us
constexpr int RC_MERGE_UNITS = 11;   // what parts and their merge cost
constexpr int RC_L2_BLOCKS = 768;    // 100 MB: what of the 126 MB L2 a launch's keys and values may take
constexpr int RC_PLAN_BINS = 1024;   // weights (K/V tiles, items) are told apart up to this

struct RcPlan {
  int2* items;
  int32_t* header;                // number of items, work counter, whether order[] is valid, CTAs of a split launch
  int32_t* order;                 // work indices, heaviest first (launches of at most RC_SORT_MAX work items); K/V tiles of each behind them
  // Split launch (null: not wanted): CTA c takes the K/V tiles from start[c] = (work index, tile) up to start[c + 1].
  // merge[c]: what the merge does at cut c: parts of the item it is the first cut of (0: nothing to do), first token of the
  // item's rows, rows (tokens x heads), group.
  int2* start; int4* merge; int32_t* unit_cu;
  int n_cta;                      // CTAs of the attention launch
  const int32_t* cu; const int32_t* pos0; const int32_t* slot; const int32_t* route_cu; const int32_t* hist;
  int n_seq, G, Hq, s;
  int prefix_len;   // > 0: every sequence sees rows g*prefix_len .. of the "route" tensors (shared prefix)
  int64_t self_rows;
  int64_t route_rows;   // rows of the packed route tensors / entries of route_idx
  int item_tiles;            // query tiles of a work item: 1, or 2 (a pair)
  int n_levels, max_items;   // work items of the longest sequence, capacity of items[]
  int32_t* status;
};

// One work item as published by the scheduler warp (16 ints in shared memory).
struct RcItem {
  int n_tiles;      // -1: no more work
  int g, seq0, L, tok0, kv_end, pos0, rA0, lenA, nA, b_valid;
  int H;            // rows that precede the sequence's own tokens in the self part (earlier turns), all visible
  int64_t base;
  int part;         // slot of this CTA's part of a split item, -1: the whole item
};

// Work index w -> item; false when the caller's index arrays are inconsistent
// (flagged in the status word; the scheduler skips the item).
__device__ __forceinline__ bool rc_load_item(const RcPlan& p, int w, RcItem& it) {
  const int2 e = p.items[w / p.G];
  it.g = w % p.G;
  const int b = e.x;
  const int TQ = 128 / p.s;
  it.seq0 = p.cu[b];
  it.L = p.cu[b + 1] - it.seq0;
  it.tok0 = e.y * p.item_tiles * TQ;
  it.b_valid = p.item_tiles > 1 && it.tok0 + TQ < it.L;
  it.H = p.hist ? p.hist[b] : 0;
  it.kv_end = it.H + min(it.L, it.tok0 + p.item_tiles * TQ);   // self rows the item can see: the history, then its causal range
  it.base = p.slot ? (int64_t)p.slot[b] : (int64_t)it.seq0;
  it.pos0 = p.pos0 ? p.pos0[b] : 0;
  it.rA0 = 0; it.lenA = 0;
  bool route_ok = true;
  if (p.route_cu) {
    it.rA0 = p.route_cu[b * p.G + it.g]; it.lenA = p.route_cu[b * p.G + it.g + 1] - it.rA0;
    route_ok = (int64_t)it.rA0 + it.lenA <= p.route_rows;   // e.g. after a compaction that overflowed its capacity
  }
  else if (p.prefix_len > 0) { it.rA0 = it.g * p.prefix_len; it.lenA = p.prefix_len; }
  it.nA = (it.lenA + RC_TILE_N - 1) / RC_TILE_N;
  it.n_tiles = it.nA + (it.kv_end + RC_TILE_N - 1) / RC_TILE_N;
  const bool ok = it.L > 0 && it.tok0 < it.L && it.lenA >= 0 && it.rA0 >= 0 && it.base >= 0 && it.H >= 0 &&
                  it.base + it.H + it.L <= p.self_rows && it.seq0 >= 0 && route_ok;
  if (!ok) rc_set_status(p.status, route_ok ? RECACHE_DEV_BAD_SLOT : RECACHE_DEV_OVERFLOW);
  return ok;
}

struct RcPlanSmem {
  int hist[RC_PLAN_BINS + 1];
  int warp_sum[33];
  int most;         // K/V tiles of the longest item
  int blocks;       // of 256 key and value rows (128 KB) that the launch reads
};

// Exclusive block scan of one int per thread; *total gets the sum (same pattern of calls in every thread).
__device__ __forceinline__ int rc_plan_scan(int v, RcPlanSmem& sh, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += u;
  }
  __syncthreads();
  if (lane == 31) sh.warp_sum[warp] = incl;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll 1
  for (int w = 0; w < nw; ++w) { const int x = sh.warp_sum[w]; if (w < warp) before += x; all += x; }
  *total = all;
  return before + incl - v;
}
// Turns the bin counts into the first index of each bin, bin 0 first; all threads of the block.
__device__ __forceinline__ void rc_plan_scan_bins(RcPlanSmem& sh) {
  const int per = (RC_PLAN_BINS + 1 + blockDim.x - 1) / blockDim.x;
  const int i0 = min(RC_PLAN_BINS + 1, (int)threadIdx.x * per), i1 = min(RC_PLAN_BINS + 1, i0 + per);
  int sum = 0, total;
#pragma unroll 1
  for (int i = i0; i < i1; ++i) sum += sh.hist[i];
  int at = rc_plan_scan(sum, sh, &total);
#pragma unroll 1
  for (int i = i0; i < i1; ++i) { const int c = sh.hist[i]; sh.hist[i] = at; at += c; }
  __syncthreads();
}

// A later turn (RcPlan.start given) whose items, of one query tile each, do not fill the CTAs evenly: their K/V tiles, laid end
// to end, are cut into n equal ranges, so that an item may be shared by several CTAs (their partial results are merged
// afterwards).  An item counts RC_ITEM_UNITS more than its tiles, and a cut is moved to the item's
// edge where it would leave a part of fewer than two tiles, or a part whose first tile some row of
// the item does not see.  Taken only where the longest CTA gets shorter by more than parts and merge cost.  Whole, a launch
// of one round ends with its longest item, one of more 0.8 of that after the mean CTA or, of items much alike, a little
// after as many mean items as there are rounds; ranges take a fifth longer where
// the launch reads more than L2 holds, as whole items of a sequence walk its keys in step and parts do not.  Chosen and
// measured on 602 turns of up to three rounds, in a grid and at random, on inputs that are not in L2: the slower way is taken
// at a mean cost of 0.1 % and of more than 3 % in 9 of them (0.8 % and 67 with six units for the merge, which pairs of tiles had).
//   1 request of 16 tokens, 2 heads a group, over 1000 / 4000 rows (8 items of 12 / 36 tiles): 24.8 / 32.7 us split, 23.4 / 44.3 whole
//   4 x 16 tokens over 1000 (32 items of 13) 27.1 and 24.1; 8 x 17-250 over 300-2048 (152 items of 15) 42.9 and 41.7
//   1 x 64 tokens, 4 heads, over 12,000 (16 items of 99) 42.8 and 100.8; 16 x 64 over 4000 (256 items of 37) 127 and 109
// Encoding and first turns are never split: a resource's result must not depend on what is encoded beside it,
// nor a first turn's on whether its rows are packed or gathered.  False: not worth it.
__device__ __forceinline__ bool rc_plan_split(const RcPlan& p, RcPlanSmem& sh, int n_work) {
  const int tid = threadIdx.x, n_thr = blockDim.x;
  const int32_t* tiles = p.order + RC_SORT_MAX;
  const int per = (n_work + n_thr - 1) / n_thr;
  const int w0 = min(n_work, tid * per), w1 = min(n_work, w0 + per);
  int units = 0, items = 0, total_units, n_items;
#pragma unroll 1
  for (int w = w0; w < w1; ++w)
    if (tiles[w] > 0) { units += tiles[w] + RC_ITEM_UNITS; ++items; }
  rc_plan_scan(items, sh, &n_items);
  int at = rc_plan_scan(units, sh, &total_units);
  if (n_items == 0) return false;
  const int n = min(p.n_cta, max(1, (total_units - RC_ITEM_UNITS * n_items) / 4));
  const float pace = sh.blocks > RC_L2_BLOCKS ? 1.2f : 1.f;
  const float split = pace * total_units / n + RC_ITEM_UNITS + RC_MERGE_UNITS;
  float whole = 0.f;
  if (n_items > p.n_cta)
    whole = fminf((float)total_units / p.n_cta + 0.8f * sh.most, 1.05f * total_units / n_items * ((n_items + p.n_cta - 1) / p.n_cta));
  if (split > fmaxf((float)(sh.most + RC_ITEM_UNITS), whole)) return false;
#pragma unroll 1
  for (int w = w0; w < w1; ++w) { p.unit_cu[w] = at; if (tiles[w] > 0) at += tiles[w] + RC_ITEM_UNITS; }
  __syncthreads();
#pragma unroll 1
  for (int c = tid; c <= n; c += n_thr) {
    int2 cut = make_int2(n_work, 0);
    if (c < n) {
      const int x = (int)((int64_t)total_units * c / n);
      int lo = 0, hi = n_work;                       // the last item that starts at or before x (an empty one starts where the next does)
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (p.unit_cu[mid] <= x) lo = mid; else hi = mid;
      }
      cut = make_int2(lo, x - p.unit_cu[lo] - RC_ITEM_UNITS);
      RcItem it;
      rc_load_item(p, lo, it);
      if (cut.y < 2) cut.y = 0;
      else if (it.n_tiles - cut.y < 2 || cut.y > it.nA + (it.H + it.tok0) / RC_TILE_N) cut = make_int2(lo + 1, 0);
    }
    p.start[c] = cut;
  }
  __syncthreads();
#pragma unroll 1
  for (int c = tid; c < n; c += n_thr) {
    int4 m = make_int4(0, 0, 0, 0);
    const int2 cut = p.start[c];
    if (c > 0 && cut.y > 0 && (p.start[c - 1].x != cut.x || p.start[c - 1].y == 0)) {
      RcItem it;
      rc_load_item(p, cut.x, it);
      m = make_int4(2, it.seq0 + it.tok0, min(128, (it.L - it.tok0) * p.s), it.g);
#pragma unroll 1
      for (int j = c + 1; p.start[j].x == cut.x && p.start[j].y > 0; ++j) ++m.x;
    }
    p.merge[c] = m;
  }
  if (tid == 0) p.header[3] = n;
  return true;
}

// Items = (sequence, index of one or two query tiles, as item_tiles says): sequence by sequence, the longest sequences
// first, and inside a sequence the last (heaviest) first, so that the
// launch ends on the light items of short sequences.  With the KV group as the
// fastest index of the flattened work list, the CTAs that run at the same time
// share one sequence's K/V, which then stays in L2 instead of being streamed
// from HBM once per item.  One block.  (Sequences of equal length land in an
// order that may differ between launches; no result depends on it.)
// (Nothing is unrolled: the block runs every loop for a step or two, out of a cold instruction cache, and
// the unrolled code took 0.3-0.4 us more of turns of 35-50 us.)
__device__ __forceinline__ void rc_build_plan(const RcPlan& p, RcPlanSmem& sh) {
  const int tid = threadIdx.x, n_thr = blockDim.x, n_seq = p.n_seq, tok_per_item = p.item_tiles * 128 / p.s;
  const int32_t* cu = p.cu;
  auto n_items_of = [&](int b) {
    const int len = cu[b + 1] - cu[b];
    return min(len > 0 ? (len + tok_per_item - 1) / tok_per_item : 0, p.n_levels);
  };
  // each thread owns a contiguous chunk of sequences: local sums, block scan of the chunk sums, then the items
  const int per = (n_seq + n_thr - 1) / n_thr;
  const int b0 = min(n_seq, tid * per), b1 = min(n_seq, b0 + per);
  int sum = 0, total;
#pragma unroll 1
  for (int b = b0; b < b1; ++b) {
    const int len = cu[b + 1] - cu[b];
    if (len < 0 || (len + tok_per_item - 1) / tok_per_item > p.n_levels)   // not monotone, or longer than the max_len given
      rc_set_status(p.status, RECACHE_DEV_BAD_SEQLENS);
    sum += n_items_of(b);
  }
#pragma unroll 1
  for (int i = tid; i <= RC_PLAN_BINS; i += n_thr) sh.hist[i] = 0;
  int k = rc_plan_scan(sum, sh, &total);
  const int n_items = min(total, p.max_items), n_work = n_items * p.G;
  // (an encode launch shares K/V between the items of a sequence only: beyond a thousand items the
  // sequence-major order, which keeps a sequence's K/V in L2, is worth more than the balance)
  const bool sorted = n_work <= (p.route_cu ? RC_SORT_MAX : RC_SORT_MAX / 4);
  if (tid == 0) { p.header[0] = n_items; p.header[1] = 0; p.header[2] = sorted ? 1 : 0; p.header[3] = 0; }
  if (!sorted) {
    // counting sort of the sequences by their number of items, longest first: hist[bin] = items of
    // that bin, then the first item index of the bin
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
      const int nt = n_items_of(b);
      if (nt > 0) atomicAdd(&sh.hist[RC_PLAN_BINS - min(nt, RC_PLAN_BINS)], nt);
    }
    __syncthreads();
    rc_plan_scan_bins(sh);
  }
#pragma unroll 1
  for (int b = b0; b < b1; ++b) {
    const int nt = n_items_of(b);
    if (nt == 0) continue;
    if (!sorted) k = atomicAdd(&sh.hist[RC_PLAN_BINS - min(nt, RC_PLAN_BINS)], nt);
#pragma unroll 1
    for (int l = nt - 1; l >= 0; --l, ++k)
      if (k < p.max_items) p.items[k] = make_int2(b, l);
  }
  if (!sorted) return;
  // Few work items (a prefill of a handful of requests): one CTA gets one or two of them, so their
  // order decides the tail.  Sort them by weight (K/V tiles), heaviest first, with a counting sort.
  if (tid == 0) { sh.most = 0; sh.blocks = 0; }
  __syncthreads();
  if (p.start)
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
      const int own = cu[b + 1] - cu[b] + (p.hist ? p.hist[b] : 0);
      atomicAdd(&sh.blocks, (max(p.route_cu[(b + 1) * p.G] - p.route_cu[b * p.G], 0) >> 8) + ((p.G * max(own, 0)) >> 8));
    }
  int32_t* tiles = p.order + RC_SORT_MAX;
#pragma unroll 1
  for (int w = tid; w < n_work; w += n_thr) {
    RcItem it;
    const int n = rc_load_item(p, w, it) ? it.n_tiles : 0;
    tiles[w] = n;
    atomicAdd(&sh.hist[RC_PLAN_BINS - min(n, RC_PLAN_BINS)], 1);
    if (p.start) atomicMax(&sh.most, n);
  }
  __syncthreads();
  if (p.start && rc_plan_split(p, sh, n_work)) return;
  rc_plan_scan_bins(sh);
#pragma unroll 1
  for (int w = tid; w < n_work; w += n_thr) p.order[atomicAdd(&sh.hist[RC_PLAN_BINS - min(tiles[w], RC_PLAN_BINS)], 1)] = w;
}
