// Attention in exact fp32 arithmetic (no tensor cores, accurate expf): the fp32
// path of encode and prefill, and the bf16 shapes that the tensor-core kernel
// does not cover.
//
// One CTA owns a block of up to 8 query rows (8 / s consecutive tokens of a
// sequence x the s query heads of a group).  The keys are dealt in tiles of 32 to
// eight parts (tile t belongs to part t % 8), each with an online softmax of its
// own over all its tiles; the parts' (max, sum, O) are merged through shared
// memory at the end, so nothing synchronises in between.  A warp computes a part,
// or two warps four each: where there are blocks enough to fill the GPU many times
// and keys for a few tiles only, eight warps mostly wait for one of them.  For the
// scores four lanes share a key's row, so that a warp's 16-byte loads touch 8 lines, not
// 32 (with a key to a lane the loads' tag lookups alone took 512 cycles a tile),
// and a query load from shared memory serves 16 FMA; for P V a lane owns d / 32 columns and the
// probabilities are broadcast, with the value rows loaded eight at a time ahead
// of their use.  At the few hundred rows of the calls made in earnest half the time
// is a block's start (a chain of dependent loads) and half FMA issue.  A warp per
// query row, which read every key row once per query row, took 69 us each for 1,250
// tokens in six resources and for the 160-token turn over them (4 / 2 heads of 64);
// this kernel takes 20 and 11 us, and the pass of encode, compaction and turn 44 us
// instead of 155 (the rows' softmaxes one after the other, blocks light to heavy: 53;
// four warps to a CTA: 55; 16 rows to a CTA: 80).  It was the faster one for hundreds of
// sequences of up to 32 keys (1000 of 1-8 29 us there, 37 here; of 17-32 147 and 146, 32 / 8 heads of 128 1907 and 2110).
//
// Key set of a row (token t of sequence b at local index j, head h, group g):
//   route part : rows route_cu[b*G+g] .. route_cu[b*G+g+1]-1 of k_route/v_route,
//                all visible (prefill only)
//   self part  : rows base(b) .. base(b)+j of k_self[g]/v_self[g] (causal);
//                base = slot[b] for encoding (cache rows of the resource),
//                cu[b] for prefill (rotated conversation keys).
// The query is rotated on load at position pos0[b] + j (0 + j for encoding).
// Blocks and tiles are aligned to the sequence, never to the batch: results do
// not depend on what else is in the launch.
#include <float.h>

#include <type_traits>

#include "common.cuh"

namespace {

constexpr int PARTS = 8, ROWS = 8, KT = 32, VB = 8;    // PARTS: key tile t belongs to part t % PARTS of its row; VB: value rows loaded at a time

// N consecutive elements as floats, N * sizeof(T) a multiple of 4
template <typename T, int N> __device__ __forceinline__ void load_f(const T* p, float* f);
template <> __device__ __forceinline__ void load_f<float, 2>(const float* p, float* f) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  f[0] = v.x; f[1] = v.y;
}
template <> __device__ __forceinline__ void load_f<float, 4>(const float* p, float* f) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
template <> __device__ __forceinline__ void load_f<float, 8>(const float* p, float* f) {
  load_f<float, 4>(p, f); load_f<float, 4>(p + 4, f + 4);
}
template <> __device__ __forceinline__ void load_f<__nv_bfloat16, 2>(const __nv_bfloat16* p, float* f) {
  const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
  f[0] = __uint_as_float(w << 16); f[1] = __uint_as_float(w & 0xffff0000u);
}
template <> __device__ __forceinline__ void load_f<__nv_bfloat16, 4>(const __nv_bfloat16* p, float* f) {
  load_f<__nv_bfloat16, 2>(p, f); load_f<__nv_bfloat16, 2>(p + 2, f + 2);
}
template <> __device__ __forceinline__ void load_f<__nv_bfloat16, 8>(const __nv_bfloat16* p, float* f) {
  const uint4 v = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(w[i] << 16); f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
}

template <int D> struct Smem {
  float q[ROWS][D];
  union Part {
    float p[KT][ROWS];                                   // probabilities of the tile at hand, key-major
    float o[ROWS][D];                                    // at the end: the part's O
  } part[PARTS];
  float m[PARTS][ROWS], l[PARTS][ROWS];
};

// WARPS warps to a CTA, each of which takes PARTS / WARPS parts, one after the other: which warp computes a
// part makes no difference to any result.
template <typename T, typename TO, int D, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 16 / WARPS) attn_rows_kernel(
    const T* q, TO* __restrict__ o, const int32_t* cu, int n_seq, int total,
    const int32_t* pos0, const int32_t* slot,
    const T* k_self, const T* v_self, int64_t self_rows,
    const T* k_route, const T* v_route, const int32_t* route_cu,
    int prefix_len, const int32_t* hist, int64_t route_rows, int Hq, int G, const float* __restrict__ cos_tab, const float* __restrict__ sin_tab, int max_pos,
    float scale, int32_t* status) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  Smem<D>& sh = *reinterpret_cast<Smem<D>*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = Hq / G, TQ = ROWS / s, g = blockIdx.y;
  rc_grid_wait();
  rc_grid_launch_next();

  // Block index -> (sequence, block of it).  Sequence b's blocks start at cu[b] / TQ + b, which leaves
  // every sequence at least the ceil(len / TQ) it needs.
  // (32 boundaries are probed at a time: the block's start is a chain of dependent loads and little else)
  const int x = gridDim.x - 1 - blockIdx.x;              // the last blocks of a sequence have the most keys: they begin first
  int b = 0;
  for (int width = n_seq; width > 1;) {
    const int step = (width + 31) >> 5, at = b + lane * step;
    const bool le = lane * step < width && (lane == 0 || cu[at] / TQ + at <= x);
    const int last = 31 - __clz(__ballot_sync(0xffffffffu, le));      // (the boundaries ascend)
    b += last * step;
    width = min(step, width - last * step);
  }
  const int seq0 = cu[b], L = cu[b + 1] - seq0, n_cu = cu[n_seq];
  const int slot_b = slot ? slot[b] : 0, hist_b = hist ? hist[b] : 0, pos_b = pos0 ? pos0[b] : 0;
  const int route0 = route_cu ? route_cu[b * G + g] : g * prefix_len, route1 = route_cu ? route_cu[b * G + g + 1] : route0 + prefix_len;
  if (x == 0 && g == 0 && threadIdx.x == 0 && n_cu < total) rc_set_status(status, RECACHE_DEV_BAD_SEQLENS);
  const int tok0 = (x - (seq0 / TQ + b)) * TQ;           // first token of the block, local
  if (seq0 < 0 || L < 0 || seq0 + L > total) { if (threadIdx.x == 0) rc_set_status(status, RECACHE_DEV_BAD_SEQLENS); return; }
  if (tok0 < 0 || tok0 >= L) return;
  const int64_t base = slot ? (int64_t)slot_b : (int64_t)seq0;
  const int H = hist_b;                  // earlier-turn rows at the start of the self part, all visible
  const int p0 = pos_b;
  // tokens that can be computed: inside the sequence, the rotary table and the cache
  int n_tok = min(TQ, L - tok0);
  if (base < 0 || H < 0 || base + H + tok0 + n_tok > self_rows) {
    if (threadIdx.x == 0) rc_set_status(status, RECACHE_DEV_BAD_SLOT);
    n_tok = base < 0 || H < 0 ? 0 : (int)min((int64_t)n_tok, max((int64_t)0, self_rows - base - H - tok0));
  }
  if (p0 + tok0 < 0 || p0 + tok0 + n_tok > max_pos) {
    if (threadIdx.x == 0) rc_set_status(status, RECACHE_DEV_BAD_POS);
    n_tok = p0 + tok0 < 0 ? 0 : min(n_tok, max(0, max_pos - p0 - tok0));
  }
  if (n_tok <= 0) return;
  const int n_rows = n_tok * s;                          // row r = (token tok0 + r / s, head g * s + r % s)

  // ---- rotated query rows, rounded to the storage dtype like the cached keys ----
  constexpr int HALF = D / 2;
  for (int e = threadIdx.x; e < ROWS * HALF; e += WARPS * 32) {
    const int r = e / HALF, i = e % HALF;
    float ol = 0.f, oh = 0.f;
    if (r < n_rows) {
      const T* qrow = q + ((int64_t)(seq0 + tok0 + r / s) * Hq + g * s + r % s) * D;
      const int64_t at = (int64_t)(p0 + tok0 + r / s) * HALF + i;
      const float l = rc_to_float<T>(qrow[i]), h = rc_to_float<T>(qrow[i + HALF]), c = cos_tab[at], sn = sin_tab[at];
      ol = rc_to_float<T>(rc_from_float<T>(__fmaf_rn(l, c, -__fmul_rn(h, sn))));
      oh = rc_to_float<T>(rc_from_float<T>(__fmaf_rn(h, c, __fmul_rn(l, sn))));
    }
    sh.q[r][i] = ol; sh.q[r][i + HALF] = oh;
  }
  __syncthreads();

  // ---- the row's keys: the route's packed rows, or (encoding behind a shared prefix) the group's prefix
  // rows; then the sequence's own.  A range outside the route tensors (e.g. after a compaction that
  // overflowed its capacity) is reported and read as an empty route. ----
  int n_route = 0;
  if (route_cu || prefix_len > 0) {
    if (route0 >= 0 && route1 >= route0 && (int64_t)route1 <= route_rows) n_route = route1 - route0;
    else if (threadIdx.x == 0) rc_set_status(status, RECACHE_DEV_OVERFLOW);
  }
  const int n_self = H + tok0 + n_tok, route_tiles = (n_route + KT - 1) / KT, n_tiles = route_tiles + (n_self + KT - 1) / KT;
  const int n_parts = min(PARTS, n_tiles);               // the others have no tile

  constexpr int CPL = D / 32;   // output columns per lane: CPL * lane ..
  for (int w = warp; w < n_parts; w += WARPS) {
    float acc[ROWS][CPL], m[ROWS], l[ROWS];              // l: this lane's keys only
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
      for (int c = 0; c < CPL; ++c) acc[r][c] = 0.f;
    }
    float (*ps)[ROWS] = sh.part[w].p;
    for (int t = w; t < n_tiles; t += PARTS) {
      const bool own = t >= route_tiles;                 // a tile of the sequence's own keys
      const int k0 = (own ? t - route_tiles : t) * KT, n = own ? n_self : n_route;
      const int64_t row0 = own ? (int64_t)g * self_rows + base : (int64_t)route0;
      const T* kb = (own ? k_self : k_route) + row0 * D;
      const T* vb = (own ? v_self : v_route) + row0 * D;
      const int all_see = own ? H + tok0 + 1 : n;        // keys that every row of the block sees
      const int cnt = min(KT, n - k0);
      // ---- scores: four lanes share eight keys' rows, each a quarter of their 16-byte chunks ----
      const int part = lane & 3, key8 = lane >> 2;
      float sc[4][ROWS];                                 // [keys 8 kg + key8][row], this lane's chunks only
#pragma unroll
      for (int kg = 0; kg < 4; ++kg)
#pragma unroll
        for (int r = 0; r < ROWS; ++r) sc[kg][r] = 0.f;
      constexpr int EPC = 16 / (int)sizeof(T);
      const T* kp[4];
#pragma unroll
      for (int kg = 0; kg < 4; ++kg) kp[kg] = kb + (int64_t)min(k0 + 8 * kg + key8, n - 1) * D + part * EPC;
#pragma unroll 2
      for (int i = 0; i < D; i += 4 * EPC) {
        float kv[4][EPC];
#pragma unroll
        for (int kg = 0; kg < 4; ++kg) load_f<T, EPC>(kp[kg] + i, kv[kg]);
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
          for (int e = 0; e < EPC; e += 4) {
            const float4 a = *reinterpret_cast<const float4*>(&sh.q[r][i + part * EPC + e]);
#pragma unroll
            for (int kg = 0; kg < 4; ++kg) {
              sc[kg][r] = fmaf(kv[kg][e], a.x, sc[kg][r]); sc[kg][r] = fmaf(kv[kg][e + 1], a.y, sc[kg][r]);
              sc[kg][r] = fmaf(kv[kg][e + 2], a.z, sc[kg][r]); sc[kg][r] = fmaf(kv[kg][e + 3], a.w, sc[kg][r]);
            }
          }
      }
      // the four lanes' sums, scattered: lane `part` keeps the keys of kg = part
      const int mine = 8 * part + key8, kk = k0 + mine;
      const bool b0 = part & 1, b1 = part & 2;
      float v1[ROWS];
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        float u[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          u[h] = (b0 ? sc[2 * h + 1][r] : sc[2 * h][r]) + __shfl_xor_sync(0xffffffffu, b0 ? sc[2 * h][r] : sc[2 * h + 1][r], 1);
        v1[r] = (b1 ? u[1] : u[0]) + __shfl_xor_sync(0xffffffffu, b1 ? u[0] : u[1], 2);
      }
      // the first value rows are on their way while the softmax runs
      const T* vp = vb + (int64_t)k0 * D + CPL * lane;
      float vn[VB][CPL];
      auto load_v = [&](int j0) {
#pragma unroll
        for (int j = 0; j < VB; ++j) load_f<T, CPL>(vp + (int64_t)min(j0 + j, cnt - 1) * D, vn[j]);   // (past the end: a repeat, with p = 0)
      };
      load_v(0);
      // ---- online softmax (a key past the row's own token, or past the end, counts as -inf); the rows
      // go through each step together, so that their shuffles and exponentials overlap ----
      float mx[ROWS];
      int tok = 0, head = 0;                             // of row r
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int lim = own ? min(n, H + tok0 + tok + 1) : n;
        if (++head == s) { head = 0; ++tok; }
        mx[r] = v1[r] = kk < lim ? v1[r] * scale : -INFINITY;
      }
#pragma unroll
      for (int off = 16; off; off >>= 1)
#pragma unroll
        for (int r = 0; r < ROWS; ++r) mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], off));
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const float m_new = fmaxf(m[r], mx[r]), m_use = m_new == -INFINITY ? 0.f : m_new;
        const float f = expf(m[r] - m_use);              // 0 as long as nothing was seen
        v1[r] = expf(v1[r] - m_use);
        m[r] = m_new;
        l[r] = l[r] * f + v1[r];
#pragma unroll
        for (int c = 0; c < CPL; ++c) acc[r][c] *= f;
      }
#pragma unroll
      for (int r = 0; r < ROWS; r += 4) *reinterpret_cast<float4*>(&ps[mine][r]) = make_float4(v1[r], v1[r + 1], v1[r + 2], v1[r + 3]);
      __syncwarp();
      // ---- O += P V ----
#pragma unroll
      for (int j0 = 0; j0 < KT; j0 += VB) {
        if (j0 >= cnt) break;
        float v[VB][CPL];
#pragma unroll
        for (int j = 0; j < VB; ++j)
#pragma unroll
          for (int c = 0; c < CPL; ++c) v[j][c] = vn[j][c];
        if (j0 + VB < cnt) load_v(j0 + VB);
        if (k0 + j0 + VB > all_see) {
          // some row does not see the last of these keys (or they are repeats past the end): its p = 0 would
          // make NaN of an infinite value, so such values are taken out and added for the rows that see them
          bool odd = false;
#pragma unroll
          for (int j = 0; j < VB; ++j)
#pragma unroll
            for (int c = 0; c < CPL; ++c)
              if (k0 + j0 + j >= all_see && !(fabsf(v[j][c]) <= FLT_MAX)) { v[j][c] = 0.f; odd = true; }
          if (odd) {
#pragma unroll 1
            for (int j = max(all_see - k0, j0); j < min(j0 + VB, cnt); ++j) {
              float u[CPL];
              load_f<T, CPL>(vp + (int64_t)j * D, u);
#pragma unroll
              for (int c = 0; c < CPL; ++c) {
                if (fabsf(u[c]) <= FLT_MAX) continue;
#pragma unroll
                for (int r = 0; r < ROWS; ++r)
                  if (k0 + j <= H + tok0 + r / s) acc[r][c] = fmaf(ps[j][r], u[c], acc[r][c]);
              }
            }
          }
        }
#pragma unroll
        for (int j = 0; j < VB; ++j) {
#pragma unroll
          for (int r = 0; r < ROWS; r += 4) {
            const float4 pr = *reinterpret_cast<const float4*>(&ps[j0 + j][r]);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
              acc[r][c] = fmaf(pr.x, v[j][c], acc[r][c]); acc[r + 1][c] = fmaf(pr.y, v[j][c], acc[r + 1][c]);
              acc[r + 2][c] = fmaf(pr.z, v[j][c], acc[r + 2][c]); acc[r + 3][c] = fmaf(pr.w, v[j][c], acc[r + 3][c]);
            }
          }
        }
      }
      __syncwarp();
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
#pragma unroll
      for (int off = 16; off; off >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], off);
      if (lane == 0) { sh.m[w][r] = m[r]; sh.l[w][r] = l[r]; }
#pragma unroll
      for (int c = 0; c < CPL; ++c) sh.part[w].o[r][CPL * lane + c] = acc[r][c];
    }
  }

  // ---- merge the parts ----
  __syncthreads();
  for (int r = warp; r < n_rows; r += WARPS) {
    float mw = lane < n_parts ? sh.m[lane][r] : -INFINITY, M = mw;
#pragma unroll
    for (int off = 16; off; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    const float f = mw == -INFINITY ? 0.f : expf(mw - M);
    float sum = lane < n_parts ? sh.l[lane][r] * f : 0.f;
#pragma unroll
    for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    const float inv = 1.f / sum;                         // (the self part always holds the token itself, so sum > 0)
    TO* orow = o + ((int64_t)(seq0 + tok0 + r / s) * Hq + g * s + r % s) * D;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < PARTS; ++w) {
        const float fw = __shfl_sync(0xffffffffu, f, w);
        if (w < n_parts) v = fmaf(sh.part[w].o[r][lane + 32 * c], fw, v);
      }
      orow[lane + 32 * c] = rc_from_float<TO>(v * inv);
    }
  }
}

template <typename T, typename TO>
cudaError_t launch(const recache_ctx* ctx, const AttnRowsArgs& a, cudaStream_t st) {
  const int d = ctx->desc.head_dim, Hq = ctx->desc.n_q_heads, G = ctx->desc.n_kv_heads, TQ = ROWS / (Hq / G);
  if (a.total == 0 || a.n_seq == 0) return cudaSuccess;
  const dim3 grid((unsigned)(a.total / TQ + a.n_seq), (unsigned)G);
  const float scale = (float)(1.0 / sqrt((double)d));
  RcLaunchScope scope(ctx, a.route_cu ? RC_K_PREFILL_ATTN : RC_K_ENCODE_ATTN, st);
  auto go = [&](auto kernel, size_t smem, int warps) {
    return rc_launch_overlapped(kernel, grid, warps * 32, smem, st, (const T*)a.q, (TO*)a.o, a.cu, a.n_seq, a.total, a.pos0, a.slot, (const T*)a.k_self,
                                (const T*)a.v_self, a.self_rows, (const T*)a.k_route, (const T*)a.v_route, a.route_cu, a.prefix_len, a.hist,
                                a.route_rows, Hq, G, (const float*)ctx->cos_tab, (const float*)ctx->sin_tab, ctx->desc.max_pos, scale, ctx->status);
  };
  // Two warps to a CTA (6-8 CTAs to an SM instead of 2) where the blocks fill the GPU three times over with eight and a row
  // has few keys; what the host knows of their number are averages and capacities, which is enough for a rule
  // that no result depends on.  Eight warps / two, us: 1000 resources of 33-64 tokens 601 / 288 (4 / 2 heads of 64, fp32)
  // and 6851 / 4252 (32 / 8 of 128), 300 of 128-256 739 / 531 and 8646 / 8326, but 16 of 150-1200 294 / 320 and
  // 3509 / 4057; turns of 1-8 tokens over 100 rows 107 / 87 and 945 / 1021; 236 blocks of 50 keys 14.8 / 21.5, 976 34.7 / 25.1.
  const int64_t blocks = (int64_t)grid.x * G, keys = a.total / a.n_seq / 2 + a.prefix_len + (a.route_cu ? a.route_rows / ((int64_t)a.n_seq * G) : 0) +
                                                     (a.hist ? a.self_rows / a.n_seq : 0);
  const bool few = blocks >= 6 * (ctx->sm_count > 0 ? ctx->sm_count : 148) && keys <= (d == 64 ? 200 : 96);
  auto pick = [&](auto head) {
    constexpr int D = decltype(head)::value;
    return few ? go(attn_rows_kernel<T, TO, D, 2>, sizeof(Smem<D>), 2) : go(attn_rows_kernel<T, TO, D, 8>, sizeof(Smem<D>), 8);
  };
  return d == 64 ? pick(std::integral_constant<int, 64>()) : pick(std::integral_constant<int, 128>());
}

}  // namespace

cudaError_t rc_launch_attn_rows(const recache_ctx* ctx, const AttnRowsArgs& a, cudaStream_t st) {
  if (ctx->desc.dtype == RECACHE_F32) return launch<float, float>(ctx, a, st);
  if (a.out_dtype == RECACHE_F32) return launch<__nv_bfloat16, float>(ctx, a, st);
  return launch<__nv_bfloat16, __nv_bfloat16>(ctx, a, st);
}
