// What the tensor-core attention kernels (attn_tc.cu, attn_tile.cu) share: tile sizes, launch
// parameters, and the PTX they are written in.
#pragma once
#include <cuda.h>

#include "tile_plan.cuh"

namespace rc_tc {

constexpr int D = 128;
constexpr int TILE_N = RC_TILE_N;
constexpr int BOX_BYTES = 16384;   // [128 rows][64 bf16], 128-byte swizzle
constexpr int TILE_BYTES = 32768;  // two boxes: head_dim halves
constexpr uint32_t WAIT_PROBES = 1u << 21;           // ~2.8 s of suspended probes: a wait this long is a bug, not load

struct TcParams : RcPlan {
  // gather mode: route row n of group g is row route_idx[n] of gather_k / gather_v ([G][pool_tokens][128] bf16)
  const uint8_t* gather_k; const uint8_t* gather_v; const int32_t* route_idx; int64_t pool_tokens;
  void* out;
  float* part_o; float2* part_ml;   // split launch: O [slot][128 rows][128], (maximum in log2 units, sum) [slot][128 rows]
  const float* cos_tab; const float* sin_tab; int max_pos;
  float scale_log2;
};
// The tensor maps of a launch: q, own keys and values, route keys and values.
struct TcMaps { CUtensorMap q, ks, vs, kr, vr; };

// ------------------------------------------------------------------ PTX --
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
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// 16-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros instead
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(src_bytes) : "memory");
}
// one arrival on the barrier once all earlier cp.async of this thread have landed (the barrier's
// expected count already includes it)
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
// plain bulk copy global -> shared (16-byte aligned, size a multiple of 16)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A * B with A in shared memory (mma_ss) or tensor memory (mma_ts); the 64-bit shared
// memory descriptors advance by adds on their address field.
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(d), "r"(a), "l"(db), "r"(idesc), "r"(acc) : "memory");
}
// one lane of a fully converged warp, chosen by the hardware
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}

#define RC_R32(r, o) "=r"(r[o + 0]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), \
    "=r"(r[o + 6]), "=r"(r[o + 7]), "=r"(r[o + 8]), "=r"(r[o + 9]), "=r"(r[o + 10]), "=r"(r[o + 11]),               \
    "=r"(r[o + 12]), "=r"(r[o + 13]), "=r"(r[o + 14]), "=r"(r[o + 15]), "=r"(r[o + 16]), "=r"(r[o + 17]),           \
    "=r"(r[o + 18]), "=r"(r[o + 19]), "=r"(r[o + 20]), "=r"(r[o + 21]), "=r"(r[o + 22]), "=r"(r[o + 23]),           \
    "=r"(r[o + 24]), "=r"(r[o + 25]), "=r"(r[o + 26]), "=r"(r[o + 27]), "=r"(r[o + 28]), "=r"(r[o + 29]),           \
    "=r"(r[o + 30]), "=r"(r[o + 31])
#define RC_W32(r, o) "r"(r[o + 0]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]),       \
    "r"(r[o + 6]), "r"(r[o + 7]), "r"(r[o + 8]), "r"(r[o + 9]), "r"(r[o + 10]), "r"(r[o + 11]), "r"(r[o + 12]),      \
    "r"(r[o + 13]), "r"(r[o + 14]), "r"(r[o + 15]), "r"(r[o + 16]), "r"(r[o + 17]), "r"(r[o + 18]), "r"(r[o + 19]),  \
    "r"(r[o + 20]), "r"(r[o + 21]), "r"(r[o + 22]), "r"(r[o + 23]), "r"(r[o + 24]), "r"(r[o + 25]), "r"(r[o + 26]),  \
    "r"(r[o + 27]), "r"(r[o + 28]), "r"(r[o + 29]), "r"(r[o + 30]), "r"(r[o + 31])
#define RC_LIST32_OUT "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}"
#define RC_LIST32_IN "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32}"

// 32 consecutive columns of this thread's lane
#define TMEM_LD32(taddr, r, o) \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 " RC_LIST32_OUT ", [%32];" : RC_R32(r, o) : "r"(taddr) : "memory")
#define TMEM_ST32(taddr, r, o) \
  asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], " RC_LIST32_IN ";" ::"r"(taddr), RC_W32(r, o) : "memory")

#define TMEM_LD16(taddr, r) \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];" \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), \
                 "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr) : "memory")

#define TMEM_ST16(taddr, r) \
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" \
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), \
                 "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory")

// one 32-byte store (the address is 32-byte aligned)
__device__ __forceinline__ void st_global_v8(void* ptr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e, uint32_t f,
                                             uint32_t g, uint32_t h) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(ptr), "r"(a), "r"(b), "r"(c), "r"(d), "r"(e),
               "r"(f), "r"(g), "r"(h) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Shared-memory matrix descriptors, 128-byte swizzle, 8-row groups 1024 bytes apart.
//  K-major operand (rows = M or N index, 64 bf16 of K per 128-byte row): SBO = 1024.
//  MN-major operand (rows = K index, 64 bf16 of N per row): SBO = 1024 between 8-row
//  K groups, LBO = distance between 64-wide N chunks.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32) | (1ull << 46) | (2ull << 61);
}
// kind::f16 instruction descriptor: fp32 accumulate, bf16 A and B, M = 128, N = 128
constexpr uint32_t IDESC_BASE = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t IDESC_QK = IDESC_BASE;               // A, B K-major
constexpr uint32_t IDESC_QK64 = IDESC_BASE - ((64u >> 3) << 17);   // N = 64
constexpr uint32_t IDESC_PV = IDESC_BASE | (1u << 16);  // B (= V) MN-major

// Packed fp32 pairs (one instruction, two lanes of the FMA pipe).  Operands that many share, and sums, are kept as pairs.
__device__ __forceinline__ uint64_t pair2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, uint64_t b, uint64_t c) {
  asm("{\n\t.reg .b64 ra, rd;\n\tmov.b64 ra, {%2, %3};\n\tfma.rn.f32x2 rd, ra, %4, %5;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "l"(b), "l"(c));
}
__device__ __forceinline__ void add2(uint64_t& d, float a0, float a1) {
  asm("{\n\t.reg .b64 ra;\n\tmov.b64 ra, {%1, %2};\n\tadd.rn.f32x2 %0, %0, ra;\n\t}" : "+l"(d) : "f"(a0), "f"(a1));
}
// the sum of two pairs, (a0 + a1) + (b0 + b1)
__device__ __forceinline__ float sum4(uint64_t a, uint64_t b) {
  float a0, a1, b0, b1;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a0), "=f"(a1) : "l"(a));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(b0), "=f"(b1) : "l"(b));
  return (a0 + a1) + (b0 + b1);
}
// d = a * b + c and d = a * b on pairs (one instruction each; same rounding as the scalar forms)
__device__ __forceinline__ void fma2v(float& d0, float& d1, float a0, float a1, float b0, float b1, float c0, float c1) {
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void mul2v(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&p);
}
// Rotates eight elements and their partners (64 further on, in the tile's other box) of a query row in
// shared memory.
__device__ __forceinline__ void rotate_chunk(uint8_t* qb, const float* cs, const float* sn) {
  const uint4 ulo = *reinterpret_cast<uint4*>(qb), uhi = *reinterpret_cast<uint4*>(qb + BOX_BYTES);
  const uint32_t wlo[4] = {ulo.x, ulo.y, ulo.z, ulo.w}, whi[4] = {uhi.x, uhi.y, uhi.z, uhi.w};
  uint32_t ol[4], oh[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float l0 = __uint_as_float(wlo[i] << 16), l1 = __uint_as_float(wlo[i] & 0xffff0000u);
    const float h0 = __uint_as_float(whi[i] << 16), h1 = __uint_as_float(whi[i] & 0xffff0000u);
    // lo' = lo cos - hi sin, hi' = hi cos + lo sin: the products with sin are rounded first
    // (hi * (-sin) is exactly -(hi * sin)), as in the scalar form of the other kernels
    float t0, t1, u0, u1, a0, a1, b0, b1;
    mul2v(t0, t1, h0, h1, -sn[2 * i], -sn[2 * i + 1]);
    mul2v(u0, u1, l0, l1, sn[2 * i], sn[2 * i + 1]);
    fma2v(a0, a1, l0, l1, cs[2 * i], cs[2 * i + 1], t0, t1);
    fma2v(b0, b1, h0, h1, cs[2 * i], cs[2 * i + 1], u0, u1);
    ol[i] = pack2(a0, a1);
    oh[i] = pack2(b0, b1);
  }
  *reinterpret_cast<uint4*>(qb) = make_uint4(ol[0], ol[1], ol[2], ol[3]);
  *reinterpret_cast<uint4*>(qb + BOX_BYTES) = make_uint4(oh[0], oh[1], oh[2], oh[3]);
}

using Item = RcItem;

}  // namespace rc_tc

// The attention with one query tile to a work item, and the merge of the parts of a split launch (attn_tile.cu).
cudaError_t rc_launch_attn_tile(const recache_ctx* ctx, const rc_tc::TcMaps& m, const rc_tc::TcParams& p, bool f32, bool split,
                                unsigned grid, cudaStream_t st);
