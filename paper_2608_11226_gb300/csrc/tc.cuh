// Blackwell (sm_103a) tensor-core primitives as inline PTX: tcgen05 MMA with
// TMEM accumulators, shared-memory matrix descriptors, TMEM allocation and
// loads, bulk copies and mbarriers.  Every wait is bounded: on timeout it
// returns false and the caller records an error instead of spinning forever.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace pe {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Swizzled K-major operand layouts (the byte address bits [4, 4+b) are
// XOR-ed with bits [7, 7+b)):
//   SW128: rows of 128 B (64 bf16), 8-row atoms of 1024 B, b = 3
//   SW64 : rows of  64 B (32 bf16), 8-row atoms of  512 B, b = 2
//   SW32 : rows of  32 B (16 bf16), 8-row atoms of  256 B, b = 1
// Element (r, k) of a tile with R rows and K columns (bf16) lives in K-block
// kb = k / KB (KB = 64, 32 or 16 elements) at byte
//   kb * R * RB + r * RB + (((k % KB) / 8) ^ ((r % 8) >> s)) * 16 + (k % 8) * 2
// with RB the row bytes and s = 0 for SW128, 1 for SW64, 2 for SW32; the atom
// base must be aligned to the atom size.
enum : uint32_t { kLayoutSW128 = 2, kLayoutSW64 = 4, kLayoutSW32 = 6 };

template <int RB>
__host__ __device__ __forceinline__ uint32_t swz_offset(int r, int k, int R) {
  static_assert(RB == 128 || RB == 64 || RB == 32, "row bytes of a swizzled layout");
  constexpr int KB = RB / 2;  // bf16 elements per row of a K-block
  const int kb = k / KB, kk = k % KB;
  const int chunk = kk / 8;
  const int phys = RB == 128 ? (chunk ^ (r & 7)) : RB == 64 ? (chunk ^ ((r >> 1) & 3)) : (chunk ^ ((r >> 2) & 1));
  return (uint32_t)(kb * R * RB + r * RB + phys * 16 + (kk % 8) * 2);
}

// The same bytes serve as an MN-major operand.  A tile stored as above with
// rows = K (samples) and contiguous elements = M or N (features) is the
// canonical MN-major swizzled layout: the 128/64/32-byte rows hold 64/32/16
// consecutive M (or N) elements of one K index, XOR-swizzled within 8-row
// atoms.  Its descriptor takes two strides: LBO = bytes between atoms that
// are adjacent along M/N (the next 64/32/16 elements), SBO = bytes between
// 8-row groups along K.

// tcgen05 shared-memory matrix descriptor, K-major, swizzled:
// start address >> 4 [0,14), leading-dim byte offset >> 4 [16,30) (unused
// for swizzled K-major), stride-dim byte offset >> 4 [32,46) (one 8-row atom),
// fixed 0b001 at [46,49), layout type [61,64).
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t saddr, uint32_t sbo_bytes, uint32_t layout) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1u << 46;
  d |= (uint64_t)(layout & 7u) << 61;
  return d;
}

// shared-memory matrix descriptor with both byte strides given (MN-major
// operands, and K-major SW32 tiles): start >> 4 at [0,14), LBO >> 4 at
// [16,30), SBO >> 4 at [32,46), 0b001 at [46,49), layout type at [61,64)
__device__ __forceinline__ uint64_t desc_strided(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes,
                                                 uint32_t layout) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1u << 46;
  d |= (uint64_t)(layout & 7u) << 61;
  return d;
}

// instruction descriptor for kind::f16 with bf16 A and B, fp32 D, both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// the same with A and/or B MN-major (bits 15 and 16 of the descriptor)
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int M, int N, int a_mn, int b_mn) {
  return idesc_bf16(M, N) | ((uint32_t)(a_mn & 1) << 15) | ((uint32_t)(b_mn & 1) << 16);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "}\n" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
}

// arrive on an mbarrier once every tcgen05 op issued so far by this thread completed
__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(mbar))
               : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// generic-proxy shared-memory writes -> visible to the async proxy (MMA, bulk copies)
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// TMEM allocation by one full warp; the base address is written to *slot
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane (32x32b shape: warp
// w reads lanes 32*(w%4) .. +31; taddr carries the lane in bits [16,32))
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// the same in two parts, so that other work runs while the load is in flight:
// tmem_get16 starts it (one at a time per buffer), tmem_got16 waits for every
// load of the thread and names the buffer, whose values must not be used before
__device__ __forceinline__ void tmem_get16(uint32_t taddr, float (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_got16(float (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                 "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])
               :
               : "memory");
}

// N chunks of 16 columns from taddr on, each loaded while f(j, values) works on
// the one before
template <int N, class F>
__device__ __forceinline__ void tmem_chunks(uint32_t taddr, F f) {
  float v[2][16];
  tmem_get16(taddr, v[0]);
#pragma unroll
  for (int j = 0; j < N; ++j) {
    tmem_got16(v[j & 1]);
    if (j + 1 < N) tmem_get16(taddr + (uint32_t)(16 * (j + 1)), v[(j + 1) & 1]);
    f(j, v[j & 1]);
  }
}

// 32 bytes of global memory in one load from L2 (32-byte aligned): a warp whose
// lanes read 32 different lines takes 32 L1 cycles per request of either
// width, so half as many as with 16-byte loads.  In the 72B PPO kernel issuing
// the h1 chunks took 4-5 k clk of a tile's 58 k; a 72B update of 32 steps went
// from 6.84 to 6.57 ms.
__device__ __forceinline__ void ld_global32(const void* p, uint4& lo, uint4& hi) {
  asm volatile("ld.relaxed.gpu.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
               : "l"(p)
               : "memory");
}

// ask L2 to fetch `bytes` (a multiple of 16) from p on (16-byte aligned; no wait)
__device__ __forceinline__ void bulk_prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// ---------------------------------------------------------------- mbarriers
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait for phase `parity` of the barrier: false after ~`cycles` SM cycles
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, long long cycles = 4000000000LL) {
  if (mbar_try_wait(b, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(b, parity)) {
    if (clock64() - t0 > cycles) return false;
  }
  return true;
}

// bulk copy global -> shared (size a multiple of 16 B, both addresses 16-B aligned);
// completion is signalled as transaction bytes on the mbarrier
__device__ __forceinline__ void bulk_g2s(void* dst_smem, const void* src_gmem, uint32_t bytes, uint64_t* mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst_smem)),
      "l"(src_gmem), "r"(bytes), "r"(smem_u32(mbar))
      : "memory");
}

// an L2 policy that keeps the lines of a copy: for weights that every CTA
// re-reads while the tile images stream past them
__device__ __forceinline__ uint64_t l2_keep() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ void bulk_g2s(void* dst_smem, const void* src_gmem, uint32_t bytes, uint64_t* mbar,
                                         uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_u32(dst_smem)),
      "l"(src_gmem), "r"(bytes), "r"(smem_u32(mbar)), "l"(policy)
      : "memory");
}

// bulk copy shared -> global (16-byte aligned, a multiple of 16 bytes), in the
// issuing thread's current bulk group
__device__ __forceinline__ void bulk_s2g(void* dst_gmem, const void* src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst_gmem), "r"(smem_u32(src_smem)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the copies of this thread's groups have read their shared memory
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// ... and have been written
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// a tile image (bytes, a multiple of 16 KB) from shared to global memory, 16 KB
// at a time, each read before the next is queued: a weight stage's copy then
// waits behind 16 KB of image at most
__device__ __forceinline__ void store_image(uint8_t* dst_gmem, const uint8_t* src_smem, uint32_t bytes) {
  for (uint32_t o = 0; o < bytes; o += 16384) {
    bulk_s2g(dst_gmem + o, src_smem + o, 16384);
    bulk_commit();
    bulk_wait_read();
  }
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// tanh of a pair of fp32 pre-activations to within kTanhUlps fp32 steps of
// tanhf: x P(x^2) / Q(x^2) with P and Q cubic, fitted to tanh on |x| <= 3.5 by
// weighted least squares.  The argument is clamped to +-3.5 first: tanh(3.5) =
// 0.99818 lies above the midpoint 0.99805 between the two largest bf16 values
// below and at one, so every |x| >= 3.5 rounds to +-1 as tanhf's result does;
// infinities clamp and NaN passes.  Over all 1.08e9 floats in [0, 3.5) it
// equals tanhf for 94%, differs by one step for 5%, by more than three for 16
// in a million, by kTanhUlps at most.
constexpr int kTanhUlps = 5;
__device__ __forceinline__ float2 tanh2_rational(float2 x) {
  asm("min.NaN.xorsign.abs.f32 %0, %0, 0f40600000;" : "+f"(x.x));  // 3.5 with x's sign
  asm("min.NaN.xorsign.abs.f32 %0, %0, 0f40600000;" : "+f"(x.y));
  const float2 s = __fmul2_rn(x, x);
  auto both = [](float c) { return make_float2(c, c); };
  float2 p = __ffma2_rn(both(6.116621e-06f), s, both(2.6453265e-03f));
  float2 q = __ffma2_rn(both(1.8635452e-04f), s, both(2.2691658e-02f));
  p = __ffma2_rn(p, s, both(0.1268055f));
  q = __ffma2_rn(q, s, both(0.46013883f));
  p = __ffma2_rn(p, s, both(1.0f));
  q = __ffma2_rn(q, s, both(1.0f));
  float2 r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(q.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(q.y));
  return __fmul2_rn(__fmul2_rn(x, p), r);
}

// tanh(v + bias) of N hidden pre-activations (one TMEM chunk of a thread's row;
// bias 16-byte aligned), rounded to bf16 and packed in pairs; the bias is added
// with the packed two-lane fp32 add (the same rounding as two adds).  A result
// can differ from bf16(tanhf(v + bias)) only where its fp32 value lies within
// kTanhUlps steps of a midpoint between two bf16 values, low half 0x8000 +-
// kTanhUlps: 11 of 65,536.  `least` takes the least of (low half - 0x8000 +
// kTanhUlps) mod 2^16 of the even and of the odd columns; tanh_exact settles
// the chunks where one is at most 2 kTanhUlps.
template <int N>
__device__ __forceinline__ void tanh_bf16(const float (&v)[N], const float* bias, uint32_t (&pk)[N / 2],
                                          uint32_t& least) {
  constexpr uint32_t kShift = (0x8000u + kTanhUlps) * 0x10001u;
  least = 0xFFFFFFFFu;
#pragma unroll
  for (int i = 0; i < N; i += 4) {
    const float4 b = *reinterpret_cast<const float4*>(bias + i);
    const float2 t = tanh2_rational(__fadd2_rn(make_float2(v[i], v[i + 1]), make_float2(b.x, b.y)));
    const float2 u = tanh2_rational(__fadd2_rn(make_float2(v[i + 2], v[i + 3]), make_float2(b.z, b.w)));
    pk[i / 2] = pack_bf16(t.x, t.y);
    pk[i / 2 + 1] = pack_bf16(u.x, u.y);
    least = __viaddmin_u16x2(__byte_perm(__float_as_uint(t.x), __float_as_uint(t.y), 0x5410), kShift, least);
    least = __viaddmin_u16x2(__byte_perm(__float_as_uint(u.x), __float_as_uint(u.y), 0x5410), kShift, least);
  }
}

__device__ __forceinline__ bool near_midpoint(uint32_t least) {
  return min(least & 0xFFFFu, least >> 16) <= 2 * kTanhUlps;
}

// Makes the activations of a warp's 32 rows (from row0 on; NJ chunks of 16
// accumulators from taddr, columns from c0 on) in the K-major buffer `act` those
// of tanhf; least[j]: tanh_bf16's of the thread's chunk j.  8% of a warp's chunks
// need it, and all warps of a tile wait for the last one, so the latency of a
// pass and the code it fetches count: one row of a chunk at a time, a lane per
// column, in one loop for all chunks.  A 72B rollout of 65,536 envs x 64 steps
// takes 3.75 ms, a Stress rollout of 262,144 x 8 4.18 ms; with tanhf for every
// value, about 18 issue slots and both sides of its branch, 4.20 and 4.63; with
// the rational alone, whose results are not tanhf's, 3.36 and 3.76.  (Settling
// each chunk before the next, 4.05 and 4.51.)
template <int R, int NJ>
__device__ __forceinline__ void tanh_exact(const uint32_t (&least)[NJ], uint32_t taddr, const float* bias, uint8_t* act,
                                           int row0, int c0) {
  uint32_t m = least[0];
#pragma unroll
  for (int j = 1; j < NJ; ++j) m = __vminu2(m, least[j]);
  if (!__any_sync(0xffffffffu, near_midpoint(m))) return;
  const int lane = threadIdx.x & 31;
  uint32_t near = 0;  // the thread's chunks to settle
#pragma unroll
  for (int j = 0; j < NJ; ++j) near |= near_midpoint(least[j]) ? 1u << j : 0u;
  for (;;) {
    const uint32_t key = __reduce_min_sync(0xffffffffu, near ? (uint32_t)(__ffs(near) << 5 | lane) : 0xFFFFFFFFu);
    if (key == 0xFFFFFFFFu) break;
    const int j = (int)(key >> 5) - 1, r = (int)(key & 31u), c = c0 + 16 * j + (lane & 15);
    float v[16], z = 0.0f;
    tmem_ld16(taddr + (uint32_t)(16 * j), v);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float x = __shfl_sync(0xffffffffu, v[i], r);
      if ((lane & 15) == i) z = x;
    }
    const __nv_bfloat16 h = __float2bfloat16_rn(tanhf(z + bias[c]));
    __syncwarp();  // after the rows' own stores
    *reinterpret_cast<__nv_bfloat16*>(act + swz_offset<128>(row0 + r, c, R)) = h;
    if (lane == r) near &= near - 1;
  }
}

}  // namespace tc
}  // namespace pe
