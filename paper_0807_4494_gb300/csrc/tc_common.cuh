// PTX helpers for the tcgen05 / TMEM / bulk-copy / mbarrier machinery of sm_100-family GPUs,
// used by the tensor-core contraction (contract_tc.cu) and the torus passes (torus_gemm.cu).
#pragma once

#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace ssht {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// A-operand tiles of the contraction: 128 rows x 32 K values, 128 bytes a row and part: one part for
// the split-FP16 form (32 hi parts, 32 lo parts), two for the split-BF16 form ([h | m] and [l | 0]).
constexpr int kTileRows = 128, kTileK = 32;
constexpr int kAPart = kTileRows * kTileK * 4;

// Byte offset of element (row, kbyte) in a K-major tile with 128-byte rows in the SWIZZLE_128B
// layout: 8-row x 128-byte atoms stacked along rows, the 16-byte chunk c of row r stored at
// chunk c ^ (r mod 8).  Tiles start on 1024-byte boundaries.
__host__ __device__ __forceinline__ uint32_t sw128(int row, int kbyte) {
  return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((((kbyte >> 4) ^ row) & 7) << 4) + (kbyte & 15));
}

// Instruction descriptor: D = F32, A = B = BF16 (kind::f16), both K-major, shape M x N.
__device__ __forceinline__ uint32_t idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Instruction descriptor: D = F32, A = B = FP16 (kind::f16), both K-major, shape M x N.
__device__ __forceinline__ uint32_t idesc_f16(int m, int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Orders this thread's shared-memory writes (generic proxy) before later reads of the tensor core
// (async proxy).
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The same without suspending the thread (try_wait may hold it until the phase completes).
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}

// Bounded wait for the phase of the given parity: false once limit_ns of device time has passed
// (checked after every poll) or, if abort is not null, once *abort is set (every 256 polls).  Limits below
// 10 us poll without suspending, so that a wait cannot outlast them inside one try_wait.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort, long long limit_ns) {
  const uint32_t b = smem_u32(bar);
  const bool brief = limit_ns < 10000;
  if (brief ? mbar_poll(b, parity) : mbar_test(b, parity)) return true;
  const unsigned long long t0 = globaltimer();
  for (unsigned i = 1;; ++i) {
    if (brief ? mbar_poll(b, parity) : mbar_test(b, parity)) return true;
    if ((i & 255u) == 0u && abort && *abort) return false;
    if ((long long)(globaltimer() - t0) > limit_ns) return false;
  }
}

// Waits for work this CTA has already issued (bulk copies, tensor-core operations) before it
// leaves: not cut short by the abort flag, bounded by two seconds.
constexpr long long kDrainNs = 2000000000ll;

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Thread-block clusters: the rank in the cluster, a peer's shared-memory address, a barrier of the
// whole cluster, and an arrival on a peer's mbarrier.  The arrival carries no ordinary memory accesses
// with it (what it announces are finished tensor-memory loads and finished bulk copies): its default
// scope is the CTA, because a release at cluster scope waits 1300 - 1800 clocks for the arriving
// thread's earlier accesses, which made it the longest step of the pipeline.
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_peer(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// 1-D bulk copy global -> shared, completion counted in bytes on an mbarrier.
// Both addresses 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// 1-D bulk copy shared -> global, tracked by the issuing thread's bulk groups (same alignment rules).
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until at most N of this thread's newest bulk groups still read their shared memory.
template <int N> __device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The forms for a pair of CTAs of a cluster (cta_group::2): both allocate and free together, the
// leader (rank 0) issues products of 256 rows -- 128 a CTA, each CTA holding its rows of A, half of the
// rows of B and its rows of D -- and their completion arrives at the same barrier of both CTAs.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
// kind::f16, one CTA or a pair.  The shared-memory matrix descriptors (SWIZZLE_128B, version 1, 1024 bytes between
// 8-row groups, the leading offset unused for swizzled K-major tiles) are given by their low words -- the
// start address in 16-byte units, kDescLow added -- so that stepping through a tile is one addition.
constexpr uint32_t kDescLow = 1u << 16, kDescHigh = (1024u >> 4) | (1u << 14) | (2u << 29);
template <bool PAIR>
__device__ __forceinline__ void mma_f16_lo(uint32_t dtmem, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t accum) {
  if constexpr (PAIR)
    asm volatile("{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n mov.b64 da, {%1, %4};\n mov.b64 db, {%2, %4};\n"
                 " tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, p;\n}\n"
                 ::"r"(dtmem), "r"(alo), "r"(blo), "r"(idesc), "r"(kDescHigh), "r"(accum));
  else
    asm volatile("{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n mov.b64 da, {%1, %4};\n mov.b64 db, {%2, %4};\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}\n"
                 ::"r"(dtmem), "r"(alo), "r"(blo), "r"(idesc), "r"(kDescHigh), "r"(accum));
}
// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
  return ok != 0;
}
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

// Moves registers between the warpgroups of a CTA (every warp of the warpgroup executes it): N a
// thread from here on.  The shares must add up to at most what the CTA was launched with.
template <int N> __device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }

// Arrive on an mbarrier once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 32 lanes x 32 bits, 16 consecutive columns per thread; tmem_wait_ld before the values are used.
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The power of two that brings a block's largest magnitude amax to [2^14, 2^15), and the scale that
// undoes it, with a 2^-14 of the other operand's range folded in (below 2^-126 a denormal number).
// Magnitudes below 2^-112 share 2^127, which leaves the smallest normal number 2^1 and so both of its parts
// whole; an infinity or a NaN stays what it is in the parts.
__device__ __forceinline__ float block_power(float amax, float* scale) {
  const int e = min(max((int)(__float_as_uint(amax) >> 23), 14), 254);
  *scale = __uint_as_float(e > 28 ? (uint32_t)(e - 28) << 23 : 1u << (e - 6));
  return __uint_as_float((uint32_t)(268 - e) << 23);
}

// x = hi + lo with both parts FP16, rounded to nearest (the remainder x - hi is exact in FP32): 22 to
// 24 significant bits while lo is a normal number.  Two values at a time.
__device__ __forceinline__ void split2(float a, float b, uint32_t* hi, uint32_t* lo) {
  const __half2 h = __floats2half2_rn(a, b);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
  *hi = *reinterpret_cast<const uint32_t*>(&h);
  *lo = *reinterpret_cast<const uint32_t*>(&l);
}

// The A operand's power of two: |U Delta| <= sqrt(4095 / 4 pi) < 18.1 up to L = 2048.
constexpr float kAScale = 1024.f;

// x = h + m + l with each part rounded to BF16 (8 significant bits, round to nearest): the three
// parts carry about 24 significant bits of x; each remainder is exact in FP32.
__device__ __forceinline__ void split_bf16x3(float x, uint16_t* h, uint16_t* m, uint16_t* l) {
  const __nv_bfloat16 a = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(a);
  const __nv_bfloat16 b = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(b);
  const __nv_bfloat16 c = __float2bfloat16_rn(r2);
  *h = __bfloat16_as_ushort(a);
  *m = __bfloat16_as_ushort(b);
  *l = __bfloat16_as_ushort(c);
}

// Parts of an operand tile: 1 for split-FP16, 2 for split-BF16.
template <bool BF> constexpr int kParts = BF ? 2 : 1;

// Writes an A operand's x at the byte offset off = sw128(row, 2k) of its first part.  Split-FP16: hi, and
// lo 64 bytes further on in the row (the swizzle flips bit 6 with it), of x times kAScale.  Split-BF16:
// h and m likewise, l in the second part (whose other half stays zero).
template <bool BF>
__device__ __forceinline__ void put_parts(uint8_t* tile, int part_bytes, uint32_t off, float x) {
  if constexpr (BF) {
    uint16_t h, m, l;
    split_bf16x3(x, &h, &m, &l);
    *(uint16_t*)(tile + off) = h;
    *(uint16_t*)(tile + (off ^ 64u)) = m;
    *(uint16_t*)(tile + part_bytes + off) = l;
  } else {
    (void)part_bytes;
    const float y = kAScale * x;
    const __half h = __float2half_rn(y), l = __float2half_rn(y - __half2float(h));
    *(__half*)(tile + off) = h;
    *(__half*)(tile + (off ^ 64u)) = l;
  }
}

// block_power of the largest magnitude over the warp (amax >= 0, or a NaN).
__device__ __forceinline__ float warp_power(float amax, float* scale) {
  return block_power(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax))), scale);
}

// Writes two rows (j, j + 1: a field's real and imaginary part) of a data tile if `store` (warp-uniform), the
// warp's lanes holding K = lane of both (x, y): neighbouring lanes exchange a value, so that each lane splits and
// stores two K of one row (4-byte stores).  Split-FP16: of x and y times the block's power of two `up`.
// Split-BF16: three parts; the half of the second part's row that none of them fills stays as it was zeroed.
template <bool BF>
__device__ __forceinline__ void put_rows2(uint8_t* tile, int part_bytes, int j, int lane, float x, float y, float up, bool store) {
  const bool odd = lane & 1;
  const float other = __shfl_xor_sync(0xffffffffu, odd ? x : y, 1);
  const float a = odd ? other : x, b = odd ? y : other;
  const uint32_t off = sw128(j + (lane & 1), 4 * (lane >> 1));
  if constexpr (BF) {
    uint16_t h[2], m[2], l[2];
    split_bf16x3(a, &h[0], &m[0], &l[0]);
    split_bf16x3(b, &h[1], &m[1], &l[1]);
    if (!store) return;
    *(uint32_t*)(tile + off) = h[0] | (uint32_t)h[1] << 16;
    *(uint32_t*)(tile + (off ^ 64u)) = m[0] | (uint32_t)m[1] << 16;
    *(uint32_t*)(tile + part_bytes + off) = l[0] | (uint32_t)l[1] << 16;
  } else {
    uint32_t h, l;
    split2(up * a, up * b, &h, &l);
    if (!store) return;
    *(uint32_t*)(tile + off) = h;
    *(uint32_t*)(tile + (off ^ 64u)) = l;
  }
}

}  // namespace tc
}  // namespace ssht
