// PTX wrappers for the tcgen05 / TMA / mbarrier kernels (sm_100 family).
#pragma once

#include "common.cuh"

#include <cuda_bf16.h>

#include <type_traits>

namespace tcx {

constexpr unsigned long long kWaitNs = 2000000000ull;  // bounded waits give up after 2 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long gtime() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: true when the phase completed, false on abort/timeout (after
// limit_ns of %globaltimer time).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned long long limit_ns = kWaitNs) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = gtime();
  while (true) {
    if (mbar_try(bar, parity)) return true;
    if (*abort_flag) return false;
    if (gtime() - t0 > limit_ns) {
      *abort_flag = 1;
      return false;
    }
  }
}
// The same wait made by all 32 lanes of a warp that goes on to warp-collective
// tcgen05.ld: true only when every lane saw the phase complete, so the lanes
// break out (or go on) together even when a time limit runs out between them.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                               unsigned long long limit_ns = kWaitNs) {
  const bool ok = mbar_wait(bar, parity, abort_flag, limit_ns);
  return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (SBO), descriptor version 1.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}
// One thread of a warp, picked the way the compiler knows to be one (so that what it
// computes for tcgen05 instructions can stay in uniform registers).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// sdesc() from its low word: address / 16 and the fixed fields.
__device__ __forceinline__ uint32_t sdesc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ uint64_t sdesc_at(uint32_t lo) {
  return (static_cast<uint64_t>((1024u >> 4) | (1u << 14) | (2u << 29)) << 32) | lo;
}

// Instruction descriptor: D = F32, A/B format `fmt` (bf16 = 1, tf32 = 2),
// both K-major, N x M tile.
__host__ __device__ constexpr uint32_t idesc(uint32_t fmt, int M = 128, int N = 128) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
template <bool TF32>
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if constexpr (TF32) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
  }
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
      "[%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
        "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
        "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
        "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// ---- CTA pairs: a cluster of two CTAs sharing one tcgen05.mma.cta_group::2
// (M = 256: rows 0-127 from the even CTA's shared memory, 128-255 from the
// odd CTA's at the same offsets; B split along N the same way; each CTA
// holds its 128 rows of the accumulator in its own TMEM).  Every tcgen05
// instruction of such a kernel uses .cta_group::2.
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the object at shared::cta address `a` in CTA
// `rank` of this cluster.
__device__ __forceinline__ uint32_t mapa_rank(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// Cluster-wide barrier of all threads (release / acquire).
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t a) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(a) : "memory");
}
// TMA tile load into this CTA's shared memory, completion signalled on an
// mbarrier of either CTA of the pair (`bar`: shared::cluster address).
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], "
      "[%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
// Collective TMEM allocation / release of the pair: one warp of each CTA.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
template <bool TF32>
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if constexpr (TF32) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
  }
}
// Arrive (once each) on the mbarrier at `bar`'s offset in every CTA of
// `mask` when the pair's previously issued MMAs have completed.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                   smem_u32(bar)),
               "h"(mask)
               : "memory");
}

// 16 consecutive 32-bit columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}



// A operand in TMEM: the M x K tile's row r in lane r, one 32-bit column per tf32
// element, from column `a`; B through its shared-memory descriptor.
__device__ __forceinline__ void umma_ts_tf32(uint32_t tmem_d, uint32_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}
// 16 consecutive 32-bit columns of this warp's 32 TMEM lanes, written.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15, %16};" ::"r"(taddr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// hi = tf32(x), lo = tf32(x - hi), rounded to nearest with ties away as cvt.rna does,
// in integer instructions (an addition of half a unit to the magnitude's bits and a
// mask: 97 a clock and SM against 21 conversions).  The bits of an infinity or a NaN
// would not survive that: such values take the conversion (Any).
template <bool Any>
__device__ __forceinline__ void split_tf32(const float4& x, float4& h, float4& l) {
  auto rna = [](float v) {
    return Any ? to_tf32(v) : __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xffffe000u);
  };
  h = make_float4(rna(x.x), rna(x.y), rna(x.z), rna(x.w));
  l = make_float4(rna(x.x - h.x), rna(x.y - h.y), rna(x.z - h.z), rna(x.w - h.w));
}
// Whether 32 values are all finite (one test for all: a branch per float4 kept their
// splits from overlapping, 1050 cycles a step against 600).
__device__ __forceinline__ bool all_finite(const float4 (&x)[8]) {
  float t[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) t[j] = (x[j].x + x[j].y) + (x[j].z + x[j].w);
  const float s = ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
  return s - s == 0.0f;
}

// The FP32-staged operand pipeline of the block-sparse and grouped kernels (tf32x3):
// TMA loads the FP32 128 x 32 tiles of A and B; warps of a converter group of four turn
// A into hi and lo in TMEM (row r in lane r: 32 columns each) and another group
// turns B into hi (in place) and lo in shared memory.  What bounds such a kernel is the
// shared-memory pipe (128 bytes a clock): with both operands split in shared memory a
// K-step of 32 moved 32 KB in by TMA, 32 KB out and 64 KB in by the converters and 96-128
// KB by the MMAs, 1800-2050 cycles against 1070-1420 of MMA; with A in TMEM the MMAs read
// only B and A's split is not stored: 1150-1280.
constexpr int kFsTile = 128 * 128;          // bytes of a 128 x 32 FP32 tile
constexpr int kFsStage = 3 * kFsTile;       // A, B (then its hi), B's lo
constexpr int kFsStages = 4;
constexpr int kFsSmem = kFsStages * kFsStage + 1024;
constexpr int kFsTmemA = 256;               // first TMEM column of the A stages (64 each)
constexpr int kFsTmemCols = 512;            // two accumulators of 128, four A stages
// A converter (128 threads of warps whose index mod 4 is their TMEM lane quarter).
__device__ __forceinline__ void fs_convert_a(const uint8_t* stage, uint32_t tmem, int s, int q, int lane) {
  const int row = 32 * q + lane;
  const uint32_t ta = tmem + (static_cast<uint32_t>(32 * q) << 16) + kFsTmemA + 64 * s;
  // all loads first: one warp per scheduler works on a stage, so its own instructions
  // have to hide the latencies
  float4 x[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = *reinterpret_cast<const float4*>(stage + row * 128 + ((j ^ (row & 7)) << 4));
  auto go = [&](auto any) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      float h[16], l[16];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float4 a, b;
        split_tf32<decltype(any)::value>(x[4 * half + j], a, b);
        h[4 * j] = a.x, h[4 * j + 1] = a.y, h[4 * j + 2] = a.z, h[4 * j + 3] = a.w;
        l[4 * j] = b.x, l[4 * j + 1] = b.y, l[4 * j + 2] = b.z, l[4 * j + 3] = b.w;
      }
      tmem_st16(ta + 16 * half, h);
      tmem_st16(ta + 32 + 16 * half, l);
    }
  };
  // (the stores to TMEM are of the whole warp)
  if (__all_sync(0xffffffffu, all_finite(x))) go(std::false_type{});
  else go(std::true_type{});
  tmem_st_wait();
  tc_fence_before();
}
// B converter (128 threads, t = 0..127): elementwise, so the 128-byte swizzle is kept.
__device__ __forceinline__ void fs_convert_b(uint8_t* stage, int t) {
  float4* b = reinterpret_cast<float4*>(stage + kFsTile) + t;
  float4 x[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = b[128 * i];
  auto go = [&](auto any) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float4 h, l;
      split_tf32<decltype(any)::value>(x[i], h, l);
      b[128 * i] = h;
      b[128 * i + kFsTile / 16] = l;
    }
  };
  if (all_finite(x)) go(std::false_type{});
  else go(std::true_type{});
  // the generic-proxy stores must be visible to the tensor core's reads
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// The MMAs of one stage (lo: descriptor of its first byte), in the order of the
// stored-split kernels.
__device__ __forceinline__ void fs_mma(uint32_t lo, uint32_t tmem, int s, uint32_t d, uint32_t id, bool first,
                                       bool lolo) {
  const uint32_t ta = tmem + kFsTmemA + 64 * s;
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    const uint64_t bh = sdesc_at(lo + (kFsTile >> 4) + 2 * ks), bl = sdesc_at(lo + (2 * kFsTile >> 4) + 2 * ks);
    umma_ts_tf32(d, ta + 8 * ks, bh, id, !(first && ks == 0));
    umma_ts_tf32(d, ta + 8 * ks, bl, id, 1u);
    umma_ts_tf32(d, ta + 32 + 8 * ks, bh, id, 1u);
    if (lolo) umma_ts_tf32(d, ta + 32 + 8 * ks, bl, id, 1u);
  }
}

// A warp's 32 x 32 FP32 sub-tile (row pitch ld) between global memory and registers, lane
// l holding row l: eight 16-byte accesses a lane, each of four whole 128-byte rows, and a
// turn through 4 KB of shared memory (16-byte chunks swizzled by row: no bank
// conflicts).  A lane reading or writing its own row touches 32 lines per
// instruction, 13-18 thousand cycles for the epilogue of a 128 x 128 tile.
__device__ __forceinline__ void tile_fetch(const float* src, size_t ld, int lane, float4 (&g)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
    g[i] = *reinterpret_cast<const float4*>(src + (size_t)(4 * i + (lane >> 3)) * ld + 4 * (lane & 7));
}
__device__ __forceinline__ void tile_turn_in(uint8_t* sm, int lane, const float4 (&g)[8], float (&y)[32]) {
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 4 * i + (lane >> 3);
    *reinterpret_cast<float4*>(sm + r * 128 + (((lane & 7) ^ (r & 7)) << 4)) = g[i];
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float4 v = *reinterpret_cast<const float4*>(sm + lane * 128 + ((j ^ (lane & 7)) << 4));
    y[4 * j] = v.x, y[4 * j + 1] = v.y, y[4 * j + 2] = v.z, y[4 * j + 3] = v.w;
  }
}
__device__ __forceinline__ void tile_store(uint8_t* sm, int lane, const float (&y)[32], float* dst, size_t ld) {
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j)
    *reinterpret_cast<float4*>(sm + lane * 128 + ((j ^ (lane & 7)) << 4)) =
        make_float4(y[4 * j], y[4 * j + 1], y[4 * j + 2], y[4 * j + 3]);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 4 * i + (lane >> 3);
    *reinterpret_cast<float4*>(dst + (size_t)r * ld + 4 * (lane & 7)) =
        *reinterpret_cast<const float4*>(sm + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
  }
}

// Traits of the tensor-core precisions: operand bytes, elements per 128-byte
// row (one 128B-swizzle atom), K of one MMA instruction, hi/lo split.
template <int P>
struct Prec {
  static constexpr bool tf32 = (P == TB_PREC_TF32 || P == TB_PREC_TF32X3);
  static constexpr bool split = (P == TB_PREC_TF32X3 || P == TB_PREC_BF16X3);
  static constexpr int eb = tf32 ? 4 : 2;          // operand bytes
  static constexpr int bk = 128 / eb;              // elements per 128-byte row
  static constexpr int uk = 32 / eb;               // K of one MMA instruction
  static constexpr int nop = split ? 2 : 1;        // operand arrays
  static constexpr int stage_bytes = 2 * nop * 128 * 128;
  static constexpr int stages = split ? 3 : 6;
  static constexpr int smem_bytes = stages * stage_bytes + 1024;
};

// Operand split of a row segment of 32 FP32 values into hi (and lo).
template <int P>
__device__ __forceinline__ void store_operands(const float (&y)[32], void* hi_row, void* lo_row) {
  if constexpr (Prec<P>::tf32) {
    uint4* h = reinterpret_cast<uint4*>(hi_row);
    uint4* l = reinterpret_cast<uint4*>(lo_row);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float hv[4], lv[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        hv[t] = to_tf32(y[4 * j + t]);
        lv[t] = to_tf32(y[4 * j + t] - hv[t]);
      }
      h[j] = make_uint4(__float_as_uint(hv[0]), __float_as_uint(hv[1]), __float_as_uint(hv[2]),
                        __float_as_uint(hv[3]));
      if constexpr (Prec<P>::split)
        l[j] = make_uint4(__float_as_uint(lv[0]), __float_as_uint(lv[1]), __float_as_uint(lv[2]),
                          __float_as_uint(lv[3]));
    }
  } else {
    uint4* h = reinterpret_cast<uint4*>(hi_row);
    uint4* l = reinterpret_cast<uint4*>(lo_row);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t hw[4], lw[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float a0 = y[8 * j + 2 * t], a1 = y[8 * j + 2 * t + 1];
        const __nv_bfloat16 h0 = __float2bfloat16_rn(a0), h1 = __float2bfloat16_rn(a1);
        const __nv_bfloat16 l0 = __float2bfloat16_rn(a0 - __bfloat162float(h0));
        const __nv_bfloat16 l1 = __float2bfloat16_rn(a1 - __bfloat162float(h1));
        hw[t] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        lw[t] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
      }
      h[j] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
      if constexpr (Prec<P>::split) l[j] = make_uint4(lw[0], lw[1], lw[2], lw[3]);
    }
  }
}

// Operand split of one FP32 value into hi (and lo) at element index idx.
template <int P>
__device__ __forceinline__ void store_operand1(float y, void* hi, void* lo, size_t idx) {
  if constexpr (Prec<P>::tf32) {
    const float hv = to_tf32(y);
    reinterpret_cast<uint32_t*>(hi)[idx] = __float_as_uint(hv);
    if constexpr (Prec<P>::split) reinterpret_cast<uint32_t*>(lo)[idx] = __float_as_uint(to_tf32(y - hv));
  } else {
    const __nv_bfloat16 h = __float2bfloat16_rn(y);
    reinterpret_cast<unsigned short*>(hi)[idx] = __bfloat16_as_ushort(h);
    if constexpr (Prec<P>::split)
      reinterpret_cast<unsigned short*>(lo)[idx] = __bfloat16_as_ushort(__float2bfloat16_rn(y - __bfloat162float(h)));
  }
}

}  // namespace tcx
