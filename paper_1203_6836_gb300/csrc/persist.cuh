// Pieces of the kernels that run a chain of dependent tensor-core products of
// symmetric matrices in one launch (tf32 and tf32x3).  A product of a small
// matrix is all latency: barrier, TMA, a few MMAs, epilogue, barrier.  What was
// measured on the way here, per product at n = 66 (ld = 128):
//   per-lane row stores of every operand array           14 us
//   FP32 arrays split by converter warps on every load   12 us (1.5-3.5 thousand
//     cycles from a loaded stage to its MMAs, and at large n the shared-memory
//     pipe carries the conversion beside the MMA reads: 2.1 us per 128 x 128 x 32
//     step against 0.8)
// so the operands are stored split, once, and the epilogue stages its chunk and
// its transpose in shared memory for TMA stores: no global store is scattered, and
// none needs a proxy fence before the next product's loads.  A warp of its own issues
// and awaits those stores and arrives at the barrier.
#pragma once

#include "tc_ptx.cuh"

#include <atomic>

namespace tcx {

constexpr int kRunEpi = 256;   // warps 2-9: epilogue
// warp 0 producer, 1 MMA, 10 diagonal patches or decisions, 11 stores
constexpr int kRunThreads = 64 + kRunEpi + 64;
constexpr int kRunChunk = 32 * 1024;  // staging of one 128 x 32 chunk and its transpose

// 128 x BN output units; a stage holds 32 columns of the A rows (128) and of
// the B rows (BN), hi, then lo.  Three stages, and the staging buffers that fit
// beside them.
template <int P, int BN>
struct RunCfg {
  using C = Prec<P>;
  static constexpr int a_bytes = 128 * 128;
  static constexpr int b_bytes = BN * 128;
  static constexpr int half_bytes = a_bytes + b_bytes;
  static constexpr int stage_bytes = C::nop * half_bytes;
  static constexpr int stages = 3;
  static constexpr int bufs = BN == 32 ? 3 : BN == 64 ? 2 : 1;
  static constexpr int smem = stages * stage_bytes + bufs * kRunChunk + 1024;
};

// Unit u of the nt x nt tiling's upper triangle: tile (I, J), I <= J, and the
// first of its BN columns.  With BN = 128 the tiles of a last round that leaves
// half or three quarters of the grid idle are cut into 64- or 32-column units (n =
// 2400: 190 tiles on 152 CTAs, one round of tiles and one of 32 columns).
struct RunUnits {
  int nt, tiles, full, per, U;  // per: units per cut tile
};
template <int BN>
__device__ __forceinline__ RunUnits run_units(int ld, int G) {
  RunUnits w;
  w.nt = ld / 128;
  w.tiles = w.nt * (w.nt + 1) / 2;
  w.full = 0;
  w.per = 128 / BN;
  if (BN == 128) {
    const int F = w.tiles / G, rem = w.tiles - F * G;
    w.full = F * G;
    w.per = 4 * rem <= G ? 4 : 2 * rem <= G ? 2 : 1;
  }
  w.U = w.full + (w.tiles - w.full) * w.per;
  return w;
}
struct RunUnit {
  int I, J, c0, nc;
};
template <int BN>
__device__ __forceinline__ RunUnit run_unit(const RunUnits& w, int u) {
  RunUnit r;
  int t = u;
  r.c0 = 0;
  r.nc = 128;
  if (u >= w.full) {
    const int v = u - w.full;
    t = w.full + v / w.per;
    r.nc = 128 / w.per;
    r.c0 = (v % w.per) * r.nc;
  }
  int i = 0;
  while (t >= w.nt - i) {
    t -= w.nt - i;
    ++i;
  }
  r.I = i;
  r.J = i + t;
  return r;
}

__device__ __forceinline__ void fence_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Grid barrier: every CTA that has units adds one per phase to a counter that
// is zero at the start of the call; phase p is over when it reaches p times
// their number.  (A cluster, a power of two, may hold CTAs without units.  Nothing would
// pace them: the others could be two phases ahead, rewriting the buffers from which an
// idle one still takes its decision.  They leave at once.)  The CTAs must be co-resident
// (a cooperative launch, or a grid of one cluster).  A wait gives up after kWaitNs, or
// once another CTA has recorded an error.
__device__ __forceinline__ void run_arrive(unsigned* bar) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}
__device__ __forceinline__ bool run_wait(const unsigned* bar, unsigned target, const int* err, volatile int* abort) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
  if (v >= target) return true;
  const unsigned long long t0 = gtime();
  while (true) {
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
    if (v >= target) return true;
    if (*abort) return false;
    if (*reinterpret_cast<const volatile int*>(err) || gtime() - t0 > kWaitNs) {
      *abort = 1;
      return false;
    }
  }
}
// Whether this CTA is the last of n to leave (one thread, after it has recorded the CTA's
// error, if any).  It writes the report: whether one of them gave up is known only then.
__device__ __forceinline__ bool run_last(unsigned* left, unsigned n) {
  unsigned v;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(v) : "l"(left) : "memory");
  return v + 1 == n;
}
// Barrier of the 256 epilogue threads; epi_any: the same, true in all of them
// when `v` is in any.
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ bool epi_any(int v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.or.pred q, 1, 256, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(v)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// All but the last N committed groups of stores have read their shared-memory
// source / all writes are done.
template <int N>
__device__ __forceinline__ void tma_store_read_wait() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void tma_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// The TMA loads of one stage: 32 columns from k0 of the A rows and of the unit's B
// rows, hi and lo (map index 1 and 2).  A cut unit of a BN = 128 grid loads its rows
// in 32-row boxes (b32), so the tile is the rows the MMAs read and nothing more.
template <int P, int BN>
__device__ __forceinline__ void load_stage(uint8_t* base, uint64_t* full, const CUtensorMap (&ma)[3],
                                           const CUtensorMap (&mb)[3], const CUtensorMap (&b32)[3], const RunUnit& un,
                                           int k0) {
  using Q = RunCfg<P, BN>;
  const int yb = un.J * 128 + un.c0;
  mbar_expect_tx(full, Q::C::nop * (Q::a_bytes + un.nc * 128));
#pragma unroll
  for (int h = 0; h < Q::C::nop; ++h) {
    uint8_t* t = base + h * Q::half_bytes;
    tma_load_2d(t, &ma[1 + h], full, k0, un.I * 128);
    if (BN < 128 || un.nc == 128) {
      tma_load_2d(t + Q::a_bytes, &mb[1 + h], full, k0, yb);
    } else {
      for (int b = 0; b < un.nc; b += 32) tma_load_2d(t + Q::a_bytes + b * 128, &b32[1 + h], full, k0, yb + b);
    }
  }
}

// The diagonal of a stage's operand tile (rows row0 .. row0 + rows, the 32 columns
// from k0) becomes the split of s * (id + t * d[k]) (one warp, one element a lane).
// I +- 2E and 2I - W differ from a multiple of E and W by a power of two only there,
// so their products are taken with the stored operands of E and W, this patch and a
// factor in the epilogue (exact: powers of two scale through the split and the
// sums), instead of storing them.
template <int P>
__device__ __forceinline__ void patch_diag(uint8_t* tile, int lo_off, int row0, int rows, int k0, int lane,
                                           const float* d, float id, float t, float s, int lim) {
  const int k = k0 + lane, r = k - row0;
  if (r < 0 || r >= rows || k >= lim) return;
  const float v = s * (id + t * __ldcg(d + k)), h = to_tf32(v);
  uint8_t* p = tile + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4;
  *reinterpret_cast<float*>(p) = h;
  if constexpr (Prec<P>::split) *reinterpret_cast<float*>(p + lo_off) = to_tf32(v - h);
}

// The MMAs of one stage (lo: descriptor of its first byte): a K-slice of 32, in the
// order of the stored-split kernels (hi hi, hi lo, lo hi, and lo lo for a square), so
// the sums round alike.
template <int P, int BN>
__device__ __forceinline__ void stage_mma(uint32_t lo, uint32_t d, uint32_t id, bool first, bool lolo) {
  using C = Prec<P>;
  using Q = RunCfg<P, BN>;
  constexpr uint32_t kB = Q::a_bytes >> 4, kLo = Q::half_bytes >> 4;
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    const uint32_t a = lo + 2 * ks;
    umma<true>(d, sdesc_at(a), sdesc_at(a + kB), id, !(first && ks == 0));
    if constexpr (C::split) {
      umma<true>(d, sdesc_at(a), sdesc_at(a + kLo + kB), id, 1u);
      umma<true>(d, sdesc_at(a + kLo), sdesc_at(a + kB), id, 1u);
      if (lolo) umma<true>(d, sdesc_at(a + kLo), sdesc_at(a + kLo + kB), id, 1u);
    }
  }
}

// A 128 x 32 chunk of an off-diagonal tile and its transpose, 16 columns of one
// row per epilogue thread (row 32 q + lane, columns 16 half ..), into the staging
// buffer in the layout of the 128-byte-swizzled boxes.  Free of bank conflicts.
__device__ __forceinline__ void stage_chunk(uint8_t* st, const float (&y)[16], int q, int half, int lane) {
  const int row = 32 * q + lane;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    *reinterpret_cast<float4*>(st + row * 128 + (((4 * half + j) ^ (row & 7)) << 4)) =
        make_float4(y[4 * j], y[4 * j + 1], y[4 * j + 2], y[4 * j + 3]);
  uint8_t* m = st + 16 * 1024 + q * 4096 + (lane & 3) * 4;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int r = 16 * half + j;
    *reinterpret_cast<float*>(m + r * 128 + (((lane >> 2) ^ (r & 7)) << 4)) = y[j];
  }
}
// Its TMA stores (one thread): rows from r0, columns from c0; m128 / m32 are the
// array's maps of 128- and 32-row boxes.
__device__ __forceinline__ void store_chunk(const uint8_t* st, const CUtensorMap* m128, const CUtensorMap* m32, int r0,
                                            int c0) {
  tma_store_2d(m128, st, c0, r0);
#pragma unroll
  for (int b = 0; b < 4; ++b) tma_store_2d(m32, st + 16 * 1024 + b * 4096, r0 + 32 * b, c0);
  tma_store_commit();
}
// The same for chunk k (columns 32 k ..) of a diagonal tile, of which the upper
// triangle is kept and mirrored: the 32 x 32 block on the diagonal is made
// symmetric in the staging buffer, the blocks above it are staged as above, the
// ones below are left to the chunks they mirror.
__device__ __forceinline__ void stage_chunk_diag(uint8_t* st, const float (&y)[16], int q, int half, int lane, int k) {
  if (q < k) {
    stage_chunk(st, y, q, half, lane);
  } else if (q == k) {
    uint8_t* b = st + q * 4096;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int c = 16 * half + j;
      if (c < lane) continue;
      *reinterpret_cast<float*>(b + lane * 128 + (((c >> 2) ^ (lane & 7)) << 4) + (c & 3) * 4) = y[j];
      *reinterpret_cast<float*>(b + c * 128 + (((lane >> 2) ^ (c & 7)) << 4) + (lane & 3) * 4) = y[j];
    }
  }
}
__device__ __forceinline__ void store_chunk_diag(const uint8_t* st, const CUtensorMap* m32, int r0, int k) {
  const int c0 = r0 + 32 * k;
  for (int b = 0; b <= k; ++b) {
    tma_store_2d(m32, st + b * 4096, c0, r0 + 32 * b);
    if (b < k) tma_store_2d(m32, st + 16 * 1024 + b * 4096, r0 + 32 * b, c0);
  }
  tma_store_commit();
}

// The staging buffers as a ring between the epilogue warps and the store warp; `used`
// counts the arrays each side has put through it, over the whole kernel.
struct StageRing {
  uint8_t* buf;
  uint64_t *full, *free;  // 8 epilogue warps have written / the stores have read
};
// How a chunk is stored: off the diagonal with its transpose; chunk 0-3 of a diagonal
// tile, mirrored from its upper triangle; or as it is.
constexpr int kOff = -1, kAsIs = 4;

// One array of a chunk (all 8 epilogue warps).  (After a wait that gave up the buffer is
// written all the same: the call fails, and the warps stay together.)
template <int P, int BN>
__device__ __forceinline__ void ring_put(const StageRing& r, int& used, const float (&y)[16], int q, int half, int lane,
                                         int mode, volatile int* abort, unsigned long long wl) {
  constexpr int NB = RunCfg<P, BN>::bufs;
  const int b = used % NB;
  if (used >= NB) mbar_wait_warp(&r.free[b], ((used / NB) - 1) & 1, abort, wl);
  uint8_t* st = r.buf + b * kRunChunk;
  if (mode < 0 || mode >= kAsIs) stage_chunk(st, y, q, half, lane);
  else stage_chunk_diag(st, y, q, half, lane, mode);
  fence_async_shared();
  __syncwarp();
  if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&r.full[b])) : "memory");
  ++used;
}
// hi and lo of 16 values.
template <int P, int BN>
__device__ __forceinline__ void ring_put_split(const StageRing& r, int& used, const float (&y)[16], int q, int half,
                                               int lane, int mode, volatile int* abort, unsigned long long wl) {
  float v[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = to_tf32(y[j]);
  ring_put<P, BN>(r, used, v, q, half, lane, mode, abort, wl);
  if constexpr (Prec<P>::split) {
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = to_tf32(y[j] - v[j]);
    ring_put<P, BN>(r, used, v, q, half, lane, mode, abort, wl);
  }
}
// The store warp's side (one thread): issues the array's TMA stores and frees the buffer
// whose stores have read it.
template <int P, int BN>
__device__ __forceinline__ bool ring_store(const StageRing& r, int& used, const CUtensorMap* m128,
                                           const CUtensorMap* m32, int r0, int c0, int mode, volatile int* abort,
                                           unsigned long long wl) {
  constexpr int NB = RunCfg<P, BN>::bufs;
  const int b = used % NB;
  if (!mbar_wait(&r.full[b], (used / NB) & 1, abort, wl)) return false;
  const uint8_t* st = r.buf + b * kRunChunk;
  if (mode < 0) {
    store_chunk(st, m128, m32, r0, c0);
  } else if (mode >= kAsIs) {
    tma_store_2d(m128, st, c0, r0);
    tma_store_commit();
  } else {
    store_chunk_diag(st, m32, r0, mode);
  }
  // the group before the last NB - 1 has been read
  tma_store_read_wait<NB - 1>();
  if (used >= NB - 1) {
    const int f = (used - (NB - 1)) % NB;
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&r.free[f])) : "memory");
  }
  ++used;
  return true;
}

}  // namespace tcx

// The launch of a chain over an ld x ld matrix.  Where the barrier's CTAs are
// co-resident: a grid that is one cluster (up to 16 CTAs), or a cooperative
// launch.  Captured steps run beside those of other trajectories, where a grid
// that waits for the whole chip would hold them up: they take one cluster, a
// cooperative grid of at most half the chip (one CTA a tile), or (false) the
// launched form.  So do products of more than kRunSteps 128 x 128 x 32 steps a CTA (0.2 s
// at 0.8 us each: from ld = 33 000 on the whole chip): the waits between products last a whole
// one and give up after 2 s, and a launch is nothing beside it.
constexpr long long kRunSteps = 250000;
struct RunShape {
  int bn, grid, cluster;
};
inline bool tb_run_shape(const tb_ctx* ctx, int ld, int captured, RunShape* r) {
  const int nt = ld / 128, T = nt * (nt + 1) / 2;
  int most = tb_persistent_grid(ctx, captured ? 16 : 1 << 30);
  if (captured && T > most) {
    if (2 * T > ctx->sm_count || T > tb_persistent_grid(ctx, 1 << 30)) return false;
    most = T;
  }
  r->bn = 4 * T <= most ? 32 : 2 * T <= most ? 64 : 128;
  const int U = T * (128 / r->bn);
  r->grid = U < most ? U : most;
  r->cluster = r->grid <= 16;
  if (r->cluster) {
    int c = 1;  // a power of two: at most one round more, or CTAs that leave at once
    while (c < r->grid && 2 * c <= most) c *= 2;
    r->grid = c;
  }
  return (long long)((T + r->grid - 1) / r->grid) * (ld / 32) <= kRunSteps;
}

// Whether a cluster of 1, 2, .. 16 CTAs of one kernel fits a device: 0 not asked
// yet, 1 yes, -1 no.
struct RunFits {
  std::atomic<signed char> known[64][5];
};

// The maps of one matrix: 128-, BN- and 32-row boxes of its FP32 master, hi and lo.
template <int P, int BN>
int tb_run_maps(tb_ctx* ctx, float* m, void* hi, void* lo, int ld, CUtensorMap (&a)[3], CUtensorMap (&b)[3],
                CUtensorMap (&s)[3]) {
  void* const arr[3] = {m, hi, lo};
  for (int h = 0; h < (tcx::Prec<P>::split ? 3 : 2); ++h) {
    int rc = sp2_tc_make_map(ctx, P, arr[h], ld, &a[h], 128, 128);
    if (!rc) rc = sp2_tc_make_map(ctx, P, arr[h], ld, &s[h], 128, 32);
    if (!rc && BN == 64) rc = sp2_tc_make_map(ctx, P, arr[h], ld, &b[h], 128, BN);
    if (rc) return rc;
    if (BN != 64) b[h] = BN == 32 ? s[h] : a[h];
  }
  return TB_OK;
}

// Launches it; *ran stays 0 where no cluster of this size fits the device.
template <typename K, typename... A>
int tb_run_launch(tb_ctx* ctx, K kernel, RunFits* fits, int threads, int smem, int cluster, int grid, int* ran, cudaStream_t s,
                  const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cluster) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = grid;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    std::atomic<signed char>& known = fits->known[ctx->device & 63][31 - __builtin_clz((unsigned)grid)];
    if (!known.load()) {
      if (grid > 8) TB_CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      int fit = 0;
      if (cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg) != cudaSuccess) fit = 0;
      (void)cudaGetLastError();
      known.store(fit > 0 ? 1 : -1);
    }
    if (known.load() < 0) return TB_OK;
  } else {
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
  }
  TB_CUDA_TRY(ctx, cudaLaunchKernelEx(&cfg, kernel, args...));
  *ran = 1;
  return TB_OK;
}
