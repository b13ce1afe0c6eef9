// Thresholded block-sparse SP2 (row a5): the linear-scaling form of the
// purification (Sec. III.B, Table I tau > 0 rows).
//
// Reading: after X0 and after every projection, every 32 x 32 block of X whose
// Frobenius norm is below tau is set to zero (the paper drops elements below
// tau; the 32 x 32 block rule is the block-sparse reading).
//
// GB300 layout: X is stored as 128 x 128 super-blocks (one tcgen05 tile) in a
// block-sparse-row structure, ping-ponged between two buffers.  A super-block
// is stored when at least one of its sixteen 32 x 32 sub-blocks survives the
// drop rule; dropped sub-blocks inside a stored super-block hold zeros, so the
// arithmetic is the same as dropping 32 x 32 blocks.  For n <= 131072 there are
// at most 1024 super-rows and each row's pattern is a 1024-bit bitmap.
//
// Per projection (all on the device, no host synchronisation):
//   symbolic  reduce the trace partials of X_k and take the stop/branch decision
//           (every CTA the same); each row has bitmaps of its stored and its live
//           (not all-zero) super-blocks, written with the pattern and by the numeric
//           kernel; candidates of row I = OR of the live bitmaps of its live
//           columns; every block scans the rows' counts for the output slots; each upper output block
//           (I <= J; X^2 and its pattern are symmetric) gets the list of common
//           K (live in both rows I and J) as pairs of source slots; the upper
//           blocks are listed in (band of 8 block rows, column, row) order;
//   numeric  a persistent tcgen05 kernel walks that list: TMA loads the (I,K)
//           and (J,K) tiles of every pair into shared memory (tf32x3: the FP32
//           blocks, split into hi and lo by eight converter warps, A into TMEM and B in
//           place; other precisions: their stored splits), the MMA accumulates in TMEM
//           (double-buffered between blocks), the epilogue applies the branch
//           (X^2 or 2X - X^2), zeroes every 32 x 32 sub-block with ||.||_F <
//           tau (one warp owns a 32-row band, so a sub-block norm is a warp
//           reduction), writes block (I,J) and, transposed, its mirror (J,I),
//           and accumulates FP64 trace partials.
// The final iterate is written to the dense FP64 D or, with BSR input and
// output (dm_sp2_sparse), to a BSR D.
//
// The same engine computes C = alpha A B + gamma S + delta I for two
// different symmetric, commuting matrices (the candidate pattern is that of
// A B and B A together, so it is symmetric; the diagonal blocks keep their
// upper triangle and mirror it), which is what the block-sparse Fermi
// expansion (dm_fermi_sparse, row f2) is built from, with exact affine steps
// alpha X + delta I on X's pattern.

#include "common.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace {

using namespace tcx;

constexpr int SB = 128;            // super-block side (tcgen05 tile)
constexpr int MW = 32;             // bitmap words per row (1024 super-rows: n <= 131072)
constexpr int kMaxNsb = MW * 32;
constexpr int kThreads = 192;      // numeric kernel: TMA, MMA, 4 epilogue warps
// tf32x3 keeps only the FP32 master of every block: the numeric kernel loads the
// masters and eight converter warps split them, A into TMEM and B in shared memory
// (tc_ptx.cuh; the same rounding the stored splits had, so the products are bitwise
// those of stored splits), at half the operand bytes and a third of the stores
template <int P>
constexpr bool kStaged = P == TB_PREC_TF32X3;
template <int P>
constexpr int kNumThreads = kStaged<P> ? 448 : kThreads;
template <int P>
constexpr int kNumStages = kStaged<P> ? kFsStages : Prec<P>::stages;
template <int P>
constexpr int kNumStageBytes = kStaged<P> ? kFsStage : Prec<P>::stage_bytes;
template <int P>
constexpr int kNumSmem = kStaged<P> ? kFsSmem : Prec<P>::smem_bytes;
constexpr int kTiles = SB * SB;    // elements per super-block
constexpr int kMaxGrid = 256;      // cap of the persistent numeric grid (which is also at most the SM count)
constexpr int kBand = 8;           // block rows whose outputs the numeric kernel walks together

inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

struct Buf {
  int* row_ptr;      // [nsb + 1]
  int* col;          // [cap]
  uint32_t* stored;  // [nsb * MW]
  uint32_t* live;    // [nsb * MW]
  float* val;        // [cap * kTiles] FP32 master
  void* hi;          // [cap * kTiles] stored operand splits (null with kStaged)
  void* lo;
};

// An upper output block of the numeric kernel: all that its warps need to know of it in two
// loads, which they make a block ahead (a chain of six dependent loads before).
struct __align__(16) Unit {
  int o, p0, np, om;  // slot, first pair and pairs, slot of the mirror
  int I, J, oi, pad;  // block row and column, slot in S (or -1)
};
__device__ __forceinline__ Unit load_unit(const Unit* u) {
  const int4 a = reinterpret_cast<const int4*>(u)[0], b = reinterpret_cast<const int4*>(u)[1];
  return Unit{a.x, a.y, a.z, a.w, b.x, b.y, b.z, 0};
}

struct Sym {
  uint32_t* cand;    // [nsb * MW]
  int* cnt;          // [nsb]
  int* rowp;         // [nsb] pairs of a row's upper blocks
  int* ucnt;         // [nsb] upper blocks of a row
  int* old_idx;      // [cap]
  int2* pcnt;        // [cap] pairs of the earlier blocks of the block's row, of the block
  int2* pairs;       // [pcap]
  int* scal;         // [4]: blocks of the new pattern, pairs, upper blocks
  Unit* list;        // [cap] upper output blocks, band by band
  int* npl;          // [cap] their pairs
  Unit* order;       // [cap] the same in the numeric kernel's order
  uint16_t* flags;   // [nsb * nsb] X0 sub-block keep masks
};

struct Args {
  int n, ld, nsb, cap, pcap;
  int mw;                 // bitmap words in use: ceil(nsb / 32)
  double nocc, tau2, floor, tol;
  int rule, k, max_iter;
  SP2State* st;
  const double* parts_in;
  int nparts_in;
  double* parts_out;
  // start X0 = x0_s (x0_e I - H); x0_s = 0: the SP2 start from the Gershgorin
  // bounds in st (e = eps_max, s = 1/(eps_max - eps_min))
  double x0_e, x0_s;
  int keep_diag;          // every pattern stores the diagonal blocks
  int same_ab;            // the product's operands are one matrix
};

// Epilogue of a product C = alpha A B + gamma S + delta I: (alpha, gamma) =
// (a1, g1) when branch is set and bit k of the SP2 branch record is, else
// (a0, g0); delta on the diagonal of the n x n block.  lolo: also the lo x lo
// split product (squares, where it keeps the diagonal unbiased).
struct Epi {
  float a0, g0, a1, g1, d;
  int branch, lolo;
};

__device__ __forceinline__ int popc_below(const uint32_t* m, int bit) {
  int r = 0;
  for (int w = 0; w < (bit >> 5); ++w) r += __popc(m[w]);
  const uint32_t part = m[bit >> 5] & ((1u << (bit & 31)) - 1u);
  return r + __popc(part);
}

// Row of slot o of b: the last row whose start is <= o.
__device__ __forceinline__ int slot_row(const Buf& b, int nsb, int o) {
  int lo = 0, hi = nsb;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (b.row_ptr[mid] <= o) lo = mid;
    else hi = mid;
  }
  return lo;
}

// ------------------------------------------------------------------ init

// emin/emax from the Gershgorin partials (one block).
__global__ void k_bsr_bounds(const double* bparts, int nb, SP2State* st) {
  double a = INFINITY, b = -INFINITY;
  for (int i = threadIdx.x; i < nb; i += 32) {
    a = fmin(a, bparts[2 * i]);
    b = fmax(b, bparts[2 * i + 1]);
  }
  a = warp_min(a);
  b = warp_max(b);
  if (threadIdx.x == 0) {
    st->emin = a;
    st->emax = b;
  }
}

// (e, s) of the start X0 = s (e I - H).
__device__ __forceinline__ void x0_affine(const Args& a, double* e, double* s) {
  if (a.x0_s != 0.0) {
    *e = a.x0_e;
    *s = a.x0_s;
    return;
  }
  const double emin = a.st->emin, emax = a.st->emax;
  double w = emax - emin;
  if (!(w > 0.0)) w = 1.0;
  *e = emax;
  *s = 1.0 / w;
}

// Whether any lane's value is not zero (an integer test and a vote: a few cycles,
// where an FP64 instruction of a warp takes 76 of its scheduler).
// The halves come from a move that the compiler does not see through: it turns the
// test of a double's bits into a comparison in FP64.
__device__ __forceinline__ bool nonzero_bits(double x) {
  uint32_t lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(x));
  return ((hi << 1) | lo) != 0u;
}
__device__ __forceinline__ bool any_nonzero(double x) { return __any_sync(0xffffffffu, nonzero_bits(x)); }

// Values to be added in FP64, gathered first: zeros add nothing, and where no lane holds a
// value in both p and v the two are one value a lane.  flush(p) when some lane has two.  In
// a molecular H a row of 32 elements holds one or two that are not zero, so that about five
// rows share an FP64 instruction (at 76 cycles a warp and scheduler it costs more than the
// test, the vote and the merge together).  The caller flushes the last p.
template <class Fn>
__device__ __forceinline__ void gather_add(double v, double& p, Fn flush) {
  const bool nv = nonzero_bits(v);
  if (__any_sync(0xffffffffu, nv && nonzero_bits(p))) {
    flush(p);
    p = v;
  } else if (nv) {
    p = v;
  }
}

// Keep mask of a super-block of X0 = s (e I - H) from the elements x(r, c) of e I - H: a
// 32 x 32 sub-block is kept where s^2 sum x^2 >= tau^2 (scale2 = s^2; one FMA per element:
// GB300's FP64 rate is low).  Each of the 8 warps takes two sub-blocks: its lanes the
// columns, so that a row is one coalesced load, 16 in flight, and a sub-block's sum stays
// in one warp, few FP64 instructions to a sub-block (gather_add).  Called by
// every thread of the block, which all get the mask.  (Sums of each of the 16 sub-blocks in
// every warp, combined through shared memory, took 80 FP64 additions a warp and a serial
// sum of 128: 849 us for the 16383 atoms of a vapour, 194 us now.)
template <class X>
__device__ __forceinline__ uint16_t block_keep(const Args& a, double scale2, X x) {
  __shared__ unsigned s_mask;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) s_mask = 0u;
  __syncthreads();
#pragma unroll 1
  for (int q = warp; q < 16; q += 8) {
    const int r0 = 32 * (q >> 2), c = 32 * (q & 3) + lane;
    double acc = 0.0, p = 0.0;
    auto flush = [&](double y) { acc = fma(y, y, acc); };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = x(r0 + 16 * h + k, c);
#pragma unroll
      for (int k = 0; k < 16; ++k) gather_add(v[k], p, flush);
    }
    if (any_nonzero(p)) {
      flush(p);
      acc = warp_sum(acc) * scale2;
      if (lane == 0 && acc >= a.tau2 && acc > 0.0) atomicOr(&s_mask, 1u << q);
    }
  }
  __syncthreads();
  const uint16_t f = (uint16_t)s_mask;
  __syncthreads();  // s_mask is reused by the next block of a grid-stride loop
  return f;
}

// The same from H's super-block (I, J) at h (row stride ld; null: zero).
__device__ uint16_t x0_keep(const Args& a, const double* h, size_t ld, int I, int J, double e, double scale2) {
  const int ne = max(0, a.n - I * SB), nc = max(0, a.n - J * SB);  // rows and columns inside the matrix
  if (h && I != J && ne >= SB && nc >= SB)
    return block_keep(a, scale2, [&](int r, int c) { return h[r * ld + c]; });
  return block_keep(a, scale2, [&](int r, int c) {
    if (r >= ne || c >= nc) return 0.0;
    const double x = h ? h[r * ld + c] : 0.0;
    return I == J && r == c ? e - x : x;
  });
}

__device__ __forceinline__ uint16_t mask_transposed(uint16_t f) {
  uint16_t t = 0;
  for (int q = 0; q < 16; ++q)
    if ((f >> q) & 1) t |= (uint16_t)(1u << ((q & 3) * 4 + (q >> 2)));
  return t;
}

// One block per upper super-block (I, J) of X0 = s (e I - H): its keep mask, and below the
// diagonal the twin's mask transposed, so that the pattern is exactly symmetric (the
// products compute upper blocks and mirror them).
__global__ void __launch_bounds__(256) k_bsr_init_flags(const double* __restrict__ H, Args a, Sym sy) {
  const int I = blockIdx.y, J = blockIdx.x;
  if (I > J) return;
  double emax, inv;
  x0_affine(a, &emax, &inv);
  const uint16_t f = x0_keep(a, H + (size_t)I * SB * a.n + J * SB, a.n, I, J, emax, inv * inv);
  if (threadIdx.x == 0) {
    sy.flags[(size_t)I * a.nsb + J] = f;
    if (I != J) sy.flags[(size_t)J * a.nsb + I] = mask_transposed(f);
  }
}

// Row I of X0: live bitmap of its kept super-blocks; stored = live (and the
// diagonal block with keep_diag); count of stored blocks.
__global__ void k_bsr_init_rows(Args a, Sym sy, Buf b) {
  const int I = blockIdx.x;
  __shared__ uint32_t m[MW];
  if (threadIdx.x < MW) m[threadIdx.x] = 0u;
  __syncthreads();
  for (int J = threadIdx.x; J < a.nsb; J += blockDim.x)
    if (sy.flags[(size_t)I * a.nsb + J]) atomicOr(&m[J >> 5], 1u << (J & 31));
  __syncthreads();
  if (threadIdx.x < MW) {
    const uint32_t diag = (a.keep_diag && (I >> 5) == (int)threadIdx.x) ? 1u << (I & 31) : 0u;
    b.stored[I * MW + threadIdx.x] = m[threadIdx.x] | diag;
    b.live[I * MW + threadIdx.x] = m[threadIdx.x];
    m[threadIdx.x] |= diag;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int c = 0;
    for (int w = 0; w < MW; ++w) c += __popc(m[w]);
    sy.cnt[I] = c;
  }
}

// Exclusive scan of cnt[0..nsb) into row_ptr (one block); total into scal[0].
// One warp: lane l scans rows [l * per, (l + 1) * per) after an exclusive
// warp scan of the lanes' sums.
__global__ void k_bsr_scan_rows(Args a, Sym sy, int* row_ptr) {
  if (a.st->done || a.st->err) return;
  const int lane = threadIdx.x & 31, per = (a.nsb + 31) / 32;
  const int lo = min(a.nsb, lane * per), hi = min(a.nsb, lo + per);
  int mine = 0;
  for (int i = lo; i < hi; ++i) mine += sy.cnt[i];
  int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  int run = incl - mine;
  for (int i = lo; i < hi; ++i) {
    row_ptr[i] = run;
    run += sy.cnt[i];
  }
  if (lane == 31) {
    row_ptr[a.nsb] = incl;
    sy.scal[0] = incl;
    if (incl > a.cap) atomicExch(&a.st->err, TB_ERR_OOM);
  }
}

// Fill the X0 blocks of row I, kFillSplit thread blocks sharing its stored blocks: values
// with dropped sub-blocks zeroed, operand splits, trace partials of each thread block.
// src(J, &ld): H's super-block (I, J) (null: zero).  A warp takes a sub-block at a time, its
// lanes the columns: whole-row loads and stores; dropped sub-blocks and rows that are all
// zero take no FP64 work.  (One thread block a row, 32 elements of a row to a thread: 325 us
// for 16383 atoms, 51 us now.)
constexpr int kFillSplit = 4;
template <int P, class Src>
__device__ void x0_fill_row(const Args& a, const Sym& sy, const Buf& b, Src src) {
  __shared__ uint16_t s_col[kMaxNsb];
  __shared__ float s_t[8][32][33];  // stored splits: a sub-block to be read by rows
  __shared__ double s1[8], s2[8];
  const int I = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double emax, inv;
  x0_affine(a, &emax, &inv);
  const uint32_t* st = b.stored + I * MW;
  for (int J = threadIdx.x; J < a.nsb; J += blockDim.x)
    if ((st[J >> 5] >> (J & 31)) & 1u) s_col[popc_below(st, J)] = (uint16_t)J;
  __syncthreads();
  double t1 = 0.0, t2 = 0.0;
  const int o0 = b.row_ptr[I], cnt = b.row_ptr[I + 1] - o0;
  const int ne = max(0, a.n - I * SB);
  for (int k = blockIdx.y; k < cnt; k += kFillSplit) {
    const int J = s_col[k], o = o0 + k;
    const uint16_t f = sy.flags[(size_t)I * a.nsb + J];
    const int nc = max(0, a.n - J * SB);
    size_t ld = 0;
    const double* h = src(J, &ld);
    if (threadIdx.x == 0) b.col[o] = J;
#pragma unroll 1
    for (int q = warp; q < 16; q += 8) {
      const int r0 = 32 * (q >> 2), c0 = 32 * (q & 3), c = c0 + lane;
      float* dst = b.val + (size_t)o * kTiles + (size_t)r0 * SB + c0;
      if ((f >> q) & 1) {
        const bool dsub = I == J && r0 == c0;
        float yd = 0.0f;
#pragma unroll
        for (int rb = 0; rb < 32; rb += 16) {
          double x[16];
#pragma unroll
          for (int r = 0; r < 16; ++r)
            x[r] = h && r0 + rb + r < ne && c < nc ? h[(r0 + rb + r) * ld + c] : 0.0;
#pragma unroll
          for (int r = 0; r < 16; ++r) {
            float y = 0.0f;
            if (dsub) {
              const bool on = rb + r == lane && r0 + lane < ne;
              y = (float)(((on ? emax : 0.0) - x[r]) * inv);
              if (on) yd = y;
            } else if (any_nonzero(x[r])) {
              y = (float)(-x[r] * inv) + 0.0f;  // + 0: the zeros of X0 are positive
            }
            if (__any_sync(0xffffffffu, y != 0.0f)) {
              const double d = abs_to_f64(y);
              t2 = fma(d, d, t2);
            }
            dst[(size_t)(rb + r) * SB + lane] = y;
            if constexpr (!kStaged<P>) s_t[warp][rb + r][lane] = y;
          }
        }
        if (dsub) t1 += (double)yd;
      } else {
#pragma unroll
        for (int r = 0; r < 32; r += 4)
          *reinterpret_cast<float4*>(dst + (size_t)(r + (lane >> 3)) * SB + 4 * (lane & 7)) =
              make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (!kStaged<P>)
          for (int r = 0; r < 32; ++r) s_t[warp][r][lane] = 0.0f;
      }
      if constexpr (!kStaged<P>) {
        __syncwarp();
        float y[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) y[j] = s_t[warp][lane][j];
        __syncwarp();
        const size_t e0 = (size_t)o * kTiles + (size_t)(r0 + lane) * SB + c0;
        char* hp = static_cast<char*>(b.hi) + e0 * Prec<P>::eb;
        char* lp = b.lo ? static_cast<char*>(b.lo) + e0 * Prec<P>::eb : hp;
        store_operands<P>(y, hp, lp);
      }
    }
  }
  t1 = warp_sum(t1);
  t2 = warp_sum(t2);
  if (lane == 0) {
    s1[warp] = t1;
    s2[warp] = t2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double x = 0, y = 0;
    for (int q = 0; q < 8; ++q) {
      x += s1[q];
      y += s2[q];
    }
    double* p = a.parts_out + 3 * (I * kFillSplit + blockIdx.y);
    p[0] = x;
    p[1] = y;
    p[2] = 0.0;
  }
}

template <int P>
__global__ void __launch_bounds__(256) k_bsr_init_fill(const double* __restrict__ H, Args a, Sym sy, Buf b) {
  if (a.st->err) return;
  x0_fill_row<P>(a, sy, b, [&](int J, size_t* ld) {
    *ld = a.n;
    return H + (size_t)blockIdx.x * SB * a.n + J * SB;
  });
}

// ---- BSR input (dm_sp2_sparse): H given as 128 x 128 FP64 blocks

// Slot of block (I, J) in a BSR row (binary search over its sorted columns), or -1.
__device__ __forceinline__ int bsr_find(const int* __restrict__ row_ptr, const int* __restrict__ col, int I, int J) {
  int lo = row_ptr[I], hi = row_ptr[I + 1] - 1;
  while (lo <= hi) {
    const int mid = (lo + hi) >> 1;
    const int c = col[mid];
    if (c == J) return mid;
    if (c < J) lo = mid + 1;
    else hi = mid - 1;
  }
  return -1;
}

// Gershgorin partials of block row I (kBndSplit blocks of 256 threads, 16 rows each): warp w
// takes rows w + 8k, lane l the columns 32 c + l, so each block is read as 8 independent
// coalesced loads a lane, two blocks at a time, and the row sums stay in registers until one
// warp sum per row; min(H_ii - r_i) and max(H_ii + r_i) over the rows go into
// bparts[2 (I kBndSplit + y)].  One addition an element would make the FP64 pipe the bound
// (1.1 ms for the 1.2 GB of a 16383-atom H); the elements are gathered (gather_add) first:
// 0.40 ms, against 0.18 ms for the bytes.
constexpr int kBndSplit = 8;
__global__ void __launch_bounds__(256) k_bsr_bounds_in(tb_bsr H, double* __restrict__ bparts) {
  __shared__ double smin[8], smax[8];
  constexpr int kRows = 16 / kBndSplit;  // rows per warp
  const int I = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = blockIdx.y * (SB / kBndSplit) + warp;
  bparts += 2 * (I * kBndSplit + blockIdx.y);
  if (*H.status != TB_OK) {  // an incomplete H (k_bsr_status_in fails the call)
    if (threadIdx.x == 0) bparts[0] = bparts[1] = 0.0;
    return;
  }
  double rad[kRows], dia[kRows], pend[kRows];
#pragma unroll
  for (int k = 0; k < kRows; ++k) rad[k] = dia[k] = pend[k] = 0.0;
  const int o1 = H.row_ptr[I + 1];
  for (int o = H.row_ptr[I]; o < o1; o += 2) {
    const bool two = o + 1 < o1;
    const bool dblk[2] = {H.col[o] == I, two && H.col[o + 1] == I};
    double x[2][kRows][4];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int k = 0; k < kRows; ++k)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
          x[t][k][cc] = t == 0 || two ? H.val[(size_t)(o + t) * kTiles + (r0 + 8 * k) * SB + 32 * cc + lane] : 0.0;
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int k = 0; k < kRows; ++k)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          double v = x[t][k][cc];
          if (dblk[t] && 32 * cc + lane == r0 + 8 * k) {
            dia[k] = v;
            v = 0.0;
          }
          gather_add(v, pend[k], [&](double y) { rad[k] += fabs(y); });
        }
  }
#pragma unroll
  for (int k = 0; k < kRows; ++k) rad[k] += fabs(pend[k]);
  double lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const double rs = warp_sum(rad[k]), c = warp_sum(dia[k]);  // one lane holds the diagonal element
    if (I * SB + r0 + 8 * k < H.n) {
      lo = fmin(lo, c - rs);
      hi = fmax(hi, c + rs);
    }
  }
  if (lane == 0) {
    smin[warp] = lo;
    smax[warp] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = smin[0], b = smax[0];
    for (int w = 1; w < 8; ++w) {
      a = fmin(a, smin[w]);
      b = fmax(b, smax[w]);
    }
    bparts[0] = a;
    bparts[1] = b;
  }
}

// As k_bsr_init_flags, from the blocks of a BSR H (an absent block of H is
// zero in X0 off the diagonal).
// An H whose build overflowed its capacity fails the call (TB_ERR_OOM).
__global__ void k_bsr_status_in(const int* Hstatus, SP2State* st) {
  if (*Hstatus != TB_OK) st->err = TB_ERR_OOM;
}

// Row of slot o of a BSR matrix: the last row whose start is <= o.
__device__ __forceinline__ int bsr_row_of(const int* __restrict__ row_ptr, int nsb, int o) {
  int lo = 0, hi = nsb;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (row_ptr[mid] <= o) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Keep masks of X0 from a BSR H, one block per stored upper block of H (grid-stride;
// the masks start zeroed, and a block H does not store is zero in X0 off the
// diagonal); k_bsr_init_flags_diag covers diagonal blocks H does not store.
__global__ void __launch_bounds__(256) k_bsr_init_flags_in(tb_bsr H, Args a, Sym sy) {
  if (*H.status != TB_OK) return;  // the call fails through k_bsr_status_in
  const int nblk = min(H.row_ptr[H.nsb], H.cap);
  double emax, inv;
  x0_affine(a, &emax, &inv);
  for (int o = blockIdx.x; o < nblk; o += gridDim.x) {
    const int I = bsr_row_of(H.row_ptr, H.nsb, o), J = H.col[o];
    if (I > J) continue;  // its mask is its twin's transposed (or 0: H stores none)
    const uint16_t f = x0_keep(a, H.val + (size_t)o * kTiles, SB, I, J, emax, inv * inv);
    if (threadIdx.x == 0) {
      sy.flags[(size_t)I * a.nsb + J] = f;
      if (I != J && f && bsr_find(H.row_ptr, H.col, J, I) >= 0)
        sy.flags[(size_t)J * a.nsb + I] = mask_transposed(f);
    }
  }
}

__global__ void __launch_bounds__(256) k_bsr_init_flags_diag(tb_bsr H, Args a, Sym sy) {
  const int I = blockIdx.x;
  if (*H.status != TB_OK || bsr_find(H.row_ptr, H.col, I, I) >= 0) return;
  double emax, inv;
  x0_affine(a, &emax, &inv);
  const uint16_t f = x0_keep(a, nullptr, 0, I, I, emax, inv * inv);
  if (threadIdx.x == 0) sy.flags[(size_t)I * a.nsb + I] = f;
}

// As k_bsr_init_fill, from the blocks of a BSR H.
template <int P>
__global__ void __launch_bounds__(256) k_bsr_init_fill_in(tb_bsr H, Args a, Sym sy, Buf b) {
  if (a.st->err) return;
  x0_fill_row<P>(a, sy, b, [&](int J, size_t* ld) {
    *ld = SB;
    const int slot = bsr_find(H.row_ptr, H.col, blockIdx.x, J);
    return slot >= 0 ? H.val + (size_t)slot * kTiles : nullptr;
  });
}

// ------------------------------------------------------- per projection

// Whether the call is finished or failed, the same for every thread of the block also where
// another block of this launch sets the error.
__device__ __forceinline__ bool stopped(const SP2State* st) {
  return __syncthreads_or(threadIdx.x == 0 && (st->done || st->err));
}

// Decision for projection k, the same in every block (256 threads): whether the phase stops.
__device__ bool bsr_decide(const Args& a) {
  __shared__ int s_stop;
  SP2State* st = a.st;
  if (threadIdx.x < 32) {
    double x = 0, y = 0;
    for (int i = threadIdx.x; i < a.nparts_in; i += 32) {
      x += a.parts_in[3 * i];
      y += a.parts_in[3 * i + 1];
    }
    x = warp_sum(x);
    y = warp_sum(y);
    if (threadIdx.x == 0) {
      SP2StepArgs d{};
      d.nocc = a.nocc;
      d.tol = a.tol;
      d.floor = a.floor;
      d.rule = a.rule;
      d.k = a.k;
      d.max_iter = a.max_iter;
      int br = 0, capped = 0;
      const int stop = sp2_decide(d, x, y, st->t1, st->t2, true, &br, &capped);
      s_stop = stop;
      if (blockIdx.x == 0) {
        st->t1[a.k] = x;
        st->t2[a.k] = y;
        if (stop) {
          st->iters = a.k;
          st->capped = capped;
          st->done = 1;
        } else if (br) {
          st->branch[a.k >> 6] |= 1ull << (a.k & 63);
        }
      }
    }
  }
  __syncthreads();
  return s_stop;
}

// Candidate columns of row I of A B: the OR of B's live rows over A's live
// columns of row I; unless A and B are one matrix also the same with A and B
// exchanged (the pattern of B A = (A B)^T), so that the pattern is symmetric
// as the upper-block computation with mirrors needs; S's live blocks; the
// diagonal block with keep_diag.  With `decide` the projection's decision first.  A and B are symmetric (rows = columns).
__global__ void __launch_bounds__(256) k_bsr_cand(Args a, Buf A, Buf B, Buf S, Sym sy, bool decide) {
  __shared__ uint32_t c[MW];
  if (stopped(a.st)) return;
  if (decide && bsr_decide(a)) return;
  const int I = blockIdx.x;
  if (threadIdx.x < MW) c[threadIdx.x] = 0u;
  __syncthreads();
  for (int side = 0; side < (a.same_ab ? 1 : 2); ++side) {
    const uint32_t* li = (side ? B.live : A.live) + I * MW;
    const uint32_t* rows = side ? A.live : B.live;
    for (int K = threadIdx.x; K < a.nsb; K += blockDim.x)
      if ((li[K >> 5] >> (K & 31)) & 1u)
        for (int w = 0; w < a.mw; ++w) {
          const uint32_t v = rows[K * MW + w];
          if (v) atomicOr(&c[w], v);
        }
  }
  __syncthreads();
  if (threadIdx.x < MW) {
    uint32_t v = c[threadIdx.x];
    if (S.live) v |= S.live[I * MW + threadIdx.x];
    if (a.keep_diag && (I >> 5) == (int)threadIdx.x) v |= 1u << (I & 31);
    sy.cand[I * MW + threadIdx.x] = v;
    c[threadIdx.x] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < MW; ++w) s += __popc(c[w]);
    sy.cnt[I] = s;
  }
}

// Sum of v over the rows before I, and over all nsb rows (256 threads; every thread gets
// both): each block of a symbolic kernel scans the rows' counts for itself, instead of a
// launch of one block before it.
__device__ void rows_prefix(const int* __restrict__ v, int nsb, int I, long long* before, long long* total) {
  __shared__ long long s_b[8], s_t[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  long long b = 0, t = 0;
  for (int i = threadIdx.x; i < nsb; i += 256) {
    const int x = v[i];
    t += x;
    if (i < I) b += x;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    b += __shfl_xor_sync(0xffffffffu, b, d);
    t += __shfl_xor_sync(0xffffffffu, t, d);
  }
  if (lane == 0) {
    s_b[warp] = b;
    s_t[warp] = t;
  }
  __syncthreads();
  b = t = 0;
  for (int w = 0; w < 8; ++w) {
    b += s_b[w];
    t += s_t[w];
  }
  *before = b;
  *total = t;
}

// Output blocks of row I: its start, and for each block the column, the slot of S_IJ (or
// -1) and the pairs of the row's blocks before it; the row's pairs and upper blocks.
__global__ void __launch_bounds__(256) k_bsr_fill_out(Args a, Buf A, Buf B, Buf S, Buf bn, Sym sy) {
  __shared__ int s_w[8];
  if (stopped(a.st)) return;
  const int I = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  long long base, total;
  rows_prefix(sy.cnt, a.nsb, I, &base, &total);
  if (threadIdx.x == 0) {
    bn.row_ptr[I] = (int)base;
    if (I == 0) {
      bn.row_ptr[a.nsb] = (int)total;
      sy.scal[0] = (int)total;
      if (total > a.cap) atomicExch(&a.st->err, TB_ERR_OOM);
    }
  }
  if (total > a.cap) return;
  const uint32_t* ci = sy.cand + I * MW;
  const uint32_t* si = S.stored ? S.stored + I * MW : nullptr;
  const uint32_t* li = A.live + I * MW;
  if (threadIdx.x < MW) {  // the numeric kernel adds the live ones
    bn.stored[I * MW + threadIdx.x] = ci[threadIdx.x];
    bn.live[I * MW + threadIdx.x] = 0u;
  }
  int run = 0, upper = 0;
  long long prod = 0;  // a block above the diagonal has a mirror with as many products
  for (int J0 = 0; J0 < a.nsb; J0 += 256) {
    const int J = J0 + (int)threadIdx.x;
    const bool has = J < a.nsb && ((ci[J >> 5] >> (J & 31)) & 1u);
    int pc = 0;
    if (has && J >= I) {  // the product is symmetric: blocks below the diagonal are written as mirrors
      const uint32_t* lj = B.live + J * MW;
      for (int w = 0; w < a.mw; ++w) pc += __popc(li[w] & lj[w]);
      ++upper;
      prod += J > I ? 2 * pc : pc;
    }
    int incl = pc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    int before = run;
    for (int w = 0; w < 8; ++w) {
      if (w < warp) before += s_w[w];
      run += s_w[w];
    }
    __syncthreads();
    if (has) {
      const int o = (int)base + popc_below(ci, J);
      bn.col[o] = J;
      sy.old_idx[o] = (si && ((si[J >> 5] >> (J & 31)) & 1u)) ? S.row_ptr[I] + popc_below(si, J) : -1;
      sy.pcnt[o] = make_int2(before + incl - pc, pc);
    }
  }
  upper = __reduce_add_sync(0xffffffffu, upper);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) prod += __shfl_xor_sync(0xffffffffu, prod, d);
  if (lane == 0) {
    s_w[warp] = upper;
    if (prod) atomicAdd(&a.st->block_products, (unsigned long long)prod);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int u = 0;
    for (int w = 0; w < 8; ++w) u += s_w[w];
    sy.rowp[I] = run;
    sy.ucnt[I] = u;
  }
}

// The numeric kernel's lists, in one launch:
// - blocks below nsb * kPairSplit: the pairs (slot of A_IK, slot of B_JK) of every upper
//   output block (I, J), (A B)_IJ = sum_K A_IK B_JK^T for a symmetric B: a warp per output
//   block, its lanes the columns K of a bitmap word, so that the pairs are written
//   coalesced (a thread per output block: 11 us a projection at 256 block rows, and the
//   scan of the pair counts before it another 11);
// - the others: the upper output blocks (I <= J) in (band of kBand block rows, column J,
//   row I) order.  The persistent numeric kernel takes them in this order, so the CTAs
//   working at the same time cover a few columns of one band: they share the (I, K) tiles
//   of the band's rows and the (J, K) tiles of those columns in L2 instead of each
//   streaming its own.  A warp per band and bitmap word, its lanes the columns (a warp per
//   band walking the columns: 22 us a projection).
constexpr int kPairSplit = 4;
__global__ void __launch_bounds__(256) k_bsr_pairs(Args a, Buf A, Buf B, Buf bn, Sym sy) {
  if (stopped(a.st)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const int npb = a.nsb * kPairSplit;
  const bool listing = (int)blockIdx.x >= npb;
  const int I = listing ? 0 : blockIdx.x / kPairSplit;
  long long before, total;
  rows_prefix(sy.rowp, a.nsb, I, &before, &total);
  if (blockIdx.x == 0 && threadIdx.x == 0 && total > a.pcap) atomicExch(&a.st->err, TB_ERR_OOM);
  if (total > a.pcap) return;
  if (!listing) {
    const int part = blockIdx.x % kPairSplit;
    const uint32_t al = A.live[I * MW + lane], as = A.stored[I * MW + lane];
    const int ra0 = A.row_ptr[I], o1 = bn.row_ptr[I + 1];
    for (int o = bn.row_ptr[I] + part * 8 + warp; o < o1; o += kPairSplit * 8) {
      const int J = bn.col[o];
      if (J < I) continue;
      int p = (int)before + sy.pcnt[o].x;
      const uint32_t m_l = al & B.live[J * MW + lane], bs = B.stored[J * MW + lane];
      int ra = ra0, rb = B.row_ptr[J];
      for (int w = 0; w < a.mw; ++w) {
        const uint32_t m = __shfl_sync(0xffffffffu, m_l, w), sa = __shfl_sync(0xffffffffu, as, w),
                       sb = __shfl_sync(0xffffffffu, bs, w);
        if ((m >> lane) & 1u)
          sy.pairs[p + __popc(m & below)] = make_int2(ra + __popc(sa & below), rb + __popc(sb & below));
        p += __popc(m);
        ra += __popc(sa);
        rb += __popc(sb);
      }
    }
    return;
  }
  const int id = ((int)blockIdx.x - npb) * 8 + warp, band = id / a.mw, w = id % a.mw, I0 = band * kBand;
  if (id == 0) {
    int u = 0;
    for (int i = lane; i < a.nsb; i += 32) u += sy.ucnt[i];
    u = __reduce_add_sync(0xffffffffu, u);
    if (lane == 0) sy.scal[2] = u;
  }
  if (I0 >= a.nsb) return;
  int pos = 0, pairs0 = 0;  // entries and pairs before the band
  for (int i = lane; i < I0; i += 32) {
    pos += sy.ucnt[i];
    pairs0 += sy.rowp[i];
  }
  pairs0 = __reduce_add_sync(0xffffffffu, pairs0);
  uint32_t word[kBand];  // word w of the band's rows, columns J >= I only
  int slot[kBand];       // slot of the first block of that word
  const int J = 32 * w + lane;
  int mine = 0;
#pragma unroll
  for (int r = 0; r < kBand; ++r) {
    const int Ir = I0 + r;
    const uint32_t c = Ir < a.nsb ? sy.cand[Ir * MW + lane] : 0u;  // lane: the word
    const int lo = Ir - 32 * lane;                                 // keep bits J >= I
    const uint32_t up = lo >= 32 ? 0u : lo > 0 ? c & ~((1u << lo) - 1u) : c;
    if (lane < w) pos += __popc(up);
    slot[r] = __reduce_add_sync(0xffffffffu, lane < w ? __popc(c) : 0);
    if (Ir < a.nsb) slot[r] += bn.row_ptr[Ir];
    const uint32_t cw = __shfl_sync(0xffffffffu, c, w);
    slot[r] += __popc(cw & below);
    word[r] = __shfl_sync(0xffffffffu, up, w);
    mine += (word[r] >> lane) & 1u;
  }
  pos = __reduce_add_sync(0xffffffffu, pos);
  int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  pos += incl - mine;
  if (!mine) return;
  // slot of the mirror (J, I): the band's rows lie in one word of row J
  const uint32_t* cj = sy.cand + J * MW;
  const int mir = bn.row_ptr[J] + popc_below(cj, I0);
  const uint32_t wj = cj[I0 >> 5] >> (I0 & 31);
  int2 pc[kBand];
  int oi[kBand], rp[kBand];
#pragma unroll
  for (int r = 0; r < kBand; ++r) {  // loads of all rows in flight together
    const int o = (word[r] >> lane) & 1u ? slot[r] : 0;
    pc[r] = sy.pcnt[o];
    oi[r] = sy.old_idx[o];
    rp[r] = I0 + r < a.nsb ? sy.rowp[I0 + r] : 0;
  }
#pragma unroll
  for (int r = 0; r < kBand; ++r) {
    if ((word[r] >> lane) & 1u) {
      sy.npl[pos] = pc[r].y;
      int4* u = reinterpret_cast<int4*>(sy.list + pos++);
      u[0] = make_int4(slot[r], pairs0 + pc[r].x, pc[r].y, J > I0 + r ? mir + __popc(wj & ((1u << r) - 1u)) : slot[r]);
      u[1] = make_int4(I0 + r, J, oi[r], 0);
    }
    pairs0 += rp[r];
  }
}

// The numeric kernel's order: the band list sorted (stably) into classes of falling pair
// counts (four to an octave), which its thread blocks take in rounds of alternating
// direction: no two of them differ by more than about one block's work, where the band list
// in rounds left the mean one a quarter of the time idle (16383 atoms: 154 -> 126 us a
// projection; a liquid of 4096 atoms 39.0 -> 35.6 ms in all).  Within a class the bands stay
// together.  A thread block per class.
constexpr int kClasses = 44;  // up to 1024 pairs: ten octaves and one
__device__ __forceinline__ int pair_class(int np) {
  return kClasses - 1 - (int)((__float_as_uint((float)(np + 1)) - 0x3f800000u) >> 21);
}
__global__ void __launch_bounds__(1024) k_bsr_balance(Args a, Sym sy) {
  __shared__ int s_w[2][32], s_c[2];
  if (a.st->done || a.st->err) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nu = sy.scal[2], c = blockIdx.x;
  if (threadIdx.x < 2) s_c[threadIdx.x] = 0;
  __syncthreads();
  int before = 0, own = 0;
#pragma unroll 4
  for (int u = threadIdx.x; u < nu; u += 1024) {
    const int k = pair_class(sy.npl[u]);
    before += k < c;
    own += k == c;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  own = __reduce_add_sync(0xffffffffu, own);
  if (lane == 0 && before) atomicAdd(&s_c[0], before);
  if (lane == 0 && own) atomicAdd(&s_c[1], own);
  __syncthreads();
  if (s_c[1] == 0) return;
  int pos = s_c[0];
  for (int u0 = 0, t = 0; u0 < nu; u0 += 1024, t ^= 1) {
    const int u = u0 + (int)threadIdx.x;
    const bool mine = u < nu && pair_class(sy.npl[u]) == c;
    const unsigned m = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) s_w[t][warp] = __popc(m);
    __syncthreads();  // the other half of s_w is rewritten after the next one
    const int w = s_w[t][lane];
    const int at = pos + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0);
    pos += __reduce_add_sync(0xffffffffu, w);
    if (mine) {
      const int4* src = reinterpret_cast<const int4*>(sy.list + u);
      int4* dst = reinterpret_cast<int4*>(sy.order + at + __popc(m & ((1u << lane) - 1u)));
      const int4 x = src[0], y = src[1];
      dst[0] = x;
      dst[1] = y;
    }
  }
}

// Unit of thread block b of g in round k.
__device__ __forceinline__ int unit_of(int k) {
  const int g = gridDim.x, b = blockIdx.x;
  return k * g + ((k & 1) ? g - 1 - b : b);
}

// Persistent numeric projection.
template <int P>
__global__ void __launch_bounds__(kNumThreads<P>, 1)
    k_bsr_step_tc(Args a, const __grid_constant__ CUtensorMap ah, const __grid_constant__ CUtensorMap al,
                  const __grid_constant__ CUtensorMap bh, const __grid_constant__ CUtensorMap bl, Buf S, Buf bn,
                  Sym sy, Epi ep) {
  using C = Prec<P>;
  constexpr int NS = kNumStages<P>;
  constexpr uint32_t kCols = kStaged<P> ? kFsTmemCols : 2 * SB;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[NS], empty[NS], tfull[2], tempty[2], mdone, conv[NS];
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_abort;
  __shared__ double s_red[4][3];
  __shared__ __align__(16) float s_sym[4][32][36];  // per epilogue warp: one 32 x 32 sub-block
  SP2State* st = a.st;
  if (st->done || st->err) return;
  const int br = ep.branch ? (int)((st->branch[a.k >> 6] >> (a.k & 63)) & 1ull) : 0;
  const float alpha = br ? ep.a1 : ep.a0, gamma = br ? ep.g1 : ep.g0;
  const int nu = sy.scal[2];  // upper output blocks, walked in sy.order
  // an FP32 sum of squares below this is below tau^2 (thresholds whose squares could
  // underflow take the FP64 sum)
  const float drop32 = a.tau2 > 1e-24 ? (float)(0.9999 * a.tau2) : -1.0f;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&conv[s], 8);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
    }
    mbar_init(&mdone, 1);
    s_abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  constexpr int chunks = SB / C::bk;  // k-steps of one super-block

  if (warp == 0 && lane == 0) {
    prefetch_map(&ah);
    prefetch_map(&bh);
    if (C::split) {
      prefetch_map(&al);
      prefetch_map(&bl);
    }
    int g = 0, issued = 0;
    int4 next = blockIdx.x < nu ? *reinterpret_cast<const int4*>(sy.order + blockIdx.x) : make_int4(0, 0, 0, 0);
    for (int r = 0; unit_of(r) < nu && !s_abort; ++r) {
      const int p0 = next.y, p1 = next.y + next.z;
      if (unit_of(r + 1) < nu) next = *reinterpret_cast<const int4*>(sy.order + unit_of(r + 1));
      int2 pr1 = p0 < p1 ? sy.pairs[p0] : make_int2(0, 0);
      for (int p = p0; p < p1 && !s_abort; ++p) {
        const int2 pr = pr1;
        if (p + 1 < p1) pr1 = sy.pairs[p + 1];
        for (int c = 0; c < chunks; ++c, ++g) {
          const int s = g % NS;
          if (g >= NS && !mbar_wait(&empty[s], ((g / NS) - 1) & 1, &s_abort)) break;
          uint8_t* base = smem + s * kNumStageBytes<P>;
          // staged: the FP32 masters into the hi positions only
          mbar_expect_tx(&full[s], kStaged<P> ? 2 * kFsTile : C::stage_bytes);
          tma_load_2d(base, &ah, &full[s], c * C::bk, pr.x * SB);
          tma_load_2d(base + 128 * 128, &bh, &full[s], c * C::bk, pr.y * SB);
          if constexpr (C::split && !kStaged<P>) {
            tma_load_2d(base + 2 * 128 * 128, &al, &full[s], c * C::bk, pr.x * SB);
            tma_load_2d(base + 3 * 128 * 128, &bl, &full[s], c * C::bk, pr.y * SB);
          }
          issued = g + 1;
        }
      }
    }
    if (s_abort) {
      for (int q = (issued > NS ? issued - NS : 0); q < issued; ++q) {
        const unsigned long long t0 = gtime();
        while (!mbar_try(&full[q % NS], (q / NS) & 1) && gtime() - t0 < kWaitNs) {
        }
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      const uint32_t lo0 = sdesc_lo(smem_u32(smem));
      constexpr uint32_t id = idesc(C::tf32 ? 2u : 1u);
      int g = 0, it = 0;
      int next = blockIdx.x < nu ? sy.order[blockIdx.x].np : 0;
      for (int r = 0; unit_of(r) < nu && !s_abort; ++r) {
        const int np = next;
        if (unit_of(r + 1) < nu) next = sy.order[unit_of(r + 1)].np;
        const int buf = it & 1;
        if (it >= 2 && !mbar_wait(&tempty[buf], ((it >> 1) - 1) & 1, &s_abort)) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * SB;
        bool first = true;
        for (int p = 0; p < np && !s_abort; ++p) {
          for (int c = 0; c < chunks; ++c, ++g) {
            const int s = g % NS;
            if (!mbar_wait(kStaged<P> ? &conv[s] : &full[s], (g / NS) & 1, &s_abort)) break;
            tc_fence_after();
            const uint32_t base = lo0 + s * (kNumStageBytes<P> >> 4);
            if constexpr (kStaged<P>) {
              fs_mma(base, tmem, s, d, id, first, ep.lolo);
              first = false;
            } else {
#pragma unroll
              for (int ks = 0; ks < C::bk / C::uk; ++ks) {
                const uint32_t koff = ks * 2;
                const uint64_t dah = sdesc_at(base + koff), dbh = sdesc_at(base + (kFsTile >> 4) + koff);
                umma<C::tf32>(d, dah, dbh, id, first ? 0u : 1u);
                first = false;
                if constexpr (C::split) {
                  const uint64_t dal = sdesc_at(base + (2 * kFsTile >> 4) + koff), dbl = sdesc_at(base + (3 * kFsTile >> 4) + koff);
                  umma<C::tf32>(d, dah, dbl, id, 1u);
                  umma<C::tf32>(d, dal, dbh, id, 1u);
                  // lo x lo: in a square it keeps the diagonal blocks' sums of squares unbiased
                  if (ep.lolo) umma<C::tf32>(d, dal, dbl, id, 1u);
                }
              }
            }
            umma_commit(&empty[s]);
          }
        }
        umma_commit(&tfull[buf]);
        ++it;
      }
      // arrives once every MMA this thread issued has completed
      umma_commit(&mdone);
    }
    __syncwarp();
  } else if (kStaged<P> && warp >= 6) {
    // converters: warps 6-9 A, 10-13 B
    int g = 0, next = blockIdx.x < nu ? sy.order[blockIdx.x].np : 0;
    for (int r = 0; unit_of(r) < nu && !s_abort; ++r) {
      const int npc = next * chunks;
      if (unit_of(r + 1) < nu) next = sy.order[unit_of(r + 1)].np;
      for (int i = 0; i < npc && !s_abort; ++i, ++g) {
        const int s = g % NS;
        if (!mbar_wait_warp(&full[s], (g / NS) & 1, &s_abort)) break;
        uint8_t* stage = smem + s * kFsStage;
        if (warp < 10) fs_convert_a(stage, tmem, s, warp & 3, lane);
        else fs_convert_b(stage, threadIdx.x - 320);
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&conv[s])) : "memory");
      }
    }
  } else if (warp >= 2) {
    const int q = warp & 3;
    const int row = 32 * q + lane;
    double t1 = 0.0, t2 = 0.0;
    int it = 0;
    Unit next{};
    if (blockIdx.x < nu) next = load_unit(sy.order + blockIdx.x);
    for (int r = 0; unit_of(r) < nu; ++r) {
      const Unit un = next;
      if (unit_of(r + 1) < nu) next = load_unit(sy.order + unit_of(r + 1));
      const int buf = it & 1;
      ++it;
      const int o = un.o, om = un.om, I = un.I, J = un.J, oi = un.oi;
      const bool has = un.np > 0, mirror = J > I;
      // a diagonal block of a product of two matrices is not exactly symmetric
      // in rounding (A B against B A): its upper triangle is kept and mirrored
      const bool symd = I == J && !a.same_ab;
      float* xmir = bn.val + (size_t)om * kTiles;
      // this warp's 32 rows of S_IJ and of the new block; the sub-tile of S that a step needs
      // is fetched a step (the first one, the products) ahead
      const float* xold = S.val + (size_t)(oi >= 0 ? oi : 0) * kTiles + (size_t)(32 * q) * SB;
      const int c_first = symd ? q : 0;  // sub-blocks before it are written as mirrors
      float4 xg[8];
      if (oi >= 0) tile_fetch(xold + 32 * c_first, SB, lane, xg);
      if (!mbar_wait_warp(&tfull[buf], ((it - 1) >> 1) & 1, &s_abort)) break;
      tc_fence_after();
      float* xnew = bn.val + (size_t)o * kTiles + (size_t)(32 * q) * SB;
      // stored splits (not with kStaged)
      char* hrow = kStaged<P> ? nullptr : static_cast<char*>(bn.hi) + ((size_t)o * kTiles + (size_t)row * SB) * C::eb;
      char* lrow = bn.lo ? static_cast<char*>(bn.lo) + ((size_t)o * kTiles + (size_t)row * SB) * C::eb : hrow;
      int kept = 0;
#pragma unroll 1
      for (int c = c_first; c < 4; ++c) {
        uint32_t v[32];
        if (has) {
          tmem_ld32(tmem + (static_cast<uint32_t>(32 * q) << 16) + buf * SB + 32 * c, v);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = 0u;
        }
        // S's sub-tile
        float xs[32];
        if (oi >= 0) {
          tile_turn_in(reinterpret_cast<uint8_t*>(s_sym[q]), lane, xg, xs);
          if (c < 3) tile_fetch(xold + 32 * (c + 1), SB, lane, xg);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) xs[j] = 0.0f;
        }
        float y[32];
        double ss = 0.0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float cxx = __uint_as_float(v[j]);
          y[j] = fmaf(gamma, xs[j], alpha * cxx);
          if (ep.d != 0.0f && I == J && row == 32 * c + j && I * SB + row < a.n) y[j] += ep.d;
        }
        if (symd && c == q) {
          // the 32 x 32 diagonal sub-block: element (l, j) with j < l from lane j
          __syncwarp();  // every lane is done with what tile_turn_in or tile_store left there
#pragma unroll
          for (int j = 0; j < 32; ++j) s_sym[q][lane][j] = y[j];
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j < lane) y[j] = s_sym[q][j][lane];
          __syncwarp();
        }
        // The FP32 sum of the squares decides the sub-blocks that are clearly dropped (its
        // rounding, 37 steps of 2^-24, is a fortieth of drop32's margin): only the others take FP64 work.
        float s32 = 0.0f;
#pragma unroll
        for (int j = 0; j < 32; ++j) s32 = fmaf(y[j], y[j], s32);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s32 += __shfl_xor_sync(0xffffffffu, s32, d);
        const bool open = !(s32 < drop32);
        if (open) {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const double d = abs_to_f64(y[j]);
            ss = fma(d, d, ss);
          }
        }
        // squared Frobenius norm of sub-block (q, c); this lane's share of it is also its
        // share of ||X||_F^2 when the sub-block is kept.  (The FP64 pipe, at 1.7 results per
        // clock and SM, bounds the blocks of few products: one FMA per element and no
        // conversion leaves 5 us of the 19 us that two of each took.)
        const double mine = ss;
        if (open) ss = warp_sum(ss);
        const bool keep = open && ss >= a.tau2 && ss > 0.0;
        if (!keep) {
#pragma unroll
          for (int j = 0; j < 32; ++j) y[j] = 0.0f;
        } else {
          kept = 1;
        }
        const double u2 = keep ? mine : 0.0;
        if (I == J && c == q) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j == lane) t1 += (double)y[j];
        }
        const bool twice = mirror || (symd && c > q);
        t2 += twice ? 2.0 * u2 : u2;
        tile_store(reinterpret_cast<uint8_t*>(s_sym[q]), lane, y, xnew + 32 * c, SB);
        if constexpr (!kStaged<P>) store_operands<P>(y, hrow + 32 * c * C::eb, lrow + 32 * c * C::eb);
        if (twice) {
          // element (row, 32c + j) of block (I, J) is element (32c + j, row) of
          // block (J, I) (of this block itself for symd): for each j the 32
          // lanes write 32 consecutive values
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const size_t e = (size_t)(32 * c + j) * SB + row;
            xmir[e] = y[j];
            if constexpr (!kStaged<P>) store_operand1<P>(y[j], bn.hi, bn.lo ? bn.lo : bn.hi, (size_t)om * kTiles + e);
          }
        }
      }
      tc_fence_before();
      if (lane == 0) {
        // the block is live when any of its 32-row bands kept a sub-block
        if (kept) {
          atomicOr(&bn.live[I * MW + (J >> 5)], 1u << (J & 31));
          if (mirror) atomicOr(&bn.live[J * MW + (I >> 5)], 1u << (I & 31));
        }
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[buf])) : "memory");
      }
    }
    t1 = warp_sum(t1);
    t2 = warp_sum(t2);
    if (lane == 0) {
      s_red[q][0] = t1;
      s_red[q][1] = t2;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 64) {
    a.parts_out[3 * blockIdx.x] = s_red[0][0] + s_red[1][0] + s_red[2][0] + s_red[3][0];
    a.parts_out[3 * blockIdx.x + 1] = s_red[0][1] + s_red[1][1] + s_red[2][1] + s_red[3][1];
    a.parts_out[3 * blockIdx.x + 2] = 0.0;
    if (s_abort) atomicExch(&st->err, TB_ERR_TIMEOUT);
  }
  if (warp == 1) {
    tc_fence_after();
    if (lane == 0) {
      // wait (bounded) until every issued MMA has retired before TMEM is freed
      const unsigned long long t0 = gtime();
      while (!mbar_try(&mdone, 0) && gtime() - t0 < kWaitNs) {
      }
    }
    __syncwarp();
    tmem_dealloc(tmem, kCols);
  }
}

// Final iterate (buffer chosen by the iteration count) -> dense FP64 D.
__global__ void k_bsr_to_dense(const SP2State* st, Args a, Buf b0, Buf b1, Sym sy0, Sym sy1, double* D) {
  if (st->err) return;  // D stays zero; the report carries the error
  const Buf& b = (st->iters & 1) ? b1 : b0;
  const int nblk = min(b.row_ptr[a.nsb], a.cap);
  for (int o = blockIdx.x; o < nblk; o += gridDim.x) {
    const int I = slot_row(b, a.nsb, o), J = b.col[o];
    for (int e = threadIdx.x; e < kTiles; e += blockDim.x) {
      const int r = I * SB + e / SB, c = J * SB + e % SB;
      if (r < a.n && c < a.n) D[(size_t)r * a.n + c] = (double)b.val[(size_t)o * kTiles + e];
    }
  }
}

// out = alpha X + delta I on X's pattern (X stores every diagonal block when
// delta != 0): values, operand splits and bitmaps.  Exact up to
// the FP32 rounding of the values; nothing is dropped.
template <int P>
__global__ void __launch_bounds__(256) k_bsr_affine(Args a, Buf X, Buf out, float alpha, float delta) {
  if (a.st->done || a.st->err) return;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  for (int i = tid; i <= a.nsb; i += nth) out.row_ptr[i] = X.row_ptr[i];
  for (int i = tid; i < a.nsb * MW; i += nth) {
    const int I = i / MW, w = i % MW;
    out.stored[i] = X.stored[i];
    out.live[i] = X.live[i] | ((delta != 0.0f && (I >> 5) == w) ? 1u << (I & 31) : 0u);
  }
  const int nblk = X.row_ptr[a.nsb];
  for (int o = blockIdx.x; o < nblk; o += gridDim.x) {
    const int I = slot_row(X, a.nsb, o), J = X.col[o];
    const bool diag = I == J && delta != 0.0f;
    if (threadIdx.x == 0) out.col[o] = J;
    if constexpr (kStaged<P>) {
      // 16 bytes a lane, consecutive across the block, several loads in flight (a thread
      // per 32-value segment took 0.31 ms for what memory moves in 0.05)
      const float4* src = reinterpret_cast<const float4*>(X.val + (size_t)o * kTiles);
      float4* dst = reinterpret_cast<float4*>(out.val + (size_t)o * kTiles);
#pragma unroll 8
      for (int e = threadIdx.x; e < kTiles / 4; e += 256) {
        float4 x = src[e];
        x.x *= alpha;
        x.y *= alpha;
        x.z *= alpha;
        x.w *= alpha;
        if (diag) {
          const int r = e / (SB / 4), d = r - 4 * (e % (SB / 4));
          if (I * SB + r < a.n) {
            if (d == 0) x.x += delta;
            if (d == 1) x.y += delta;
            if (d == 2) x.z += delta;
            if (d == 3) x.w += delta;
          }
        }
        dst[e] = x;
      }
    } else {
      for (int seg = threadIdx.x; seg < SB * 4; seg += blockDim.x) {
        const int r = seg >> 2, cs = seg & 3;
        const size_t e0 = (size_t)o * kTiles + (size_t)r * SB + 32 * cs;
        float y[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          y[j] = alpha * X.val[e0 + j];
          if (diag && r == 32 * cs + j && I * SB + r < a.n) y[j] += delta;
        }
        float* dst = out.val + e0;
#pragma unroll
        for (int j = 0; j < 32; ++j) dst[j] = y[j];
        char* hp = static_cast<char*>(out.hi) + e0 * Prec<P>::eb;
        char* lp = out.lo ? static_cast<char*>(out.lo) + e0 * Prec<P>::eb : hp;
        store_operands<P>(y, hp, lp);
      }
    }
  }
}

// Final iterate -> BSR D (structure and FP64 values, plus dshift on the
// diagonal of the n x n block); TB_ERR_OOM in D.status when it holds more
// blocks than D.cap.  sel < 0: the SP2 iterate (buffer by the iteration
// count), else buffer sel.
__global__ void k_bsr_to_bsr(const SP2State* st, Args a, Buf b0, Buf b1, int sel, double dshift, tb_bsr D) {
  const Buf& b = (sel < 0 ? (st->iters & 1) : sel) ? b1 : b0;
  // after an error the iterate may never have been written: no blocks
  const int nblk = st->err ? 0 : min(b.row_ptr[a.nsb], a.cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) *D.status = nblk > D.cap ? TB_ERR_OOM : TB_OK;
  if (nblk > D.cap || st->err) {
    // an empty matrix: no row holds a block
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= a.nsb; i += gridDim.x * blockDim.x) D.row_ptr[i] = 0;
    return;
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= a.nsb; i += gridDim.x * blockDim.x)
    D.row_ptr[i] = b.row_ptr[i];
  for (int o = blockIdx.x; o < nblk; o += gridDim.x) {
    const int J = b.col[o];
    if (threadIdx.x == 0) D.col[o] = J;
    const int I = dshift != 0.0 ? slot_row(b, a.nsb, o) : -1;
    const float* src = b.val + (size_t)o * kTiles;
    double* dst = D.val + (size_t)o * kTiles;
    for (int e = threadIdx.x; e < kTiles; e += blockDim.x) {
      const int r = e / SB;
      const bool dg = I == J && r == e % SB && I * SB + r < a.n;
      dst[e] = (double)src[e] + (dg ? dshift : 0.0);
    }
  }
}

__global__ void k_bsr_report(SP2State* st, Args a, Buf b0, Buf b1, tb_sp2_report* rep, int* nblk_out) {
  const Buf& b = (st->iters & 1) ? b1 : b0;
  if (nblk_out) *nblk_out = min(b.row_ptr[a.nsb], a.cap);
  if (!rep) return;
  const double t1 = st->t1[st->iters], t2 = st->t2[st->iters];
  int status = TB_OK;
  if (st->err) status = st->err;
  else if (fabs(t1 - a.nocc) > 0.25) status = TB_ERR_GAP;
  rep->status = status;
  rep->iters = st->iters;
  rep->refine_iters = 0;
  rep->n = a.n;
  rep->eps_min = st->emin;
  rep->eps_max = st->emax;
  rep->trace = t1;
  rep->idem_trace = t1 - t2;
  rep->idem_fro = -1.0;
  rep->branch_bits[0] = st->branch[0];
  rep->branch_bits[1] = st->branch[1];
  rep->refine_bits = 0;
  rep->block_products = (long long)st->block_products;
  rep->blocks = min(b.row_ptr[a.nsb], a.cap);
}

constexpr int kMaxBufs = 7;  // matrices of the Fermi expansion (SP2: two)

struct BsrLayout {
  int n, ld, nsb, cap, pcap, nbuf;
  bool staged;  // tf32x3: FP32 masters only, no stored operand splits
  size_t off_state, off_bparts, off_parts, off_scal, off_flags, off_cand, off_cnt, off_oldidx,
      off_rowp, off_ucnt, off_pcnt, off_pairs, off_list, off_npl, off_order;
  size_t off_rp[kMaxBufs], off_col[kMaxBufs], off_st[kMaxBufs], off_lv[kMaxBufs],
      off_val[kMaxBufs], off_hi[kMaxBufs], off_lo[kMaxBufs];
  size_t total;
  int nparts;
};

// Workspace of nbuf block-sparse matrices of bpr blocks per block row on
// average (0: every block) and the shared symbolic arrays.
BsrLayout bsr_layout(int n, int prec, int bpr, int nbuf) {
  BsrLayout L{};
  L.n = n;
  L.ld = round_up(std::max(n, 1), SB);
  L.nsb = L.ld / SB;
  L.nbuf = nbuf;
  const int per_row = (bpr <= 0 || bpr > L.nsb) ? L.nsb : bpr;
  L.cap = L.nsb * per_row;
  L.pcap = L.cap * per_row;
  L.nparts = std::max(kFillSplit * L.nsb, kMaxGrid);
  size_t o = 0;
  auto take = [&](size_t bytes) {
    size_t r = o;
    o += (bytes + 1023) / 1024 * 1024;
    return r;
  };
  const size_t eb = (prec == TB_PREC_TF32 || prec == TB_PREC_TF32X3) ? 4 : 2;
  const bool split = prec == TB_PREC_TF32X3 || prec == TB_PREC_BF16X3;
  L.staged = prec == TB_PREC_TF32X3;
  L.off_state = take(sizeof(SP2State));
  L.off_bparts = take(sizeof(double) * 2 * std::max((n + 7) / 8, kBndSplit * L.nsb));
  L.off_parts = take(sizeof(double) * 3 * 2 * L.nparts);
  L.off_scal = take(sizeof(int) * 4);
  L.off_flags = take(sizeof(uint16_t) * (size_t)L.nsb * L.nsb);
  L.off_cand = take(sizeof(uint32_t) * MW * L.nsb);
  L.off_cnt = take(sizeof(int) * L.nsb);
  L.off_rowp = take(sizeof(int) * L.nsb);
  L.off_ucnt = take(sizeof(int) * L.nsb);
  L.off_oldidx = take(sizeof(int) * L.cap);
  L.off_pcnt = take(sizeof(int2) * L.cap);
  L.off_pairs = take(sizeof(int2) * (size_t)L.pcap);
  L.off_list = take(sizeof(Unit) * L.cap);
  L.off_npl = take(sizeof(int) * L.cap);
  L.off_order = take(sizeof(Unit) * L.cap);
  for (int b = 0; b < nbuf; ++b) {
    L.off_rp[b] = take(sizeof(int) * (L.nsb + 1));
    L.off_col[b] = take(sizeof(int) * L.cap);
    L.off_st[b] = take(sizeof(uint32_t) * MW * L.nsb);
    L.off_lv[b] = take(sizeof(uint32_t) * MW * L.nsb);
    L.off_val[b] = take(sizeof(float) * (size_t)L.cap * kTiles);
    L.off_hi[b] = L.staged ? 0 : take(eb * (size_t)L.cap * kTiles);
    L.off_lo[b] = (split && !L.staged) ? take(eb * (size_t)L.cap * kTiles) : 0;
  }
  L.total = o;
  return L;
}

int make_block_map(tb_ctx* ctx, int prec, const void* base, int rows, CUtensorMap* map) {
  const bool tf = prec == TB_PREC_TF32 || prec == TB_PREC_TF32X3;
  const size_t eb = tf ? 4 : 2;
  const cuuint64_t dims[2] = {(cuuint64_t)SB, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)(SB * eb)};
  const cuuint32_t box[2] = {(cuuint32_t)(128 / eb), 128};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = ctx->encode_tiled(map, tf ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                                 const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                 CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return tb_fail(ctx, TB_ERR_CUDA, "cuTensorMapEncodeTiled (blocks) failed (%d)", (int)r);
  return TB_OK;
}

// One block-sparse matrix of the workspace and the tensor maps of its operands.
struct Mat {
  Buf b;
  CUtensorMap mh, ml;
};

// The workspace bound to its parts.
struct Engine {
  BsrLayout L;
  SP2State* st;
  double* bparts;
  double* parts;  // two slots of 3 * nparts
  Sym sy;
  Mat m[kMaxBufs];
};

int bind_engine(tb_ctx* ctx, int prec, const BsrLayout& L, void* ws, Engine* e) {
  char* base = static_cast<char*>(ws);
  e->L = L;
  e->st = reinterpret_cast<SP2State*>(base + L.off_state);
  e->bparts = reinterpret_cast<double*>(base + L.off_bparts);
  e->parts = reinterpret_cast<double*>(base + L.off_parts);
  Sym& sy = e->sy;
  sy.cand = reinterpret_cast<uint32_t*>(base + L.off_cand);
  sy.cnt = reinterpret_cast<int*>(base + L.off_cnt);
  sy.rowp = reinterpret_cast<int*>(base + L.off_rowp);
  sy.ucnt = reinterpret_cast<int*>(base + L.off_ucnt);
  sy.old_idx = reinterpret_cast<int*>(base + L.off_oldidx);
  sy.pcnt = reinterpret_cast<int2*>(base + L.off_pcnt);
  sy.pairs = reinterpret_cast<int2*>(base + L.off_pairs);
  sy.scal = reinterpret_cast<int*>(base + L.off_scal);
  sy.list = reinterpret_cast<Unit*>(base + L.off_list);
  sy.npl = reinterpret_cast<int*>(base + L.off_npl);
  sy.order = reinterpret_cast<Unit*>(base + L.off_order);
  sy.flags = reinterpret_cast<uint16_t*>(base + L.off_flags);
  for (int i = 0; i < L.nbuf; ++i) {
    Buf& b = e->m[i].b;
    b.row_ptr = reinterpret_cast<int*>(base + L.off_rp[i]);
    b.col = reinterpret_cast<int*>(base + L.off_col[i]);
    b.stored = reinterpret_cast<uint32_t*>(base + L.off_st[i]);
    b.live = reinterpret_cast<uint32_t*>(base + L.off_lv[i]);
    b.val = reinterpret_cast<float*>(base + L.off_val[i]);
    b.hi = L.staged ? nullptr : base + L.off_hi[i];
    b.lo = L.off_lo[i] ? base + L.off_lo[i] : nullptr;
    // staged: the numeric kernel reads the FP32 masters (tf32 tiles of the same shape)
    int rc = make_block_map(ctx, prec, L.staged ? static_cast<void*>(b.val) : b.hi, L.cap * SB, &e->m[i].mh);
    if (rc) return rc;
    if (b.lo) {
      if ((rc = make_block_map(ctx, prec, b.lo, L.cap * SB, &e->m[i].ml))) return rc;
    } else {
      e->m[i].ml = e->m[i].mh;
    }
  }
  return TB_OK;
}

Args engine_args(const Engine& e, double tau) {
  Args a{};
  a.n = e.L.n;
  a.ld = e.L.ld;
  a.nsb = e.L.nsb;
  a.mw = (e.L.nsb + 31) / 32;
  a.cap = e.L.cap;
  a.pcap = e.L.pcap;
  a.tau2 = tau * tau;
  a.st = e.st;
  return a;
}

// X0 = s (e I - H) into out, with the drop, from a dense H (Hb null) or a BSR
// H; trace partials per block row into a.parts_out.
template <int P>
int launch_start(tb_ctx* ctx, Engine& e, const Args& a, const double* H, const tb_bsr* Hb, Mat& out,
                 cudaStream_t s) {
  const int nsb = e.L.nsb;
  if (Hb) {
    TB_CUDA_TRY(ctx, cudaMemsetAsync(e.sy.flags, 0, sizeof(uint16_t) * (size_t)nsb * nsb, s));
    k_bsr_init_flags_in<<<std::max(1, std::min(Hb->cap, 8192)), 256, 0, s>>>(*Hb, a, e.sy);
    TB_LAUNCH_CHECK(ctx);
    k_bsr_init_flags_diag<<<nsb, 256, 0, s>>>(*Hb, a, e.sy);
  } else {
    k_bsr_init_flags<<<dim3(nsb, nsb), 256, 0, s>>>(H, a, e.sy);
  }
  TB_LAUNCH_CHECK(ctx);
  k_bsr_init_rows<<<nsb, 256, 0, s>>>(a, e.sy, out.b);
  TB_LAUNCH_CHECK(ctx);
  k_bsr_scan_rows<<<1, 32, 0, s>>>(a, e.sy, out.b.row_ptr);
  TB_LAUNCH_CHECK(ctx);
  if (Hb) k_bsr_init_fill_in<P><<<dim3(nsb, kFillSplit), 256, 0, s>>>(*Hb, a, e.sy, out.b);
  else k_bsr_init_fill<P><<<dim3(nsb, kFillSplit), 256, 0, s>>>(H, a, e.sy, out.b);
  TB_LAUNCH_CHECK(ctx);
  return TB_OK;
}

// out = alpha A B + gamma S + delta I (S may be null), thresholded: the
// symbolic phase, then the persistent numeric kernel (trace partials per CTA
// into a.parts_out).  A and B are symmetric and their bitmaps current; out
// is none of A, B, S.  prof_k >= 0 marks the numeric launch for profiling.
template <int P>
int launch_product(tb_ctx* ctx, Engine& e, Args a, const Mat& A, const Mat& B, const Mat* S, Mat& out, Epi ep,
                   int grid, cudaStream_t s, bool decide = false, int prof_k = -1) {
  a.same_ab = &A == &B;
  const Buf none{};
  const Buf& Sb = S ? S->b : none;
  const int nsb = e.L.nsb;
  k_bsr_cand<<<nsb, 256, 0, s>>>(a, A.b, B.b, Sb, e.sy, decide);
  k_bsr_fill_out<<<nsb, 256, 0, s>>>(a, A.b, B.b, Sb, out.b, e.sy);
  const int nlist = (nsb + kBand - 1) / kBand * a.mw;  // a warp each
  k_bsr_pairs<<<nsb * kPairSplit + (nlist + 7) / 8, 256, 0, s>>>(a, A.b, B.b, out.b, e.sy);
  k_bsr_balance<<<kClasses, 1024, 0, s>>>(a, e.sy);
  TB_LAUNCH_CHECK(ctx);
  if (prof_k >= 0) tb_prof_mark(ctx, 1, 2 * prof_k, s);
  k_bsr_step_tc<P><<<grid, kNumThreads<P>, kNumSmem<P>, s>>>(a, A.mh, A.ml, B.mh, B.ml, Sb, out.b, e.sy, ep);
  TB_LAUNCH_CHECK(ctx);
  if (prof_k >= 0) tb_prof_mark(ctx, 1, 2 * prof_k + 1, s);
  return TB_OK;
}

template <int P>
int prepare_numeric(tb_ctx* ctx, int* grid) {
  static unsigned long long attr_done = 0;
  if (int rc = tb_smem_attr(ctx, k_bsr_step_tc<P>, kNumSmem<P>, &attr_done)) return rc;
  *grid = tb_persistent_grid(ctx, kMaxGrid);
  return TB_OK;
}

// H dense (Hb null) or BSR (Hb); D dense or BSR (Db).
template <int P>
int run_bsr(tb_ctx* ctx, const double* H, const tb_bsr* Hb, int n, double nocc, const tb_sp2_opts* o, double* D,
            tb_bsr* Db, void* ws, size_t ws_bytes, tb_sp2_report* rep, cudaStream_t s) {
  const BsrLayout L = bsr_layout(n, o->precision, o->bsr_blocks_per_row, 2);
  if (ws_bytes < L.total)
    return tb_fail(ctx, TB_ERR_ARG, "workspace %zu bytes < required %zu (block-sparse)", ws_bytes, L.total);
  Engine e;
  int rc = bind_engine(ctx, o->precision, L, ws, &e);
  if (rc) return rc;
  SP2State* st = e.st;
  double* slot[2] = {e.parts, e.parts + 3 * (size_t)L.nparts};
  Args a = engine_args(e, o->tau);
  a.nocc = nocc;
  a.tol = o->tol;
  a.rule = o->rule;
  a.max_iter = o->max_iter;
  {
    const double u = (o->precision == TB_PREC_TF32X3 || o->precision == TB_PREC_BF16X3) ? 0x1p-24
                     : o->precision == TB_PREC_TF32 ? 0x1p-11 : 0x1p-8;
    a.floor = 2.0 * n * u;
  }
  ctx->prof_n[0] = ctx->prof_n[1] = 0;
  TB_CUDA_TRY(ctx, cudaMemsetAsync(st, 0, sizeof(SP2State), s));
  if (Hb) {
    k_bsr_status_in<<<1, 1, 0, s>>>(Hb->status, st);
    TB_LAUNCH_CHECK(ctx);
    k_bsr_bounds_in<<<dim3(L.nsb, kBndSplit), 256, 0, s>>>(*Hb, e.bparts);
    TB_LAUNCH_CHECK(ctx);
    k_bsr_bounds<<<1, 32, 0, s>>>(e.bparts, kBndSplit * L.nsb, st);
  } else {
    const int nb = (n + 7) / 8;
    if ((rc = sp2_launch_bounds(ctx, H, n, e.bparts, s))) return rc;
    k_bsr_bounds<<<1, 32, 0, s>>>(e.bparts, nb, st);
  }
  TB_LAUNCH_CHECK(ctx);
  a.parts_out = slot[0];
  if ((rc = launch_start<P>(ctx, e, a, H, Hb, e.m[0], s))) return rc;

  int grid = 0;
  if ((rc = prepare_numeric<P>(ctx, &grid))) return rc;
  // X^2 (branch 0) or 2X - X^2 (branch 1), the lo x lo product of a square
  const Epi sp2_epi{1.0f, 0.0f, -1.0f, 2.0f, 0.0f, 1, 1};
  tb_prof_mark(ctx, 0, 0, s);
  for (int k = 0; k <= o->max_iter; ++k) {
    a.k = k;
    a.parts_in = slot[k & 1];
    a.nparts_in = k == 0 ? kFillSplit * L.nsb : grid;
    a.parts_out = slot[(k + 1) & 1];
    Mat& bo = e.m[k & 1];
    Mat& bn = e.m[(k + 1) & 1];
    if ((rc = launch_product<P>(ctx, e, a, bo, bo, &bo, bn, sp2_epi, grid, s, true, k))) return rc;
    tb_prof_mark(ctx, 0, k + 1, s);
  }
  if (Db) {
    k_bsr_to_bsr<<<std::min(4096, std::max(1, L.cap)), 256, 0, s>>>(st, a, e.m[0].b, e.m[1].b, -1, 0.0, *Db);
  } else {
    TB_CUDA_TRY(ctx, cudaMemsetAsync(D, 0, sizeof(double) * (size_t)n * n, s));
    k_bsr_to_dense<<<std::min(4096, std::max(1, L.cap)), 256, 0, s>>>(st, a, e.m[0].b, e.m[1].b, e.sy, e.sy, D);
  }
  TB_LAUNCH_CHECK(ctx);
  k_bsr_report<<<1, 1, 0, s>>>(st, a, e.m[0].b, e.m[1].b, rep, nullptr);
  TB_LAUNCH_CHECK(ctx);
  return TB_OK;
}

// ------------------------------------------------ block-sparse Fermi expansion

constexpr int kFoeBufs = 7;  // E (two, alternating), Y, A, Z, T, W
constexpr int kFoeMinM = 8;

__global__ void k_bsr_fail(SP2State* st, int code) { st->err = code; }

__global__ void k_bsr_fermi_report(tb_fermi_report* rep, double* mu_out, int status, int iters, int m, int n,
                                   double mu, double trace, double trace_dd, double emin, double emax) {
  if (mu_out && status == TB_OK) *mu_out = mu;
  if (!rep) return;
  rep->status = status;
  rep->mu_iters = iters;
  rep->m = m;
  rep->n = n;
  rep->mu = mu;
  rep->trace = trace;
  rep->trace_dd = trace_dd;
  rep->eps_min = emin;
  rep->eps_max = emax;
}

// The recursive Fermi-operator expansion of dm_fermi on thresholded
// block-sparse products (every product and the start drop 32 x 32 blocks
// with Frobenius norm < tau; the affine steps are exact), the chemical
// potential by the host: one expansion per step, two traces read back.
template <int P>
int run_bsr_fermi(tb_ctx* ctx, const tb_bsr* Hb, int n, double nocc, double kT, const tb_fermi_opts* o,
                  double tau, int bpr, tb_bsr* Db, double* mu_dev, void* ws, size_t ws_bytes,
                  tb_fermi_report* rep, cudaStream_t s) {
  const BsrLayout L = bsr_layout(n, o->precision, bpr, kFoeBufs);
  if (ws_bytes < L.total)
    return tb_fail(ctx, TB_ERR_ARG, "workspace %zu bytes < required %zu (block-sparse)", ws_bytes, L.total);
  Engine e;
  int rc = bind_engine(ctx, o->precision, L, ws, &e);
  if (rc) return rc;
  SP2State* st = e.st;
  Args a = engine_args(e, tau);
  a.keep_diag = 1;
  a.parts_out = e.parts;
  const int m_max = o->m > 0 ? o->m : 14;
  const int ns = o->ns_iters > 0 ? o->ns_iters : 3;
  const double tol = o->trace_tol > 0.0 ? o->trace_tol : 1e-6 + 1e-9 * nocc;
  const double beta = 1.0 / kT;
  TB_CUDA_TRY(ctx, cudaMemsetAsync(st, 0, sizeof(SP2State), s));
  k_bsr_status_in<<<1, 1, 0, s>>>(Hb->status, st);
  k_bsr_bounds_in<<<dim3(L.nsb, kBndSplit), 256, 0, s>>>(*Hb, e.bparts);
  k_bsr_bounds<<<1, 32, 0, s>>>(e.bparts, kBndSplit * L.nsb, st);
  TB_LAUNCH_CHECK(ctx);
  SP2State hs;
  double mu0 = NAN;
  TB_CUDA_TRY(ctx, cudaMemcpyAsync(&hs, st, sizeof(SP2State), cudaMemcpyDeviceToHost, s));
  if (mu_dev) TB_CUDA_TRY(ctx, cudaMemcpyAsync(&mu0, mu_dev, sizeof(double), cudaMemcpyDeviceToHost, s));
  TB_CUDA_TRY(ctx, cudaStreamSynchronize(s));
  const double emin = hs.emin, emax = hs.emax;
  double lo = emin - 40.0 * kT - 1.0, hi = emax + 40.0 * kT + 1.0;
  int m = std::min(kFoeMinM, m_max);
  while (m < m_max && !(beta * (hi - lo) <= std::ldexp(1.0, m + 1))) ++m;
  double mu = (std::isfinite(mu0) && mu0 > lo && mu0 < hi) ? mu0 : 0.5 * (emin + emax);
  int status = hs.err ? hs.err : TB_ERR_NOT_CONVERGED;
  if (!hs.err && !(beta * (hi - lo) <= std::ldexp(1.0, m + 1))) status = TB_ERR_ARG;  // start undefined
  int grid = 0;
  if ((rc = prepare_numeric<P>(ctx, &grid))) return rc;
  std::vector<double> hp(3 * (size_t)grid);
  Mat* E[2] = {&e.m[0], &e.m[1]};
  Mat* Y = &e.m[2];
  Mat* A = &e.m[3];
  Mat* Z = &e.m[4];
  Mat* T = &e.m[5];
  Mat* W = &e.m[6];
  auto affine = [&](const Mat& X, Mat& out, float alpha, float delta) -> int {
    k_bsr_affine<P><<<std::min(4096, std::max(1, L.cap)), 256, 0, s>>>(a, X.b, out.b, alpha, delta);
    TB_LAUNCH_CHECK(ctx);
    return TB_OK;
  };
  auto product = [&](const Mat& X1, const Mat& X2, const Mat* S, Mat& out, Epi ep) -> int {
    int r = launch_product<P>(ctx, e, a, X1, X2, S, out, ep, grid, s);
    if (r) return r;
    TB_LAUNCH_CHECK(ctx);
    return TB_OK;
  };
  const Epi plain{1.0f, 0.0f, 1.0f, 0.0f, 0.0f, 0, 0};
  auto with = [](float alpha, float gamma, float delta, int lolo) { return Epi{alpha, gamma, alpha, gamma, delta, 0, lolo}; };
  int it = 0, fin = 0;
  double trd = NAN, t1 = NAN;
  for (it = 1; status == TB_ERR_NOT_CONVERGED && it <= o->mu_iters; ++it) {
    // L = beta/2^(m+2) (mu I - H), then E0 = L - 4/3 L L^2
    a.x0_e = mu;
    a.x0_s = beta / std::ldexp(1.0, m + 2);
    if ((rc = launch_start<P>(ctx, e, a, nullptr, Hb, *Y, s))) return rc;
    a.x0_s = 0.0;
    if ((rc = product(*Y, *Y, nullptr, *A, with(1.0f, 0.0f, 0.0f, 1)))) return rc;
    if ((rc = product(*Y, *A, Y, *E[0], with(-4.0f / 3.0f, 1.0f, 0.0f, 0)))) return rc;
    int cur = 0;
    for (int step = 0; step < m; ++step) {
      Mat* Zc = Z;
      Mat* Yc = Y;
      // W = (I - 2E)(I + 2E), A = 2I - W
      if ((rc = affine(*E[cur], *T, -2.0f, 1.0f)) || (rc = affine(*E[cur], *Y, 2.0f, 1.0f))) return rc;
      if ((rc = product(*T, *Y, nullptr, *W, plain))) return rc;
      if ((rc = affine(*W, *A, -1.0f, 2.0f))) return rc;
      // Z1 = (32 A A - 144 A + 210 I) / 99, then Newton-Schulz Z <- Z (2I - A Z)
      if ((rc = product(*A, *A, A, *Zc, with(32.0f / 99.0f, -144.0f / 99.0f, 210.0f / 99.0f, 1)))) return rc;
      for (int k = 1; k < ns; ++k) {
        if ((rc = product(*A, *Zc, nullptr, *T, with(-1.0f, 0.0f, 2.0f, 0)))) return rc;
        if ((rc = product(*Zc, *T, nullptr, *Yc, plain))) return rc;
        std::swap(Zc, Yc);
      }
      // E <- E + E (Z W): the last product's partials are Tr E and ||E||_F^2
      if ((rc = product(*Zc, *W, nullptr, *T, plain))) return rc;
      if ((rc = product(*E[cur], *T, E[cur], *E[1 - cur], with(1.0f, 1.0f, 0.0f, 0)))) return rc;
      cur = 1 - cur;
    }
    TB_CUDA_TRY(ctx, cudaMemcpyAsync(hp.data(), e.parts, sizeof(double) * hp.size(), cudaMemcpyDeviceToHost, s));
    TB_CUDA_TRY(ctx, cudaMemcpyAsync(&hs, st, sizeof(SP2State), cudaMemcpyDeviceToHost, s));
    TB_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    if (hs.err) {
      status = hs.err;
      break;
    }
    double tr = 0.0, fro = 0.0;
    for (int i = 0; i < grid; ++i) {
      tr += hp[3 * i];
      fro += hp[3 * i + 1];
    }
    fin = cur;
    trd = 0.5 * n + tr;
    t1 = 0.25 * n - fro;  // Tr D(I - D) = n/4 - ||E||_F^2
    const double dev = trd - nocc;
    if (fabs(dev) <= tol) {
      status = TB_OK;
      break;
    }
    if (it == o->mu_iters) break;
    if (dev < 0.0) lo = mu;
    else hi = mu;
    mu = foe_next_mu(mu, dev, t1, beta, tol, lo, hi);
  }
  it = std::min(it, o->mu_iters);
  // D = I/2 + E; after an error (the state's flag, raised here for one the
  // host found) an empty matrix
  if (status != TB_OK && status != TB_ERR_NOT_CONVERGED) k_bsr_fail<<<1, 1, 0, s>>>(st, status);
  k_bsr_to_bsr<<<std::min(4096, std::max(1, L.cap)), 256, 0, s>>>(st, a, E[0]->b, E[1]->b, fin, 0.5, *Db);
  TB_LAUNCH_CHECK(ctx);
  k_bsr_fermi_report<<<1, 1, 0, s>>>(rep, mu_dev, status, it, m, n, mu, trd, t1, emin, emax);
  TB_LAUNCH_CHECK(ctx);
  return TB_OK;
}

}  // namespace

int dm_sp2_bsr_workspace(int n, const tb_sp2_opts* o, int nsm, size_t* bytes) {
  if (n > kMaxNsb * SB) return TB_ERR_UNSUPPORTED;
  (void)nsm;
  *bytes = bsr_layout(n, o->precision, o->bsr_blocks_per_row, 2).total;
  return TB_OK;
}

int dm_sp2_bsr(tb_ctx* ctx, const double* H, int n, double nocc, const tb_sp2_opts* o, double* D, void* ws,
               size_t ws_bytes, tb_sp2_report* rep, cudaStream_t s) {
  if (n > kMaxNsb * SB) return tb_fail(ctx, TB_ERR_UNSUPPORTED, "block-sparse SP2 supports n <= %d", kMaxNsb * SB);
  switch (o->precision) {
    case TB_PREC_TF32: return run_bsr<TB_PREC_TF32>(ctx, H, nullptr, n, nocc, o, D, nullptr, ws, ws_bytes, rep, s);
    case TB_PREC_TF32X3: return run_bsr<TB_PREC_TF32X3>(ctx, H, nullptr, n, nocc, o, D, nullptr, ws, ws_bytes, rep, s);
    case TB_PREC_BF16: return run_bsr<TB_PREC_BF16>(ctx, H, nullptr, n, nocc, o, D, nullptr, ws, ws_bytes, rep, s);
    case TB_PREC_BF16X3: return run_bsr<TB_PREC_BF16X3>(ctx, H, nullptr, n, nocc, o, D, nullptr, ws, ws_bytes, rep, s);
    default: return tb_fail(ctx, TB_ERR_UNSUPPORTED, "block-sparse SP2 needs a tensor-core precision");
  }
}

extern "C" int dm_sp2_sparse(tb_ctx* ctx, const tb_bsr* H, double nocc, const tb_sp2_opts* o, tb_bsr* D, void* ws,
                             size_t ws_bytes, tb_sp2_report* rep, void* stream) {
  if (!ctx) return TB_ERR_ARG;
  if (!H || !D || !o || !ws) return tb_fail(ctx, TB_ERR_ARG, "null argument to dm_sp2_sparse");
  const int n = H->n;
  if (n < 1 || D->n != n || H->nsb != (n + SB - 1) / SB || D->nsb != H->nsb)
    return tb_fail(ctx, TB_ERR_ARG, "dm_sp2_sparse: inconsistent BSR sizes");
  if (!H->row_ptr || !H->col || !H->val || !D->row_ptr || !D->col || !D->val || !D->status)
    return tb_fail(ctx, TB_ERR_ARG, "dm_sp2_sparse: null BSR array");
  if (!(o->tau > 0.0)) return tb_fail(ctx, TB_ERR_ARG, "dm_sp2_sparse needs tau > 0");
  if (n > kMaxNsb * SB) return tb_fail(ctx, TB_ERR_UNSUPPORTED, "block-sparse SP2 supports n <= %d", kMaxNsb * SB);
  if (!(nocc >= 0.0) || nocc > n) return tb_fail(ctx, TB_ERR_ARG, "n_occ %g outside [0, n]", nocc);
  if (o->max_iter < 1 || o->max_iter > SP2_MAX_ITER)
    return tb_fail(ctx, TB_ERR_ARG, "max_iter %d outside 1..%d", o->max_iter, SP2_MAX_ITER);
  if ((reinterpret_cast<uintptr_t>(ws) & 1023) != 0) return tb_fail(ctx, TB_ERR_ARG, "workspace must be 1024-byte aligned");
  cudaStream_t s = as_stream(stream);
  switch (o->precision) {
    case TB_PREC_TF32: return run_bsr<TB_PREC_TF32>(ctx, nullptr, H, n, nocc, o, nullptr, D, ws, ws_bytes, rep, s);
    case TB_PREC_TF32X3: return run_bsr<TB_PREC_TF32X3>(ctx, nullptr, H, n, nocc, o, nullptr, D, ws, ws_bytes, rep, s);
    case TB_PREC_BF16: return run_bsr<TB_PREC_BF16>(ctx, nullptr, H, n, nocc, o, nullptr, D, ws, ws_bytes, rep, s);
    case TB_PREC_BF16X3: return run_bsr<TB_PREC_BF16X3>(ctx, nullptr, H, n, nocc, o, nullptr, D, ws, ws_bytes, rep, s);
    default: return tb_fail(ctx, TB_ERR_UNSUPPORTED, "block-sparse SP2 needs a tensor-core precision");
  }
}

extern "C" int dm_fermi_sparse_workspace_size(int n, const tb_fermi_opts* o, int blocks_per_row, size_t* bytes) {
  if (n < 1 || !o || !bytes) return TB_ERR_ARG;
  if (n > kMaxNsb * SB) return TB_ERR_UNSUPPORTED;
  *bytes = bsr_layout(n, o->precision, blocks_per_row, kFoeBufs).total;
  return TB_OK;
}

extern "C" int dm_fermi_sparse(tb_ctx* ctx, const tb_bsr* H, double nocc, double kT, const tb_fermi_opts* o,
                               double tau, int blocks_per_row, tb_bsr* D, double* mu, void* ws, size_t ws_bytes,
                               tb_fermi_report* rep, void* stream) {
  if (!ctx) return TB_ERR_ARG;
  if (!H || !D || !o || !ws) return tb_fail(ctx, TB_ERR_ARG, "null argument to dm_fermi_sparse");
  const int n = H->n;
  if (n < 1 || D->n != n || H->nsb != (n + SB - 1) / SB || D->nsb != H->nsb)
    return tb_fail(ctx, TB_ERR_ARG, "dm_fermi_sparse: inconsistent BSR sizes");
  if (!H->row_ptr || !H->col || !H->val || !H->status || !D->row_ptr || !D->col || !D->val || !D->status)
    return tb_fail(ctx, TB_ERR_ARG, "dm_fermi_sparse: null BSR array");
  if (!(tau > 0.0)) return tb_fail(ctx, TB_ERR_ARG, "dm_fermi_sparse needs tau > 0");
  if (!(kT > 0.0)) return tb_fail(ctx, TB_ERR_ARG, "dm_fermi_sparse needs kT > 0");
  if (n > kMaxNsb * SB) return tb_fail(ctx, TB_ERR_UNSUPPORTED, "block-sparse expansion supports n <= %d", kMaxNsb * SB);
  if (!(nocc >= 0.0) || nocc > n) return tb_fail(ctx, TB_ERR_ARG, "n_occ %g outside [0, n]", nocc);
  if (o->mu_iters < 1 || o->mu_iters > 100) return tb_fail(ctx, TB_ERR_ARG, "mu_iters %d outside 1..100", o->mu_iters);
  if (o->m < 0 || o->m > 30 || o->ns_iters < 0 || o->ns_iters > 8)
    return tb_fail(ctx, TB_ERR_ARG, "dm_fermi_sparse: m or ns_iters out of range");
  if ((reinterpret_cast<uintptr_t>(ws) & 1023) != 0) return tb_fail(ctx, TB_ERR_ARG, "workspace must be 1024-byte aligned");
  cudaStream_t s = as_stream(stream);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  TB_CUDA_TRY(ctx, cudaStreamIsCapturing(s, &cap));
  if (cap != cudaStreamCaptureStatusNone)
    return tb_fail(ctx, TB_ERR_UNSUPPORTED, "dm_fermi_sparse reads traces on the host: not capturable");
  switch (o->precision) {
    case TB_PREC_TF32:
      return run_bsr_fermi<TB_PREC_TF32>(ctx, H, n, nocc, kT, o, tau, blocks_per_row, D, mu, ws, ws_bytes, rep, s);
    case TB_PREC_TF32X3:
      return run_bsr_fermi<TB_PREC_TF32X3>(ctx, H, n, nocc, kT, o, tau, blocks_per_row, D, mu, ws, ws_bytes, rep, s);
    case TB_PREC_BF16:
      return run_bsr_fermi<TB_PREC_BF16>(ctx, H, n, nocc, kT, o, tau, blocks_per_row, D, mu, ws, ws_bytes, rep, s);
    case TB_PREC_BF16X3:
      return run_bsr_fermi<TB_PREC_BF16X3>(ctx, H, n, nocc, kT, o, tau, blocks_per_row, D, mu, ws, ws_bytes, rep, s);
    default: return tb_fail(ctx, TB_ERR_UNSUPPORTED, "block-sparse expansion needs a tensor-core precision");
  }
}
