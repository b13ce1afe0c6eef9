// dm_fermi's expansion loop in one launch (tf32, tf32x3): every product of every
// expansion, the elementwise steps between them and the chemical-potential
// decisions run in one persistent grid, the products separated by a grid
// barrier.
//
// What bounds the launched form: an expansion is ~70 dependent products with
// ~60 elementwise launches between them, and outside a captured graph the host
// enqueues it mu_iters (30) times for every m_max (14) doubling steps, nearly
// all of them launches that return at once: 29 ms for n = 192, where the
// products that run take well under 1 ms.  Here
//   - the loops are on the device, so nothing is enqueued that does not run;
//   - the elementwise passes are gone: I + 2E, I - 2E and A = 2I - W are multiplied
//     as E and W with a patched diagonal (patch_diag), and a result that is only
//     multiplied further has no FP32 master;
//   - a unit (128 x BN of the upper triangle) always belongs to the same CTA,
//     so the FP32 values an epilogue adds (E, W, L) are its own earlier stores,
//     and only the TMA producer waits at the barriers (the stores are another warp's, so
//     a value of the product just before is read behind that wait all the same).
// Same operand values, products and order of accumulation per element as the
// launched form (k_gemm_tc): the matrices are bitwise the same.
//
// BN (32, 64 or 128 columns) is the narrowest unit whose products still fit the
// grid in one round: a product of a small matrix is one unit deep on every CTA,
// so its time is that of one unit, while large matrices take 128 columns, where
// a CTA loads 64 KB of operands per 128 x 128 x 32 step (40 KB for 32 columns).

#include "foe.cuh"
#include "persist.cuh"

namespace {

using namespace tcx;

struct FoeMaps {
  CUtensorMap a[kFoeMats][3];  // 128-row boxes of the FP32 master, hi and lo
  CUtensorMap b[kFoeMats][3];  // BN-row boxes
  CUtensorMap s[kFoeMats][3];  // 32-row boxes
};

// matrices, in the order in which dm_fermi lays them out (1, the launched form's A,
// holds the diagonals of E and W)
enum { ME0 = 0, MA = 1, MZ = 2, MT = 3, MY = 4, ME1 = 5, MW = 6 };

enum Kind { kLL, kE0, kW, kZ1, kT, kY, kZW, kE, kEW };

struct Prod {
  int a, b, out;  // operands and result
  int e;          // FP32 matrix added in the epilogue, or -1
  int kind;
  int lolo;       // a square: also the lo lo MMA, which keeps its diagonal unbiased
  int last;       // traces are wanted: the last E and the two products after it
  int patch;      // operands with a patched diagonal: bit 0 A, bit 1 B
};

// Product p of an expansion of m doubling steps with `ns` steps per inverse.
__device__ __forceinline__ Prod prod_of(int p, int m, int ns) {
  const int per = 2 * ns + 2;
  const int steps = m * per;
  // Z and Y swap in every Newton-Schulz step
  auto zb = [&](int swaps) { return (swaps & 1) ? MY : MZ; };
  if (p == 0) return Prod{MT, MT, MW, -1, kLL, 1, 0, 0};
  if (p == 1) return Prod{MT, MW, ME0, MT, kE0, 0, m == 0, 0};
  const int q = p - 2;
  const int s = q < steps ? q / per : m, j = q - s * per;
  const int sw = s * (ns - 1);  // swaps before this step
  const int X = (s & 1) ? ME1 : ME0, Xn = (s & 1) ? ME0 : ME1;
  const int Z = zb(sw);
  if (j == 0) return Prod{X, X, MW, -1, kW, 0, s == m, 3};  // W = (I - 2E)(I + 2E)
  if (s == m) return Prod{X, MW, Z, -1, kEW, 0, 1, 0};
  if (j == 1) return Prod{MW, MW, Z, MW, kZ1, 1, 0, 3};
  const int Zf = zb(sw + ns - 1);
  if (j == per - 2) return Prod{Zf, MW, MT, -1, kZW, 0, 0, 0};
  if (j == per - 1) return Prod{X, MT, Xn, X, kE, 0, s == m - 1, 0};
  const int k = (j - 2) >> 1;  // Newton-Schulz step
  const int Zk = zb(sw + k), Yk = zb(sw + k + 1);
  if (((j - 2) & 1) == 0) return Prod{MW, Zk, MT, -1, kT, 0, 0, 1};
  return Prod{Zk, MT, Yk, -1, kY, 0, 0, 0};
}

template <int P, int BN>
__global__ void __launch_bounds__(kRunThreads, 1) k_foe_run(const FoeRunArgs a, const __grid_constant__ FoeMaps mp) {
  using Q = RunCfg<P, BN>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[Q::stages], conv[Q::stages], empty[Q::stages], tfull[2], tempty[2], go, mdone;
  __shared__ __align__(8) uint64_t sfull[Q::bufs], sfree[Q::bufs];
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_abort;
  __shared__ int s_go;
  __shared__ FoeState fs;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const StageRing ring{smem + Q::stages * Q::stage_bytes, sfull, sfree};
  const unsigned G = gridDim.x;
  const RunUnits wu = run_units<BN>(a.ld, (int)G);
  const unsigned Gw = min(G, (unsigned)wu.U);  // the CTAs that arrive at the barriers
  if (blockIdx.x >= Gw) return;                // no units
  // Pipeline wait limit.  A wait that spans the grid barrier (a product's first stage and first
  // accumulator, what the stores and the patches wait for) is not the pipeline's: kWaitNs.
  const unsigned long long wl = a.wait_ns ? a.wait_ns : kWaitNs;
  const int nk = a.ld / 32;
  unsigned* bar = &a.st->bar;
  const int* err = &a.st->err;
  for (int i = threadIdx.x; i < (int)(sizeof(FoeState) / 4); i += kRunThreads)
    reinterpret_cast<int*>(&fs)[i] = reinterpret_cast<const int*>(a.st)[i];
  if (threadIdx.x == 0) {
    for (int s = 0; s < Q::stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&conv[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 8);
    }
    for (int b = 0; b < Q::bufs; ++b) {
      mbar_init(&sfull[b], 8);
      mbar_init(&sfree[b], 1);
    }
    mbar_init(&go, 1);
    mbar_init(&mdone, 1);
    s_abort = 0;
    s_go = !a.st->done;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, 2 * BN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const int m = fs.meff;
  const int np = 2 + m * (2 * a.ns + 2) + 2;

  int g = 0, t_mma = 0, t_epi = 0, issued = 0;  // g: stages gone through by this role
  int used = 0;                                 // arrays put through the staging ring
  uint32_t cpar = 0, gopar = 0;                 // parities of the next conv (a bit per stage) and go phase
  const int mine = (wu.U - 1 - (int)blockIdx.x) / (int)G + 1;  // units of this CTA
  unsigned phase = 0;                           // barrier phases completed before this expansion
  while (s_go) {
    if (warp == 0 && lane == 0) {
      // ------------------------------------------------------------ producer
      for (int p = 0; p < np && !s_abort; ++p) {
        const Prod r = prod_of(p, m, a.ns);
        prefetch_map(&mp.a[r.a][1]);
        prefetch_map(&mp.b[r.b][1]);
        if (P == TB_PREC_TF32X3) {
          prefetch_map(&mp.a[r.a][2]);
          prefetch_map(&mp.b[r.b][2]);
        }
        if (!run_wait(bar, (phase + p + 1) * Gw, err, &s_abort)) break;
        fence_async_all();
        if (r.patch) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&go)) : "memory");
        for (int u = blockIdx.x; u < wu.U && !s_abort; u += G) {
          const RunUnit un = run_unit<BN>(wu, u);
          for (int kb = 0; kb < nk; ++kb, ++g) {
            const int s = g % Q::stages;
            if (g >= Q::stages && !mbar_wait(&empty[s], ((g / Q::stages) - 1) & 1, &s_abort, wl)) break;
            uint8_t* base = smem + s * Q::stage_bytes;
            load_stage<P, BN>(base, &full[s], mp.a[r.a], mp.b[r.b], mp.s[r.b], un, kb * 32);
            issued = g + 1;
          }
        }
      }
    } else if (warp == 1) {
      if (elect_one()) {
        // ------------------------------------------------------------ MMA issuer
        const uint32_t lo0 = sdesc_lo(smem_u32(smem));
        for (int p = 0; p < np && !s_abort; ++p) {
          const Prod r = prod_of(p, m, a.ns);
          const bool lolo = r.lolo;
          for (int u = blockIdx.x; u < wu.U && !s_abort; u += G, ++t_mma) {
            const RunUnit un = run_unit<BN>(wu, u);
            const uint32_t id = idesc(2u, 128, un.nc);
            const int buf = t_mma & 1;
            if (t_mma >= 2 && !mbar_wait(&tempty[buf], ((t_mma >> 1) - 1) & 1, &s_abort, wl)) break;
            tc_fence_after();
            for (int kb = 0; kb < nk; ++kb, ++g) {
              const int s = g % Q::stages;
              const unsigned long long lim = kb == 0 && u == (int)blockIdx.x ? kWaitNs : wl;
              if (r.patch) {
                if (!mbar_wait(&conv[s], (cpar >> s) & 1, &s_abort, lim)) break;
                cpar ^= 1u << s;
              } else if (!mbar_wait(&full[s], (g / Q::stages) & 1, &s_abort, lim)) {
                break;
              }
              tc_fence_after();
              stage_mma<P, BN>(lo0 + s * (Q::stage_bytes >> 4), tmem + buf * BN, id, kb == 0, lolo);
              umma_commit(&empty[s]);
            }
            umma_commit(&tfull[buf]);
          }
        }
      }
      __syncwarp();
    } else if (warp == 11) {
      // ------------------------------------------------------------ stores
      for (int p = 0; p < np && lane == 0 && !s_abort; ++p) {
        const Prod r = prod_of(p, m, a.ns);
        const bool master = r.kind == kE0 || r.kind == kE || r.kind == kW || r.kind == kEW;
        const int h0 = master ? 0 : 1, h1 = r.kind == kEW ? 1 : Q::C::split ? 3 : 2;
        for (int u = blockIdx.x; u < wu.U && !s_abort; u += G) {
          const RunUnit un = run_unit<BN>(wu, u);
          for (int c = 0; c < un.nc; c += 32)
            for (int h = h0; h < h1; ++h)
              if (!ring_store<P, BN>(ring, used, &mp.a[r.out][h], &mp.s[r.out][h], un.I * 128, un.J * 128 + un.c0 + c,
                                     un.I == un.J ? (un.c0 + c) >> 5 : kOff, &s_abort, kWaitNs))
                break;
        }
        tma_store_wait();
        if (!s_abort) run_arrive(bar);
      }
    } else if (warp == 10) {
      // ------------------------------------------------------------ diagonal patches
      // Every stage of a patched product passes through this warp.  It waits for the
      // product (go) before its stages: a parity wait tells a phase only from the one
      // before it, and this warp skips the products in between.
      for (int p = 0; p < np && !s_abort; ++p) {
        const Prod r = prod_of(p, m, a.ns);
        // W: (I - 2E)/-2 and (I + 2E)/2; else -A = W - 2I
        const bool w = r.kind == kW;
        const float* d = a.m[MA] + (w ? 0 : a.ld);
        const int lim = w ? a.n : a.ld;
        if (!r.patch) {
          g += mine * nk;
          continue;
        }
        if (!mbar_wait_warp(&go, gopar, &s_abort, kWaitNs)) break;
        gopar ^= 1u;
        for (int u = blockIdx.x; u < wu.U && !s_abort; u += G) {
          const RunUnit un = run_unit<BN>(wu, u);
          const int yb = un.J * 128 + un.c0;
          for (int kb = 0; kb < nk; ++kb, ++g) {
            const int s = g % Q::stages;
            if (!mbar_wait_warp(&full[s], (g / Q::stages) & 1, &s_abort, wl)) break;
            uint8_t* base = smem + s * Q::stage_bytes;
            if (r.patch & 1)
              patch_diag<P>(base, Q::half_bytes, un.I * 128, 128, kb * 32, lane, d, w ? 1.0f : 2.0f,
                            w ? -2.0f : -1.0f, w ? -0.5f : -1.0f, lim);
            if (r.patch & 2)
              patch_diag<P>(base + Q::a_bytes, Q::half_bytes, yb, un.nc, kb * 32, lane, d, w ? 1.0f : 2.0f,
                            w ? 2.0f : -1.0f, w ? 0.5f : -1.0f, lim);
            fence_async_shared();  // the stores are visible to the tensor core's reads
            __syncwarp();
            if (lane == 0)
              asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&conv[s])) : "memory");
          }
        }
      }
    } else if (warp >= 2) {
      // ------------------------------------------------------------ epilogue
      const int eid = threadIdx.x - 64;
      // L = -c (H - mu I) on the n x n block, zero in the padding, of this
      // CTA's units (the tile and its mirror image, each from its own place in H)
      {
        const double mu = fs.mu, c = fs.c;
        float* L = a.m[MT];
        auto put = [&](int r, int col) {
          double x = 0.0;
          if (r < a.n && col < a.n) x = (r == col ? c * mu : 0.0) - c * a.H[(size_t)r * a.n + col];
          const size_t e = (size_t)r * a.ld + col;
          L[e] = (float)x;
          store_operand1<P>((float)x, a.hi[MT], a.lo[MT], e);
        };
        for (int u = blockIdx.x; u < wu.U; u += G) {
          const RunUnit un = run_unit<BN>(wu, u);
          const int sh = 31 - __clz(un.nc), r0 = un.I * 128, q0 = un.J * 128 + un.c0;
#pragma unroll 4
          for (int e = eid; e < 128 * un.nc; e += kRunEpi) put(r0 + (e >> sh), q0 + (e & (un.nc - 1)));
          if (un.I != un.J) {
#pragma unroll 4
            for (int e = eid; e < 128 * un.nc; e += kRunEpi) put(q0 + (e >> 7), r0 + (e & 127));
          }
        }
        fence_async_all();
        epi_sync();
        if (eid == 0) run_arrive(bar);
      }
      const int q = warp & 3, half = (warp - 2) >> 2;
      for (int p = 0; p < np && !s_abort; ++p) {
        const Prod r = prod_of(p, m, a.ns);
        double* const trace = r.kind == kW ? a.partsw : r.kind == kEW ? a.parts3 : a.parts;
        const float al = r.kind == kE0 ? -4.0f / 3.0f : r.kind == kZ1 ? 32.0f / 99.0f : r.kind == kW ? -4.0f : 1.0f;
        const float be = r.kind == kZ1 ? -144.0f / 99.0f : 1.0f;
        const float gam = r.kind == kT ? 2.0f : r.kind == kZ1 ? 210.0f / 99.0f : 0.0f;
        const bool master = r.kind == kE0 || r.kind == kE || r.kind == kW || r.kind == kEW;
        for (int u = blockIdx.x; u < wu.U; u += G, ++t_epi) {
          const int buf = t_epi & 1;
          const RunUnit un = run_unit<BN>(wu, u);
          const int r0 = un.I * 128, gr = r0 + 32 * q + lane;
          const bool diag = un.I == un.J;
          // The FP32 values added: this CTA's own earlier stores, past L1 (TMA wrote them).
          // E and L are at least one grid barrier old here, so they are fetched while the
          // MMAs run.  W (kZ1) is the product just before, whose stores another warp may
          // still be issuing: it is fetched behind tfull, which comes after the barrier that
          // this CTA's store warp arrives at when its stores are written.
          float ev[16];
          auto load_e = [&](int row, int col) {
            const float4* e4 = reinterpret_cast<const float4*>(a.m[r.e] + (size_t)row * a.ld + col);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 t = __ldcg(e4 + j);
              ev[4 * j] = t.x;
              ev[4 * j + 1] = t.y;
              ev[4 * j + 2] = t.z;
              ev[4 * j + 3] = t.w;
            }
          };
          if (r.e >= 0 && r.kind != kZ1) load_e(gr, un.J * 128 + un.c0 + 16 * half);
          if (!mbar_wait_warp(&tfull[buf], (t_epi >> 1) & 1, &s_abort, u == (int)blockIdx.x ? kWaitNs : wl)) break;
          if (r.kind == kZ1) load_e(gr, un.J * 128 + un.c0 + 16 * half);
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < un.nc; c += 32) {
            uint32_t v[16];
            tmem_ld16(tmem + (static_cast<uint32_t>(32 * q) << 16) + buf * BN + c + 16 * half, v);
            const int chunk0 = un.J * 128 + un.c0 + c, col0 = chunk0 + 16 * half;
            const int dj = gr - col0;  // the diagonal's column in these 16
            float y[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) y[j] = al * __uint_as_float(v[j]);
            if (r.e >= 0) {
              if (r.kind == kZ1) {  // A = 2I - W
#pragma unroll
                for (int j = 0; j < 16; ++j) ev[j] = (j == dj ? 2.0f : 0.0f) - ev[j];
              }
#pragma unroll
              for (int j = 0; j < 16; ++j) y[j] = fmaf(be, ev[j], y[j]);
              if (c + 32 < un.nc) load_e(gr, col0 + 32);
            }
            const int dk = diag ? (un.c0 + c) >> 5 : kOff;
            if (diag) {
              if (gr < a.n) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (j == dj) y[j] += gam;
              }
              if (dk == q) {
                // this warp's rows hold the chunk's diagonal: kept for the patches, and
                // a trace slot for 16 of its elements, whatever the grid
                float x = 0.0f;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (j == dj) x = y[j];
                if (dj >= 0 && dj < 16) {
                  if (r.kind == kE0 || r.kind == kE) a.m[MA][gr] = x;
                  if (r.kind == kW) a.m[MA][a.ld + gr] = x;
                }
                if (r.last) {
                  const double t1 = warp_sum((double)x);
                  if (lane == 0) trace[un.I * 8 + 2 * dk + half] = t1;
                }
              }
            }
            if (master) ring_put<P, BN>(ring, used, y, q, half, lane, dk, &s_abort, wl);
            if (r.kind != kEW) ring_put_split<P, BN>(ring, used, y, q, half, lane, dk, &s_abort, wl);
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[buf])) : "memory");
        }
      }
    }
    phase += np + 1;
    __syncthreads();
    // the chemical-potential step, the same in every CTA
    if (warp == 0) {
      const bool ok = run_wait(bar, phase * Gw, err, &s_abort);
      if (__all_sync(0xffffffffu, ok)) {
        double x = 0.0, y = 0.0, z = 0.0;
        for (int i = lane; i < 8 * wu.nt; i += 32) {
          x += __ldcg(a.parts + i);
          y += __ldcg(a.partsw + i);
          z += __ldcg(a.parts3 + i);
        }
        x = warp_sum(x);
        y = warp_sum(y);
        z = warp_sum(z);
        if (lane == 0) foe_mu_step(&fs, x, y, z, a.n, a.nocc, a.beta, a.tol, a.max_it);
      } else if (lane == 0) {
        s_abort = 1;
      }
      if (lane == 0) s_go = !fs.done && !s_abort;
    }
    __syncthreads();
  }
  // D = E + I/2, with the canonical shift, of this CTA's units (past L1: the
  // lower half of a diagonal tile is another CTA's, the rest TMA wrote)
  if (!s_abort && !fs.err) {
    const float* E = a.m[(m & 1) ? ME1 : ME0];
    const float *W = a.m[MW], *U = a.m[((m * (a.ns - 1)) & 1) ? MY : MZ];
    const float u = (float)fs.u;
    const bool shift = !fs.nocorr;
    auto put = [&](int r, int col) {
      if (r >= a.n || col >= a.n) return;
      const size_t e = (size_t)r * a.ld + col;
      float x = __ldcg(E + e);
      if (shift) x = foe_shifted(x, __ldcg(W + e), __ldcg(U + e), u);
      a.D[(size_t)r * a.n + col] = (double)x + (r == col ? 0.5 : 0.0);
    };
    for (int i = blockIdx.x; i < wu.U; i += G) {
      const RunUnit un = run_unit<BN>(wu, i);
      const int sh = 31 - __clz(un.nc), r0 = un.I * 128, q0 = un.J * 128 + un.c0;
#pragma unroll 4
      for (int e = threadIdx.x; e < 128 * un.nc; e += kRunThreads) put(r0 + (e >> sh), q0 + (e & (un.nc - 1)));
      if (un.I != un.J) {
#pragma unroll 4
        for (int e = threadIdx.x; e < 128 * un.nc; e += kRunThreads) put(q0 + (e >> 7), r0 + (e & 127));
      }
    }
  }
  if (threadIdx.x == 0 && s_abort) atomicExch(&a.st->err, TB_ERR_TIMEOUT);
  if (warp == 0 && lane == 0 && s_abort) {
    // let every issued copy land before the CTA can exit
    for (int q = (issued > Q::stages ? issued - Q::stages : 0); q < issued; ++q) {
      const unsigned long long t0 = gtime();
      while (!mbar_try(&full[q % Q::stages], (q / Q::stages) & 1) && gtime() - t0 < kWaitNs) {
      }
    }
  }
  if (threadIdx.x == 0 && run_last(&a.st->left, Gw))
    foe_report(&fs, *reinterpret_cast<const volatile int*>(err), a.n, a.nocc, a.tol, a.mu_out, a.rep);
  tc_fence_before();
  if (warp == 1) {
    if (elect_one()) {
      // every issued MMA retired (bounded) before TMEM is freed
      umma_commit(&mdone);
      const unsigned long long t0 = gtime();
      while (!mbar_try(&mdone, 0) && gtime() - t0 < kWaitNs) {
      }
    }
    __syncwarp();
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * BN);
  }
}

template <int P, int BN>
int launch(tb_ctx* ctx, const FoeRunArgs& a, int cluster, int grid, int* ran, cudaStream_t s) {
  using Q = RunCfg<P, BN>;
  FoeMaps mp{};
  for (int i = 0; i < kFoeMats; ++i) {
    const int rc = tb_run_maps<P, BN>(ctx, a.m[i], a.hi[i], a.lo[i], a.ld, mp.a[i], mp.b[i], mp.s[i]);
    if (rc) return rc;
  }
  static unsigned long long attr_done = 0;
  if (int rc = tb_smem_attr(ctx, k_foe_run<P, BN>, Q::smem, &attr_done)) return rc;
  static RunFits fits;
  return tb_run_launch(ctx, k_foe_run<P, BN>, &fits, kRunThreads, Q::smem, cluster, grid, ran, s, a, mp);
}

template <int P>
int launch_bn(tb_ctx* ctx, const FoeRunArgs& a, const RunShape& r, int* ran, cudaStream_t s) {
  switch (r.bn) {
    case 32: return launch<P, 32>(ctx, a, r.cluster, r.grid, ran, s);
    case 64: return launch<P, 64>(ctx, a, r.cluster, r.grid, ran, s);
    default: return launch<P, 128>(ctx, a, r.cluster, r.grid, ran, s);
  }
}

}  // namespace

int foe_run(tb_ctx* ctx, int precision, const FoeRunArgs& a, int captured, int* ran, cudaStream_t s) {
  *ran = 0;
  if (precision != TB_PREC_TF32 && precision != TB_PREC_TF32X3) return TB_OK;
  RunShape r;
  if (!tb_run_shape(ctx, a.ld, captured, &r)) return TB_OK;
  for (int round = 0; round < 2 && !*ran; ++round) {
    const int rc = precision == TB_PREC_TF32 ? launch_bn<TB_PREC_TF32>(ctx, a, r, ran, s)
                                             : launch_bn<TB_PREC_TF32X3>(ctx, a, r, ran, s);
    if (rc || !r.cluster) return rc;
    r.cluster = 0;  // no cluster of this size fits the device: a cooperative launch
  }
  return TB_OK;
}
