// The tensor-core main phase of dm_sp2 (tf32, tf32x3) in one launch: X0, every
// projection and the stop/branch decisions run in one persistent grid, the
// projections separated by a grid barrier (persist.cuh).
//
// What bounds the launched form of small matrices: a projection of a 600 x 600 matrix is
// a few microseconds of work on 15 CTAs, each launch costs about as much again, and
// the host enqueues max_iter + 1 (100) launches, most of which return at once: 1.3 ms
// for 16 projections.  Here nothing runs after the stop, a small matrix is spread
// over more CTAs (32- or 64-column units), and the operands are stored by TMA.
// The projections compute the same products in the same order of accumulation as
// k_sp2_step_tc: X is bitwise the same.  The FP64 trace partials have a slot per 128 x
// 32 chunk, so the sums do not depend on the grid.
//
// Where CTA pairs are the faster form (sp2_tc_pairs in gemm_tc.cu) dm_sp2 takes that one,
// launched: it halves the operand bytes per flop, and a launch is 1% of its projection.

#include "persist.cuh"
#include "sp2_run.cuh"

namespace {

using namespace tcx;

struct Sp2Maps {
  CUtensorMap a[2][3];  // the two iterates: 128-row boxes of the FP32 master, hi and lo
  CUtensorMap b[2][3];  // BN-row boxes
  CUtensorMap s[2][3];  // 32-row boxes
};

// Two barriers: the operands of X_{k+1} are stored (ops), and its trace partials (tr).  The
// product of projection k needs only the first, the epilogue's branch and the stop the
// second, so the MMAs run while the FP64 sums, their barrier and the decision are still
// under way (11 of 29 thousand cycles of a projection at n = 48); what a stop leaves of
// the product is not used.
template <int P, int BN>
__global__ void __launch_bounds__(kRunThreads, 1) k_sp2_run(const Sp2RunArgs g0, const __grid_constant__ Sp2Maps mp) {
  using Q = RunCfg<P, BN>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[Q::stages], empty[Q::stages], tfull[2], tempty[2], mdone;
  __shared__ __align__(8) uint64_t sfull[Q::bufs], sfree[Q::bufs];
  __shared__ __align__(8) uint64_t dec[2], decfree[2];  // by parity of the projection
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_abort;
  __shared__ int s_dec[2];  // 1 stop, 2 the branch 2X - X^2
  __shared__ double s_red[2][8][2];
  __shared__ double s_lo, s_hi;

  const SP2StepArgs& a = g0.a;
  SP2State* st = a.st;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const StageRing ring{smem + Q::stages * Q::stage_bytes, sfull, sfree};
  const unsigned G = gridDim.x;
  const RunUnits wu = run_units<BN>(a.ld, (int)G);
  const unsigned Gw = min(G, (unsigned)wu.U);  // the CTAs that arrive at the barriers
  if (blockIdx.x >= Gw) return;                // no units
  // Pipeline wait limit.  A wait that spans a grid barrier (a projection's first stage and first
  // accumulator, the decisions, what the stores wait for) is not the pipeline's: kWaitNs.
  const unsigned long long wl = a.wait_ns ? a.wait_ns : kWaitNs;
  const int nk = a.ld / 32;
  const int slots = 4 * wu.tiles;
  if (threadIdx.x == 0) {
    for (int s = 0; s < Q::stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 8);
      mbar_init(&dec[b], 1);
      mbar_init(&decfree[b], 11);  // producer, MMA issuer, 8 epilogue warps, store warp
    }
    for (int b = 0; b < Q::bufs; ++b) {
      mbar_init(&sfull[b], 8);
      mbar_init(&sfree[b], 1);
    }
    mbar_init(&mdone, 1);
    s_abort = 0;
    fence_barrier_init();
  }
  if (warp == 0) {
    // Gershgorin bounds from the rows' partials
    double lo = INFINITY, hi = -INFINITY;
    for (int i = lane; i < g0.nbparts; i += 32) {
      lo = fmin(lo, g0.bparts[2 * i]);
      hi = fmax(hi, g0.bparts[2 * i + 1]);
    }
    lo = warp_min(lo);
    hi = warp_max(hi);
    if (lane == 0) {
      s_lo = lo;
      s_hi = hi;
      if (blockIdx.x == 0) {
        st->emin = lo;
        st->emax = hi;
      }
    }
  }
  if (warp == 1) tmem_alloc(&tmem_base, 2 * BN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const int q = warp & 3, half = (warp - 2) >> 2;
  auto arrive = [](uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
  };
  // The decision of projection k, by one thread; -1 when the wait gave up.
  auto decision = [&](int k) -> int {
    if (!mbar_wait(&dec[k & 1], (k >> 1) & 1, &s_abort, kWaitNs)) return -1;
    const int d = *reinterpret_cast<volatile int*>(&s_dec[k & 1]);
    arrive(&decfree[k & 1]);
    return d;
  };
  auto slot_of = [&](const RunUnit& un, int c) {
    return 4 * (un.I * wu.nt - un.I * (un.I - 1) / 2 + un.J - un.I) + ((un.c0 + c) >> 5);
  };

  if (warp == 0) {
    if (lane == 0) {
      // -------------------------------------------------------------- producer
      int g = 0, issued = 0;
      for (int k = 0;; ++k) {
        const int ib = k & 1;
        prefetch_map(&mp.a[ib][1]);
        prefetch_map(&mp.b[ib][1]);
        if (Q::C::split) {
          prefetch_map(&mp.a[ib][2]);
          prefetch_map(&mp.b[ib][2]);
        }
        if (!run_wait(g0.bar, (unsigned)(k + 1) * Gw, &st->err, &s_abort)) break;
        fence_async_all();
        int d = 0, i = 0;
        bool asked = false;
        for (int u = blockIdx.x; u < wu.U && !s_abort; u += G, ++i) {
          if (i == 2) {  // two accumulators without the epilogue
            asked = true;
            d = decision(k);
            if (d < 0 || (d & 1)) break;
          }
          const RunUnit un = run_unit<BN>(wu, u);
          for (int kb = 0; kb < nk; ++kb, ++g) {
            const int s = g % Q::stages;
            if (g >= Q::stages && !mbar_wait(&empty[s], ((g / Q::stages) - 1) & 1, &s_abort, wl)) break;
            load_stage<P, BN>(smem + s * Q::stage_bytes, &full[s], mp.a[ib], mp.b[ib], mp.s[ib], un, kb * 32);
            issued = g + 1;
          }
        }
        if (!asked) d = decision(k);
        if (d < 0 || (d & 1) || s_abort) break;
      }
      // let every issued copy land before the CTA can exit
      for (int i = (issued > Q::stages ? issued - Q::stages : 0); i < issued; ++i) {
        const unsigned long long t0 = gtime();
        while (!mbar_try(&full[i % Q::stages], (i / Q::stages) & 1) && gtime() - t0 < kWaitNs) {
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (elect_one()) {
      // ------------------------------------------------------------ MMA issuer
      const uint32_t lo0 = sdesc_lo(smem_u32(smem));
      int g = 0, t = 0;
      for (int k = 0;; ++k) {
        int d = 0, i = 0;
        bool asked = false;
        for (int u = blockIdx.x; u < wu.U && !s_abort; u += G, ++t, ++i) {
          if (i == 2) {
            asked = true;
            d = decision(k);
            if (d < 0 || (d & 1)) break;
          }
          const RunUnit un = run_unit<BN>(wu, u);
          const uint32_t id = idesc(2u, 128, un.nc);
          const int buf = t & 1;
          if (t >= 2 && !mbar_wait(&tempty[buf], ((t >> 1) - 1) & 1, &s_abort, wl)) break;
          tc_fence_after();
          for (int kb = 0; kb < nk; ++kb, ++g) {
            const int s = g % Q::stages;
            if (!mbar_wait(&full[s], (g / Q::stages) & 1, &s_abort, kb == 0 && i == 0 ? kWaitNs : wl)) break;
            tc_fence_after();
            stage_mma<P, BN>(lo0 + s * (Q::stage_bytes >> 4), tmem + buf * BN, id, kb == 0, false);
            umma_commit(&empty[s]);
          }
          umma_commit(&tfull[buf]);
        }
        if (!asked) d = decision(k);
        if (d < 0 || (d & 1) || s_abort) break;
      }
    }
    __syncwarp();
  } else if (warp == 10) {
    // -------------------------------------------------------------- decisions
    SP2StepArgs b = a;
    double e1 = 0.0, e2 = 0.0, e3 = 0.0;  // Tr X - Tr X^2 of the last projections (lane 0)
    unsigned long long branch[2] = {0, 0};
    for (int k = 0;; ++k) {
      bool ok = run_wait(g0.bar_tr, (unsigned)(k + 1) * Gw, &st->err, &s_abort);
      // lanes 0-15 sum Tr X, 16-31 ||X||_F^2
      double x = 0.0;
      for (int i = lane & 15; i < slots; i += 16) x += __ldcg(g0.parts[k & 1] + 2 * i + (lane >> 4));
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      const double y = __shfl_sync(0xffffffffu, x, 16);
      ok = __all_sync(0xffffffffu, ok);
      int stop = 1;
      if (lane == 0) {
        // the slot of two projections ago has been read by everyone
        if (k >= 2 && !mbar_wait(&decfree[k & 1], ((k >> 1) - 1) & 1, &s_abort, kWaitNs)) ok = false;
        int br = 0, capped = 0;
        if (ok && !s_abort) {
          b.k = k;
          stop = sp2_decide_e(b, x, y, e1, e2, e3, true, &br, &capped);
          s_dec[k & 1] = stop | (br << 1);
          arrive(&dec[k & 1]);
          e3 = e2;
          e2 = e1;
          e1 = x - y;
          if (br) branch[k >> 6] |= 1ull << (k & 63);
          if (blockIdx.x == 0) {
            st->t1[k] = x;
            st->t2[k] = y;
            if (stop) {
              st->iters = k;
              st->capped = capped;
              st->branch[0] = branch[0];
              st->branch[1] = branch[1];
              st->done = 1;
            }
          }
        } else {
          s_abort = 1;
          s_dec[k & 1] = 1;
          arrive(&dec[k & 1]);
        }
      }
      if (__shfl_sync(0xffffffffu, stop, 0)) break;
    }
  } else if (warp == 11) {
    // -------------------------------------------------------------- stores
    if (lane == 0) {
      int used = 0;
      for (int k = 0;; ++k) {
        const int d = decision(k);
        if (d < 0 || (d & 1)) break;
        const int ob = (k & 1) ^ 1;
        for (int u = blockIdx.x; u < wu.U && !s_abort; u += G) {
          const RunUnit un = run_unit<BN>(wu, u);
          for (int c = 0; c < un.nc; c += 32)
            for (int h = 0; h < (Q::C::split ? 3 : 2); ++h)
              if (!ring_store<P, BN>(ring, used, &mp.a[ob][h], &mp.s[ob][h], un.I * 128, un.J * 128 + un.c0 + c,
                                     un.I == un.J ? kAsIs : kOff, &s_abort, kWaitNs))
                break;
        }
        tma_store_wait();
        if (s_abort) break;
        run_arrive(g0.bar);
      }
      tma_store_wait();
    }
  } else {
    // -------------------------------------------------------------- epilogue (warps 2-9)
    const int eid = threadIdx.x - 64;
    int sp = 0;  // parity of the partial sums' buffer
    // (t1, t2) of a chunk into its slot: the warps' sums meet in s_red, the first warp adds
    // them; all 256 epilogue threads
    auto put_parts = [&](double* parts, int slot, double t1, double t2, bool diag) {
      t2 = warp_sum(t2);
      if (diag) t1 = warp_sum(t1);
      if (lane == 0) {
        s_red[sp][warp - 2][0] = t1;
        s_red[sp][warp - 2][1] = t2;
      }
      epi_sync();
      if (warp == 2) {
        double t = lane < 16 ? s_red[sp][lane & 7][lane >> 3] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0 || lane == 8) parts[2 * slot + (lane >> 3)] = t;
      }
      sp ^= 1;
    };
    {
      // X0 = (emax I - H)/(emax - emin), zero outside n x n, and its trace partials
      const double emin = s_lo, emax = s_hi;
      double w = emax - emin;
      if (!(w > 0.0)) w = 1.0;  // H = c I: X0 = 0 (no gap; reported through the trace)
      const double inv = 1.0 / w;
      double t1 = 0.0, t2 = 0.0;
      auto put = [&](int r, int c) {
        double x = 0.0;
        if (r < a.n && c < a.n) x = ((r == c ? emax : 0.0) - g0.H[(size_t)r * a.n + c]) * inv;
        const float xf = (float)x;
        const size_t e = (size_t)r * a.ld + c;
        g0.M[0][e] = xf;
        store_operand1<P>(xf, g0.hi[0], g0.lo[0], e);
        const double d = abs_to_f64(xf);
        if (r == c) t1 += (double)xf;
        t2 = fma(d, d, t2);
      };
      for (int u = blockIdx.x; u < wu.U; u += G) {
        const RunUnit un = run_unit<BN>(wu, u);
        for (int c = 0; c < un.nc; c += 32) {
          const int r0 = un.I * 128, c0 = un.J * 128 + un.c0 + c;
          t1 = t2 = 0.0;
#pragma unroll 4
          for (int e = eid; e < 4096; e += kRunEpi) put(r0 + (e >> 5), c0 + (e & 31));
          if (un.I != un.J) {
#pragma unroll 4
            for (int e = eid; e < 4096; e += kRunEpi) put(c0 + (e >> 7), r0 + (e & 127));
          }
          put_parts(g0.parts[0], slot_of(un, c), t1, t2, un.I == un.J);
        }
      }
      fence_async_all();
      epi_sync();
      if (eid == 0) {
        run_arrive(g0.bar);
        run_arrive(g0.bar_tr);
      }
    }
    int t = 0, used = 0;
    for (int k = 0;; ++k) {
      const int ib = k & 1, ob = ib ^ 1;
      int d = 0;
      bool asked = false;
      for (int u = blockIdx.x; u < wu.U; u += G, ++t) {
        const RunUnit un = run_unit<BN>(wu, u);
        const int buf = t & 1;
        const int r0 = un.I * 128, gr = r0 + 32 * q + lane;
        const bool diag = un.I == un.J;
        const bool ok = mbar_wait_warp(&tfull[buf], (t >> 1) & 1, &s_abort, asked ? wl : kWaitNs);
        // X_k (this CTA's own earlier stores, past L1: TMA wrote them), fetched before the
        // branch that may not take it is known
        float xv[16];
        auto load_x = [&](int col) {
          const float4* x4 = reinterpret_cast<const float4*>((ib ? g0.M[1] : g0.M[0]) + (size_t)gr * a.ld + col);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 v = __ldcg(x4 + j);
            xv[4 * j] = v.x;
            xv[4 * j + 1] = v.y;
            xv[4 * j + 2] = v.z;
            xv[4 * j + 3] = v.w;
          }
        };
        load_x(un.J * 128 + un.c0 + 16 * half);
        if (!asked) {
          asked = true;
          if (lane == 0) d = decision(k);
          d = __shfl_sync(0xffffffffu, d, 0);
        }
        // the warps meet in every chunk below, so they leave together
        if (epi_any(!ok || d < 0)) {
          d = -1;
          break;
        }
        if (d & 1) break;
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < un.nc; c += 32) {
          uint32_t v[16];
          tmem_ld16(tmem + (static_cast<uint32_t>(32 * q) << 16) + buf * BN + c + 16 * half, v);
          const int col0 = un.J * 128 + un.c0 + c + 16 * half;
          float y[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) y[j] = __uint_as_float(v[j]);
          if (d & 2) {
#pragma unroll
            for (int j = 0; j < 16; ++j) y[j] = fmaf(2.0f, xv[j], -y[j]);
            if (c + 32 < un.nc) load_x(col0 + 32);
          }
          const int mode = diag ? kAsIs : kOff;
          ring_put<P, BN>(ring, used, y, q, half, lane, mode, &s_abort, wl);
          ring_put_split<P, BN>(ring, used, y, q, half, lane, mode, &s_abort, wl);
          // traces, while the stores drain (rows of the padding are zero: nothing to sum)
          double t1 = 0.0, t2 = 0.0;
          if (r0 + 32 * q < a.n) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const double x = abs_to_f64(y[j]);
              t2 = fma(x, x, t2);
            }
          }
          if (diag) {
            float x = 0.0f;
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (j == gr - col0) x = y[j];
            t1 = (double)x;
          } else {
            t2 *= 2.0;  // the mirrored tile counts too
          }
          put_parts(ob ? g0.parts[1] : g0.parts[0], slot_of(un, c), t1, t2, diag);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive(&tempty[buf]);
      }
      if (d < 0 || (d & 1)) break;
      __syncwarp();  // the slots are the first warp's stores
      if (eid == 0) run_arrive(g0.bar_tr);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_abort) atomicExch(&st->err, TB_ERR_TIMEOUT);
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
int launch(tb_ctx* ctx, const Sp2RunArgs& g, const RunShape& r, int* ran, cudaStream_t s) {
  using Q = RunCfg<P, BN>;
  Sp2Maps mp{};
  for (int i = 0; i < 2; ++i) {
    const int rc = tb_run_maps<P, BN>(ctx, g.M[i], g.hi[i], g.lo[i], g.a.ld, mp.a[i], mp.b[i], mp.s[i]);
    if (rc) return rc;
  }
  static unsigned long long attr_done = 0;
  if (int rc = tb_smem_attr(ctx, k_sp2_run<P, BN>, Q::smem, &attr_done)) return rc;
  static RunFits fits;
  return tb_run_launch(ctx, k_sp2_run<P, BN>, &fits, kRunThreads, Q::smem, r.cluster, r.grid, ran, s, g, mp);
}

template <int P>
int launch_bn(tb_ctx* ctx, const Sp2RunArgs& g, const RunShape& r, int* ran, cudaStream_t s) {
  switch (r.bn) {
    case 32: return launch<P, 32>(ctx, g, r, ran, s);
    case 64: return launch<P, 64>(ctx, g, r, ran, s);
    default: return launch<P, 128>(ctx, g, r, ran, s);
  }
}

}  // namespace

int sp2_run(tb_ctx* ctx, int precision, const Sp2RunArgs& g, int captured, int* ran, cudaStream_t s) {
  *ran = 0;
  if (precision != TB_PREC_TF32 && precision != TB_PREC_TF32X3) return TB_OK;
  if (sp2_tc_pairs(ctx, g.a.ld) > 0) return TB_OK;
  RunShape r;
  if (!tb_run_shape(ctx, g.a.ld, captured, &r)) return TB_OK;
  for (int round = 0; round < 2 && !*ran; ++round) {
    const int rc = precision == TB_PREC_TF32 ? launch_bn<TB_PREC_TF32>(ctx, g, r, ran, s)
                                             : launch_bn<TB_PREC_TF32X3>(ctx, g, r, ran, s);
    if (rc || !r.cluster) return rc;
    r.cluster = 0;  // no cluster of this size fits the device: a cooperative launch
  }
  return TB_OK;
}
