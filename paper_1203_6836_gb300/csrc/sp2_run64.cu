// The FP64 SP2 path (TB_PREC_FP64) of small matrices in one launch: X0, every
// projection, the decisions, D and the report.
//
// What bounds the launched form: a projection of a 48 x 48 matrix is about a microsecond
// of FP64 work (GB300: two FP64 results per clock and SM), a launch costs more, and
// outside a captured graph the host enqueues max_iter + 1 of them.  Here the
// projections are separated by a grid barrier, and only the upper triangle of the
// symmetric X^2 is computed and mirrored, which halves the FP64 work of every size.
//
// A unit is a T x T tile: 8 x 8 up to n = 136 (153 units: one per SM), where the 256
// threads split K in four, 16 x 16 above.  8 x 8 tiles cost 16 bytes of operands per
// FMA pair from shared memory, which the FP64 rate leaves time for many times over.
//
// n <= 512; above that a projection has work enough for its launch (sp2.cu).

#include "persist.cuh"
#include "sp2_run.cuh"

#include <algorithm>

namespace {

using namespace tcx;

constexpr int kThr = 256;
constexpr int kKC = 64;  // columns of the panels staged at a time

template <int T>
__global__ void __launch_bounds__(kThr) k_sp2_run64(const Sp2Run64Args g) {
  constexpr int KG = kThr / (T * T);  // K groups per unit
  constexpr int kPer = T * kKC / kThr;  // panel entries per thread and operand
  __shared__ double As[T][kKC + 1], Bs[T][kKC + 1];
  __shared__ double red[kThr];
  __shared__ double s_red[8][2];
  __shared__ double s_lo, s_hi;
  __shared__ int s_dec;
  __shared__ volatile int s_abort;
  SP2StepArgs a = g.a;
  SP2State* st = a.st;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned G = gridDim.x;
  const int nt = (a.n + T - 1) / T, U = nt * (nt + 1) / 2;
  const unsigned Gw = min(G, (unsigned)U);
  if (blockIdx.x >= Gw) return;  // no units (persist.cuh, grid barrier)
  const int kn = nt * T;  // columns in use; the padding up to it is zero
  auto tile = [&](int u, int* I, int* J) {
    int i = 0;
    while (u >= nt - i) {
      u -= nt - i;
      ++i;
    }
    *I = i;
    *J = i + u;
  };
  if (threadIdx.x == 0) s_abort = 0;
  if (warp == 0) {
    double lo = INFINITY, hi = -INFINITY;
    for (int i = lane; i < g.nbparts; i += 32) {
      lo = fmin(lo, g.bparts[2 * i]);
      hi = fmax(hi, g.bparts[2 * i + 1]);
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
  __syncthreads();
  // (t1, t2) of a unit into its slot (all threads)
  auto put_parts = [&](double* parts, int u, double t1, double t2) {
    t1 = warp_sum(t1);
    t2 = warp_sum(t2);
    if (lane == 0) {
      s_red[warp][0] = t1;
      s_red[warp][1] = t2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
      double t = 0.0;
      for (int w = 0; w < kThr / 32; ++w) t += s_red[w][threadIdx.x];
      parts[2 * u + threadIdx.x] = t;
    }
    __syncthreads();
  };
  {
    // X0 = (emax I - H)/(emax - emin), zero outside n x n
    const double emax = s_hi;
    double w = emax - s_lo;
    if (!(w > 0.0)) w = 1.0;  // H = c I: X0 = 0 (no gap; reported through the trace)
    const double inv = 1.0 / w;
    for (int u = blockIdx.x; u < U; u += G) {
      int I, J;
      tile(u, &I, &J);
      double t1 = 0.0, t2 = 0.0;
      auto put = [&](int r, int c) {
        double x = 0.0;
        if (r < a.n && c < a.n) x = ((r == c ? emax : 0.0) - g.H[(size_t)r * a.n + c]) * inv;
        g.F[0][(size_t)r * a.ld + c] = x;
        if (r == c) t1 += x;
        t2 += x * x;
      };
      const int e = threadIdx.x;
      if (e < T * T) {
        put(I * T + e / T, J * T + e % T);
        if (I != J) put(J * T + e / T, I * T + e % T);
      }
      put_parts(g.parts[0], u, t1, t2);
    }
    if (threadIdx.x == 0) run_arrive(g.bar);
  }
  for (int k = 0;; ++k) {
    const double* X = g.F[k & 1];
    double* Y = g.F[(k & 1) ^ 1];
    if (threadIdx.x == 0 && !run_wait(g.bar, (unsigned)(k + 1) * Gw, &st->err, &s_abort)) s_abort = 1;
    __syncthreads();
    // the first panels of the first unit, fetched past L1 (other SMs wrote them)
    // beside the partials
    double pa[kPer], pb[kPer], xrc = 0.0;
    int I = 0, J = 0;
    auto fetch = [&](int k0) {
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int e = threadIdx.x + i * kThr, r = e / kKC, c = k0 + e % kKC;
        pa[i] = c < kn ? __ldcg(X + (size_t)(I * T + r) * a.ld + c) : 0.0;
        pb[i] = c < kn ? __ldcg(X + (size_t)(J * T + r) * a.ld + c) : 0.0;
      }
    };
    const int oi = (threadIdx.x % (T * T)) / T, oj = threadIdx.x % T, kg = threadIdx.x / (T * T);
    tile(blockIdx.x, &I, &J);
    fetch(0);
    xrc = __ldcg(X + (size_t)(I * T + oi) * a.ld + J * T + oj);
    if (warp == 0) {
      double x = 0.0, y = 0.0;
      for (int i = lane; i < U; i += 32) {
        x += __ldcg(g.parts[k & 1] + 2 * i);
        y += __ldcg(g.parts[k & 1] + 2 * i + 1);
      }
      x = warp_sum(x);
      y = warp_sum(y);
      if (lane == 0) {
        int br = 0, capped = 0, stop = 1;
        if (!s_abort) {
          a.k = k;
          stop = sp2_decide_e(a, x, y, 0.0, 0.0, 0.0, false, &br, &capped);
          if (blockIdx.x == 0) {
            st->t1[k] = x;
            st->t2[k] = y;
            if (stop) {
              st->iters = k;
              st->capped = capped;
              st->done = 1;
            } else if (br) {
              st->branch[k >> 6] |= 1ull << (k & 63);
            }
          }
        }
        s_dec = stop | (br << 1);
      }
    }
    __syncthreads();
    const int dec = s_dec;
    if (dec & 1) {
      if (!s_abort) {
        // D, of this CTA's units, mirrored
        for (int u = blockIdx.x; u < U; u += G) {
          tile(u, &I, &J);
          const int e = threadIdx.x, r = I * T + e / T, c = J * T + e % T;
          if (e < T * T && r < a.n && c < a.n) {
            const double x = __ldcg(X + (size_t)r * a.ld + c);
            g.D[(size_t)r * a.n + c] = x;
            if (I != J) g.D[(size_t)c * a.n + r] = x;
          }
        }
      }
      break;
    }
    for (int u = blockIdx.x; u < U; u += G) {
      if (u != (int)blockIdx.x) {
        tile(u, &I, &J);
        fetch(0);
        xrc = __ldcg(X + (size_t)(I * T + oi) * a.ld + J * T + oj);
      }
      double acc = 0.0;
      for (int k0 = 0; k0 < kn; k0 += kKC) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          const int e = threadIdx.x + i * kThr, r = e / kKC, c = e % kKC;
          As[r][c] = pa[i];
          Bs[r][c] = pb[i];
        }
        __syncthreads();
        if (k0 + kKC < kn) fetch(k0 + kKC);
        const int ke = min(kKC, kn - k0);  // a multiple of T, hence of KG
#pragma unroll 8
        for (int c = kg; c < ke; c += KG) acc = fma(As[oi][c], Bs[oj][c], acc);
        __syncthreads();
      }
      if (KG > 1) {
        red[threadIdx.x] = acc;
        __syncthreads();
        if (threadIdx.x < T * T) {
#pragma unroll
          for (int q = 1; q < KG; ++q) acc += red[threadIdx.x + q * T * T];
        }
      }
      double t1 = 0.0, t2 = 0.0;
      if (threadIdx.x < T * T) {
        const int r = I * T + oi, c = J * T + oj;
        const double y = (dec & 2) ? 2.0 * xrc - acc : acc;
        Y[(size_t)r * a.ld + c] = y;
        if (I != J) Y[(size_t)c * a.ld + r] = y;
        if (r == c) t1 = y;
        t2 = (I != J ? 2.0 : 1.0) * (y * y);
      }
      put_parts(g.parts[(k & 1) ^ 1], u, t1, t2);
    }
    if (threadIdx.x == 0) run_arrive(g.bar);
  }
  if (threadIdx.x == 0) {
    if (s_abort) atomicExch(&st->err, TB_ERR_TIMEOUT);
    if (run_last(&st->left, Gw) && g.rep) sp2_fill_report(st, 0, a.n, a.nocc, g.rep);
  }
}

template <int T>
int launch(tb_ctx* ctx, const Sp2Run64Args& g, cudaStream_t s) {
  const int nt = (g.a.n + T - 1) / T, U = nt * (nt + 1) / 2;
  // The whole chip, also under capture: three of these blocks fit an SM, so chains of several
  // captured steps run side by side.  (Held to half the chip, as the chains that fill an SM's
  // shared memory are, a captured call of n = 192 took 460 us for its 78 units on 76 blocks,
  // 258 on the whole chip, 326 launched; n = 512 4.10 ms, 2.38, 4.03.  Four such calls at once,
  // us a call: n = 192 197 / 144 / 206, n = 512 1913 / 2189 / 3765.)
  const int G = std::min(U, tb_persistent_grid(ctx, 1 << 30));
  static RunFits fits;
  int ran = 0, c = 1;
  if (G <= 16) {
    while (c < G) c *= 2;
    if (ctx->grid_limit > 0 && c > ctx->grid_limit) c /= 2;
    const int rc = tb_run_launch(ctx, k_sp2_run64<T>, &fits, kThr, 0, 1, c, &ran, s, g);
    if (rc || ran) return rc;
  }
  return tb_run_launch(ctx, k_sp2_run64<T>, &fits, kThr, 0, 0, G, &ran, s, g);
}

}  // namespace

int sp2_run64(tb_ctx* ctx, const Sp2Run64Args& g, cudaStream_t s) {
  return g.a.n <= 136 ? launch<8>(ctx, g, s) : launch<16>(ctx, g, s);
}
