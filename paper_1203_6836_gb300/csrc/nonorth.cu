// Non-orthogonal formulation (row f3, App. D.1): the congruence factor
// Z = S^{-1/2} (Z^T S Z = I, Eq. Congr), H_perp = Z^T H Z, the density matrix
// rho = Z rho_perp Z^T of rho_perp = theta(mu0 I - H_perp) (dm_sp2) or the
// Fermi-Dirac matrix (dm_fermi) (Eq. DM_perp), and the energy-weighted
// density matrix W = Z (H_perp rho_perp + rho_perp H_perp) Z^T / 2 of the
// Pulay force.
//
// Z by the coupled Newton-Schulz iteration (GEMM only): with c >= lambda_max(S)
// (Gershgorin), Y_0 = S/c, Z_0 = I and
//   T_k = (3 I - Z_k Y_k)/2,  Y_{k+1} = Y_k T_k,  Z_{k+1} = T_k Z_k,
// Y_k -> (S/c)^{1/2} and Z_k -> (S/c)^{-1/2}, quadratically once
// ||I - S/c|| < 1 (the eigenvalues of S/c lie in (0, 1]); Z = Z_k / sqrt(c).
// Since Z_k Y_k = 3 I - 2 T_k, the residual max |Z_k Y_k - I| = 2 max |I - T_k|
// comes from T_k without another product; the iteration stops on the device
// at 1e-13, or below 1e-9 once the residual no longer halves (the rounding
// floor of the FP64 products at large n).  Up to n = 512 the whole iteration is one
// launch (k_ns_run); above, a fixed sequence of launches that return at once after
// the stop.
//
// All products are FP64 GEMMs on the FP64 units (no tensor-core FP64 on
// GB300): T x T output tiles, bounds-guarded for any n, row-major with
// stride n.  The FP64 rate bounds them (100 us for n = 384), so a product that is
// symmetric (every one of the iteration, whose factors are polynomials in S, and the
// second of each congruence Z M Z) computes its upper triangle only and mirrors it.

#include "common.cuh"
#include "persist.cuh"

#include <algorithm>

namespace {

constexpr int kMaxNS = 24;     // Newton-Schulz iterations at most (about 12 reach 1e-13 for cond(S) = 100)
constexpr double kNSTol = 1e-13;
constexpr double kNSFloor = 1e-9;  // below it, a residual that no longer halves is the rounding floor
constexpr int kK = 16;         // GEMM k-step
constexpr int kSmallN = 512;   // 16 x 16 tiles, and the Newton-Schulz iteration in one launch

struct NonorthState {
  double res;      // last Newton-Schulz residual
  int done;        // the iteration has converged
  int iters;
  int err;
  unsigned bar;    // grid barrier of k_ns_run
  unsigned left;   // its CTAs that have finished
  unsigned long long cmax;               // largest row sum of |S|, as bits (which order alike)
  unsigned long long tmax[kMaxNS];       // max |I - T_k| of each iteration, as bits
};

struct Layout {
  size_t off_state, off_mat, mat_bytes, off_inner, total;
  size_t inner_bytes;
};

constexpr int kMats = 7;  // Z, Y, T, P (scratch), H_perp, rho_perp, Q (scratch)

Layout make_layout(int n, size_t inner) {
  Layout L{};
  size_t o = 0;
  auto take = [&](size_t b) {
    const size_t r = o;
    o += (b + 1023) / 1024 * 1024;
    return r;
  };
  L.off_state = take(sizeof(NonorthState));
  L.mat_bytes = (sizeof(double) * (size_t)n * n + 1023) / 1024 * 1024;
  L.off_mat = take(L.mat_bytes * kMats);
  L.inner_bytes = inner;
  L.off_inner = take(inner);
  L.total = o;
  return L;
}

// C = alpha A B + beta E + gamma I (E may be null), n x n row-major; skipped
// when *skip is set; sym: C is symmetric (its upper triangle, mirrored: inside a diagonal
// tile too, where the two halves differ in rounding).  T x T tile per CTA, 256 threads with
// (T/16)^2 outputs.
template <int T>
__global__ void __launch_bounds__(256) k_gemm64(int n, double alpha, const double* __restrict__ A,
                                                const double* __restrict__ B, double beta,
                                                const double* __restrict__ E, double gamma,
                                                double* __restrict__ C, const int* skip, int sym) {
  constexpr int R = T / 16;
  __shared__ double As[kK][T + 1];
  __shared__ double Bs[kK][T + 1];
  if (skip && *skip) return;
  if (sym && blockIdx.x < blockIdx.y) return;  // the mirror of its twin
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int row0 = blockIdx.y * T, col0 = blockIdx.x * T;
  double acc[R][R];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) acc[i][j] = 0.0;
  for (int k0 = 0; k0 < n; k0 += kK) {
    for (int e = threadIdx.x; e < T * kK; e += 256) {
      const int r = e / kK, kk = e % kK;
      const int gr = row0 + r, gk = k0 + kk;
      As[kk][r] = (gr < n && gk < n) ? A[(size_t)gr * n + gk] : 0.0;
      const int kb = e / T, c = e % T;
      const int gkb = k0 + kb, gc = col0 + c;
      Bs[kb][c] = (gkb < n && gc < n) ? B[(size_t)gkb * n + gc] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kK; ++kk) {
      double av[R], bv[R];
#pragma unroll
      for (int i = 0; i < R; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < R; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int r = row0 + ty + 16 * i, c = col0 + tx + 16 * j;
      if (r >= n || c >= n || (sym && c < r)) continue;
      const size_t e = (size_t)r * n + c;
      double v = alpha * acc[i][j];
      if (E) v += beta * E[e];
      if (r == c) v += gamma;
      C[e] = v;
      if (sym) C[(size_t)c * n + r] = v;
    }
}

int gemm(tb_ctx* ctx, int n, double alpha, const double* A, const double* B, double beta, const double* E,
         double gamma, double* C, const int* skip, int sym, cudaStream_t s) {
  if (n <= kSmallN) {
    const dim3 g((n + 15) / 16, (n + 15) / 16);
    k_gemm64<16><<<g, 256, 0, s>>>(n, alpha, A, B, beta, E, gamma, C, skip, sym);
  } else {
    const dim3 g((n + 63) / 64, (n + 63) / 64);
    k_gemm64<64><<<g, 256, 0, s>>>(n, alpha, A, B, beta, E, gamma, C, skip, sym);
  }
  TB_LAUNCH_CHECK(ctx);
  return TB_OK;
}

// The largest row sum of |S| into st->cmax (zero at the start): a warp per row.
__device__ __forceinline__ void row_bound(const double* __restrict__ S, int n, int row, int lane, NonorthState* st) {
  double r = 0.0;
  for (int j = lane; j < n; j += 32) r += fabs(S[(size_t)row * n + j]);
  r = warp_sum(r);
  if (lane == 0) atomicMax(&st->cmax, (unsigned long long)__double_as_longlong(r));
}
__device__ __forceinline__ double bound_of(unsigned long long bits) {
  const double m = __longlong_as_double((long long)bits);
  return m > 0.0 ? m : 1.0;
}
// max |I - T| as bits, NaN above every number.
__device__ __forceinline__ unsigned long long dev_bits(double t, bool diag) {
  return (unsigned long long)__double_as_longlong(fabs(diag ? 1.0 - t : t));
}
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long m) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
    m = v > m ? v : m;
  }
  return m;
}

__global__ void __launch_bounds__(256) k_ns_bound(const double* __restrict__ S, int n, NonorthState* st) {
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row < n) row_bound(S, n, row, threadIdx.x & 31, st);
}

// The Newton-Schulz iteration in one launch (n <= kSmallN): the row bound, Y_0 and Z_0, then
// per iteration T (its deviation from I reduced on the way) and, after a grid barrier and
// the stop decision that every CTA takes alike, Y T and T Z together.  Launched, the
// iteration was 144 launches (one reading T on a single SM, two copies) of which it
// needs a quarter; n = 384, 6 iterations: 2.9 ms.  16 x 16 units of the upper triangle.
constexpr int kNsThr = 256, kNsKC = 64;
struct NsArgs {
  const double* S;
  double *Z[2], *Y[2], *T;  // the iterates, alternating; T also takes the result
  int n;
  NonorthState* st;
  tb_nonorth_report* rep;
};
__global__ void __launch_bounds__(kNsThr) k_ns_run(const NsArgs g) {
  using namespace tcx;
  __shared__ double As[16][kNsKC + 1], Bs[16][kNsKC + 1];
  __shared__ unsigned long long s_m[kNsThr / 32];
  __shared__ volatile int s_abort;
  __shared__ int s_ok;
  const int n = g.n, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = (n + 15) / 16, U = nt * (nt + 1) / 2;
  const unsigned G = gridDim.x;
  NonorthState* st = g.st;
  unsigned phase = 0;
  if (threadIdx.x == 0) s_abort = 0;
  // ends a phase: every CTA's stores are visible after it; false when a wait gave up
  auto meet = [&]() -> bool {
    __syncthreads();
    if (threadIdx.x == 0) {
      run_arrive(&st->bar);
      s_ok = run_wait(&st->bar, ++phase * G, &st->err, &s_abort);
    }
    __syncthreads();
    return s_ok;
  };
  auto tile = [&](int u, int* I, int* J) {
    int i = 0;
    while (u >= nt - i) {
      u -= nt - i;
      ++i;
    }
    *I = i;
    *J = i + u;
  };
  const int oi = threadIdx.x >> 4, oj = threadIdx.x & 15;
  // element (oi, oj) of tile (I, J) of A B, B symmetric (operands past L1: other SMs wrote them)
  auto product = [&](const double* A, const double* B, int I, int J) -> double {
    double pa[4], pb[4], acc = 0.0;
    auto fetch = [&](int k0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = threadIdx.x + i * kNsThr, r = e / kNsKC, c = k0 + e % kNsKC;
        pa[i] = (c < n && I * 16 + r < n) ? __ldcg(A + (size_t)(I * 16 + r) * n + c) : 0.0;
        pb[i] = (c < n && J * 16 + r < n) ? __ldcg(B + (size_t)(J * 16 + r) * n + c) : 0.0;
      }
    };
    fetch(0);
    for (int k0 = 0; k0 < n; k0 += kNsKC) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = threadIdx.x + i * kNsThr, r = e / kNsKC, c = e % kNsKC;
        As[r][c] = pa[i];
        Bs[r][c] = pb[i];
      }
      __syncthreads();
      if (k0 + kNsKC < n) fetch(k0 + kNsKC);
      const int ke = min(kNsKC, (n - k0 + 3) & ~3);
#pragma unroll 8
      for (int c = 0; c < ke; ++c) acc = fma(As[oi][c], Bs[oj][c], acc);
    }
    return acc;
  };
  auto put = [&](double* C, int I, int J, double v) {
    const int r = I * 16 + oi, c = J * 16 + oj;
    if (r >= n || c >= n || c < r) return;
    C[(size_t)r * n + c] = v;
    C[(size_t)c * n + r] = v;
  };
  for (int row = blockIdx.x * (kNsThr / 32) + warp; row < n; row += G * (kNsThr / 32)) row_bound(g.S, n, row, lane, st);
  bool ok = meet();
  const double c = bound_of(__ldcg(&st->cmax));
  {
    const double inv = 1.0 / c;
    for (int u = blockIdx.x; u < U && ok; u += G) {
      int I, J;
      tile(u, &I, &J);
      auto init = [&](int r, int q) {
        if (r >= n || q >= n) return;
        g.Y[0][(size_t)r * n + q] = g.S[(size_t)r * n + q] * inv;
        g.Z[0][(size_t)r * n + q] = r == q ? 1.0 : 0.0;
      };
      init(I * 16 + oi, J * 16 + oj);
      if (I != J) init(J * 16 + oi, I * 16 + oj);
    }
    ok = ok && meet();
  }
  double res = INFINITY;
  int it = 0, done = 0, cur = 0;
  for (; it < kMaxNS && !done && ok; ++it) {
    unsigned long long m = 0;
    for (int u = blockIdx.x; u < U; u += G) {
      int I, J;
      tile(u, &I, &J);
      double t = -0.5 * product(g.Z[cur], g.Y[cur], I, J);  // T = 3/2 I - Z Y / 2
      const bool dg = I == J && oi == oj;
      if (dg) t += 1.5;
      put(g.T, I, J, t);
      if (J * 16 + oj < n && I * 16 + oi <= J * 16 + oj) {  // the elements that put() stores
        const unsigned long long b = dev_bits(t, dg);
        m = b > m ? b : m;
      }
    }
    m = warp_max_bits(m);
    if (lane == 0) s_m[warp] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kNsThr / 32; ++w) m = s_m[w] > m ? s_m[w] : m;
      atomicMax(&st->tmax[it], m);
    }
    if (!(ok = meet())) break;
    const double r = 2.0 * __longlong_as_double((long long)__ldcg(&st->tmax[it])), prev = res;
    res = r;
    // converged, or stalled at the FP64 rounding floor of the products
    done = r <= kNSTol || (r <= kNSFloor && r >= 0.5 * prev);
    if (done) continue;
    for (int u = blockIdx.x; u < 2 * U; u += G) {
      int I, J;
      tile(u < U ? u : u - U, &I, &J);
      if (u < U) put(g.Y[cur ^ 1], I, J, product(g.Y[cur], g.T, I, J));
      else put(g.Z[cur ^ 1], I, J, product(g.T, g.Z[cur], I, J));
    }
    ok = meet();
    cur ^= 1;
  }
  // Z / sqrt(c) into T's place
  const double f = 1.0 / sqrt(c);
  for (int u = blockIdx.x; u < U && ok; u += G) {
    int I, J;
    tile(u, &I, &J);
    const int r = I * 16 + oi, q = J * 16 + oj;
    if (r < n && q < n) put(g.T, I, J, f * __ldcg(g.Z[cur] + (size_t)r * n + q));
  }
  if (threadIdx.x == 0) {
    if (!ok) atomicExch(&st->err, TB_ERR_TIMEOUT);
    if (run_last(&st->left, G) && g.rep) {
      const int err = *reinterpret_cast<volatile int*>(&st->err);
      g.rep->status = err ? err : done ? TB_OK : TB_ERR_NOT_CONVERGED;
      g.rep->ns_iters = it;
      g.rep->ns_residual = res;
    }
  }
}

// Y = S / c, Z = I.
__global__ void k_ns_init(const double* __restrict__ S, int n, const NonorthState* st, double* __restrict__ Y,
                          double* __restrict__ Z) {
  const double c = bound_of(st->cmax), inv = 1.0 / c;
  const size_t total = (size_t)n * n;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    Y[e] = S[e] * inv;
    Z[e] = (e / n == e % n) ? 1.0 : 0.0;
  }
}

// max |I - T_k|, then the stop decision.
__global__ void __launch_bounds__(256) k_ns_dev(const double* __restrict__ T, int n, NonorthState* st, int it) {
  if (st->done) return;
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  unsigned long long m = 0;
  if (row < n)
    for (int j = lane; j < n; j += 32) {
      const unsigned long long b = dev_bits(T[(size_t)row * n + j], j == row);
      m = b > m ? b : m;
    }
  m = warp_max_bits(m);
  if (lane == 0) atomicMax(&st->tmax[it], m);
}
__global__ void k_ns_check(NonorthState* st, int it) {
  if (st->done) return;
  const double r = 2.0 * __longlong_as_double((long long)st->tmax[it]), prev = it ? st->res : INFINITY;
  st->res = r;
  st->iters = it + 1;
  // converged, or stalled at the FP64 rounding floor of the products
  if (r <= kNSTol || (r <= kNSFloor && r >= 0.5 * prev)) st->done = 1;
}

// Z <- Z / sqrt(c) (the final factor), report.
__global__ void k_ns_finish(double* __restrict__ Z, int n, const NonorthState* st, tb_nonorth_report* rep) {
  const double f = 1.0 / sqrt(bound_of(st->cmax));
  const size_t total = (size_t)n * n;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x)
    Z[e] *= f;
  if (rep && blockIdx.x == 0 && threadIdx.x == 0) {
    rep->status = st->done ? TB_OK : TB_ERR_NOT_CONVERGED;
    rep->ns_iters = st->iters;
    rep->ns_residual = st->res;
  }
}

// W = (W' + W'^T) / 2 in place.
__global__ void k_symmetrize(double* __restrict__ W, int n) {
  const size_t total = (size_t)n * n;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const size_t r = e / n, c = e % n;
    if (r < c) {
      const double a = W[e], b = W[c * n + r];
      const double m = 0.5 * (a + b);
      W[e] = m;
      W[c * n + r] = m;
    }
  }
}

// dst = src unless *skip.
__global__ void k_copy_unless(const double* __restrict__ src, double* __restrict__ dst, int n, const int* skip) {
  if (*skip) return;
  const size_t total = (size_t)n * n;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x)
    dst[e] = src[e];
}

size_t inner_bytes(int n, double kT, const tb_sp2_opts* so, const tb_fermi_opts* fo, int* rc) {
  size_t b = 0;
  *rc = kT > 0.0 ? dm_fermi_workspace_size(n, fo, &b) : dm_sp2_workspace_size(n, so, &b);
  return b;
}

}  // namespace

extern "C" int dm_nonorth_workspace_size(int n, double kT, const tb_sp2_opts* so, const tb_fermi_opts* fo,
                                         size_t* bytes) {
  if (n < 1 || !bytes || (kT > 0.0 ? !fo : !so)) return TB_ERR_ARG;
  int rc = TB_OK;
  const size_t inner = inner_bytes(n, kT, so, fo, &rc);
  if (rc) return rc;
  *bytes = make_layout(n, inner).total;
  return TB_OK;
}

extern "C" int dm_nonorth(tb_ctx* ctx, const double* H, const double* S, int n, double n_occ, double kT,
                          const tb_sp2_opts* so, const tb_fermi_opts* fo, double* mu, double* rho, double* W,
                          void* ws, size_t ws_bytes, tb_sp2_report* sp2_report, tb_fermi_report* fermi_report,
                          tb_nonorth_report* report, void* stream) {
  if (!ctx) return TB_ERR_ARG;
  if (!H || !S || !rho || !W || !ws) return tb_fail(ctx, TB_ERR_ARG, "null argument to dm_nonorth");
  if (n < 1) return tb_fail(ctx, TB_ERR_ARG, "n = %d", n);
  if (kT > 0.0 ? (!fo || !mu) : !so) return tb_fail(ctx, TB_ERR_ARG, "dm_nonorth: missing solver options");
  int rc = TB_OK;
  const size_t inner = inner_bytes(n, kT, so, fo, &rc);
  if (rc) return tb_fail(ctx, rc, "dm_nonorth: inner workspace query failed");
  const Layout L = make_layout(n, inner);
  if (ws_bytes < L.total) return tb_fail(ctx, TB_ERR_ARG, "workspace %zu bytes < required %zu", ws_bytes, L.total);
  if ((reinterpret_cast<uintptr_t>(ws) & 1023) != 0) return tb_fail(ctx, TB_ERR_ARG, "workspace must be 1024-byte aligned");
  cudaStream_t s = as_stream(stream);
  char* base = static_cast<char*>(ws);
  NonorthState* st = reinterpret_cast<NonorthState*>(base + L.off_state);
  double* M[kMats];
  for (int i = 0; i < kMats; ++i) M[i] = reinterpret_cast<double*>(base + L.off_mat + i * L.mat_bytes);
  double *Z = M[0], *Y = M[1], *T = M[2], *P = M[3], *Hp = M[4], *Dp = M[5], *Q = M[6];
  const int eb = std::min(1184, (int)(((size_t)n * n + 255) / 256));

  // Z = S^{-1/2} by coupled Newton-Schulz
  TB_CUDA_TRY(ctx, cudaMemsetAsync(st, 0, sizeof(NonorthState), s));
  if (n <= kSmallN) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    TB_CUDA_TRY(ctx, cudaStreamIsCapturing(s, &cs));
    const int nt = (n + 15) / 16, U = nt * (nt + 1) / 2;
    // captured steps run beside those of other trajectories: half the chip at most
    const int G = std::min(U, tb_persistent_grid(ctx, cs != cudaStreamCaptureStatusNone ? ctx->sm_count / 2 : 1 << 30));
    NsArgs a{S, {Z, P}, {Y, Q}, T, n, st, report};
    int ran = 0;
    if ((rc = tb_run_launch(ctx, k_ns_run, nullptr, kNsThr, 0, 0, G, &ran, s, a))) return rc;
    std::swap(Z, T);
  } else {
    // each update goes through P and a copy, so the current iterate stays in Z and Y
    // whichever launch the stop skips
    k_ns_bound<<<(n + 7) / 8, 256, 0, s>>>(S, n, st);
    TB_LAUNCH_CHECK(ctx);
    k_ns_init<<<eb, 256, 0, s>>>(S, n, st, Y, Z);
    TB_LAUNCH_CHECK(ctx);
    const int* skip = &st->done;
    for (int it = 0; it < kMaxNS; ++it) {
      if ((rc = gemm(ctx, n, -0.5, Z, Y, 0.0, nullptr, 1.5, T, skip, 1, s))) return rc;  // T = 3/2 I - Z Y / 2
      k_ns_dev<<<(n + 7) / 8, 256, 0, s>>>(T, n, st, it);
      TB_LAUNCH_CHECK(ctx);
      k_ns_check<<<1, 1, 0, s>>>(st, it);
      TB_LAUNCH_CHECK(ctx);
      if ((rc = gemm(ctx, n, 1.0, Y, T, 0.0, nullptr, 0.0, P, skip, 1, s))) return rc;
      k_copy_unless<<<eb, 256, 0, s>>>(P, Y, n, skip);
      TB_LAUNCH_CHECK(ctx);
      if ((rc = gemm(ctx, n, 1.0, T, Z, 0.0, nullptr, 0.0, P, skip, 1, s))) return rc;
      k_copy_unless<<<eb, 256, 0, s>>>(P, Z, n, skip);
      TB_LAUNCH_CHECK(ctx);
    }
    k_ns_finish<<<eb, 256, 0, s>>>(Z, n, st, report);
    TB_LAUNCH_CHECK(ctx);
  }

  // H_perp = Z H Z (Z symmetric)
  if ((rc = gemm(ctx, n, 1.0, Z, H, 0.0, nullptr, 0.0, P, nullptr, 0, s))) return rc;
  if ((rc = gemm(ctx, n, 1.0, P, Z, 0.0, nullptr, 0.0, Hp, nullptr, 1, s))) return rc;
  // rho_perp
  void* iws = base + L.off_inner;
  if (kT > 0.0)
    rc = dm_fermi(ctx, Hp, n, n_occ, kT, fo, Dp, mu, iws, L.inner_bytes, fermi_report, s);
  else
    rc = dm_sp2(ctx, Hp, n, n_occ, so, Dp, iws, L.inner_bytes, sp2_report, s);
  if (rc) return rc;
  // rho = Z rho_perp Z
  if ((rc = gemm(ctx, n, 1.0, Z, Dp, 0.0, nullptr, 0.0, P, nullptr, 0, s))) return rc;
  if ((rc = gemm(ctx, n, 1.0, P, Z, 0.0, nullptr, 0.0, rho, nullptr, 1, s))) return rc;
  // W = Z (H_perp rho_perp + rho_perp H_perp) Z / 2 = Z sym(H_perp rho_perp) Z
  if ((rc = gemm(ctx, n, 1.0, Hp, Dp, 0.0, nullptr, 0.0, Q, nullptr, 0, s))) return rc;
  k_symmetrize<<<eb, 256, 0, s>>>(Q, n);
  TB_LAUNCH_CHECK(ctx);
  if ((rc = gemm(ctx, n, 1.0, Z, Q, 0.0, nullptr, 0.0, P, nullptr, 0, s))) return rc;
  if ((rc = gemm(ctx, n, 1.0, P, Z, 0.0, nullptr, 0.0, W, nullptr, 1, s))) return rc;
  return TB_OK;
}
