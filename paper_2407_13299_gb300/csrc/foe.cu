// Chebyshev Fermi-operator expansion at finite electronic temperature (the
// finite-temperature method Sec. "Introduction" names: the Fermi Operator
// Expansion of Goedecker and Teter, Phys. Rev. B 51, 9455).
//
// P = f(H), f(e) = 1 / (1 + exp((e - mu) / kT)). H is scaled into [-1, 1] by a
// spectral enclosure [e_min, e_max] (a = centre, b = half-width, b = 1 for a
// point): H_s = (H - a I) / b. g(x) = f(a + b x) is expanded in M Chebyshev
// terms with coefficients from Gauss-Chebyshev quadrature on N = 2M nodes,
//   theta_j = pi (2j + 1) / (2N), x_j = cos(theta_j),
//   c_k = (2 / N) sum_j g(x_j) cos(k theta_j),
// and P = (c_0 / 2) I + sum_{k>=1} c_k T_k(H_s) with T_{k+1} = 2 H_s T_k - T_{k-1}.
// The products H_s T_k are formed by the product kernels of the library, whose
// output step makes them the next term and adds it to P (EPI_CHEB: a separate
// pass read and wrote 5 n^2 doubles for it; n = 2048: 20 us of a 160 us step);
// this file holds the scalar set-up (enclosure, mu, coefficients) and the
// elementwise passes.
//
// Second evaluation of the same series (Paterson-Stockmeyer, after Liang et
// al., J. Chem. Phys. 119, 4117 (2003)): q = ceil(sqrt(M)) baby steps T_1 .. T_q
// are kept, the series is folded into sum_{m<r} T_m(y) B_m with y = T_q and
// B_m = sum_{j<q} w_{m,j} T_j (T_{qm+j} = 2 T_m(y) T_j - T_{qm-j}), and summed
// by Clenshaw's recurrence in y. Its kernels here: the weighted combination
// with the Clenshaw update, the
// Frobenius products <T_{qm}, T_j> and the trace assembly of canonical use,
// and the block folding of the coefficients.
//
// With a target n_occ, mu solves sum_k c_k(mu) tr T_k = n_occ. Writing
// w_j = t_0 / 2 + sum_{k>=1} t_k cos(k theta_j) (t_k = tr T_k from a first pass
// of the recurrence), the expansion's trace is (2 / N) sum_j g_mu(x_j) w_j, and
// mu is found by at least 100 bisection halvings of [e_min - 40 kT, e_max + 40 kT].
//
// cos(k theta_j) is evaluated as cospi(r / 2N) with r = k (2j + 1) mod 4N, an
// exact integer reduction, so large k lose no accuracy to the argument.
// Every sum runs in a fixed order: results are reproducible bit for bit.

#include <algorithm>

#include "dmp_internal.cuh"

namespace dmp {

namespace {

constexpr int kReduceThreads = 1024;
constexpr double kMuBracketKT = 40.0;
constexpr int kMuHalvings = 100;
constexpr int kMuLevels = 7;  // halvings per round of the bisection
constexpr int kMuNodes = (1 << kMuLevels) - 1;
constexpr int kSumThreads = 256;

// Fermi-Dirac occupation without overflow.
__device__ __forceinline__ double fermi(double e, double mu, double kT) {
  const double z = (e - mu) / kT;
  if (z > 0.0) {
    const double ez = exp(-z);
    return ez / (1.0 + ez);
  }
  return 1.0 / (1.0 + exp(z));
}

// cos(k theta_j), theta_j = pi (2j + 1) / (2N)
__device__ __forceinline__ double cos_k_theta(int64_t k, int64_t j, int64_t N) {
  // k < M and 2 j + 1 < 2 N = 4 M: the product stays below 2^31 (M <= 16384)
  const uint32_t r = (static_cast<uint32_t>(k) * static_cast<uint32_t>(2 * j + 1)) % static_cast<uint32_t>(4 * N);
  return cospi(static_cast<double>(r) / static_cast<double>(2 * N));
}

__device__ __forceinline__ double node_x(int64_t j, int64_t N) {
  return cospi(static_cast<double>(2 * j + 1) / static_cast<double>(2 * N));
}

// Block-wide sum in a fixed tree (blockDim.x == kReduceThreads); every thread
// gets the total.
__device__ double block_sum(double v, double* red) {
  const int t = threadIdx.x;
  red[t] = v;
  __syncthreads();
  for (int o = kReduceThreads / 2; o > 0; o >>= 1) {
    if (t < o) red[t] += red[t + o];
    __syncthreads();
  }
  const double total = red[0];
  __syncthreads();
  return total;
}

// The enclosure that scales H: the caller's, else the Gershgorin bounds.
__global__ void foe_scale_kernel(const PurifyState* st, double e_min, double e_max, int use_given,
                                 FoeScalars* sc) {
  const double lo = use_given ? e_min : st->h_min;
  const double hi = use_given ? e_max : st->h_max;
  double b = 0.5 * (hi - lo);
  if (!(b > 0.0)) b = 1.0;
  sc->e_min = lo;
  sc->e_max = hi;
  sc->a = 0.5 * (hi + lo);
  sc->b = b;
  sc->nonfinite = st->nonfinite;
  sc->ticket = 0;
}

// Block-wide sum over kSumThreads threads, to thread 0 (fixed order).
__device__ __forceinline__ double block_sum256(double v, double* red) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kSumThreads / 32; ++w) t += red[w];
  return t;
}

// One CTA per node j: w_j = t_0 / 2 + sum_{k=1}^{M-1} t_k cos(k theta_j), and the
// node's energy e_j = a + b x_j. (A thread per node walked its M cosines one
// after the other: 367 us at M = 200, 9 now.)
__global__ void __launch_bounds__(kSumThreads)
foe_weights_kernel(const FoeScalars* sc, const double* traces, int M, double* w,
                   double* e) {
  chain_wait();
  chain_next();
  __shared__ double red[kSumThreads / 32];
  const int64_t N = 2 * static_cast<int64_t>(M);
  const int64_t j = blockIdx.x;
  double acc = 0.0;
  for (int k = 1 + threadIdx.x; k < M; k += kSumThreads) acc += traces[k] * cos_k_theta(k, j, N);
  const double total = block_sum256(acc, red);
  if (threadIdx.x == 0) {
    w[j] = 0.5 * traces[0] + total;
    e[j] = sc->a + sc->b * node_x(j, N);
  }
}

// The bisection for mu in rounds of kMuLevels halvings: CTA i evaluates the
// expansion's trace at midpoint i + 1 (heap order) of the tree of intervals the
// next halvings can reach, so a round costs one evaluation's time, and the path
// taken is the plain bisection's. ws holds, for even and odd rounds, the round's
// interval and the traces at its midpoints (one CTA halving 100 times: 1.17 ms
// at M = 200, bound by the FP64 pipe of one SM; 15 rounds: 0.16 ms; 31 midpoints
// and 20 rounds would add five launches for the same evaluation time).
struct MuRound {
  double lo, hi;
  double tr[kMuNodes + 1];
};

// The interval round `round` starts from; every thread of the block gets it.
__device__ __forceinline__ void mu_interval(const FoeScalars* sc, double kT, double n_occ, int round,
                                            const MuRound* ws, double* tr, double& lo, double& hi) {
  if (round == 0) {
    lo = sc->e_min - kMuBracketKT * kT;
    hi = sc->e_max + kMuBracketKT * kT;
    return;
  }
  const MuRound& last = ws[(round - 1) & 1];
  for (int i = threadIdx.x; i < kMuNodes; i += blockDim.x) tr[i] = last.tr[i];
  lo = last.lo;
  hi = last.hi;
  __syncthreads();
  for (int level = 0, i = 1; level < kMuLevels; ++level) {
    const double mid = 0.5 * (lo + hi);
    const bool up = tr[i - 1] < n_occ;
    lo = up ? mid : lo;
    hi = up ? hi : mid;
    i = 2 * i + (up ? 1 : 0);
  }
}

__global__ void __launch_bounds__(kSumThreads)
foe_mu_round_kernel(const FoeScalars* sc, double kT, double n_occ, int M, const double* w,
                    const double* e, int round, MuRound* ws) {
  chain_wait();
  chain_next();
  __shared__ double tr[kMuNodes];
  __shared__ double red[kSumThreads / 32];
  double lo, hi;
  mu_interval(sc, kT, n_occ, round, ws, tr, lo, hi);
  MuRound& out = ws[round & 1];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    out.lo = lo;
    out.hi = hi;
  }
  // down the tree to this CTA's midpoint: the bits of its heap index after the first
  const int node = static_cast<int>(blockIdx.x) + 1;
  for (int bit = 30 - __clz(node); bit >= 0; --bit) {
    const double mid = 0.5 * (lo + hi);
    if ((node >> bit) & 1) {
      lo = mid;
    } else {
      hi = mid;
    }
  }
  const double mid = 0.5 * (lo + hi);
  const int N = 2 * M;
  double part = 0.0;
  for (int j = threadIdx.x; j < N; j += kSumThreads) part += fermi(e[j], mid, kT) * w[j];
  const double total = block_sum256(part, red);
  if (threadIdx.x == 0) out.tr[node - 1] = (2.0 / static_cast<double>(N)) * total;
}

// g(x_j) at mu (the bisection's when `rounds` > 0, else the given one). gx may be e.
__global__ void __launch_bounds__(kSumThreads)
foe_occupation_kernel(FoeScalars* sc, double kT, double mu_given, double n_occ, int rounds, int M, const MuRound* ws,
                      const double* e, double* gx) {
  chain_wait();
  chain_next();
  __shared__ double tr[kMuNodes];
  double mu = mu_given;
  if (rounds > 0) {
    double lo, hi;
    mu_interval(sc, kT, n_occ, rounds, ws, tr, lo, hi);
    mu = 0.5 * (lo + hi);
  }
  const int64_t N = 2 * static_cast<int64_t>(M);
  const int64_t j = static_cast<int64_t>(blockIdx.x) * kSumThreads + threadIdx.x;
  if (j < N) gx[j] = fermi(rounds > 0 ? e[j] : sc->a + sc->b * node_x(j, N), mu, kT);
  if (j == 0) sc->mu = mu;
}

// One CTA per k: c_k = (2 / N) sum_j g(x_j) cos(k theta_j). (A thread per k:
// 621 us at M = 200, 9 now.)
__global__ void __launch_bounds__(kSumThreads)
foe_coeff_kernel(const double* gx, int M, double* coeffs) {
  chain_wait();
  chain_next();
  __shared__ double red[kSumThreads / 32];
  const int64_t N = 2 * static_cast<int64_t>(M);
  const int k = blockIdx.x;
  double acc = 0.0;
  for (int64_t j = threadIdx.x; j < N; j += kSumThreads) acc += gx[j] * cos_k_theta(k, j, N);
  const double total = block_sum256(acc, red);
  if (threadIdx.x == 0) coeffs[k] = (2.0 / static_cast<double>(N)) * total;
}

// H_s = (H - a I) / b (upper triangle of H read, mirrored), T_0 = I, T_1 = H_s
// (each when its pointer is non-null), and, with coefficients,
// P = (c_0 / 2) I + c_1 H_s. Matrices of leading dimension n except H (ldh)
// and P (ldp). 32 x 32 blocks on and above the diagonal, mirrored through
// shared memory.
__global__ void __launch_bounds__(256)
foe_init_kernel(const double* H, int64_t ldh, int64_t n, const FoeScalars* sc,
                const double* coeffs, double* Hs, double* T0,
                double* T1, double* P, int64_t ldp, int T) {
  chain_wait();
  chain_next();
  __shared__ double tile[32][33];
  int bi, bj;
  upper_tile(blockIdx.x, T, bi, bj);
  const double a = sc->a, b = sc->b;
  const double c0h = coeffs ? 0.5 * coeffs[0] : 0.0;
  const double c1 = coeffs ? coeffs[1] : 0.0;
  const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
  for (int y = y0; y < 32; y += 8) {
    const int64_t r = 32 * static_cast<int64_t>(bi) + y, c = 32 * static_cast<int64_t>(bj) + x;
    if (r < n && c < n) tile[y][x] = H[r * ldh + c];
  }
  __syncthreads();
  for (int half = 0; half < (bi == bj ? 1 : 2); ++half) {
    // half 1: the mirrored block
    const int64_t br = half ? bj : bi, bc = half ? bi : bj;
    for (int y = y0; y < 32; y += 8) {
      const int64_t r = 32 * br + y, c = 32 * bc + x;
      if (r >= n || c >= n) continue;
      const bool flip = half != 0 || r > c;
      const double h = flip ? tile[x][y] : tile[y][x];
      const double d = r == c ? 1.0 : 0.0;
      const double hs = (h - (r == c ? a : 0.0)) / b;
      Hs[r * n + c] = hs;
      if (T0) T0[r * n + c] = d;
      if (T1) T1[r * n + c] = hs;
      if (coeffs) P[r * ldp + c] = c0h * d + c1 * hs;
    }
  }
}

// out = sum_i A_ii in a fixed order (one CTA).
// out[blockIdx.x] for the blockIdx.x-th matrix, `stride` doubles apart.
__global__ void __launch_bounds__(kReduceThreads)
foe_trace_kernel(const double* A, int64_t lda, int64_t stride, int64_t n, double* out) {
  chain_wait();
  chain_next();
  __shared__ double red[kReduceThreads];
  A += blockIdx.x * stride;
  double part = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += kReduceThreads) part += A[i * lda + i];
  const double total = block_sum(part, red);
  if (threadIdx.x == 0) out[blockIdx.x] = total;
}

// ---- Paterson-Stockmeyer evaluation (Liang et al., J. Chem. Phys. 119, 4117):
// baby steps T_1 .. T_q kept in q slots of n x n (T_0 = I implicit), y = T_q.

// out = ((w_0 I + w_1 T_1 + ... + w_{nt-1} T_{nt-1}) + alpha Y) - Bm2, the Y and
// Bm2 terms only when their pointers are non-null. T_t lives at T + (t - 1) tstride.
// out (leading dimension ldo) may be Bm2 (in place). Every matrix is symmetric:
// 32 x 32 blocks on and above the diagonal are formed and mirrored, which halves
// the FP64 operations that bound the kernel (nt + 1 per element; n = 2048, nt =
// 15: 115 us over the full matrix, 66 now).
__global__ void __launch_bounds__(256)
foe_combine_kernel(const double* Tm, int64_t tstride, int nt, const double* w,
                   const double* Y, double alpha, const double* Bm2, double* out, int64_t ldo, int64_t n,
                   int T) {
  chain_wait();
  chain_next();
  __shared__ double tile[32][33];
  int bi, bj;
  upper_tile(blockIdx.x, T, bi, bj);
  const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
  const int64_t c = 32 * static_cast<int64_t>(bj) + x;
  double v[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) v[u] = 32 * static_cast<int64_t>(bi) + y0 + 8 * u == c ? w[0] : 0.0;
  const int64_t r0 = 32 * static_cast<int64_t>(bi) + y0;
  for (int t = 1; t < nt; ++t) {
    const double* A = Tm + (t - 1) * tstride + r0 * n + c;
    const double wt = w[t];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c < n && r0 + 8 * u < n) v[u] += wt * A[8 * u * n];
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t r = r0 + 8 * u;
    if (r >= n || c >= n) continue;
    if (Y) v[u] += alpha * Y[r * n + c];
    if (Bm2) v[u] -= Bm2[r * n + c];
    out[r * ldo + c] = v[u];
    tile[y0 + 8 * u][x] = v[u];
  }
  if (bi == bj) return;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t r = 32 * static_cast<int64_t>(bj) + y0 + 8 * u, cc = 32 * static_cast<int64_t>(bi) + x;
    if (r < n && cc < n) out[r * ldo + cc] = tile[x][y0 + 8 * u];
  }
}

// Frobenius products <G, T_t> of symmetric matrices, t = 0 .. nt - 1: kDotTerms
// of t >= 1 per blockIdx.y, and t = 0 (T_0 = I: the trace of G) with the first of
// them. From the upper triangles: the diagonal's halves and the strict upper
// part, doubled at the end. Bound by the FP64 pipe, one operation per upper
// element and t (n = 2048, nt = 15: 51 us of it; 120 us over the full matrices
// with a read of G for every t, 85 now). The last block sums the blocks'
// parts in a fixed order.
constexpr int kDotTerms = 7;

__global__ void __launch_bounds__(256)
foe_dots_kernel(const double* G, const double* T, int64_t tstride, int nt, int64_t n,
                double* partials, double* out, FoeScalars* sc) {
  chain_wait();
  chain_next();
  __shared__ double red[8][8];
  __shared__ double tot[8];
  __shared__ bool last;
  const int t0 = 1 + kDotTerms * blockIdx.y;
  const int cnt = min(kDotTerms, nt - t0);
  double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  const double* base = T + (t0 - 1) * tstride;  // T_t0
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
    for (int64_t j = i + threadIdx.x; j < n; j += blockDim.x) {
      const int64_t at = i * n + j;
      double g = G[at];
      double a[kDotTerms];
#pragma unroll
      for (int u = 0; u < kDotTerms; ++u)
        if (u < cnt) a[u] = base[u * tstride + at];
      if (j == i) {
        g *= 0.5;
        acc[kDotTerms] += g;
      }
#pragma unroll
      for (int u = 0; u < kDotTerms; ++u)
        if (u < cnt) acc[u] += g * a[u];
    }
  }
  block_totals<8>(acc, red, tot);
  double* part = partials + static_cast<int64_t>(blockIdx.x) * nt;
  if (static_cast<int>(threadIdx.x) < cnt) part[t0 + threadIdx.x] = tot[threadIdx.x];
  if (blockIdx.y == 0 && threadIdx.x == kDotTerms) part[0] = tot[kDotTerms];
  __threadfence();  // the partials before the count
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&sc->ticket, 1) == static_cast<int>(gridDim.x * gridDim.y) - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();  // every block's partials before the reads
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t = w; t < nt; t += 8) {
    double v = 0.0;
    for (int b = lane; b < static_cast<int>(gridDim.x); b += 32)
      v += __ldcg(partials + static_cast<int64_t>(b) * nt + t);
    v = warp_sum(v);
    if (lane == 0) out[t] = 2.0 * v;
  }
  if (threadIdx.x == 0) sc->ticket = 0;
}

// tr T_k for every k < M from tr T_0 = n, the baby-step traces (k < q) and the
// Frobenius products ip[m q + j] = <T_{qm}, T_j> (j = 0: tr T_{qm}):
// tr T_{qm+j} = 2 ip[m q + j] - tr T_{qm-j}. One CTA; a block m needs block m - 1.
__global__ void __launch_bounds__(128)
foe_ps_traces_kernel(double* traces, const double* ip, int q, int M, int64_t n) {
  chain_wait();
  chain_next();
  if (threadIdx.x == 0) traces[0] = static_cast<double>(n);
  __syncthreads();
  for (int m = 1; q * m < M; ++m) {
    for (int j = threadIdx.x; j < q && q * m + j < M; j += blockDim.x)
      traces[q * m + j] = j == 0 ? ip[m * q] : 2.0 * ip[m * q + j] - traces[q * m - j];
    __syncthreads();
  }
}

// The weights w[m][j] of B_m = sum_{j<q} w[m][j] T_j, P = sum_{m<r} T_m(y) B_m:
// a_k = c_k (a_0 = c_0 / 2, zero past M), folded from the top block down
// (T_{qm+j} = 2 T_m(y) T_j - T_{qm-j}). One CTA; a holds r q doubles.
__global__ void __launch_bounds__(128)
foe_fold_kernel(const double* coeffs, int M, int q, int r, double* a, double* w) {
  chain_wait();
  chain_next();
  for (int k = threadIdx.x; k < r * q; k += blockDim.x) a[k] = k == 0 ? 0.5 * coeffs[0] : (k < M ? coeffs[k] : 0.0);
  __syncthreads();
  for (int m = r - 1; m > 0; --m) {
    for (int j = threadIdx.x; j < q; j += blockDim.x) {
      const double d = a[q * m + j];
      w[m * q + j] = j == 0 ? d : 2.0 * d;
      if (j > 0) a[q * m - j] -= d;
    }
    __syncthreads();
  }
  for (int j = threadIdx.x; j < q; j += blockDim.x) w[j] = a[j];
}

// 32 x 32 blocks on and above the diagonal
int upper_blocks(int64_t n, int& T) {
  T = static_cast<int>((n + 31) / 32);
  return T * (T + 1) / 2;
}

}  // namespace

cudaError_t launch_foe_scale(const PurifyState* state, double e_min, double e_max, int use_given, FoeScalars* sc,
                             cudaStream_t st) {
  ProfScope prof(DMP_PROF_INIT, st);
  foe_scale_kernel<<<1, 1, 0, st>>>(state, e_min, e_max, use_given, sc);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_foe_coefficients(FoeScalars* sc, double kT, double mu, double n_occ, const double* traces, int M,
                                    double* w, double* gx, double* coeffs, cudaStream_t st) {
  ProfScope prof(DMP_PROF_INIT, st);
  const int64_t N = 2 * static_cast<int64_t>(M);
  const int canonical = traces != nullptr;
  const int rounds = canonical ? (kMuHalvings + kMuLevels - 1) / kMuLevels : 0;
  MuRound* ws = reinterpret_cast<MuRound*>(coeffs);  // written by the last kernel only
  if (canonical) {
    launch_chained(foe_weights_kernel, static_cast<unsigned>(N), kSumThreads, st, sc, traces, M, w, gx);
    for (int r = 0; r < rounds; ++r)
      launch_chained(foe_mu_round_kernel, kMuNodes, kSumThreads, st, sc, kT, n_occ, M, w, gx, r, ws);
    count_launch(1 + rounds);
  }
  launch_chained(foe_occupation_kernel, static_cast<unsigned>((N + kSumThreads - 1) / kSumThreads), kSumThreads, st,
      sc, kT, mu, n_occ, rounds, M, ws, gx, gx);
  launch_chained(foe_coeff_kernel, static_cast<unsigned>(M), kSumThreads, st, gx, M, coeffs);
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_foe_init(const double* H, int64_t ldh, int64_t n, const FoeScalars* sc, const double* coeffs,
                            double* Hs, double* T0, double* T1, double* P, int64_t ldp, cudaStream_t st) {
  ProfScope prof(DMP_PROF_OTHER, st);
  int T;
  const int blocks = upper_blocks(n, T);
  launch_chained(foe_init_kernel, blocks, 256, st, H, ldh, n, sc, coeffs, Hs, T0, T1, P, ldp, T);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_foe_combine(const double* T, int nt, const double* w, const double* Y, double alpha,
                               const double* Bm2, double* out, int64_t ldo, int64_t n, cudaStream_t st) {
  ProfScope prof(DMP_PROF_OTHER, st);
  int blocks_T;
  const int blocks = upper_blocks(n, blocks_T);
  launch_chained(foe_combine_kernel, blocks, 256, st, T, n * n, nt, w, Y, alpha, Bm2, out, ldo, n, blocks_T);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_foe_dots(const double* G, const double* T, int nt, int64_t n, double* partials, double* out,
                            FoeScalars* sc, cudaStream_t st) {
  if (nt < 1) return cudaSuccess;
  ProfScope prof(DMP_PROF_MEASURE, st);
  const dim3 grid(kFoeDotBlocks, static_cast<unsigned>(std::max(1, (nt - 1 + kDotTerms - 1) / kDotTerms)));
  launch_chained(foe_dots_kernel, grid, 256, st, G, T, n * n, nt, n, partials, out, sc);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_foe_ps_traces(double* traces, const double* ip, int q, int M, int64_t n, cudaStream_t st) {
  ProfScope prof(DMP_PROF_MEASURE, st);
  launch_chained(foe_ps_traces_kernel, 1, 128, st, traces, ip, q, M, n);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_foe_fold(const double* coeffs, int M, int q, int r, double* a, double* w, cudaStream_t st) {
  ProfScope prof(DMP_PROF_INIT, st);
  launch_chained(foe_fold_kernel, 1, 128, st, coeffs, M, q, r, a, w);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_foe_trace(const double* A, int64_t lda, int64_t n, double* out, cudaStream_t st) {
  ProfScope prof(DMP_PROF_MEASURE, st);
  launch_chained(foe_trace_kernel, 1, kReduceThreads, st, A, lda, 0, n, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_foe_traces(const double* T, int count, int64_t n, double* out, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  ProfScope prof(DMP_PROF_MEASURE, st);
  launch_chained(foe_trace_kernel, static_cast<unsigned>(count), kReduceThreads, st, T, n, n * n, n, out);
  count_launch();
  return cudaGetLastError();
}

}  // namespace dmp
