// Initial guess, per-iterate measures and the stopping rules of canonical
// purification (the Palser-Manolopoulos method cited in Sec. "Introduction";
// halt rules of Sec. "Implementation Details"). All in float64.
//
// Symmetry: only the upper triangle of H is read (element (i, j) is taken as
// H[min(i,j)][max(i,j)]), so P_0 and every iterate are exactly symmetric. The
// measures of an iterate use that symmetry too: each reduction reads the upper
// triangle and doubles the strictly-upper part.
//
// Reductions are deterministic: fixed grid, fixed per-thread order, fixed tree.
//
// Also here: the elementwise SP2 step and TRS4 factor, the refinement weights
// and energy, and the FP32-storage rounding of every matrix these kernels
// store (stored_value, DMP_FLAG_FP32_STORAGE).

#include <algorithm>

#include "dmp_internal.cuh"

namespace dmp {

namespace {

constexpr int kRowThreads = 256;
constexpr int kColChunks = 32;

// Strictly-upper row sums U_i = sum_{j>i} |H_ij| and the diagonal, one CTA per row.
__global__ void __launch_bounds__(kRowThreads)
gersh_rows_kernel(const double* __restrict__ H, int64_t n, int64_t ldh, double* __restrict__ U,
                  double* __restrict__ D, int* __restrict__ flag) {
  const int64_t i = blockIdx.x;
  __shared__ double red[kRowThreads / 32];
  double sacc = 0.0;
  bool bad = false;
  const double* row = H + i * ldh;
  for (int64_t j = i + 1 + threadIdx.x; j < n; j += kRowThreads) {
    const double v = row[j];
    bad |= !isfinite(v);
    sacc += fabs(v);
  }
  sacc = warp_sum(sacc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sacc;
  if (bad) atomicExch(flag, 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kRowThreads / 32; ++w) t += red[w];
    U[i] = t;
    const double d = row[i];
    if (!isfinite(d)) atomicExch(flag, 1);
    D[i] = d;
  }
}

// Column partial sums of the strict upper triangle: Cp[chunk][c] = sum over rows
// r < c of the chunk of |H_rc|. Threads own columns, so reads are coalesced.
__global__ void gersh_cols_kernel(const double* __restrict__ H, int64_t n, int64_t ldh,
                                  double* __restrict__ Cp) {
  const int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int chunk = blockIdx.y;
  if (c >= n) return;
  const int64_t rows_per = (n + kColChunks - 1) / kColChunks;
  const int64_t r0 = chunk * rows_per;
  const int64_t r1 = min(r0 + rows_per, c);
  double sacc = 0.0;
  for (int64_t r = r0; r < r1; ++r) sacc += fabs(H[r * ldh + c]);
  Cp[static_cast<int64_t>(chunk) * n + c] = sacc;
}

// Bounds, mu, lambda -> state. One CTA.
__global__ void __launch_bounds__(1024)
gersh_final_kernel(int64_t n, int64_t n_occ, const double* __restrict__ U, const double* __restrict__ D,
                   const double* __restrict__ Cp, PurifyState* st, const int* flag) {
  __shared__ double s_lo[1024], s_hi[1024], s_tr[1024];
  __shared__ int s_ilo[1024], s_ihi[1024];
  const int t = threadIdx.x;
  double lo = 1.0 / 0.0, hi = -1.0 / 0.0, tr = 0.0;
  int ilo = 0x7fffffff, ihi = 0x7fffffff;
  for (int64_t i = t; i < n; i += blockDim.x) {
    double rad = U[i];
    for (int ch = 0; ch < kColChunks; ++ch) rad += Cp[static_cast<int64_t>(ch) * n + i];
    const double l = D[i] - rad, h = D[i] + rad;
    if (l < lo) { lo = l; ilo = static_cast<int>(i); }
    if (h > hi) { hi = h; ihi = static_cast<int>(i); }
    tr += D[i];
  }
  s_lo[t] = lo; s_hi[t] = hi; s_tr[t] = tr; s_ilo[t] = ilo; s_ihi[t] = ihi;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (t < o) {
      // keep the first index on ties
      if (s_lo[t + o] < s_lo[t] || (s_lo[t + o] == s_lo[t] && s_ilo[t + o] < s_ilo[t])) {
        s_lo[t] = s_lo[t + o];
        s_ilo[t] = s_ilo[t + o];
      }
      if (s_hi[t + o] > s_hi[t] || (s_hi[t + o] == s_hi[t] && s_ihi[t + o] < s_ihi[t])) {
        s_hi[t] = s_hi[t + o];
        s_ihi[t] = s_ihi[t + o];
      }
      s_tr[t] += s_tr[t + o];
    }
    __syncthreads();
  }
  if (t == 0) {
    const double dn = static_cast<double>(n);
    const double mu = s_tr[0] / dn;
    st->h_min = s_lo[0];
    st->h_max = s_hi[0];
    st->row_min = s_ilo[0];
    st->row_max = s_ihi[0];
    st->mu = mu;
    if (*flag) {
      st->nonfinite = 1;
      st->status = DMP_ERR_NONFINITE;
      st->done = 1;
      st->lam = 0.0;
      return;
    }
    if (!(s_hi[0] > mu && mu > s_lo[0])) {  // H is a multiple of the identity
      st->status = DMP_ERR_INVALID_ARG;
      st->done = 1;
      st->lam = 0.0;
      return;
    }
    st->n_occ_d = static_cast<double>(n_occ);
    const double lam1 = static_cast<double>(n_occ) / (s_hi[0] - mu);
    const double lam2 = static_cast<double>(n - n_occ) / (mu - s_lo[0]);
    st->lam_branch = lam1 <= lam2 ? 1 : 2;
    st->lam = lam1 <= lam2 ? lam1 : lam2;
  }
}

// P0 = (lambda/n)(mu I - H) + (n_occ/n) I on 32 x 32 upper tiles, mirrored.
__global__ void p0_kernel(const double* __restrict__ H, int64_t n, int64_t ldh, int64_t n_occ,
                          const PurifyState* st, double* __restrict__ P, int64_t ldp, int T) {
  __shared__ double tile[32][33];
  int bi, bj;
  upper_tile(blockIdx.x, T, bi, bj);
  const double dn = static_cast<double>(n);
  const double a = st->lam / dn, mu = st->mu, occ = static_cast<double>(n_occ) / dn;
  // SP2 / TRS4: X_0 = (h_max I - H) / (h_max - h_min)
  const bool var = st->method != DMP_METHOD_PM;
  const bool r32 = st->store32 != 0;
  const double hmax = st->h_max, width = st->h_max - st->h_min;
  const int64_t r0 = static_cast<int64_t>(bi) * 32, c0 = static_cast<int64_t>(bj) * 32;
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int64_t r = r0 + y, c = c0 + threadIdx.x;
    if (r < n && c < n) tile[y][threadIdx.x] = H[r * ldh + c];
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int x = threadIdx.x;
    const int64_t r = r0 + y, c = c0 + x;
    if (r < n && c < n) {
      double v;
      if (bi == bj) {
        // on the diagonal tile the lower half takes the mirror of the upper half
        const double h = (y <= x) ? tile[y][x] : tile[x][y];
        if (var) {
          v = (r == c) ? (hmax - h) / width : -h / width;
        } else {
          v = (r == c) ? a * (mu - h) + occ : -a * h;
        }
      } else {
        v = var ? -tile[y][x] / width : -a * tile[y][x];
      }
      P[r * ldp + c] = stored_value(v, r32);
    }
  }
  if (bi != bj) {
    for (int y = threadIdx.y; y < 32; y += blockDim.y) {
      // write the transposed tile: P[c0 + y][r0 + x] = -a H[r0 + x][c0 + y]
      const int64_t r = c0 + y, c = r0 + threadIdx.x;
      if (r < n && c < n)
        P[r * ldp + c] = stored_value(var ? -tile[threadIdx.x][y] / width : -a * tile[threadIdx.x][y], r32);
    }
  }
}

// Per-block partial measures of the iterate over the upper triangle: rows
// i = blockIdx.x + k * gridDim.x.
//   0: sum P_ii      1: sum X2_ii
//   2: diag P X2     3: upper P X2
//   4: diag (X2-P)^2 5: upper (X2-P)^2
//   6: diag P H      7: upper P H
//   8: diag X2^2      9: upper X2^2      (NQ = 10: SP2 / TRS4)
//
// The last block to finish sums the partials in a fixed order (thread t the
// blocks t, t + 256, ..; warp trees; the eight warps in order) and applies the
// stopping rules: NQ = 8 canonical purification (pm_decide), NQ = 10 SP2 / TRS4
// (variant_decide). At large sizes bound by the FP64 pipe, four operations per
// upper element (n = 8192: 0.30 ms, 0.22 ms for the operations alone); at small
// ones by the block sums: an add takes the pipe as long for one lane as for 32,
// so warp_sums adds 6 times for the sums that every thread has a part of, and
// those that only thread 0 has are not summed at all (n = 256: 31 us for two
// kernels before, 12.7 with all ten summed by 9 adds a warp, 11.4 now; n = 999,
// SP2 / TRS4: 30 to 24).
template <int NQ>
__global__ void __launch_bounds__(256)
measure_kernel(const double* P, int64_t ldp, const double* X2, int64_t ldx,
               const double* H, int64_t ldh, int64_t n, double* part, PurifyState* st) {
  chain_wait();
  chain_next();
  if (st->done) return;
  bool four = false;
  double d_xx = 0.0, a_xx[4] = {0.0, 0.0, 0.0, 0.0};
  // four independent accumulator sets (entries j, j + 256, j + 512, j + 768 of
  // a step) keep twelve loads in flight per thread; combined in order below
  double a_px[4] = {0.0, 0.0, 0.0, 0.0}, a_id[4] = {0.0, 0.0, 0.0, 0.0}, a_ph[4] = {0.0, 0.0, 0.0, 0.0};
  double d_p = 0.0, d_x = 0.0, d_px = 0.0, d_id = 0.0, d_ph = 0.0;
  const int64_t B = blockDim.x;
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
    const double* pr = P + i * ldp;
    const double* xr = X2 + i * ldx;
    const double* hr = H + i * ldh;
    if (threadIdx.x == 0) {
      const double p = pr[i], x = xr[i], h = hr[i];
      d_p += p;
      d_x += x;
      d_px += p * x;
      d_id += (x - p) * (x - p);
      d_ph += p * h;
      if (NQ == 10) d_xx += x * x;
    }
    int64_t j = i + 1 + threadIdx.x;
    for (; j + 3 * B < n; j += 4 * B) {
      four = true;
      double p[4], x[4], h[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        p[u] = pr[j + u * B];
        x[u] = xr[j + u * B];
        h[u] = hr[j + u * B];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a_px[u] += p[u] * x[u];
        a_id[u] += (x[u] - p[u]) * (x[u] - p[u]);
        a_ph[u] += p[u] * h[u];
        if (NQ == 10) a_xx[u] += x[u] * x[u];
      }
    }
    for (; j < n; j += B) {
      const double p = pr[j], x = xr[j], h = hr[j];
      a_px[0] += p * x;
      a_id[0] += (x - p) * (x - p);
      a_ph[0] += p * h;
      if (NQ == 10) a_xx[0] += x * x;
    }
  }
  // the block's sums: the diagonal's from thread 0, which alone has any (the adds
  // of zeros to them are left out; + 0.0 is what is left of them), and three or
  // four from every thread. Sets that stayed zero in the whole warp are not added.
  double u[4] = {a_px[0], a_id[0], a_ph[0], a_xx[0]};
  if (__any_sync(0xffffffffu, four)) {
    u[0] = (a_px[0] + a_px[1]) + (a_px[2] + a_px[3]);
    u[1] = (a_id[0] + a_id[1]) + (a_id[2] + a_id[3]);
    u[2] = (a_ph[0] + a_ph[1]) + (a_ph[2] + a_ph[3]);
    u[3] = (a_xx[0] + a_xx[1]) + (a_xx[2] + a_xx[3]);
  }
  __shared__ double red[8][NQ];
  __shared__ double tot[NQ];
  __shared__ bool last;
  double* mine = part + static_cast<int64_t>(blockIdx.x) * NQ;
  const double c = warp_sums<4>(u);
  if ((threadIdx.x & 7) == 0) red[threadIdx.x >> 5][(threadIdx.x >> 3) & 3] = c;
  if (threadIdx.x == 0) {
    mine[0] = d_p + 0.0;
    mine[1] = d_x + 0.0;
    mine[2] = d_px + 0.0;
    mine[4] = d_id + 0.0;
    mine[6] = d_ph + 0.0;
    if (NQ == 10) mine[NQ - 2] = d_xx + 0.0;
  }
  __syncthreads();
  if (threadIdx.x < (NQ - 2) / 2) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
    mine[3 + 2 * threadIdx.x] = t;
  }
  __threadfence();  // the partials before the count
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();  // every block's partials before the reads
  double v[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q)
    v[q] = threadIdx.x < gridDim.x ? __ldcg(part + static_cast<int64_t>(threadIdx.x) * NQ + q) : 0.0;
  for (int b = threadIdx.x + blockDim.x; b < static_cast<int>(gridDim.x); b += blockDim.x) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] += __ldcg(part + static_cast<int64_t>(b) * NQ + q);
  }
  block_totals<NQ>(v, red, tot);
  if (threadIdx.x == 0) {
    st->ticket = 0;
    if (NQ == 8) {
      pm_decide(st, tot);
    } else {
      variant_decide(st, tot);
      st->no_product = st->done != 0 || st->step_kind == 0;
    }
  }
}

// The elementwise half of an SP2 / TRS4 step, enqueued before the host knows the
// step's kind: X <- alpha X + b2 X2 in place (kind 0), or the TRS4 factor
// Z = zd I + zx X + zx2 X2 of F + gamma G = X2 Z (kind 1), over the full n x n. A
// block holds up to 1024 entries of a row, four per thread, whose loads do not
// wait for one another (n = 999: 11 us; 20 with a loop over rows and entries, and
// 4 more for a second kernel that finds that the step is of the other kind).
constexpr int kElemCols = 1024;

dim3 elem_grid(int64_t n) {
  return dim3(static_cast<unsigned>((n + kElemCols - 1) / kElemCols), static_cast<unsigned>(std::min<int64_t>(n, 65535)));
}

__global__ void __launch_bounds__(256)
variant_step_kernel(double* X, int64_t ldx, const double* X2, int64_t ldx2, double* Z, int64_t ldz, int64_t n,
                    const PurifyState* st) {
  chain_wait();
  chain_next();
  if (st->done != 0) return;
  const bool product = st->step_kind != 0;
  const double a = product ? st->zx : st->alpha, b = product ? st->zx2 : st->b2, d = st->zd;
  double* out = product ? Z : X;
  const int64_t ldo = product ? ldz : ldx;
  const bool r32 = st->store32 != 0;
  const int64_t j0 = static_cast<int64_t>(blockIdx.x) * kElemCols + threadIdx.x;
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
    double x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t j = j0 + 256 * u;
      x[u] = j < n ? X[i * ldx + j] : 0.0;
      y[u] = j < n ? X2[i * ldx2 + j] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t j = j0 + 256 * u;
      double v = a * x[u] + b * y[u];
      if (product && j == i) v += d;
      if (j < n) out[i * ldo + j] = stored_value(v, r32);
    }
  }
}

// The update weights of a McWeeny step (c = 1/2): alpha = 0, b2 = 3, b3 = -2.
__global__ void refine_weights_kernel(PurifyState* st) {
  st->alpha = 0.0;
  st->b2 = 3.0;
  st->b3 = -2.0;
}

// Per-block partial sums of tr(P H) over the upper triangle: [0] diagonal, [1] strictly upper.
__global__ void __launch_bounds__(256)
energy_kernel(const double* __restrict__ P, int64_t ldp, const double* __restrict__ H, int64_t ldh, int64_t n,
              double* __restrict__ part) {
  double d = 0.0, u = 0.0;
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
    const double* pr = P + i * ldp;
    const double* hr = H + i * ldh;
    if (threadIdx.x == 0) d += pr[i] * hr[i];
    for (int64_t j = i + 1 + threadIdx.x; j < n; j += blockDim.x) u += pr[j] * hr[j];
  }
  d = warp_sum(d);
  u = warp_sum(u);
  __shared__ double red[8][2];
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = d;
    red[threadIdx.x >> 5][1] = u;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
    part[static_cast<int64_t>(blockIdx.x) * 2 + threadIdx.x] = t;
  }
}

__global__ void __launch_bounds__(256)
energy_final_kernel(const double* __restrict__ part, int nblocks, PurifyState* st) {
  double d = 0.0, u = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    d += part[2 * b];
    u += part[2 * b + 1];
  }
  d = warp_sum(d);
  u = warp_sum(u);
  __shared__ double red[8][2];
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = d;
    red[threadIdx.x >> 5][1] = u;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double td = 0.0, tu = 0.0;
    for (int w = 0; w < 8; ++w) {
      td += red[w][0];
      tu += red[w][1];
    }
    st->energy_refined = td + 2.0 * tu;
  }
}

// Blocks past the last row would add zeros only.
unsigned measure_blocks(int64_t n) { return static_cast<unsigned>(std::min<int64_t>(n, kMeasureBlocks)); }

}  // namespace

cudaError_t launch_measure_variant(const double* X, int64_t ldx, const double* X2, int64_t ldx2, const double* H,
                                   int64_t ldh, int64_t n, double* partials, PurifyState* state, cudaStream_t st) {
  ProfScope prof(DMP_PROF_MEASURE, st);
  launch_chained(measure_kernel<10>, measure_blocks(n), 256, st, X, ldx, X2, ldx2, H, ldh, n, partials, state);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_variant_step(double* X, int64_t ldx, const double* X2, int64_t ldx2, double* Z, int64_t ldz,
                                int64_t n, const PurifyState* state, cudaStream_t st) {
  ProfScope prof(DMP_PROF_OTHER, st);
  launch_chained(variant_step_kernel, elem_grid(n), 256, st, X, ldx, X2, ldx2, Z, ldz, n, state);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_refine_weights(PurifyState* state, cudaStream_t st) {
  ProfScope prof(DMP_PROF_OTHER, st);
  refine_weights_kernel<<<1, 1, 0, st>>>(state);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_energy(const double* P, int64_t ldp, const double* H, int64_t ldh, int64_t n, double* partials,
                          PurifyState* state, cudaStream_t st) {
  ProfScope prof(DMP_PROF_MEASURE, st);
  energy_kernel<<<kMeasureBlocks, 256, 0, st>>>(P, ldp, H, ldh, n, partials);
  energy_final_kernel<<<1, 256, 0, st>>>(partials, kMeasureBlocks, state);
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_gershgorin_init(const double* H, int64_t n, int64_t ldh, int64_t n_occ,
                                   double* rowbuf, PurifyState* state, double* P, int64_t ldp,
                                   cudaStream_t st) {
  double* U = rowbuf;
  double* D = rowbuf + n;
  double* Cp = rowbuf + 2 * n;
  int* flag = reinterpret_cast<int*>(rowbuf + 2 * n + static_cast<int64_t>(kColChunks) * n);
  cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  ProfScope prof(DMP_PROF_INIT, st);
  gersh_rows_kernel<<<static_cast<unsigned>(n), kRowThreads, 0, st>>>(H, n, ldh, U, D, flag);
  dim3 cg(static_cast<unsigned>((n + 127) / 128), kColChunks);
  gersh_cols_kernel<<<cg, 128, 0, st>>>(H, n, ldh, Cp);
  gersh_final_kernel<<<1, 1024, 0, st>>>(n, n_occ, U, D, Cp, state, flag);
  const int T = static_cast<int>((n + 31) / 32);
  p0_kernel<<<T * (T + 1) / 2, dim3(32, 8), 0, st>>>(H, n, ldh, n_occ, state, P, ldp, T);
  count_launch(4);
  return cudaGetLastError();
}

size_t gershgorin_rowbuf_bytes(int64_t n) {
  return static_cast<size_t>((2 + kColChunks) * n + 1) * sizeof(double);
}

cudaError_t launch_measure(const double* P, int64_t ldp, const double* X2, int64_t ldx,
                           const double* H, int64_t ldh, int64_t n, double* partials,
                           PurifyState* state, cudaStream_t st) {
  ProfScope prof(DMP_PROF_MEASURE, st);
  launch_chained(measure_kernel<8>, measure_blocks(n), 256, st, P, ldp, X2, ldx, H, ldh, n, partials, state);
  count_launch();
  return cudaGetLastError();
}

}  // namespace dmp
