// Reverse mode through canonical purification: the elementwise and reduction
// kernels of dm_purify_backward. The products run on the same executors as the
// forward.
//
// Step k (c frozen at its forward value, branch frozen; the dependence of c on
// P kept), all matrices symmetric except Y:
//   Y = G P,  X2 = P^2,  V = (Y + Y^T / 2) P
//   g = alpha G + b2 (Y + Y^T) + b3 (V + V^T) + (dL/dc) dc/dP
//   dL/dc = alpha' <G, P> + b2' <G, X2> + b3' <Y, X2>     (<G, P^3> = <G P, P^2>)
//   dc/dP = ((2 P - 3 X2) t_d - t_n (I - 2 P)) / t_d^2,  t_d = tr(P - X2), t_n = c t_d
// and the new G is the symmetric part of g (the loss sees P only through
// symmetric matrices, so the symmetric part carries every directional
// derivative along symmetric perturbations).
//
// V + V^T = G P^2 + P G P + P^2 G with G and P symmetric: one general product in
// the place of G P^2 and P G P. The result moves by 1 to 2 % of the products' own
// error (which the forward's exceeds by far: the gradient's error stays the same
// to three digits): with 42 digit bits and more by less than 1e-9 of the gradient.
// With fewer (INT8 and BF16 below 6 slices, E4M3 below 9) the two products, and
// the order of the sums, stay as they are defined: a last-bit difference moves
// digits there (E4M3 s = 7, n = 1500: the merged product moves the gradient by
// 1.4e-8, s = 8 by 5e-10).
//
// Initial guess P_0 = (lambda/n)(mu I - H) + (n_occ/n) I, with mu = tr(H)/n
// and lambda = min(n_occ/(h_max - mu), (n - n_occ)/(mu - h_min)) from the
// Gershgorin bounds, whose extreme rows a (max) and b (min) enter through
// h = H_aa + sum_j |H_aj| (and the same with a minus sign for b).

#include "dmp_internal.cuh"

namespace dmp {

namespace {

// Weights of the frozen step at c, their c-derivatives and dL/dc.
__device__ void step_scalars(const double* s, double c, AdjScalars* out) {
  double a, b2, b3, da, db2, db3;
  if (c >= 0.5) {
    a = 0.0;
    b2 = (1.0 + c) / c;
    b3 = -1.0 / c;
    da = 0.0;
    db2 = -1.0 / (c * c);
    db3 = 1.0 / (c * c);
  } else {
    const double d = 1.0 - c;
    a = (1.0 - 2.0 * c) / d;
    b2 = (1.0 + c) / d;
    b3 = -1.0 / d;
    da = -1.0 / (d * d);
    db2 = 2.0 / (d * d);
    db3 = -1.0 / (d * d);
  }
  const double td = s[0] - s[1];
  out->alpha = a;
  out->b2 = b2;
  out->b3 = b3;
  out->td = td;
  out->tn = c * td;
  out->dLdc = da * s[2] + db2 * s[3] + db3 * s[4];
}

// True in the block that finishes last, with the sums over all blocks of the NQ
// partials of each in s (8 warps: warp q sums quantity q; fixed order). One
// thread adding them block by block waited for one memory latency per block.
template <int NQ>
__device__ __forceinline__ bool last_block_sums(double* part, int32_t* ticket, double* s) {
  __shared__ bool last;
  __threadfence();  // the partials before the count
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();  // every block's partials before the reads
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q < NQ) {
    double v = 0.0;
    for (int b = lane; b < static_cast<int>(gridDim.x); b += 32) v += __ldcg(part + static_cast<int64_t>(b) * NQ + q);
    v = warp_sum(v);
    if (lane == 0) s[q] = v;
  }
  if (threadIdx.x == 0) *ticket = 0;
  __syncthreads();
  return true;
}

// Sums over all elements:
//   0: tr P   1: tr X2   2: <G, P>   3: <G, X2>   4: <Y, X2>
// and, in the last block, the step's scalars from them. Four elements of each
// matrix in flight per thread; n = 1024: 5 us of the FP64 pipe, 20 in all (27 with
// one element in flight, 63 with a single thread's final sums in their own kernel).
__global__ void __launch_bounds__(256)
adj_reduce_kernel(const double* P, const double* X2, const double* G,
                  const double* Y, int64_t n, double* part, int32_t* ticket, double c,
                  AdjScalars* out) {
  chain_wait();
  chain_next();
  __shared__ double red[8][8];
  __shared__ double tot[8];
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t first = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  for (int64_t i = first; i < n; i += step) {
    v[0] += P[i * n + i];
    v[1] += X2[i * n + i];
  }
  for (int64_t i = first; i < n * n; i += 4 * step) {
    double p[4], x[4], g[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t at = i + u * step;
      const bool in = at < n * n;
      p[u] = in ? P[at] : 0.0;
      x[u] = in ? X2[at] : 0.0;
      g[u] = in ? G[at] : 0.0;
      y[u] = in ? Y[at] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[2] += g[u] * p[u];
      v[3] += g[u] * x[u];
      v[4] += y[u] * x[u];
    }
  }
  block_totals<8>(v, red, tot);
  if (threadIdx.x < 5) part[static_cast<int64_t>(blockIdx.x) * 5 + threadIdx.x] = tot[threadIdx.x];
  if (last_block_sums<5>(part, ticket, tot) && threadIdx.x == 0) step_scalars(tot, c, out);
}

// W = Y + Y^T / 2, 32 x 32 block pairs (upper_tile), transposed through shared memory.
__global__ void __launch_bounds__(256)
adj_half_kernel(const double* Y, int64_t n, double* W, int T) {
  chain_wait();
  chain_next();
  __shared__ double a[32][33], b[32][33];
  int bi, bj;
  upper_tile(blockIdx.x, T, bi, bj);
  const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
  const int64_t i0 = 32 * static_cast<int64_t>(bi), j0 = 32 * static_cast<int64_t>(bj);
#pragma unroll
  for (int y = y0; y < 32; y += 8) {
    if (i0 + y < n && j0 + x < n) a[y][x] = Y[(i0 + y) * n + j0 + x];
    if (j0 + y < n && i0 + x < n) b[y][x] = Y[(j0 + y) * n + i0 + x];
  }
  __syncthreads();
#pragma unroll
  for (int y = y0; y < 32; y += 8) {
    if (i0 + y < n && j0 + x < n) W[(i0 + y) * n + j0 + x] = a[y][x] + 0.5 * b[x][y];
    if (bi != bj && j0 + y < n && i0 + x < n) W[(j0 + y) * n + i0 + x] = b[y][x] + 0.5 * a[x][y];
  }
}

// G_new = sym(g), both blocks of a 32 x 32 block pair per CTA: Y and V are read
// and G_new written along rows on both sides of the diagonal (a thread per
// element pair read and wrote the lower side with a stride of n). (dL/dc) dc/dP
// is cp P + cx X2 + ci I. n = 1024: 20 us.
__global__ void __launch_bounds__(256)
adj_step_kernel(const double* G, const double* Y, const double* V,
                const double* P, const double* X2, int64_t n,
                const AdjScalars* sc, double* Gn, int T) {
  chain_wait();
  chain_next();
  __shared__ double low[32][33];  // b2 Y + b3 V of the lower block, then G_new of the upper
  int bi, bj;
  upper_tile(blockIdx.x, T, bi, bj);
  const double a = sc->alpha, b2 = sc->b2, b3 = sc->b3;
  const double td = sc->td, tn = sc->tn, k = sc->dLdc / (td * td);
  const double cp = 2.0 * (td + tn) * k, cx = -3.0 * td * k, ci = -tn * k;
  const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
  const int64_t i0 = 32 * static_cast<int64_t>(bi), j0 = 32 * static_cast<int64_t>(bj);
#pragma unroll
  for (int y = y0; y < 32; y += 8) {
    if (j0 + y < n && i0 + x < n) {
      const int64_t ji = (j0 + y) * n + i0 + x;
      low[y][x] = __fma_rn(b3, V[ji], __dmul_rn(b2, Y[ji]));
    }
  }
  __syncthreads();
  double v[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t i = i0 + y0 + 8 * u, j = j0 + x;
    if (i >= n || j >= n) continue;
    const int64_t ij = i * n + j;
    // G, P, X2 are symmetric; Y and V are not
    const double dc = __fma_rn(cp, P[ij], cx * X2[ij]);
    // one rounding order for both elements of a pair: G_new is symmetric to the last bit
    const double yv = __dadd_rn(__fma_rn(b3, V[ij], __dmul_rn(b2, Y[ij])), low[x][y0 + 8 * u]);
    v[u] = __fma_rn(a, G[ij], __dadd_rn(yv, dc));
    if (i == j) v[u] += ci;
    Gn[ij] = v[u];
  }
  if (bi == bj) return;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) low[y0 + 8 * u][x] = v[u];
  __syncthreads();
#pragma unroll
  for (int y = y0; y < 32; y += 8)
    if (j0 + y < n && i0 + x < n) Gn[(j0 + y) * n + i0 + x] = low[x][y];
}

// ---- the step with the two products apart (YP = G P^2, ZP = P G P, Z = Y^T).
// With so few digits a last-bit difference in a step moves digits of the next
// one, and the gradient by more than 1e-9: the sums and the terms keep one order.

// Partial sums over all elements, rows i = blockIdx.x + k gridDim.x:
//   0: tr P   1: tr X2   2: <G, P>   3: <G, X2>   4: <Z, X2>
__global__ void __launch_bounds__(256)
adj_reduce_apart_kernel(const double* __restrict__ P, const double* __restrict__ X2, const double* __restrict__ G,
                  const double* __restrict__ Z, int64_t n, double* __restrict__ part) {
  double v[5] = {0, 0, 0, 0, 0};
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
    const int64_t o = i * n;
    if (threadIdx.x == 0) {
      v[0] += P[o + i];
      v[1] += X2[o + i];
    }
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
      const double p = P[o + j], x = X2[o + j];
      v[2] += G[o + j] * p;
      v[3] += G[o + j] * x;
      v[4] += Z[o + j] * x;
    }
  }
  __shared__ double red[8][5];
#pragma unroll
  for (int q = 0; q < 5; ++q) v[q] = warp_sum(v[q]);
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int q = 0; q < 5; ++q) red[threadIdx.x >> 5][q] = v[q];
  __syncthreads();
  if (threadIdx.x < 5) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
    part[static_cast<int64_t>(blockIdx.x) * 5 + threadIdx.x] = t;
  }
}

// The sums in block order, one thread each, and the step's scalars.
__global__ void adj_scalars_kernel(const double* __restrict__ part, int nblocks, double c,
                                   AdjScalars* __restrict__ out) {
  __shared__ double s[5];
  if (threadIdx.x < 5) {
    double t = 0.0;
#pragma unroll 8
    for (int b = 0; b < nblocks; ++b) t += part[static_cast<int64_t>(b) * 5 + threadIdx.x];
    s[threadIdx.x] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) step_scalars(s, c, out);
}

// G_new = sym(g), one thread per element pair on the upper triangle.
__global__ void adj_step_apart_kernel(const double* __restrict__ G, const double* __restrict__ Y,
                                const double* __restrict__ YP, const double* __restrict__ ZP,
                                const double* __restrict__ P, const double* __restrict__ X2, int64_t n,
                                const AdjScalars* __restrict__ sc, double* __restrict__ Gn) {
  const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t i = blockIdx.y;
  if (j < i || j >= n) return;
  const double a = sc->alpha, b2 = sc->b2, b3 = sc->b3;
  const double td = sc->td, tn = sc->tn, k = sc->dLdc / (td * td);
  const int64_t ij = i * n + j, ji = j * n + i;
  const double dij = (i == j) ? 1.0 : 0.0;
  // G, P, X2 are symmetric; Y, YP, ZP are not
  const double dc = ((2.0 * P[ij] - 3.0 * X2[ij]) * td - tn * (dij - 2.0 * P[ij])) * k;
  const double yy = Y[ij] + Y[ji];
  const double gij = a * G[ij] + b2 * yy + b3 * (YP[ij] + ZP[ij] + YP[ji]) + dc;
  const double gji = a * G[ij] + b2 * yy + b3 * (YP[ji] + ZP[ji] + YP[ij]) + dc;
  const double v = 0.5 * (gij + gji);
  Gn[ij] = v;
  Gn[ji] = v;
}

// Symmetric part of a general n x n matrix (leading dimension ld) into dense out.
__global__ void sym_part_kernel(const double* __restrict__ A, int64_t ld, int64_t n, double* __restrict__ out) {
  const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t i = blockIdx.y;
  if (j < i || j >= n) return;
  const double v = 0.5 * (A[i * ld + j] + A[j * ld + i]);
  out[i * n + j] = v;
  out[j * n + i] = v;
}

// Partial sums for the initial-guess adjoint: 0: tr G0, 1: <G0, H> (H read as
// its upper triangle mirrored, G0 symmetric).
__device__ void p0_scalars(const double* sums, P0Adjoint* s) {
  const double tr = sums[0], dg = sums[1], up = sums[2];
  const double n = s->n, lam = s->lam, mu = s->mu;
  const double G0H = dg + 2.0 * up;
  const double dLdlam = (mu * tr - G0H) / n;
  double dLdmu = (lam / n) * tr;
  double dhmax = 0.0, dhmin = 0.0;
  if (s->lam_branch == 1) {
    const double d = (s->h_max - mu) * (s->h_max - mu);
    dLdmu += dLdlam * s->n_occ / d;
    dhmax = -dLdlam * s->n_occ / d;
  } else {
    const double d = (mu - s->h_min) * (mu - s->h_min);
    dLdmu += -dLdlam * (n - s->n_occ) / d;
    dhmin = dLdlam * (n - s->n_occ) / d;
  }
  s->diag_add = dLdmu / n;
  s->dhmax = s->bounds_grad ? dhmax : 0.0;
  s->dhmin = s->bounds_grad ? dhmin : 0.0;
}

__global__ void __launch_bounds__(256)
p0_reduce_kernel(const double* __restrict__ G0, const double* __restrict__ H, int64_t ldh, int64_t n,
                 double* __restrict__ part, int32_t* ticket, P0Adjoint* s) {
  __shared__ double red[8][8];
  __shared__ double tot[8];
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // tr G0, the diagonal of <G0, H>, its upper triangle
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
    if (threadIdx.x == 0) {
      v[0] += G0[i * n + i];
      v[1] += G0[i * n + i] * H[i * ldh + i];
    }
    for (int64_t j = i + 1 + threadIdx.x; j < n; j += blockDim.x) v[2] += G0[i * n + j] * H[i * ldh + j];
  }
  block_totals<8>(v, red, tot);
  if (threadIdx.x < 3) part[static_cast<int64_t>(blockIdx.x) * 3 + threadIdx.x] = tot[threadIdx.x];
  if (last_block_sums<3>(part, ticket, tot) && threadIdx.x == 0) p0_scalars(tot, s);
}

// dL/dH (symmetric part): -(lambda/n) G0 + (dL/dmu / n) I + Gershgorin row terms.
__global__ void p0_adjoint_kernel(const double* __restrict__ G0, const double* __restrict__ H, int64_t ldh,
                                  int64_t n, const P0Adjoint* __restrict__ s, double* __restrict__ out,
                                  int64_t ldo) {
  const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t i = blockIdx.y;
  if (j < i || j >= n) return;
  const double a = s->lam / s->n;
  double v = -a * G0[i * n + j];
  const int64_t ra = s->row_max, rb = s->row_min;
  const double h = H[i * ldh + j];  // upper triangle, mirrored for (j, i)
  if (i == j) {
    v += s->diag_add;
    if (i == ra) v += s->dhmax;
    if (i == rb) v += s->dhmin;
  } else {
    // the extreme row's radius holds |H_ij| once: half of it on each mirror
    const double sg = (h > 0.0) ? 1.0 : (h < 0.0 ? -1.0 : 0.0);
    if (i == ra || j == ra) v += 0.5 * s->dhmax * sg;
    if (i == rb || j == rb) v -= 0.5 * s->dhmin * sg;
  }
  out[i * ldo + j] = v;
  out[j * ldo + i] = v;
}

}  // namespace

constexpr int kAdjBlocks = 304;

cudaError_t launch_adj_half(const double* Y, int64_t n, double* W, cudaStream_t st) {
  ProfScope prof(DMP_PROF_OTHER, st);
  const int T = static_cast<int>((n + 31) / 32);
  launch_chained(adj_half_kernel, T * (T + 1) / 2, 256, st, Y, n, W, T);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_adj_reduce(const double* P, const double* X2, const double* G, const double* Y, int64_t n,
                              double* part, int32_t* ticket, double c, AdjScalars* sc, cudaStream_t st) {
  ProfScope prof(DMP_PROF_MEASURE, st);
  launch_chained(adj_reduce_kernel, kAdjBlocks, 256, st, P, X2, G, Y, n, part, ticket, c, sc);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_adj_step(const double* G, const double* Y, const double* V, const double* P, const double* X2,
                            int64_t n, const AdjScalars* sc, double* Gn, cudaStream_t st) {
  ProfScope prof(DMP_PROF_OTHER, st);
  const int T = static_cast<int>((n + 31) / 32);
  launch_chained(adj_step_kernel, T * (T + 1) / 2, 256, st, G, Y, V, P, X2, n, sc, Gn, T);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_adj_apart(const double* G, const double* Y, const double* Z, const double* YP, const double* ZP,
                             const double* P, const double* X2, int64_t n, double* part, double c, AdjScalars* sc,
                             double* Gn, cudaStream_t st) {
  {
    ProfScope prof(DMP_PROF_MEASURE, st);
    adj_reduce_apart_kernel<<<kAdjBlocks, 256, 0, st>>>(P, X2, G, Z, n, part);
    adj_scalars_kernel<<<1, 32, 0, st>>>(part, kAdjBlocks, c, sc);
  }
  ProfScope prof(DMP_PROF_OTHER, st);
  dim3 grid(static_cast<unsigned>((n + 255) / 256), static_cast<unsigned>(n));
  adj_step_apart_kernel<<<grid, 256, 0, st>>>(G, Y, YP, ZP, P, X2, n, sc, Gn);
  count_launch(3);
  return cudaGetLastError();
}

cudaError_t launch_sym_part(const double* A, int64_t ld, int64_t n, double* out, cudaStream_t st) {
  ProfScope prof(DMP_PROF_OTHER, st);
  dim3 grid(static_cast<unsigned>((n + 255) / 256), static_cast<unsigned>(n));
  sym_part_kernel<<<grid, 256, 0, st>>>(A, ld, n, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_p0_adjoint(const double* G0, const double* H, int64_t ldh, int64_t n, double* part,
                              int32_t* ticket, P0Adjoint* s, double* out, int64_t ldo, cudaStream_t st) {
  ProfScope prof(DMP_PROF_INIT, st);
  p0_reduce_kernel<<<kAdjBlocks, 256, 0, st>>>(G0, H, ldh, n, part, ticket, s);
  dim3 grid(static_cast<unsigned>((n + 255) / 256), static_cast<unsigned>(n));
  p0_adjoint_kernel<<<grid, 256, 0, st>>>(G0, H, ldh, n, s, out, ldo);
  count_launch(2);
  return cudaGetLastError();
}

}  // namespace dmp
