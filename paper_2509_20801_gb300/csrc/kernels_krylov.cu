// FP64 complex kernels of the flexible GMRES outer iteration: classical
// Gram-Schmidt passes (multi-dot and multi-axpy fused with the norm of the
// result), the solution update x += Z y, norms and scaling.
//
// All reductions are deterministic: every block writes its partial sums to
// a fixed slot and a second kernel adds the slots in a fixed order.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace stdd {

namespace {

constexpr int TPB = 256;
constexpr int NBLK = 152 * 4;   // partial-sum blocks: 4 per SM
constexpr int GROUP = 8;        // vectors of a multi-dot block
constexpr int MAXM = 512;       // longest basis handled by the axpy kernels

template <typename T> __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// block-wide sum of one double; result valid in thread 0
__device__ __forceinline__ double block_sum(double v, double *sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double s = 0;
  if (warp == 0) {
    s = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
    s = warp_sum(s);
  }
  return s;
}

// N = 2 GROUP values of a thread added over the warp, value q left in lanes
// 2 q and 2 q + 1: halving the values each round takes N exchanges where N
// separate sums take 5 N.
template <int N> __device__ __forceinline__ double warp_sums(double (&v)[N], int lane) {
  static_assert(N == 16, "sixteen values");
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1) {
    const int o = h * 32 / N;          // lanes exchanged with
    const bool up = lane & o;
#pragma unroll
    for (int q = 0; q < h; ++q) {
      const double keep = up ? v[q + h] : v[q], send = up ? v[q] : v[q + h];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  // pairs of lanes still hold halves
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// partial[z][blk][i] = sum conj(V_i) w over the block's chunk, i in the
// block's group of GROUP vectors; with self_norm, entry m is (sum |w|^2, 0).
// grid = (chunks, groups, bases).  A block sums one group, so its reduction
// over the warps is paid once for a chunk of some thousand elements; with all
// groups in every block, chunks of two elements a thread and a block-wide sum
// for each component, the reductions took two thirds of the time (262,144
// nodes, 40 vectors: 212 us; the FP64 pipe needs 76).  Eight bases of 262,144
// nodes and some 25 vectors take 432 us in one launch, near the pipe's time.
__global__ void __launch_bounds__(TPB) k_mdot(KrylovBatch B, const double2 *__restrict__ Vb, int64_t ldv, int m,
                                              int64_t n, double2 *__restrict__ partial, int self_norm) {
  __shared__ double sh[TPB / 32][2 * GROUP + 1];
  const double2 *V = Vb + B.off[blockIdx.z], *w = V + (int64_t)m * ldv;
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t g0 = (int64_t)blockIdx.x * chunk, g1 = min(n, g0 + chunk);
  const int i0 = blockIdx.y * GROUP, gi = min(GROUP, m - i0);
  const bool own = self_norm && blockIdx.y == 0;
  const int mt = m + (self_norm ? 1 : 0);
  double acc[2 * GROUP], nrm = 0.0;
#pragma unroll
  for (int q = 0; q < 2 * GROUP; ++q) acc[q] = 0.0;
  const double2 *Vg = V + (int64_t)i0 * ldv;
  for (int64_t g = g0 + threadIdx.x; g < g1; g += TPB) {
    const double2 wv = w[g];
    double2 v[GROUP];
#pragma unroll
    for (int q = 0; q < GROUP; ++q)
      if (q < gi) v[q] = Vg[(int64_t)q * ldv + g];
#pragma unroll
    for (int q = 0; q < GROUP; ++q)
      if (q < gi) {
        acc[2 * q] = fma(v[q].x, wv.x, fma(v[q].y, wv.y, acc[2 * q]));
        acc[2 * q + 1] = fma(v[q].x, wv.y, fma(-v[q].y, wv.x, acc[2 * q + 1]));
      }
    if (own) nrm = fma(wv.x, wv.x, fma(wv.y, wv.y, nrm));
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double s = warp_sums(acc, lane);
  if (own) nrm = warp_sum(nrm);
  if ((lane & 1) == 0) sh[warp][lane >> 1] = s;
  if (lane == 0) sh[warp][2 * GROUP] = nrm;
  __syncthreads();
  if (threadIdx.x < 2 * GROUP + 1) {
    const int c = threadIdx.x;
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < TPB / 32; ++k) t += sh[k][c];
    double *out = reinterpret_cast<double *>(partial + ((int64_t)blockIdx.z * gridDim.x + blockIdx.x) * mt);
    if (c < 2 * gi) out[2 * i0 + c] = t;
    if (c == 2 * GROUP && own) {
      out[2 * m] = t;
      out[2 * m + 1] = 0.0;
    }
  }
}

// h[z][i] = sum over blocks of partial[z][blk][i], fixed order; one warp per i
__global__ void k_reduce_c(KrylovBatch B, const double2 *__restrict__ partial, int nblk, int m,
                           double2 *__restrict__ h, int64_t ldh) {
  const int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (i >= m) return;
  const double2 *P = partial + (int64_t)blockIdx.y * nblk * m;
  double sr = 0, si = 0;
  for (int b = lane; b < nblk; b += 32) {
    const double2 v = P[(int64_t)b * m + i];
    sr += v.x;
    si += v.y;
  }
  sr = warp_sum(sr);
  si = warp_sum(si);
  if (lane == 0) h[B.q[blockIdx.y] * ldh + i] = make_double2(sr, si);
}

// out[z] = sum of partial[z][0..nblk), a stride of ldo doubles between bases
__global__ void k_reduce_r(KrylovBatch B, const double *__restrict__ partial, int nblk, double *__restrict__ out,
                           int64_t ldo) {
  const int lane = threadIdx.x & 31;
  const double *P = partial + (int64_t)blockIdx.x * nblk;
  double s = 0;
  for (int b = lane; b < nblk; b += 32) s += P[b];
  s = warp_sum(s);
  if (lane == 0) out[B.q[blockIdx.x] * ldo] = s;
}

// w -= sum_i h[z][i] V_i and the partial sums of ||w||^2; grid = (chunks,
// bases).  Four vectors' values are in flight at a time (72 us for 40 vectors
// of 262,144 nodes; 320 us for eight bases of some 25 vectors in one launch):
// four multiply-adds an entry at the FP64 pipe's rate.
__global__ void __launch_bounds__(TPB) k_maxpy_norm(KrylovBatch B, double2 *__restrict__ Vb, int64_t ldv, int m,
                                                    const double2 *__restrict__ h, int64_t ldh, int64_t n,
                                                    double *__restrict__ partial) {
  __shared__ double2 hs[MAXM];
  __shared__ double sh[TPB / 32];
  const double2 *hz = h + B.q[blockIdx.y] * ldh;
  for (int i = threadIdx.x; i < m; i += TPB) hs[i] = hz[i];
  __syncthreads();
  const double2 *V = Vb + B.off[blockIdx.y];
  double2 *w = Vb + B.off[blockIdx.y] + (int64_t)m * ldv;
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t g0 = (int64_t)blockIdx.x * chunk, g1 = min(n, g0 + chunk);
  double nrm = 0;
  for (int64_t g = g0 + threadIdx.x; g < g1; g += TPB) {
    double2 acc = w[g];
#pragma unroll 4
    for (int i = 0; i < m; ++i) acc = cfms(hs[i], V[(int64_t)i * ldv + g], acc);
    w[g] = acc;
    nrm = fma(acc.x, acc.x, fma(acc.y, acc.y, nrm));
  }
  const double s = block_sum(nrm, sh);
  if (threadIdx.x == 0) partial[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// V_m scaled to norm 1 by its squared norm, every basis
__global__ void __launch_bounds__(TPB) k_scale_basis(KrylovBatch B, double2 *__restrict__ Vb, int64_t ldv, int m,
                                                     const double *__restrict__ nrm2, int64_t ldn, int64_t n) {
  double2 *w = Vb + B.off[blockIdx.y] + (int64_t)m * ldv;
  const double a = 1.0 / sqrt(nrm2[B.q[blockIdx.y] * ldn]);
  for (int64_t g = (int64_t)blockIdx.x * TPB + threadIdx.x; g < n; g += (int64_t)gridDim.x * TPB) {
    const double2 v = w[g];
    w[g] = make_double2(a * v.x, a * v.y);
  }
}

__global__ void __launch_bounds__(TPB) k_maxpy(const double2 *__restrict__ Z, int64_t ldz, int m,
                                               const double2 *__restrict__ y, double2 *__restrict__ x,
                                               int64_t n) {
  __shared__ double2 ys[MAXM];
  for (int i = threadIdx.x; i < m; i += TPB) ys[i] = y[i];
  __syncthreads();
  for (int64_t g = (int64_t)blockIdx.x * TPB + threadIdx.x; g < n; g += (int64_t)gridDim.x * TPB) {
    double2 acc = x[g];
    for (int i = 0; i < m; ++i) acc = cfma(ys[i], Z[(int64_t)i * ldz + g], acc);
    x[g] = acc;
  }
}

__global__ void __launch_bounds__(TPB) k_norm2(const double2 *__restrict__ x, int64_t n,
                                               double *__restrict__ partial) {
  __shared__ double sh[TPB / 32];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t g0 = (int64_t)blockIdx.x * chunk, g1 = min(n, g0 + chunk);
  double nrm = 0;
  for (int64_t g = g0 + threadIdx.x; g < g1; g += TPB) {
    const double2 v = x[g];
    nrm = fma(v.x, v.x, fma(v.y, v.y, nrm));
  }
  const double s = block_sum(nrm, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void __launch_bounds__(TPB) k_scale(const double2 *__restrict__ x, const double *__restrict__ nrm2,
                                               double2 *__restrict__ y, int64_t n) {
  const double a = 1.0 / sqrt(nrm2[0]);
  for (int64_t g = (int64_t)blockIdx.x * TPB + threadIdx.x; g < n; g += (int64_t)gridDim.x * TPB) {
    const double2 v = x[g];
    y[g] = make_double2(a * v.x, a * v.y);
  }
}

inline int nblocks_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>(NBLK, (n + TPB - 1) / TPB)); }

}  // namespace

namespace {
// Chunks of a basis whose vectors fall into `groups`: NBLK blocks over the
// groups, each of at least two elements a thread.  The number of bases does
// not enter: the chunks set the order of the sums, and a right-hand side's
// must not depend on how many others still iterate.
int chunks_for(int64_t n, int64_t groups) {
  const int64_t most = std::max<int64_t>(1, NBLK / std::max<int64_t>(1, groups));
  return (int)std::max<int64_t>(1, std::min<int64_t>(most, (n + 2 * TPB - 1) / (2 * TPB)));
}
}  // namespace

int64_t krylov_partial_pairs(int m, int bases) {
  // chunks x (vectors + 1) of a basis: NBLK / groups chunks of 8 groups + 1
  // values at most, or one chunk of every vector
  return (int64_t)std::min(bases, KRYLOV_BATCH) * std::max(NBLK * (GROUP + 1), m + 2);
}

void launch_mdot(const KrylovBatch &B, const double2 *V, int64_t ldv, int m, int64_t n, double2 *partial, double2 *h,
                 int64_t ldh, cudaStream_t st, int self_norm) {
  const int groups = (m + GROUP - 1) / GROUP, mt = m + (self_norm ? 1 : 0);
  const int nb = chunks_for(n, groups);
  k_mdot<<<dim3(nb, groups, B.n), TPB, 0, st>>>(B, V, ldv, m, n, partial, self_norm);
  k_reduce_c<<<dim3((mt + 7) / 8, B.n), 256, 0, st>>>(B, partial, nb, mt, h, ldh);
  count_launch(2);
}

void launch_maxpy_norm(const KrylovBatch &B, double2 *V, int64_t ldv, int m, const double2 *h, int64_t ldh, int64_t n,
                       double *partial, double *nrm2, int64_t ldn, cudaStream_t st) {
  const int nb = chunks_for(n, 1);
  k_maxpy_norm<<<dim3(nb, B.n), TPB, 0, st>>>(B, V, ldv, m, h, ldh, n, partial);
  k_reduce_r<<<B.n, 32, 0, st>>>(B, partial, nb, nrm2, ldn);
  count_launch(2);
}

void launch_scale_basis(const KrylovBatch &B, double2 *V, int64_t ldv, int m, const double *nrm2, int64_t ldn,
                        int64_t n, cudaStream_t st) {
  k_scale_basis<<<dim3(chunks_for(n, 1), B.n), TPB, 0, st>>>(B, V, ldv, m, nrm2, ldn, n);
  count_launch();
}

void launch_maxpy(const double2 *Z, int64_t ldz, int m, const double2 *y, double2 *x, int64_t n,
                  cudaStream_t st) {
  k_maxpy<<<nblocks_for(n), TPB, 0, st>>>(Z, ldz, m, y, x, n);
  count_launch();
}

void launch_norm2(const double2 *x, int64_t n, double *partial, double *nrm2, cudaStream_t st) {
  const int nb = nblocks_for(n);
  k_norm2<<<nb, TPB, 0, st>>>(x, n, partial);
  KrylovBatch one = {};
  one.n = 1;
  k_reduce_r<<<1, 32, 0, st>>>(one, partial, nb, nrm2, 0);
  count_launch(2);
}

void launch_scale(const double2 *x, const double *inv_norm2, double2 *y, int64_t n, cudaStream_t st) {
  k_scale<<<nblocks_for(n), TPB, 0, st>>>(x, inv_norm2, y, n);
  count_launch();
}

}  // namespace stdd
