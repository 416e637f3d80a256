// Single-step pivoted Cholesky decomposition (Eq. 21) on the GPU.
//
// The matrix is Hermitian positive semidefinite, M = B B^H (N x N), given by
// a generator B [N][r] whose columns stand in for two-electron integrals
// computed on demand: column p of M is B conj(B[p]). Step k picks the largest
// remaining diagonal element d_p, stops when d_p < tau, and otherwise forms
//   l_k = (M[:, p] - sum_{j<k} l_j conj(l_j[p])) / sqrt(d_p),  d -= |l_k|^2.
// Every element of M - sum_k l_k l_k^H is then below tau in magnitude (the
// remainder is positive semidefinite with every diagonal element below tau).
//
// Every vector lies in the span of B's columns, l_k = B w_k, so the
// correction over the earlier vectors is taken on the r coefficients,
//   w_k = (conj(B[p]) - sum_{j<k} w_j conj(l_j[p])) / sqrt(d_p),
// instead of on the N elements: a step is one product with B (N r complex
// multiply-adds) instead of N (r + k). Two launches a step: `pivot` finishes
// the argmax and forms w_k; `vector` forms l_k, updates the diagonal and
// leaves each block's largest element for the next pivot. The pivots stay on
// the device; the host looks once per STEP_BATCH steps whether to stop.
// Bound: the FP64 pipe (4 N r multiply-adds a step at about 0.6 T/s; B's 16 N
// r bytes would take a third of that). N = 43681, r = 320, 240 vectors: 86.9 ->
// 35.0 ms (0.77 TF/s), the error against FP64 in torch 9.4e-14 -> 8.3e-14.
#include <algorithm>
#include <cmath>
#include <vector>

#include "engine.h"

namespace cdfns {

namespace {

constexpr int THREADS = 256;
constexpr long MAX_BLOCKS = 8192;                       // partial maxima
constexpr int STEP_BATCH = 32;
constexpr int SMEM_R = 2048;                            // coefficients kept in shared memory

struct Largest {
  double v;
  long i;
  // the larger value, of equal ones the smaller index; i < 0: none
  __device__ __forceinline__ void take(double v2, long i2) {
    if (i2 >= 0 && (i < 0 || v2 > v || (v2 == v && i2 < i))) {
      v = v2;
      i = i2;
    }
  }
};

__device__ __forceinline__ Largest block_largest(Largest m) {
  __shared__ double sv[THREADS / 32];
  __shared__ long si[THREADS / 32];
  for (int o = 16; o > 0; o >>= 1)
    m.take(__shfl_xor_sync(0xffffffffu, m.v, o), __shfl_xor_sync(0xffffffffu, m.i, o));
  if ((threadIdx.x & 31) == 0) {
    sv[threadIdx.x >> 5] = m.v;
    si[threadIdx.x >> 5] = m.i;
  }
  __syncthreads();
  Largest t{-1.0, -1};
  for (int w = 0; w < THREADS / 32; ++w) t.take(sv[w], si[w]);
  __syncthreads();
  return t;  // the same in every thread
}

// FIRST: d[q] = sum_s |B[q][s]|^2. Otherwise l = B w, L[q] = l, d[q] -= |l|^2.
// LANES threads per row of B: 8 (128 contiguous bytes a load, three shuffles
// for four rows at once), a warp, or the block, so that few rows still fill
// the SMs; w in shared memory.
template <bool FIRST, int LANES>
__global__ void __launch_bounds__(THREADS)
    vector_kernel(const double2 *__restrict__ B, long N, int r, const double2 *__restrict__ w,
                  const long *__restrict__ piv, double2 *__restrict__ L, double *__restrict__ d,
                  double *bv, long *bi) {
  if (!FIRST && *piv < 0) return;  // the decomposition has stopped
  __shared__ double2 sw[SMEM_R];
  const double2 *ws = w;
  if (!FIRST && r <= SMEM_R) {
    for (int s = threadIdx.x; s < r; s += THREADS) sw[s] = w[s];
    __syncthreads();
    ws = sw;
  }
  constexpr int ROWS = THREADS / LANES;  // per block and pass
  const int lane = threadIdx.x & (LANES - 1);
  Largest m{-1.0, -1};
  for (long q0 = blockIdx.x * static_cast<long>(ROWS); q0 < N; q0 += static_cast<long>(gridDim.x) * ROWS) {
    const long q = q0 + threadIdx.x / LANES;
    double xr = 0.0, xi = 0.0;
    if (q < N) {
      const double2 *row = B + q * r;
      double yr = 0.0, yi = 0.0;
#pragma unroll 4
      for (int s = lane; s < r; s += LANES) {
        const double2 b = row[s];
        if (FIRST) {
          xr = fma(b.x, b.x, xr);
          yr = fma(b.y, b.y, yr);
        } else {
          const double2 c = ws[s];
          xr = fma(b.x, c.x, xr);
          yr = fma(-b.y, c.y, yr);
          xi = fma(b.x, c.y, xi);
          yi = fma(b.y, c.x, yi);
        }
      }
      xr += yr;
      xi += yi;
    }
    for (int o = (LANES < 32 ? LANES : 32) / 2; o > 0; o >>= 1) {
      xr += __shfl_xor_sync(0xffffffffu, xr, o);
      if (!FIRST) xi += __shfl_xor_sync(0xffffffffu, xi, o);
    }
    if (LANES > 32) {  // the block's warps, pairwise
      __shared__ double2 part[THREADS / 32];
      if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = make_double2(xr, xi);
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int s = 1; s < THREADS / 32; s *= 2)
          for (int g = 0; g < THREADS / 32; g += 2 * s) part[g] = cadd(part[g], part[g + s]);
        xr = part[0].x;
        xi = part[0].y;
      }
      __syncthreads();
    }
    if (q < N && lane == 0) {
      double x;
      if (FIRST) {
        x = xr;
      } else {
        L[q] = make_double2(xr, xi);
        x = d[q] - (xr * xr + xi * xi);
      }
      d[q] = x;
      if (x > m.v) {  // ascending q: the first of equal values stays, NaN never does
        m.v = x;
        m.i = q;
      }
    }
  }
  m = block_largest(m);
  if (threadIdx.x == 0) {
    bv[blockIdx.x] = m.v;
    bi[blockIdx.x] = m.i;
  }
}

// Step k: the pivot from the partial maxima (every block by itself; -1 once
// the decomposition has stopped, -2 for a diagonal that is not finite), then
// 32 of w_k's coefficients per block, the earlier vectors spread over its
// eight warps.
__global__ void __launch_bounds__(THREADS)
    pivot_kernel(const double2 *__restrict__ B, long N, int r, double tau, int k, long nb,
                 const double *__restrict__ bv, const long *__restrict__ bi,
                 const double2 *__restrict__ L, double2 *W, long *piv) {
  if (k > 0 && piv[k - 1] < 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) piv[k] = piv[k - 1];
    return;
  }
  Largest m{-1.0, -1};
  for (long b = threadIdx.x; b < nb; b += THREADS) m.take(bv[b], bi[b]);
  m = block_largest(m);
  const bool bad = m.i >= 0 && !isfinite(m.v);
  const bool stop = bad || m.i < 0 || !(m.v >= tau) || !(m.v > 0.0);
  if (blockIdx.x == 0 && threadIdx.x == 0) piv[k] = bad ? -2 : (stop ? -1 : m.i);
  if (stop) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int s = blockIdx.x * 32 + tx;
  double2 a = make_double2(0.0, 0.0);
  if (s < r) {
#pragma unroll 4
    for (int j = ty; j < k; j += THREADS / 32) {
      const double2 l = L[j * N + m.i], w = W[static_cast<long>(j) * r + s];
      a = cfma(w, make_double2(l.x, -l.y), a);
    }
  }
  __shared__ double2 part[THREADS / 32][33];
  part[ty][tx] = a;
  __syncthreads();
  if (ty == 0 && s < r) {
    for (int g = 1; g < THREADS / 32; ++g) a = cadd(a, part[g][tx]);
    const double2 b = B[m.i * r + s];
    const double f = 1.0 / sqrt(m.v);
    W[static_cast<long>(k) * r + s] = make_double2(f * (b.x - a.x), f * (-b.y - a.y));
  }
}

}  // namespace

int pivoted_cholesky(const cplx *B, long N, int r, double tau, int max_vec, cplx *L, long *piv,
                     Allocator *al, cudaStream_t st, int num_sms) {
  // a step in us with 8 / 32 / 256 threads a row: 300 x 2100 98 / 40 / 24,
  // 1000 x 1000 54 / 30 / 38, 1000 x 4000 182 / 61 / 57, 2500 x 100 20 / 30 / 44,
  // 5000 x 800 74 / 68 / 100
  const int lanes = N > 16L * num_sms ? 8 : N > 2L * num_sms ? 32 : THREADS;
  auto first = lanes == 8 ? vector_kernel<true, 8> : lanes == 32 ? vector_kernel<true, 32> : vector_kernel<true, THREADS>;
  auto next = lanes == 8 ? vector_kernel<false, 8> : lanes == 32 ? vector_kernel<false, 32> : vector_kernel<false, THREADS>;
  const long rows = THREADS / lanes;
  const long nb = std::min<long>(MAX_BLOCKS, (N + rows - 1) / rows);
  const unsigned grid = static_cast<unsigned>(nb);
  Buf d(al, sizeof(double) * N), W(al, sizeof(cplx) * max_vec * r);
  Buf bv(al, sizeof(double) * nb), bi(al, sizeof(long) * nb), pv(al, sizeof(long) * max_vec);
  first<<<grid, THREADS, 0, st>>>(B, N, r, nullptr, nullptr, nullptr, d.as<double>(), bv.as<double>(),
                                  bi.as<long>());
  LAUNCH_CHECK();
  count_launch();
  std::vector<long> hp(max_vec);
  int n = 0;
  for (int k0 = 0; k0 < max_vec; k0 += STEP_BATCH) {
    const int k1 = std::min(max_vec, k0 + STEP_BATCH);
    for (int k = k0; k < k1; ++k) {
      pivot_kernel<<<static_cast<unsigned>((r + 31) / 32), THREADS, 0, st>>>(
          B, N, r, tau, k, nb, bv.as<double>(), bi.as<long>(), L, W.c(), pv.as<long>());
      LAUNCH_CHECK();
      next<<<grid, THREADS, 0, st>>>(B, N, r, W.c() + static_cast<long>(k) * r, pv.as<long>() + k,
                                     L + static_cast<long>(k) * N, d.as<double>(), bv.as<double>(),
                                     bi.as<long>());
      LAUNCH_CHECK();
      count_launch(2);
    }
    CUDA_CHECK(cudaMemcpyAsync(hp.data() + k0, pv.as<long>() + k0, sizeof(long) * (k1 - k0),
                               cudaMemcpyDeviceToHost, st));
    CUDA_CHECK(cudaStreamSynchronize(st));
    while (n < k1 && hp[n] >= 0) ++n;
    if (n < k1) {
      if (hp[n] == -2) fail(CC_ERR_NUMERIC, "cholesky: non-finite diagonal");
      break;
    }
  }
  if (piv) std::copy(hp.begin(), hp.begin() + n, piv);
  return n;
}

}  // namespace cdfns
