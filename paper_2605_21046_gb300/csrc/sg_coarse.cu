// Dense inverse of the coarsest level's block operator on the device: in-place
// Gauss-Jordan elimination by blocks of 16 pivots, one launch per block
// (every launch reads the matrix of one buffer and writes the other, so no
// block waits for another).  A thread block takes a 32 x 32 tile, inverts the
// 16 x 16 pivot block itself and applies the rank-16 update.
//
// The elimination on the host cost 6.5 of the 7.4 ms of a 32^2 Q2 set-up
// (450 unknowns; also once per Monte-Carlo call); this one is 29 launches,
// bound by the serial chain through the pivot block.  Pivots are taken in
// order: the operator's symmetric part is positive definite for an elliptic
// coefficient.  A coefficient that is not may need exchanges, so the inverse X
// of C is checked on a vector v > 0 and the caller falls back to the pivoting
// elimination when |C (X v) - v| is above a bound times the largest entry of
// |C| |X| v, the size of the terms that cancel there.  For FP64 levels the bound
// is 8 roundings: elliptic operators of 450 to 2000 unknowns stay below 4, as
// the pivoting elimination does, while indefinite ones (a negative mean
// coefficient) that reach 10 to 1e5 have lost one to five digits against it.
// FP32 levels, which store X to 2^-24, take 2^-32.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "sg_bounds.h"
#include "sg_internal.h"

namespace sg {

namespace {

constexpr int kPiv = 16;    // pivots per launch
constexpr int kTile = 32;   // tile of the matrix per block

__global__ void __launch_bounds__(256) coarse_step(const double* __restrict__ A, double* __restrict__ out, int n, int k0,
                                                   int* __restrict__ singular) {
  __shared__ double P[kPiv][kPiv + 1], M[kTile][kPiv + 1], R[kTile][kPiv + 1], C[kPiv][kTile + 1];
  const int tid = threadIdx.x, r0 = blockIdx.y * kTile, c0 = blockIdx.x * kTile, kb = min(kPiv, n - k0);
  const int pi = tid / kPiv, pj = tid % kPiv;
  const long long nn = (long long)n * n;
  auto at = [&](long long r, long long c) { return SG_IN(r * n + c, nn, 511) ? A[r * n + c] : 0.0; };
  // the pivot block (padded with the identity), its rows and its columns in this tile
  P[pi][pj] = pi < kb && pj < kb ? at(k0 + pi, k0 + pj) : (pi == pj ? 1.0 : 0.0);
  for (int e = tid; e < kTile * kPiv; e += 256) {
    const int a = e / kPiv, q = e % kPiv;
    R[a][q] = r0 + a < n && q < kb ? at(r0 + a, k0 + q) : 0.0;
    const int cq = e / kTile, cc = e % kTile;
    C[cq][cc] = cq < kb && c0 + cc < n ? at(k0 + cq, c0 + cc) : 0.0;
  }
  __syncthreads();
  for (int q = 0; q < kPiv; ++q) {
    const double d = P[q][q], f = P[pi][q], g = P[q][pj], a = P[pi][pj];
    __syncthreads();
    const double inv = 1.0 / d;
    if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0 && !(fabs(inv) <= 1e300)) *singular = 1;
    if (pi == q) P[pi][pj] = pj == q ? inv : g * inv;
    else P[pi][pj] = pj == q ? -f * inv : fma(-f * inv, g, a);
    __syncthreads();
  }
  // rows outside the pivot block take R P^-1, those inside -P^-1
  for (int e = tid; e < kTile * kPiv; e += 256) {
    const int a = e / kPiv, q = e % kPiv, rk = r0 + a - k0;
    double s = 0.0;
    if (rk >= 0 && rk < kb) {
      s = -P[rk][q];
    } else {
#pragma unroll
      for (int j = 0; j < kPiv; ++j) s = fma(R[a][j], P[j][q], s);
    }
    M[a][q] = s;
  }
  __syncthreads();
  for (int e = tid; e < kTile * kTile; e += 256) {
    const int a = e / kTile, b = e % kTile, r = r0 + a, c = c0 + b;
    if (r >= n || c >= n) continue;
    const int rk = r - k0, ck = c - k0;
    double v;
    if (ck >= 0 && ck < kb) {
      v = -M[a][ck];
    } else {
      v = rk >= 0 && rk < kb ? 0.0 : at(r, c);
#pragma unroll
      for (int q = 0; q < kPiv; ++q) v = fma(-M[a][q], C[q][b], v);
    }
    if (SG_IN((long long)r * n + c, nn, 512)) out[(size_t)r * n + c] = v;
  }
}

// y = A x and ya = |A| xa, a warp per row
__global__ void coarse_mv(const double* __restrict__ A, const double* __restrict__ x, const double* __restrict__ xa,
                          double* __restrict__ y, double* __restrict__ ya, int n) {
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= n) return;
  double s = 0.0, sa = 0.0;
  for (int q = lane; q < n; q += 32) {
    const double a = SG_IN((long long)row * n + q, (long long)n * n, 513) ? A[(size_t)row * n + q] : 0.0;
    s = fma(a, x[q], s);
    sa = fma(fabs(a), xa[q], sa);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    sa += __shfl_xor_sync(0xffffffffu, sa, o);
  }
  if (lane == 0) {
    y[row] = s;
    ya[row] = sa;
  }
}

template <typename T>
__global__ void coarse_store(const double* __restrict__ a, T* __restrict__ out, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = (T)a[i];
}

}  // namespace

cudaError_t coarse_inverse_device(const std::vector<double>& C, int n, int precision, void* out, bool& ok) {
  ok = n == 0;              // a mesh without interior nodes has nothing to invert
  if (ok) return cudaSuccess;
  const size_t nn = (size_t)n * n;
  double* buf = nullptr;   // the matrix, two work buffers, five vectors, the flag
  cudaError_t e = cudaMalloc(&buf, (3 * nn + 5 * (size_t)n + 1) * sizeof(double));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cudaSuccess;    // no room beside the level: the caller's way needs none
  }
  double *A0 = buf, *w[2] = {buf + nn, buf + 2 * nn}, *v = buf + 3 * nn, *y = v + n, *ya = y + n, *z = ya + n, *za = z + n;
  int* flag = reinterpret_cast<int*>(za + n);
  std::vector<double> hv(n), hz(2 * (size_t)n);
  for (int i = 0; i < n; ++i) hv[i] = 1.0 + 0.5 * ((i * 37) % 101) / 101.0;
  e = cudaMemcpy(A0, C.data(), nn * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(v, hv.data(), n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, sizeof(int), 0);
  int singular = 0, at = 0;
  if (e == cudaSuccess) {
    const dim3 grid((n + kTile - 1) / kTile, (n + kTile - 1) / kTile);
    const double* from = A0;
    for (int k0 = 0; k0 < n; k0 += kPiv, at ^= 1) {
      coarse_step<<<grid, 256>>>(from, w[at], n, k0, flag);
      from = w[at];
    }
    coarse_mv<<<(n + 7) / 8, 256>>>(from, v, v, y, ya, n);
    coarse_mv<<<(n + 7) / 8, 256>>>(A0, y, ya, z, za, n);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(hz.data(), z, 2 * n * sizeof(double), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&singular, flag, sizeof(int), cudaMemcpyDeviceToHost);
    double off = 0.0, size = 0.0;
    bool finite = true;
    for (int i = 0; i < n; ++i) {
      finite = finite && std::isfinite(hz[i]) && std::isfinite(hz[n + i]);
      off = std::max(off, std::fabs(hz[i] - hv[i]));
      size = std::max(size, hz[n + i]);
    }
    ok = e == cudaSuccess && !singular && finite && off <= (precision == kPrecF32 ? 0x1p-32 : 8 * 0x1p-52) * size;
    if (ok) {
      const int g = (int)std::min<size_t>((nn + 255) / 256, (size_t)sm_count() * 16);
      if (precision == kPrecF32) coarse_store<float><<<g, 256>>>(from, static_cast<float*>(out), (long long)nn);
      else coarse_store<double><<<g, 256>>>(from, static_cast<double*>(out), (long long)nn);
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    }
  }
  cudaFree(buf);
  return e;
}

}  // namespace sg

SG_BOUNDS_FETCH(bounds_fetch_coarse)
