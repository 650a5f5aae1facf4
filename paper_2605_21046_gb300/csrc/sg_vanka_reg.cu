// Vanka sweep for small patches (at most 18 unknowns: 2D Q1, and Q2 up to two
// time nodes), FP32 vectors: x += omega / mult * inv(patch) * r_patch for every
// cell and row.
//
// One thread holds one cell for one block of kVankaVB rows of a class, with the
// patch's r values in registers; the lanes of a warp are 32 consecutive cells
// (x fastest).  The inverses are stored [entry][cell] in the factors' precision
// (FP32 or bf16: 256^2 Q2 V-cycle with 35 rows 0.970 and 0.946 ms), so a lane's
// entry is one coalesced load that serves kVankaVB FMAs, and a patch row's
// result is weighted and added into x as soon as it is summed - no shared
// memory and no barrier.  As in the row-diagonal apply the plane of nodes that a cell shares
// with its right neighbour is handed over by a shuffle, and only the last cell
// of a warp or of a row of cells adds it itself.
//
// Small patches leave little work per sweep, so what counts is the chain of
// latencies: the tiled kernel (staging, two barriers, sums in shared memory)
// takes 24 us on 64^2 Q2 with 35 rows and 9 to 10 us on its coarser levels.
// On few cells the lines of a patch (time node, y) go to different warps, each
// with its own copy of r, so that a warp's loads of inverses are one round.
// Larger patches stay with the other sweeps: every block of rows reads every
// inverse, and at 27 unknowns (48^2 Q2 dG(2), bf16 factors) the V-cycle is
// 0.18 ms with this sweep and 0.13 with the tensor cores.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "sg_bounds.h"
#include "sg_internal.h"

namespace sg {

namespace {

constexpr int VB = 4;            // rows of a block (kVankaVB of the tiled kernel)
constexpr int kRegWarps = 4;     // row blocks (warps) per thread block

struct RegVankaArgs {
  const float* r;
  float* x;
  const void* inv;               // [class][NP * NP][n_cells], float or bf16
  const int* blk_cls;            // [n_blk]
  const int* blk_alpha;          // [n_blk][VB] rows, -1 padded
  long long n_x, n_vec_x, inv_count;
  int n_cells, n_blk;
  int cells[2], nn[2];
  float omega;
};

template <int K, int NT, bool TRANS, typename W>
__global__ void __launch_bounds__(32 * kRegWarps) mg_vanka_reg(const RegVankaArgs p) {
  constexpr int N = K + 1, NKD = N * N, NP = NT * NKD;
  const int blk = blockIdx.y * kRegWarps + threadIdx.y;
  if (blk >= p.n_blk) return;                                   // whole warps
  const int lane = threadIdx.x, cell = blockIdx.x * 32 + lane;
  const bool valid = cell < p.n_cells;
  const int cc = valid ? cell : p.n_cells - 1;
  const int cx = cc % p.cells[0], cy = cc / p.cells[0];
  const bool lo0 = cx == 0, hi0 = cx == p.cells[0] - 1, lo1 = cy == 0, hi1 = cy == p.cells[1] - 1;
  const int sy = p.nn[0], base = cx * K + cy * K * sy;
  auto inner = [&](int a) {
    const int ax = a % N, ay = a / N;
    return valid && !(ax == 0 && lo0) && !(ax == K && hi0) && !(ay == 0 && lo1) && !(ay == K && hi1);
  };
  long long off[VB];
#pragma unroll
  for (int u = 0; u < VB; ++u) {
    const int m = __ldg(p.blk_alpha + blk * VB + u);
    off[u] = m < 0 ? -1 : (long long)m * NT * p.n_x + base;
  }
  float r[NP][VB];
#pragma unroll
  for (int i = 0; i < NT; ++i)
#pragma unroll
    for (int a = 0; a < NKD; ++a)
#pragma unroll
      for (int u = 0; u < VB; ++u) {
        const long long at = off[u] + i * p.n_x + a % N + (a / N) * sy;
        r[i * NKD + a][u] = off[u] >= 0 && inner(a) && SG_IN(at, p.n_vec_x, 801) ? __ldg(p.r + at) : 0.0f;
      }
  const bool take = valid && lane > 0 && cx > 0;                          // the left lane's last plane
  const bool give = valid && lane < 31 && cell + 1 < p.n_cells && !hi0;   // mine goes to the right lane
  const W* all = static_cast<const W*>(p.inv);
  const W* inv = all + (long long)__ldg(p.blk_cls + blk) * NP * NP * p.n_cells + cc;
  // a line of nodes (time node i, row ay) at a time: the right lane's first
  // node needs the left lane's last one
#pragma unroll 1
  for (int line = blockIdx.z; line < NT * N; line += gridDim.z) {
      const int i = line / N, ay = line % N;
      float z[N][VB];
#pragma unroll
      for (int ax = 0; ax < N; ++ax) {
        const int rho = i * NKD + ay * N + ax;
        const W* row = inv + (long long)(TRANS ? rho : rho * NP) * p.n_cells;
        const long long step = (long long)(TRANS ? NP : 1) * p.n_cells;
        float w[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q)
          w[q] = SG_IN((long long)(row - all) + q * step, p.inv_count, 802) ? (float)__ldg(row + q * step) : 0.0f;
#pragma unroll
        for (int u = 0; u < VB; ++u) z[ax][u] = 0.0f;
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
          for (int u = 0; u < VB; ++u) z[ax][u] = fmaf(w[q], r[q][u], z[ax][u]);
      }
      const float wy = (ay == 0 || ay == K) ? 0.5f * p.omega : p.omega;
      const bool in_y = valid && !(ay == 0 && lo1) && !(ay == K && hi1);
#pragma unroll
      for (int u = 0; u < VB; ++u) {
        const float left = __shfl_up_sync(0xffffffffu, z[K][u], 1);
        if (take) z[0][u] += left;
        const long long at = off[u] + i * p.n_x + ay * sy;
        if (off[u] < 0 || !in_y) continue;
#pragma unroll
        for (int ax = 0; ax < N; ++ax) {
          if ((ax == 0 && lo0) || (ax == K && (hi0 || give))) continue;
          if (SG_IN(at + ax, p.n_vec_x, 803)) atomicAdd(p.x + at + ax, (ax == 0 || ax == K ? 0.5f * wy : wy) * z[ax][u]);
        }
      }
    }
}

// The inverses by cell, [class][cell][np][npp] (zeros past np), to and from the
// order of this sweep, [class][np * np][cell]: 32 x 32 tiles through shared
// memory; cells on grid.x, which alone takes more than 65535 tiles of them.
template <typename W, bool TO_COLUMNS>
__global__ void __launch_bounds__(256) vanka_columns(const W* __restrict__ in, W* __restrict__ out, int np, int npp,
                                                     int n_cells, int n_classes) {
  __shared__ W tile[32][33];
  const int c0 = blockIdx.x * 32, e0 = blockIdx.y * 32;
  const int width = TO_COLUMNS ? np : npp;                     // entries of a patch row: without or with the zeros
  const long long n_cell = (long long)n_classes * n_cells * np * npp, n_entry = (long long)n_classes * np * np * n_cells;
  for (int cls = blockIdx.z; cls < n_classes; cls += gridDim.z) {
    const long long by_cell = (long long)cls * n_cells * np * npp, by_entry = (long long)cls * np * np * n_cells;
    for (int j = threadIdx.y; j < 32; j += 8) {
      const int c = c0 + (TO_COLUMNS ? j : threadIdx.x), e = e0 + (TO_COLUMNS ? threadIdx.x : j);
      const int row = e / width, col = e % width;
      if (c >= n_cells || e >= np * width) continue;
      const long long at = TO_COLUMNS ? by_cell + ((long long)c * np + row) * npp + col
                                      : by_entry + (long long)(row * np + col) * n_cells + c;
      const W v = col < np && SG_IN(at, TO_COLUMNS ? n_cell : n_entry, 804) ? in[at] : W(0.0f);
      if (TO_COLUMNS) tile[j][threadIdx.x] = v;
      else tile[threadIdx.x][j] = v;
    }
    __syncthreads();
    for (int j = threadIdx.y; j < 32; j += 8) {
      const int c = c0 + (TO_COLUMNS ? threadIdx.x : j), e = e0 + (TO_COLUMNS ? j : threadIdx.x);
      if (c >= n_cells || e >= np * width) continue;
      const long long at = TO_COLUMNS ? by_entry + (long long)e * n_cells + c
                                      : by_cell + ((long long)c * np + e / width) * npp + e % width;
      if (SG_IN(at, TO_COLUMNS ? n_entry : n_cell, 805)) out[at] = TO_COLUMNS ? tile[threadIdx.x][j] : tile[j][threadIdx.x];
    }
    __syncthreads();
  }
}

template <typename W>
cudaError_t reorder(bool to_columns, const void* in, void* out, int np, int npp, int n_classes, long long n_cells) {
  const int entries = np * (to_columns ? np : npp);
  const dim3 grid((unsigned)((n_cells + 31) / 32), (entries + 31) / 32, std::min(n_classes, 65535)), block(32, 8);
  const W* a = static_cast<const W*>(in);
  W* b = static_cast<W*>(out);
  if (to_columns) vanka_columns<W, true><<<grid, block>>>(a, b, np, npp, (int)n_cells, n_classes);
  else vanka_columns<W, false><<<grid, block>>>(a, b, np, npp, (int)n_cells, n_classes);
  return cudaGetLastError();
}

}  // namespace

bool vanka_reg_eligible(int dim, int k, int nt) {
  return dim == 2 && k <= 2 && nt * (k + 1) * (k + 1) <= 18;
}

cudaError_t vanka_reg_reorder(bool to_columns, const void* in, bool bf16, int np, int npp, int n_classes,
                              long long n_cells, void** out) {
  const size_t n = (size_t)n_classes * n_cells * np * (to_columns ? np : npp);
  *out = nullptr;
  cudaError_t e = cudaMalloc(out, n * (bf16 ? sizeof(__nv_bfloat16) : sizeof(float)));
  if (e != cudaSuccess) return e;
  e = bf16 ? reorder<__nv_bfloat16>(to_columns, in, *out, np, npp, n_classes, n_cells)
           : reorder<float>(to_columns, in, *out, np, npp, n_classes, n_cells);
  if (e == cudaSuccess) e = cudaStreamSynchronize(0);
  return e;
}

cudaError_t launch_vanka_reg(const HostProblem& hp, const float* r, float* x, const void* inv, bool bf16,
                             const int* blk_cls, const int* blk_alpha, int n_blk, int n_classes, float omega, int trans,
                             cudaStream_t s) {
  RegVankaArgs p;
  p.r = r;
  p.x = x;
  p.inv = inv;
  p.blk_cls = blk_cls;
  p.blk_alpha = blk_alpha;
  p.n_x = hp.n_x;
  p.n_vec_x = (long long)hp.n_xi * hp.n_t * hp.n_x;
  p.n_cells = (int)hp.n_cells;
  p.n_blk = n_blk;
  for (int d = 0; d < 2; ++d) {
    p.cells[d] = hp.cells[d];
    p.nn[d] = hp.nn[d];
  }
  p.omega = omega;
  const int np = hp.n_t * (hp.k + 1) * (hp.k + 1);
  p.inv_count = (long long)n_classes * np * np * hp.n_cells;
  dim3 grid((unsigned)((hp.n_cells + 31) / 32), (n_blk + kRegWarps - 1) / kRegWarps);
  const dim3 block(32, kRegWarps);
  // as many warps per patch as the SMs hold at once (16 each)
  const long long warps = (long long)grid.x * n_blk, room = 16 * sm_count();
  for (int split : {2, 3, 4, 6, 8})
    if (split <= hp.n_t * (hp.k + 1) && warps * split <= room) grid.z = split;
#define SG_R(KK, TT)                                                                               \
  if (hp.dim == 2 && hp.k == KK && hp.n_t == TT) {                                                 \
    if (bf16 && trans) mg_vanka_reg<KK, TT, true, __nv_bfloat16><<<grid, block, 0, s>>>(p);        \
    else if (bf16) mg_vanka_reg<KK, TT, false, __nv_bfloat16><<<grid, block, 0, s>>>(p);           \
    else if (trans) mg_vanka_reg<KK, TT, true, float><<<grid, block, 0, s>>>(p);                   \
    else mg_vanka_reg<KK, TT, false, float><<<grid, block, 0, s>>>(p);                             \
    return cudaGetLastError();                                                                     \
  }
  SG_R(1, 1) SG_R(1, 2) SG_R(1, 3) SG_R(1, 4) SG_R(2, 1) SG_R(2, 2)
#undef SG_R
  return cudaErrorInvalidValue;
}

}  // namespace sg

SG_BOUNDS_FETCH(bounds_fetch_vanka_reg)
