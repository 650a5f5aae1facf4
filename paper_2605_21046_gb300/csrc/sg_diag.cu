// The apply of row-diagonal slab operators: y += sign * A_s x_s for every row s,
//     A_s = T (x) M_x + B_t (x) K[sum_t w[s][t] a_t],
// the operators that couple no two rows - the multigrid levels (block Jacobi:
// w[alpha][t] = G_t[alpha][alpha]) and the Monte-Carlo samples
// (w[s][t] = Psi_t(xi_s)).
//
// One thread holds one cell of one row, with every nodal and Gauss-point value
// of its time nodes in registers: no value passes through shared memory and
// the kernel has no barrier.  The lanes of a warp are 32 consecutive cells (x
// fastest) of one row, so the k-strided node loads of a warp fall in a few
// lines that its other loads hit in L1, and the coefficient, stored
// [term][point][cell], is read coalesced.  The two cells of a lane and its
// right neighbour share a plane of nodes: the lane hands its part over with a
// shuffle, and only the last cell of a warp or of a row adds that plane into y
// itself (18 of 27 reductions per 3D Q2 cell and time node).
//
// The cell work is about 750 FMAs per vector (3D Q2).  Held in shared memory it
// was bound by that memory's wavefronts (28 accesses per point and row) and
// took 295 us on 32^3 Q2 with 20 rows in FP32; this kernel takes 78 us
// (the V-cycle went from 1.46 to 0.97 ms with bf16 factors, 64^2 Q2 with 35
// rows from 0.254 to 0.201 ms).
#include <cuda_runtime.h>

#include <algorithm>

#include "sg_apply_kernel.cuh"

namespace sg {

namespace {

constexpr int kDiagRows = 4;   // rows (warps) per block
static_assert(kDiagCells == 32, "a lane per cell");

template <typename T>
struct DiagArgs {
  const T* x;
  T* y;
  const T* ctab;            // [term][NQD][n_cells]
  const T* wgt;             // [rows][n_terms]
  long long n_x;
  int n_cells, rows, n_terms, mass_only, aniso;
  int cells[3], nn[3];
  T ratio[3];
  T tb[kMaxNT];             // sign * tau Bhat_ii
  double lk[kLineConsts];   // constants of the 1D passes
  T amq[kMaxAmq];           // [point][i][j] w_q |J| T[i][j] / (tau Bhat_ii)
};

// FP32 3D Q2 would take 168 registers; at 128 (no spills) four blocks share an SM.
template <class A, int DIM, int K, int NT>
__global__ void __launch_bounds__(32 * kDiagRows, (std::is_same<A, F32>::value && DIM == 3 && K == 2 ? 4 : 0)) diag_apply(const __grid_constant__ DiagArgs<typename A::T> p) {
  using T = typename A::T;
  __shared__ double s_lk[kLineConsts];
  if (std::is_same<A, F64>::value) {
    const int t = threadIdx.y * 32 + threadIdx.x;
    if (t < kLineConsts) s_lk[t] = p.lk[t];
    __syncthreads();
  }
  const Line<A, K> L(s_lk);
  constexpr int N = K + 1, NQD = Shape<DIM, K>::NQD, NL = NQD / N;
  const int lane = threadIdx.x, row = blockIdx.y * kDiagRows + threadIdx.y;
  if (row >= p.rows) return;                                  // whole warps
  const int cell = blockIdx.x * 32 + lane;
  const bool valid = cell < p.n_cells;
  const int cc = valid ? cell : p.n_cells - 1;
  const int cx = cc % p.cells[0], cyz = cc / p.cells[0];
  const int cy = DIM == 3 ? cyz % p.cells[1] : cyz, cz = DIM == 3 ? cyz / p.cells[1] : 0;
  const bool lo0 = cx == 0, hi0 = cx == p.cells[0] - 1, lo1 = cy == 0, hi1 = cy == p.cells[1] - 1;
  const bool lo2 = DIM == 3 && cz == 0, hi2 = DIM == 3 && cz == p.cells[2] - 1;
  const int sy = p.nn[0], sz = DIM == 3 ? p.nn[0] * p.nn[1] : 0;
  const int base = cx * K + cy * K * sy + cz * K * sz;
  // node a of the cell lies inside the domain
  auto inner = [&](int a) {
    const int ax = a % N, ay = (a / N) % N, az = a / (N * N);
    bool in = valid && !(ax == 0 && lo0) && !(ax == K && hi0) && !(ay == 0 && lo1) && !(ay == K && hi1);
    if (DIM == 3) in = in && !(az == 0 && lo2) && !(az == K && hi2);
    return in;
  };
  auto offset = [&](int a) { return base + a % N + ((a / N) % N) * sy + (DIM == 3 ? (a / (N * N)) * sz : 0); };
  const long long v0 = (long long)row * NT, n_vec = (long long)p.rows * NT * p.n_x;

  T v[NT][NQD];
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const T* src = p.x + (v0 + i) * p.n_x;
#pragma unroll
    for (int a = 0; a < NQD; ++a)
      v[i][a] = inner(a) && SG_IN((v0 + i) * p.n_x + offset(a), n_vec, 701) ? __ldg(src + offset(a)) : T(0);
  }
  // the row's coefficient at the cell's points
  T c[NQD];
  if (!p.mass_only) {
    const T* w = p.wgt + (long long)row * p.n_terms;
#pragma unroll
    for (int q = 0; q < NQD; ++q) c[q] = T(0);
    for (int t = 0; t < p.n_terms; ++t) {
      const T wt = __ldg(w + t);
      const T* ct = p.ctab + (long long)t * NQD * p.n_cells + cc;
#pragma unroll
      for (int q = 0; q < NQD; ++q) A::fma(wt, __ldg(ct + (long long)q * p.n_cells), c[q]);
    }
  }
  T in[N], g[N], out[N];
#pragma unroll
  for (int i = 0; i < NT; ++i)
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const int o = line_first<N>(d, l), st = line_stride<N>(d);
#pragma unroll
        for (int j = 0; j < N; ++j) in[j] = v[i][o + j * st];
        L.interp(in, out);
#pragma unroll
        for (int j = 0; j < N; ++j) v[i][o + j * st] = out[j];
      }
    }
  const bool take = valid && lane > 0 && cx > 0;                          // the left lane's last plane
  const bool give = valid && lane < 31 && cell + 1 < p.n_cells && !hi0;   // mine goes to the right lane
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    T r[NQD];
#pragma unroll
    for (int q = 0; q < NQD; ++q) {
      T s = L.mul(p.amq[(q * NT + i) * NT], v[0][q]);
#pragma unroll
      for (int j = 1; j < NT; ++j) A::fma(p.amq[(q * NT + i) * NT + j], v[j][q], s);
      r[q] = s;
    }
#pragma unroll
    for (int dd = 0; dd < DIM; ++dd) {
      const int st = line_stride<N>(dd);
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const int o = line_first<N>(dd, l);
        T rl[N];
#pragma unroll
        for (int j = 0; j < N; ++j) rl[j] = r[o + j * st];
        if (!p.mass_only) {
#pragma unroll
          for (int j = 0; j < N; ++j) in[j] = v[i][o + j * st];
          L.deriv(in, g);
#pragma unroll
          for (int j = 0; j < N; ++j) g[j] = L.mul(g[j], c[o + j * st]);
          if (dd > 0 && p.aniso) {
#pragma unroll
            for (int j = 0; j < N; ++j) g[j] = L.mul(g[j], p.ratio[dd]);
          }
          if (dd + 1 < DIM) {
            L.deriv_t(g, rl);
          } else {
            L.interp_deriv_t(rl, g, out);
          }
        } else if (dd + 1 == DIM) {
          L.interp_t(rl, out);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) r[o + j * st] = dd + 1 < DIM ? rl[j] : out[j];
      }
    }
#pragma unroll
    for (int dd = DIM - 2; dd >= 0; --dd) {
      const int st = line_stride<N>(dd);
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const int o = line_first<N>(dd, l);
#pragma unroll
        for (int j = 0; j < N; ++j) in[j] = r[o + j * st];
        L.interp_t(in, out);
#pragma unroll
        for (int j = 0; j < N; ++j) r[o + j * st] = out[j];
      }
    }
    T* dst = p.y + (v0 + i) * p.n_x;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const T left = __shfl_up_sync(0xffffffffu, r[l * N + K], 1);
      if (take) r[l * N] = L.add(r[l * N], left);
    }
#pragma unroll
    for (int a = 0; a < NQD; ++a)
      if (inner(a) && !(a % N == K && give) && SG_IN((v0 + i) * p.n_x + offset(a), n_vec, 702))
        A::add_out(dst + offset(a), L.mul(p.tb[i], r[a]));
  }
}

// ctab [cell][n_terms][NQD] -> out [used][NQD][cell], with the weight of the unscaled gradients
template <typename T>
__global__ void diag_table(const double* __restrict__ ctab, T* __restrict__ out, const int* __restrict__ used,
                           int n_used, int n_terms, int nqd, int n_cells, double weight) {
  const long long n = (long long)n_used * nqd * n_cells;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int cell = (int)(i % n_cells);
    const long long r = i / n_cells;
    const int q = (int)(r % nqd), u = (int)(r / nqd);
    out[i] = (T)(weight * ctab[((long long)cell * n_terms + used[u]) * nqd + q]);
  }
}

template <class A>
cudaError_t launch(int dim, int k, int nt, const DiagParams& q, cudaStream_t s) {
  using T = typename A::T;
  DiagArgs<T> p;
  p.x = static_cast<const T*>(q.x);
  p.y = static_cast<T*>(q.y);
  p.ctab = static_cast<const T*>(q.ctab);
  p.wgt = static_cast<const T*>(q.wgt);
  p.n_x = q.n_x;
  p.n_cells = q.n_cells;
  p.rows = q.rows;
  p.n_terms = q.n_terms;
  p.mass_only = q.mass_only;
  p.aniso = 0;
  for (int d = 0; d < 3; ++d) {
    p.cells[d] = q.cells[d];
    p.nn[d] = q.nn[d];
    p.ratio[d] = (T)q.ratio[d];
    p.aniso |= d > 0 && d < dim && q.ratio[d] != 1.0;
  }
  fill_line_consts(k, p.lk);
  const int nq = k + 1, nqd = dim == 2 ? nq * nq : nq * nq * nq;
  for (int i = 0; i < nt; ++i) p.tb[i] = (T)(q.sign * q.tb[i]);
  for (int i = 0; i < nqd * nt * nt; ++i) p.amq[i] = (T)q.amq[i];
  const dim3 grid((q.n_cells + 31) / 32, (q.rows + kDiagRows - 1) / kDiagRows), block(32, kDiagRows);
#define SG_D(D, KK, TT) \
  if (dim == D && k == KK && nt == TT) { diag_apply<A, D, KK, TT><<<grid, block, 0, s>>>(p); return cudaGetLastError(); }
  SG_D(2, 1, 1) SG_D(2, 1, 2) SG_D(2, 1, 3) SG_D(2, 1, 4)
  SG_D(2, 2, 1) SG_D(2, 2, 2) SG_D(2, 2, 3) SG_D(2, 2, 4)
  SG_D(2, 3, 1) SG_D(2, 3, 2) SG_D(2, 3, 3) SG_D(2, 3, 4)
  SG_D(3, 1, 1) SG_D(3, 1, 2) SG_D(3, 2, 1) SG_D(3, 2, 2)
#undef SG_D
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_diag_apply(int precision, int dim, int k, int nt, const DiagParams& q, cudaStream_t s) {
  return precision == kPrecF32 ? launch<F32>(dim, k, nt, q, s) : launch<F64>(dim, k, nt, q, s);
}

cudaError_t diag_coefficients(int precision, const HostProblem& hp, const double* d_ctab, const std::vector<int>& used,
                              void** out, cudaStream_t s) {
  const int nq = hp.k + 1, nqd = hp.dim == 2 ? nq * nq : nq * nq * nq;
  const size_t n = used.size() * nqd * (size_t)hp.n_cells;
  int* d_used = nullptr;
  cudaError_t e = cudaMalloc(out, std::max<size_t>(1, n) * (precision == kPrecF32 ? 4 : 8));
  if (e == cudaSuccess) e = cudaMalloc(&d_used, std::max<size_t>(1, used.size()) * sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_used, used.data(), used.size() * sizeof(int), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && n > 0) {
    const int grid = (int)std::min<size_t>((n + 255) / 256, (size_t)sm_count() * 16);
    if (precision == kPrecF32)
      diag_table<float><<<grid, 256, 0, s>>>(d_ctab, static_cast<float*>(*out), d_used, (int)used.size(), hp.n_terms, nqd,
                                             (int)hp.n_cells, grad_weight(hp.k));
    else
      diag_table<double><<<grid, 256, 0, s>>>(d_ctab, static_cast<double*>(*out), d_used, (int)used.size(), hp.n_terms,
                                              nqd, (int)hp.n_cells, grad_weight(hp.k));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(d_used);
  return e;
}

}  // namespace sg

SG_BOUNDS_FETCH(bounds_fetch_diag)
