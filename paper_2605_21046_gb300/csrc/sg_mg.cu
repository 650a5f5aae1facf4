// Block-Jacobi geometric-multigrid preconditioner of the SG slab system
// (paper, Sec. 3.5, remark on the algebraic solver): every chaos mode alpha is
// preconditioned by one V-cycle of its diagonal block
//     A_alpha = A_t (x) M_x + sum_mu [G_mu]_{alpha alpha} B_t (x) K_mu,
// with a space-time Vanka patch smoother.  All N_xi * N_t vectors go through
// the V-cycle together, so one launch smooths every mode.  A level residual is
// the row-diagonal apply with per-row weights [G_mu]_{alpha alpha} (sg_diag.cu)
// or the SG cell kernel with the diagonal coupling table.
//
// Levels halve the cells per direction while every count is even and > 2;
// coefficients are re-evaluated on every level (a per-cell scale is averaged
// over the children).  Smoother: additive Vanka, one patch per cell = its
// interior nodes x all time nodes, patch matrix = principal submatrix of the
// level block operator (summed from the element matrices of the neighbouring
// cells), exact dense inverse, damping omega, corrections divided by the
// number of patches that hold the node; nu pre- and nu post-smoothing steps.
// Transfer: canonical Q_k interpolation P (tensor product of 1D tables,
// Dirichlet rows and columns removed), restriction P^T.  Coarsest level:
// dense inverse of the interior block.  Dirichlet rows are the identity on
// every level.  The whole V-cycle is captured once into a CUDA graph.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <map>
#include <type_traits>

#include "sg_bounds.h"
#include "sg_internal.h"
#include "sg_vec.cuh"

namespace sg {

void fill_apply_params(const HostProblem& hp, const LaunchShape& ls, const void* ctab,
                       const int* grow, const int* gcol, const int* gterm, const double* gval,
                       const int* perm, const void* x, void* y, int transpose, ApplyParams& p);
cudaError_t prepare_apply_kernel(int precision, int dim, int k, int n_t, size_t smem);

namespace {

// ------------------------------------------------------------------ kernels
template <typename S, typename D>
__global__ void mg_convert(const S* __restrict__ a, D* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = (D)a[i];
}

// Additive Vanka step: x += omega / mult * inv(patch) * r_patch for every
// (cell, alpha), patch = the cell's nodes x all time nodes (Dirichlet rows
// skipped), mult = number of cells that hold the node.
//
// Per (cell, diagonal class) the step is a dense product Z = inv * R with
// inv the NP x NP patch inverse and R the patch values of the class's modes
// (NP x modes).  Persistent CTAs walk units (a chunk of C cells consecutive
// in x, a tile of mode blocks) in two pipeline stages: while one unit is
// computed, the next unit's data land in the other stage by asynchronous
// copies (cp.async):
//   * the chunk's inverses of the unit's first class (contiguous in memory:
//     cells consecutive in x), 16 bytes at a time, rows padded to an odd
//     number of 16-byte pieces so that the rows of 8 consecutive threads fall
//     in different banks;
//   * r on the chunk's node grid as [time node][node][slot], one value per
//     copy, slots = the tile's modes grouped by class in blocks of kVankaVB
//     (padding and Dirichlet nodes stored as zero).
// Every thread accumulates a register block of kVankaR patch rows x one block
// of kVankaVB slots: per patch column one broadcast 16-byte load of the patch
// values and kVankaR x kVankaVB FMAs, the inverse rows read 16 bytes at a time
// (bf16 widened in registers).  The damped, multiplicity-weighted corrections
// of neighbouring cells are summed in shared memory and added into x once per
// node with reductions (no thread waits on a load of x).  The staging and the
// write-back walk their (slot, node) pairs with per-thread increments instead
// of divisions; further classes of a tile are staged synchronously.
// Inverses are stored [class][cell][NP][npp] in W (double, float or bf16;
// npp = NP rounded up to 8).
constexpr int kVankaVB = 4;      // slots per mode block (modes of one class); slots per thread
constexpr int kVankaR = 4;       // patch rows per thread

template <typename T>
struct VankaParams {
  const T* r;
  T* x;
  const void* inv;
  const int* blk_cls;       // [n_blk] class of every mode block
  const int* blk_alpha;     // [n_blk][kVankaVB] modes, -1 padded
  int n_blk, chunk, npp;
  int tile_blocks, n_tiles; // mode blocks per tile
  long long n_x, n_cells;
  long long n_vec_x;        // values per vector set (rows x time nodes x nodes; bounds checks)
  long long inv_count;      // stored inverse values (bounds checks)
  size_t smem_values;       // bytes below the index tables in shared memory (bounds checks)
  int cells[3], nn[3];
  T omega;
};

// 16-byte pieces per shared-memory row of a staged inverse of NP values of
// `bytes` each: the pieces the row needs, made odd (bank spread).
__host__ __device__ constexpr int vanka_row_pieces(int np, int bytes) {
  return ((np * bytes + 15) / 16) % 2 == 0 ? (np * bytes + 15) / 16 + 1 : (np * bytes + 15) / 16;
}
// Slots per node in shared memory for a tile of `blocks` mode blocks.
__host__ __device__ constexpr int vanka_slots(int blocks) { return blocks * kVankaVB; }

template <typename T>
struct Vec4;
template <>
struct Vec4<float> {
  __device__ static void load(const float* p, float* o) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  }
};
template <>
struct Vec4<double> {
  __device__ static void load(const double* p, double* o) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
  }
};

// One 16-byte piece of an inverse row, widened to T.
template <typename T, typename W>
struct Piece16;
template <>
struct Piece16<float, float> {
  static constexpr int n = 4;
  __device__ static void load(const float* p, float* o) { Vec4<float>::load(p, o); }
};
template <>
struct Piece16<double, double> {
  static constexpr int n = 2;
  __device__ static void load(const double* p, double* o) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    o[0] = a.x; o[1] = a.y;
  }
};
template <>
struct Piece16<float, __nv_bfloat16> {
  static constexpr int n = 8;
  __device__ static void load(const __nv_bfloat16* p, float* o) {
    const uint4 u = *reinterpret_cast<const uint4*>(p);
    const unsigned int w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o[2 * k] = __uint_as_float(w[k] << 16);
      o[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
  }
};

template <typename T, typename W>
__device__ __forceinline__ T widen(W w) { return (T)w; }
template <>
__device__ __forceinline__ float widen<float, __nv_bfloat16>(__nv_bfloat16 w) { return __bfloat162float(w); }

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned int sa = (unsigned int)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// A copy of sizeof(T) bytes (4 or 8) from global to shared memory, asynchronous.
template <typename T>
__device__ __forceinline__ void cp_async_val(T* smem, const T* gmem) {
  const unsigned int sa = (unsigned int)__cvta_generic_to_shared(smem);
  if constexpr (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prior1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// One unit of work (a chunk of cells and a tile of mode blocks).
struct VankaUnit {
  int cx0, cy, cz, nc, b0, nb;
  long long cell0;
};

template <typename T, typename W, int DIM, int K, int NT, bool TRANS>
__global__ void __launch_bounds__(256, 2) mg_vanka(const VankaParams<T> p) {
  constexpr int N = K + 1;
  constexpr int NKD = DIM == 2 ? N * N : N * N * N;
  constexpr int NP = NT * NKD;
  constexpr int R = kVankaR, VB = kVankaVB;
  constexpr int NRG = (NP + R - 1) / R;                        // row groups per cell
  constexpr int RP = vanka_row_pieces(NP, (int)sizeof(W));     // 16-byte pieces per staged row
  constexpr int RW = RP * 16 / (int)sizeof(W);                 // values per staged row
  constexpr int QV = Piece16<T, W>::n;                         // values per piece
  constexpr int NQC = (NP + QV - 1) / QV;                      // pieces a row product reads
  constexpr int LYZ = DIM == 2 ? N : N * N;                    // nodes across y (and z)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int C = p.chunk;
  const int LX = C * K + 1;                                    // chunk nodes along x
  const int LN = LX * LYZ;
  const int SL = vanka_slots(p.tile_blocks);
  const int E = NT * LN;                                       // (time node, node) pairs per slot
  // shared memory: the corrections, then two stages of (r, inverses, node and slot tables)
  // stage b: r at Rl0 + b E SL, inverses at Is0 + b C NP RW, node table at
  // Gn0 + b LN, slot table at Sm0 + b SL
  T* Zc = reinterpret_cast<T*>(smem_raw);                      // [NT][LN][SL]
  T* Rl0 = Zc + (size_t)E * SL;                                // 2 x [NT][LN][SL]
  W* Is0 = reinterpret_cast<W*>(Zc + (size_t)3 * E * SL);      // 2 x [C][NP][RW] inverses of one class
  int* Gn0 = reinterpret_cast<int*>(Is0 + (size_t)2 * C * NP * RW);   // 2 x [LN] global node, -1 outside / boundary
  int* Sm0 = Gn0 + 2 * LN;                                     // 2 x [SL] mode of every slot, -1 padding
  const size_t rl_stage = (size_t)E * SL, is_stage = (size_t)C * NP * RW;
  const W* inv = static_cast<const W*>(p.inv);
  const int nnx = p.nn[0], nny = p.nn[1], nnz_ = p.nn[2];
  const int cpr = (p.cells[0] + C - 1) / C;                    // chunks per row of cells
  const long long n_chunks = (long long)cpr * p.cells[1] * p.cells[2];
  const long long n_units = n_chunks * p.n_tiles;
  // (slot, pair) walk of the gather and the write-back: start and increments
  const int w_sl0 = tid / E, w_e0 = tid - (tid / E) * E;
  const int w_dq = nthr / E, w_dr = nthr - (nthr / E) * E;
  const int LNSL = LN * SL, LXSL = LX * SL;

  // 32-bit index arithmetic (units and cells stay below 2^31; 64-bit
  // divisions would cost more than the rest of the bookkeeping)
  auto decode = [&](long long unit, VankaUnit& U) {
    const unsigned int uu = (unsigned int)unit, nch = (unsigned int)n_chunks;
    const unsigned int ch = uu % nch;
    const int tile = (int)(uu / nch);
    U.b0 = tile * p.tile_blocks;
    U.nb = min(p.tile_blocks, p.n_blk - U.b0);
    U.cx0 = (int)(ch % (unsigned int)cpr) * C;
    const unsigned int row = ch / (unsigned int)cpr;
    U.cy = (int)(row % (unsigned int)p.cells[1]);
    U.cz = (int)(row / (unsigned int)p.cells[1]);
    U.nc = min(C, p.cells[0] - U.cx0);
    U.cell0 = ((long long)U.cz * p.cells[1] + U.cy) * p.cells[0] + U.cx0;
  };
  // the global index of every node of the unit's chunk (-1 outside the mesh or
  // on the boundary) and the mode of every slot
  auto tables = [&](const VankaUnit& U, int* Gn, int* Sm) {
    const int lxn = U.nc * K + 1;
    for (int ln = tid; ln < LN; ln += nthr) {
      const int lx = ln % LX, lyz = ln / LX;
      const int ly = lyz % N, lz = DIM == 3 ? lyz / N : 0;
      int node = -1;
      if (lx < lxn) {
        const int gx = U.cx0 * K + lx, gy = U.cy * K + ly, gz = DIM == 3 ? U.cz * K + lz : 0;
        bool in = gx > 0 && gx < nnx - 1 && gy > 0 && gy < nny - 1;
        if (DIM == 3) in = in && gz > 0 && gz < nnz_ - 1;
        if (in) node = (int)(((long long)gz * nny + gy) * nnx + gx);
      }
      Gn[ln] = node;
    }
    for (int sl = tid; sl < SL; sl += nthr) Sm[sl] = sl < U.nb * VB ? p.blk_alpha[U.b0 * VB + sl] : -1;
  };
  // asynchronous copies of the chunk's inverses of class `cls` (contiguous in
  // memory: cells consecutive in x) in 16-byte pieces
  auto stage_inverses = [&](const VankaUnit& U, int cls, W* Is, int stage_base) {
    const long long ibeg = ((long long)cls * p.n_cells + U.cell0) * NP * p.npp;
    for (int idx = tid; idx < U.nc * NP * RP; idx += nthr) {
      const int rr = idx / RP, piece = idx - rr * RP;
      if (piece * 16 >= p.npp * (int)sizeof(W)) continue;     // the padding piece of a row
      const long long g = ibeg + (long long)rr * p.npp + piece * (16 / (int)sizeof(W));
      if (!SG_IN(g + 16 / (int)sizeof(W) - 1, p.inv_count, 202)) continue;
      if (!SG_IN((size_t)stage_base + ((size_t)rr * RW + piece * (16 / sizeof(W))) * sizeof(W), p.smem_values, 203))
        continue;
      cp_async16(Is + (size_t)rr * RW + piece * (16 / (int)sizeof(W)), inv + g);
    }
  };
  // asynchronous gather of r on the chunk's node grid (slot-major, node
  // fastest); padding slots and Dirichlet nodes are stored as zero
  auto stage_r = [&](T* Rl, const int* Gn, const int* Sm) {
    int sl = w_sl0, e = w_e0;
    while (sl < SL) {
      int i = 0;
#pragma unroll
      for (int j = 1; j < NT; ++j) i += e >= j * LN;
      const int ln = e - i * LN;
      const int mode = Sm[sl], node = Gn[ln];
      const long long gi = ((long long)mode * NT + i) * p.n_x + node;
      T* dst = Rl + (size_t)e * SL + sl;
      if (mode >= 0 && node >= 0 && SG_IN(gi, p.n_vec_x, 201)) cp_async_val(dst, p.r + gi);
      else *dst = T(0);
      e += w_dr;
      sl += w_dq;
      if (e >= E) { e -= E; ++sl; }
    }
  };

  for (int i = tid; i < E * SL; i += nthr) Zc[i] = T(0);
  long long u = blockIdx.x;
  int buf = 0;
  VankaUnit cur, nxt;
  if (u < n_units) {
    decode(u, cur);
    tables(cur, Gn0, Sm0);
  }
  __syncthreads();
  if (u < n_units) {
    stage_inverses(cur, p.blk_cls[cur.b0], Is0, (int)((size_t)3 * E * SL * sizeof(T)));
    stage_r(Rl0, Gn0, Sm0);
  }
  cp_async_commit();
  for (; u < n_units; u += gridDim.x, buf ^= 1) {
    // the next unit's tables and copies go to the other stage while this one computes
    const long long un = u + gridDim.x;
    const bool has_next = un < n_units;
    __syncthreads();                                           // the other stage is free
    if (has_next) {
      decode(un, nxt);
      tables(nxt, Gn0 + (buf ^ 1) * LN, Sm0 + (buf ^ 1) * SL);
    }
    __syncthreads();
    if (has_next) {
      stage_inverses(nxt, p.blk_cls[nxt.b0], Is0 + (buf ^ 1) * is_stage,
                     (int)((size_t)3 * E * SL * sizeof(T) + (size_t)(buf ^ 1) * is_stage * sizeof(W)));
      stage_r(Rl0 + (buf ^ 1) * rl_stage, Gn0 + (buf ^ 1) * LN, Sm0 + (buf ^ 1) * SL);
    }
    cp_async_commit();
    cp_async_wait_prior1();                                    // this unit's copies have landed
    __syncthreads();
    const T* Rl = Rl0 + buf * rl_stage;
    W* Is = Is0 + buf * is_stage;
    const int* Gn = Gn0 + buf * LN;
    const int* Sm = Sm0 + buf * SL;
    // runs of consecutive blocks of one class
    for (int rb = 0; rb < cur.nb;) {
      const int cls = p.blk_cls[cur.b0 + rb];
      int re = rb + 1;
      while (re < cur.nb && p.blk_cls[cur.b0 + re] == cls) ++re;
      const int nbr = re - rb;
      const int sa = rb * VB;
      if (rb > 0) {
        // a further class of this tile: its inverses, synchronously
        __syncthreads();
        stage_inverses(cur, cls, Is, (int)((size_t)3 * E * SL * sizeof(T) + (size_t)buf * is_stage * sizeof(W)));
        cp_async_wait_all();
        __syncthreads();
      }
      const int items = cur.nc * NRG * nbr;
      for (int it = tid; it < items; it += nthr) {
        const int rg = it % NRG, cb = it / NRG;
        const int bl = cb % nbr, c = cb / nbr;
        const int s0 = sa + bl * VB;
        int rows[R];
#pragma unroll
        for (int k = 0; k < R; ++k) rows[k] = rg + k * NRG;
        T acc[R][VB];
#pragma unroll
        for (int k = 0; k < R; ++k)
#pragma unroll
          for (int uu = 0; uu < VB; ++uu) acc[k][uu] = T(0);
        const T* pb = Rl + (size_t)(c * K) * SL + s0;
        const W* ib = Is + (size_t)c * NP * RW;
        if constexpr (!TRANS) {
          const W* ir[R];
#pragma unroll
          for (int k = 0; k < R; ++k) ir[k] = ib + (size_t)min(rows[k], NP - 1) * RW;
#pragma unroll
          for (int qc = 0; qc < NQC; ++qc) {
            T w[R][QV];
#pragma unroll
            for (int k = 0; k < R; ++k) Piece16<T, W>::load(ir[k] + qc * QV, w[k]);
#pragma unroll
            for (int j = 0; j < QV; ++j) {
              const int q = qc * QV + j;
              if (q >= NP) break;
              const int iq = q / NKD, aq = q - iq * NKD;
              const int ax = aq % N, ayz = aq / N;
              T v[VB];
              Vec4<T>::load(pb + iq * LNSL + ayz * LXSL + ax * SL, v);
#pragma unroll
              for (int k = 0; k < R; ++k)
#pragma unroll
                for (int uu = 0; uu < VB; ++uu) acc[k][uu] = fma(w[k][j], v[uu], acc[k][uu]);
            }
          }
        } else {
#pragma unroll 6
          for (int q = 0; q < NP; ++q) {
            const int iq = q / NKD, aq = q - iq * NKD;
            const int ax = aq % N, ayz = aq / N;
            T v[VB];
            Vec4<T>::load(pb + iq * LNSL + ayz * LXSL + ax * SL, v);
            const W* iqrow = ib + (size_t)q * RW;
#pragma unroll
            for (int k = 0; k < R; ++k) {
              const T w = widen<T, W>(iqrow[min(rows[k], NP - 1)]);
#pragma unroll
              for (int uu = 0; uu < VB; ++uu) acc[k][uu] = fma(w, v[uu], acc[k][uu]);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < R; ++k) {
          const int rho = rows[k];
          if (rho >= NP) continue;
          const int i = rho / NKD, a = rho - i * NKD;
          const int ax = a % N, ay = (a / N) % N, az = DIM == 3 ? a / (N * N) : 0;
          const int lna = c * K + ax + LX * (ay + (DIM == 3 ? N * az : 0));
          if (Gn[lna] < 0) continue;                 // Dirichlet row
          // patches sharing the node (cell corners and faces: the local coordinate is 0 or K)
          const int mult = (ax % K == 0 ? 2 : 1) * (ay % K == 0 ? 2 : 1) * (DIM == 3 && az % K == 0 ? 2 : 1);
          const T sc = p.omega / T(mult);
          const size_t zo = (size_t)(i * LN + lna) * SL + s0;
#pragma unroll
          for (int uu = 0; uu < VB; ++uu)
            if (SG_IN(zo + uu, (size_t)E * SL, 204)) atomicAdd(Zc + zo + uu, sc * acc[k][uu]);
        }
      }
      rb = re;
    }
    __syncthreads();
    // add the corrections into x (reductions: no thread waits on a load of x)
    // and clear them for the next unit
    {
      const int SLW = cur.nb * VB;
      int sl = w_sl0, e = w_e0;
      while (sl < SLW) {
        int i = 0;
#pragma unroll
        for (int j = 1; j < NT; ++j) i += e >= j * LN;
        const int ln = e - i * LN;
        const int mode = Sm[sl], node = Gn[ln];
        T* z = Zc + (size_t)e * SL + sl;
        if (mode >= 0 && node >= 0) {
          const long long gi = ((long long)mode * NT + i) * p.n_x + node;
          if (SG_IN(gi, p.n_vec_x, 205)) atomicAdd(p.x + gi, *z);
        }
        *z = T(0);
        e += w_dr;
        sl += w_dq;
        if (e >= E) { e -= E; ++sl; }
      }
    }
    cur = nxt;
  }
  cp_async_wait_all();
}

// Grid transfers, one launch each: the d separable 1D passes of a tile of one
// plane of output nodes, in shared memory.  A block takes one vector, one
// plane along z (3D) and a tile of rows along y: it combines the planes of its
// z list while loading, then does the x and y passes (restriction) or the y
// and x passes (interpolation) between two shared arrays, so the intermediate
// arrays never reach memory.  Bound by L2 and HBM traffic: a fine plane is
// read for every coarse plane that lists it (2.5 times on average for Q2,
// mostly from L2).  The 1D lists (coarse node <- fine nodes, fine node <-
// coarse nodes) are padded to W entries per output (weight 0, an index the
// output's neighbours use) and stored entry-major; a thread keeps one output
// column, with its list in registers, and walks the rows.
//
// LARGE: the block takes a tile of columns along x as well, with its own
// input window, and its place comes from a 1D grid, so no length of a row and
// no count of rows or planes is too large.  build_transfers takes it only where
// the other form cannot be launched: whole rows need no division per value,
// and each further tile of columns loads a halo of its own.
//
// The vectors that the next kernels reduce into are preset here, where their
// nodes are written anyway: restriction also writes the coarse level's start
// (x = 0, r = b; b vanishes on the boundary), interpolation r = b inside and 0
// on the boundary for the residual that follows.
constexpr int kAxisMax = 16;  // entries of one output of a 1D transfer list, at most (4k + 1 for k <= 3)
constexpr int kTransferThreads = 256;
constexpr int kTransferBatch = 4;   // elements of a thread whose loads are in flight together

template <typename T>
struct TransferParams {
  const T* in;              // restriction: fine residual; interpolation: coarse correction
  const T* b;               // interpolation: fine right-hand side
  T *out, *x, *r;           // restriction: b, x, r of the coarse level; interpolation: fine x (out), r
  const int* idx[3];
  const T* w[3];
  const int *range, *range_x;   // first and number of input rows (columns) of every tile
  long long n_in, n_out;    // nodes per vector
  int ni[3], no[3];         // nodes per direction of the input and output grids
  int tile, max_rows, z;    // output rows per tile, most input rows of one; 3D
  int tile_x, max_cols;     // output columns per tile, most input columns of one (LARGE)
  unsigned n_vec, planes, tiles;   // vectors, planes and tiles of rows (LARGE)
  int cb_in, cb_out;        // columns a pass takes at a time, of the input and output grids
  long long lim_in, lim_out;   // values of the vectors (bounds checks)
};

// The part of a transfer that a block takes: vector, plane, output rows
// [j0, j0 + nj) and columns [i0, i0 + ni), input rows [lo, lo + cnt) and
// columns [lox, lox + cntx).
struct TransferTile {
  int v, jz, j0, nj, i0, ni, lo, cnt, lox, cntx;
};
template <typename T, bool LARGE>
__device__ __forceinline__ TransferTile transfer_tile(const TransferParams<T>& p) {
  TransferTile t;
  unsigned ty = blockIdx.z;
  if constexpr (LARGE) {
    unsigned b = blockIdx.x;
    t.v = (int)(b % p.n_vec);
    b /= p.n_vec;
    t.jz = (int)(b % p.planes);
    b /= p.planes;
    ty = b % p.tiles;
    b /= p.tiles;
    t.i0 = (int)b * p.tile_x;
    t.ni = min(p.tile_x, p.no[0] - t.i0);
    t.lox = __ldg(p.range_x + 2 * b);
    t.cntx = __ldg(p.range_x + 2 * b + 1);
  } else {
    t.v = (int)blockIdx.x;
    t.jz = (int)blockIdx.y;
    t.i0 = t.lox = 0;
    t.ni = p.no[0];
    t.cntx = p.ni[0];
  }
  t.j0 = (int)ty * p.tile;
  t.nj = min(p.tile, p.no[1] - t.j0);
  t.lo = __ldg(p.range + 2 * ty);
  t.cnt = __ldg(p.range + 2 * ty + 1);
  return t;
}

// The tile's input rows, combined along z, into S0 (row pitch cntx).
template <typename T, int W, bool LARGE>
__device__ __forceinline__ void transfer_load(const TransferParams<T>& p, const TransferTile& t, T* S0) {
  const int jz = t.jz;
  const long long v_in = (long long)t.v * p.n_in;
  const T* src = p.in + v_in;
  const int n = t.cnt * t.cntx, off = t.lo * p.ni[0] + t.lox;
  auto at = [&](int i) {   // of the tile's value i, from its first one
    if constexpr (LARGE) return (i / t.cntx) * p.ni[0] + i % t.cntx;
    else return i;
  };
  if (p.z) {
    const int plane = p.ni[0] * p.ni[1];
    const T* pl[W];
    T wz[W];
    int m = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) {
      const T wk = __ldg(p.w[2] + k * p.no[2] + jz);
      wz[k] = wk;
      pl[k] = src + (long long)__ldg(p.idx[2] + k * p.no[2] + jz) * plane + off;
      if (wk != T(0)) m = k + 1;
    }
    for (int i0 = threadIdx.x; i0 < n; i0 += kTransferBatch * kTransferThreads) {
      T s[kTransferBatch];
#pragma unroll
      for (int g = 0; g < kTransferBatch; ++g) s[g] = T(0);
#pragma unroll
      for (int k = 0; k < W; ++k) {
        if (k >= m) break;
#pragma unroll
        for (int g = 0; g < kTransferBatch; ++g) {
          const int i = i0 + g * kTransferThreads;
          if (i < n && SG_IN(pl[k] - p.in + at(i), p.lim_in, 501)) s[g] = fma(wz[k], __ldg(pl[k] + at(i)), s[g]);
        }
      }
#pragma unroll
      for (int g = 0; g < kTransferBatch; ++g)
        if (i0 + g * kTransferThreads < n) S0[i0 + g * kTransferThreads] = s[g];
    }
  } else {
    for (int i0 = threadIdx.x; i0 < n; i0 += kTransferBatch * kTransferThreads) {
      T s[kTransferBatch];
#pragma unroll
      for (int g = 0; g < kTransferBatch; ++g) {
        const int i = i0 + g * kTransferThreads;
        s[g] = i < n && SG_IN(v_in + off + at(i), p.lim_in, 501) ? __ldg(src + off + at(i)) : T(0);
      }
#pragma unroll
      for (int g = 0; g < kTransferBatch; ++g)
        if (i0 + g * kTransferThreads < n) S0[i0 + g * kTransferThreads] = s[g];
    }
  }
}

// One 1D pass along x or y of `rows` output rows: DIR 0 out[row][c] = sum_k w in[row][idx[o0 + c] - lo],
// DIR 1 out[row][c] = sum_k w in[idx[o0 + row] - lo][c]; put(row, column, value).  n_in input rows.
template <typename T, int W, int DIR, class Put>
__device__ __forceinline__ void transfer_pass(const T* in, int pitch, int cols, int cb, int rows, const int* idx,
                                              const T* w, int n_list, int o0, int lo, int n_in, Put put) {
  const int par = kTransferThreads / cb;                       // cb columns x par rows at a time
  const int c0 = threadIdx.x % cb, r0 = threadIdx.x / cb;
  if (r0 >= par) return;
  for (int c = c0; c < cols; c += cb) {
    if constexpr (DIR == 0) {
      int at[W];
      T wt[W];
#pragma unroll
      for (int k = 0; k < W; ++k) {
        at[k] = __ldg(idx + k * n_list + o0 + c) - lo;
        wt[k] = __ldg(w + k * n_list + o0 + c);
      }
      for (int r = r0; r < rows; r += par) {
        T s = T(0);
#pragma unroll
        for (int k = 0; k < W; ++k)
          if (SG_IN(at[k], pitch, 504)) s = fma(wt[k], in[r * pitch + at[k]], s);
        put(r, c, s);
      }
    } else {
      for (int r = r0; r < rows; r += par) {
        T s = T(0);
#pragma unroll
        for (int k = 0; k < W; ++k) {
          const int at = __ldg(idx + k * n_list + o0 + r) - lo;
          if (SG_IN(at, n_in, 505)) s = fma(__ldg(w + k * n_list + o0 + r), in[at * pitch + c], s);
        }
        put(r, c, s);
      }
    }
  }
}

template <typename T, int W, bool LARGE>
__global__ void __launch_bounds__(kTransferThreads) mg_restrict(const TransferParams<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TransferTile t = transfer_tile<T, LARGE>(p);
  T* S0 = reinterpret_cast<T*>(smem_raw);                       // [max_rows][fine columns]
  T* S1 = S0 + (size_t)p.max_rows * (LARGE ? p.max_cols : p.ni[0]);   // [max_rows][coarse columns]
  transfer_load<T, W, LARGE>(p, t, S0);
  __syncthreads();
  const int ncx = p.no[0], nc = LARGE ? t.ni : ncx;
  transfer_pass<T, W, 0>(S0, t.cntx, nc, p.cb_out, t.cnt, p.idx[0], p.w[0], ncx, t.i0, t.lox, t.cnt,
                         [&](int r, int c, T v) { S1[r * nc + c] = v; });
  __syncthreads();
  const long long o0 = (long long)t.v * p.n_out + ((long long)t.jz * p.no[1] + t.j0) * ncx + t.i0;
  transfer_pass<T, W, 1>(S1, nc, nc, p.cb_out, t.nj, p.idx[1], p.w[1], p.no[1], t.j0, t.lo, t.cnt, [&](int r, int c, T v) {
    const long long o = o0 + (long long)r * ncx + c;
    if (!SG_IN(o, p.lim_out, 502)) return;
    p.out[o] = v;
    p.x[o] = T(0);
    p.r[o] = v;
  });
}

template <typename T, int W, bool LARGE>
__global__ void __launch_bounds__(kTransferThreads) mg_prolong(const TransferParams<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TransferTile t = transfer_tile<T, LARGE>(p);
  const int most = LARGE ? p.max_cols : p.ni[0];
  T* S0 = reinterpret_cast<T*>(smem_raw);                       // [max_rows][coarse columns]
  T* S1 = S0 + (size_t)p.max_rows * most;                       // [tile][coarse columns]
  T* S2 = S1 + (size_t)p.tile * most;                           // [tile][fine columns]
  transfer_load<T, W, LARGE>(p, t, S0);
  __syncthreads();
  const int nfx = p.no[0];
  transfer_pass<T, W, 1>(S0, t.cntx, t.cntx, p.cb_in, t.nj, p.idx[1], p.w[1], p.no[1], t.j0, t.lo, t.cnt,
                         [&](int r, int c, T v) { S1[r * t.cntx + c] = v; });
  __syncthreads();
  transfer_pass<T, W, 0>(S1, t.cntx, t.ni, p.cb_out, t.nj, p.idx[0], p.w[0], nfx, t.i0, t.lox, t.nj,
                         [&](int r, int c, T v) { S2[r * t.ni + c] = v; });
  __syncthreads();
  // x += S2, r = b inside (whole rows of a tile are contiguous), with the loads of a batch in flight together
  const long long o0 = (long long)t.v * p.n_out + ((long long)t.jz * p.no[1] + t.j0) * nfx + t.i0;
  const bool edge_z = p.z && (t.jz == 0 || t.jz == p.no[2] - 1);
  const int n = t.nj * t.ni;
  auto at = [&](int i) {
    if constexpr (LARGE) return o0 + (long long)(i / t.ni) * nfx + i % t.ni;
    else return o0 + i;
  };
  for (int i0 = threadIdx.x; i0 < n; i0 += kTransferBatch * kTransferThreads) {
    T xv[kTransferBatch], bv[kTransferBatch];
#pragma unroll
    for (int g = 0; g < kTransferBatch; ++g) {
      const int i = i0 + g * kTransferThreads;
      const bool in = i < n && SG_IN(at(i), p.lim_out, 503);
      xv[g] = in ? p.out[at(i)] : T(0);
      bv[g] = in ? __ldg(p.b + at(i)) : T(0);
    }
#pragma unroll
    for (int g = 0; g < kTransferBatch; ++g) {
      const int i = i0 + g * kTransferThreads;
      if (i >= n || !SG_IN(at(i), p.lim_out, 503)) continue;
      const int r = i / t.ni, c = t.i0 + i - r * t.ni, jy = t.j0 + r;
      const bool bd = edge_z || jy == 0 || jy == p.no[1] - 1 || c == 0 || c == nfx - 1;
      p.out[at(i)] = xv[g] + S2[i];
      p.r[at(i)] = bd ? T(0) : bv[g];
    }
  }
}

// Coarsest level: x[inner] = inv(C_class) b[inner] for every chaos mode.  A
// block takes 8 rows of the inverse (a warp each; columns for the transposed
// cycle) and the kCoarseModes modes of one mode block, all of one class, whose
// right-hand sides it stages in shared memory: a row is read once for four
// modes, coalesced, and reduced with shuffles.  Latency bound (450 unknowns,
// 35 modes: 10 us with a mode per block).
constexpr int kCoarseModes = kVankaVB;
constexpr int kCoarseRows = 8;

template <typename T>
__global__ void __launch_bounds__(32 * kCoarseRows) mg_coarse(const T* __restrict__ b, T* __restrict__ x,
                                                              const T* __restrict__ inv, const int* __restrict__ blk_cls,
                                                              const int* __restrict__ blk_alpha,
                                                              const long long* __restrict__ inner, int n_int, int n_t,
                                                              long long n_x, int trans, long long lim_vec,
                                                              long long lim_inv) {
  extern __shared__ __align__(16) unsigned char sm[];
  T* bs = reinterpret_cast<T*>(sm);                            // [mode][n_int]
  const int blk = blockIdx.y;
  long long base[kCoarseModes];
#pragma unroll
  for (int u = 0; u < kCoarseModes; ++u) {
    const int m = __ldg(blk_alpha + blk * kCoarseModes + u);
    base[u] = m < 0 ? -1 : (long long)m * n_t * n_x;
  }
  for (int i = threadIdx.x; i < n_int; i += blockDim.x) {
    const long long at = __ldg(inner + i);
#pragma unroll
    for (int u = 0; u < kCoarseModes; ++u) bs[u * n_int + i] = base[u] >= 0 && SG_IN(base[u] + at, lim_vec, 506) ? __ldg(b + base[u] + at) : T(0);
  }
  __syncthreads();
  const T* M = inv + (long long)__ldg(blk_cls + blk) * n_int * n_int;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * kCoarseRows + warp;
  if (i >= n_int) return;
  const T* row = trans ? M + i : M + (long long)i * n_int;
  const long long step = trans ? n_int : 1;
  T s[kCoarseModes] = {};
#pragma unroll 4
  for (int q = lane; q < n_int; q += 32) {
    const T w = SG_IN(row - inv + q * step, lim_inv, 507) ? __ldg(row + q * step) : T(0);
#pragma unroll
    for (int u = 0; u < kCoarseModes; ++u) s[u] = fma(w, bs[u * n_int + q], s[u]);
  }
#pragma unroll
  for (int u = 0; u < kCoarseModes; ++u) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
    const long long at = base[u] + __ldg(inner + i);
    if (lane == 0 && base[u] >= 0 && SG_IN(at, lim_vec, 508)) x[at] = s[u];
  }
}

// ------------------------------------------------------------------ host set-up

int grid_for(long long n, int block) {
  return (int)std::max<long long>(1, std::min<long long>((n + block - 1) / block, sg::sm_count() * 32));
}

// In-place inverse of a dense n x n matrix (Gauss-Jordan, partial pivoting).
bool invert(std::vector<double>& a, int n) {
  std::vector<double> inv(n * (size_t)n, 0.0);
  for (int i = 0; i < n; ++i) inv[(size_t)i * n + i] = 1.0;
  for (int c = 0; c < n; ++c) {
    int piv = c;
    for (int r = c + 1; r < n; ++r)
      if (std::fabs(a[(size_t)r * n + c]) > std::fabs(a[(size_t)piv * n + c])) piv = r;
    if (a[(size_t)piv * n + c] == 0.0) return false;
    if (piv != c)
      for (int k = 0; k < n; ++k) {
        std::swap(a[(size_t)c * n + k], a[(size_t)piv * n + k]);
        std::swap(inv[(size_t)c * n + k], inv[(size_t)piv * n + k]);
      }
    const double d = 1.0 / a[(size_t)c * n + c];
    for (int k = 0; k < n; ++k) {
      a[(size_t)c * n + k] *= d;
      inv[(size_t)c * n + k] *= d;
    }
#pragma omp parallel for schedule(static) if (n >= 256)
    for (int r = 0; r < n; ++r) {
      if (r == c) continue;
      const double f = a[(size_t)r * n + c];
      if (f == 0.0) continue;
      for (int k = 0; k < n; ++k) {
        a[(size_t)r * n + k] -= f * a[(size_t)c * n + k];
        inv[(size_t)r * n + k] -= f * inv[(size_t)c * n + k];
      }
    }
  }
  a.swap(inv);
  return true;
}

// Reference element matrices of a level: mass (cell independent) and, per
// cell, the stiffness with the class coefficient cbar(q) = sum_t diag[t] ctab[t][q].
struct ElementData {
  int nkd = 0, nqd = 0, dim = 2;
  std::vector<double> phi;    // [a][q]
  std::vector<double> grad;   // [d][a][q] reference derivative
  std::vector<double> wJ;     // [q]
  std::vector<double> mass;   // [a][b]
};

ElementData element_data(const HostProblem& hp) {
  ElementData e;
  const int n = hp.k + 1;
  e.dim = hp.dim;
  e.nkd = hp.dim == 2 ? n * n : n * n * n;
  e.nqd = e.nkd;
  e.phi.assign((size_t)e.nkd * e.nqd, 0.0);
  e.grad.assign((size_t)3 * e.nkd * e.nqd, 0.0);
  e.wJ.assign(e.nqd, 0.0);
  double detJ = 1.0;
  for (int d = 0; d < hp.dim; ++d) detJ *= hp.h[d];
  for (int q = 0; q < e.nqd; ++q) {
    const int qi[3] = {q % n, (q / n) % n, q / (n * n)};
    double w = detJ;
    for (int d = 0; d < hp.dim; ++d) w *= hp.wq[qi[d]];
    e.wJ[q] = w;
    for (int a = 0; a < e.nkd; ++a) {
      const int ai[3] = {a % n, (a / n) % n, a / (n * n)};
      double v = 1.0;
      for (int d = 0; d < hp.dim; ++d) v *= hp.S[qi[d] * n + ai[d]];
      e.phi[(size_t)a * e.nqd + q] = v;
      for (int dd = 0; dd < hp.dim; ++dd) {
        double g = 1.0;
        for (int d = 0; d < hp.dim; ++d) g *= d == dd ? hp.dS[qi[d] * n + ai[d]] : hp.S[qi[d] * n + ai[d]];
        e.grad[((size_t)dd * e.nkd + a) * e.nqd + q] = g;
      }
    }
  }
  e.mass.assign((size_t)e.nkd * e.nkd, 0.0);
  for (int a = 0; a < e.nkd; ++a)
    for (int b = 0; b < e.nkd; ++b) {
      double s = 0.0;
      for (int q = 0; q < e.nqd; ++q) s += e.wJ[q] * e.phi[(size_t)a * e.nqd + q] * e.phi[(size_t)b * e.nqd + q];
      e.mass[(size_t)a * e.nkd + b] = s;
    }
  return e;
}

// Element stiffness of cell c for the class coefficient (ctab holds
// w_q |J| a_t / h_0^2; direction d carries (h_0 / h_d)^2).
void element_stiffness(const HostProblem& hp, const ElementData& e, const std::vector<double>& diag,
                       long long c, std::vector<double>& K) {
  std::vector<double> cbar(e.nqd, 0.0);
  for (int t = 0; t < hp.n_terms; ++t) {
    if (diag[t] == 0.0) continue;
    const double* ct = hp.ctab.data() + ((size_t)c * hp.n_terms + t) * e.nqd;
    for (int q = 0; q < e.nqd; ++q) cbar[q] += diag[t] * ct[q];
  }
  double ratio[3];
  for (int d = 0; d < 3; ++d) ratio[d] = d < hp.dim ? (hp.h[0] * hp.h[0]) / (hp.h[d] * hp.h[d]) : 0.0;
  K.assign((size_t)e.nkd * e.nkd, 0.0);
  for (int a = 0; a < e.nkd; ++a)
    for (int b = a; b < e.nkd; ++b) {
      double s = 0.0;
      for (int d = 0; d < hp.dim; ++d) {
        const double* ga = e.grad.data() + ((size_t)d * e.nkd + a) * e.nqd;
        const double* gb = e.grad.data() + ((size_t)d * e.nkd + b) * e.nqd;
        double sd = 0.0;
        for (int q = 0; q < e.nqd; ++q) sd += cbar[q] * ga[q] * gb[q];
        s += ratio[d] * sd;
      }
      K[(size_t)a * e.nkd + b] = s;
      K[(size_t)b * e.nkd + a] = s;
    }
}

void cell_coords(const HostProblem& hp, long long c, int cc[3]) {
  cc[0] = (int)(c % hp.cells[0]);
  cc[1] = (int)((c / hp.cells[0]) % hp.cells[1]);
  cc[2] = (int)(c / ((long long)hp.cells[0] * hp.cells[1]));
}

bool node_interior(const HostProblem& hp, const int g[3]) {
  for (int d = 0; d < hp.dim; ++d)
    if (g[d] <= 0 || g[d] >= hp.nn[d] - 1) return false;
  return true;
}

// Row pitch of the stored patch inverses: np rounded up to 8 values (16-byte
// rows for bf16, float and double).
int vanka_row_pitch(int np) { return (np + 7) / 8 * 8; }

// Coarsest level: the dense interior block of one class.
void coarse_matrix(const HostProblem& hp, const ElementData& e, const std::vector<double>& diag,
                    const std::vector<long long>& node_of, std::vector<double>& out) {
  const int n = hp.k + 1, nkd = e.nkd, nt = hp.n_t;
  const int nin = (int)node_of.size();
  std::vector<int> idx(hp.n_x, -1);
  for (int i = 0; i < nin; ++i) idx[node_of[i]] = i;
  const int N = nt * nin;
  std::vector<double> C((size_t)N * N, 0.0), K;
  for (long long c = 0; c < hp.n_cells; ++c) {
    element_stiffness(hp, e, diag, c, K);
    int cc[3];
    cell_coords(hp, c, cc);
    int g[64];
    for (int a = 0; a < nkd; ++a) {
      const int ai[3] = {a % n, (a / n) % n, a / (n * n)};
      long long gl = 0, stride = 1;
      for (int d = 0; d < hp.dim; ++d) {
        gl += (long long)(cc[d] * hp.k + ai[d]) * stride;
        stride *= hp.nn[d];
      }
      g[a] = idx[gl];
    }
    for (int i = 0; i < nt; ++i)
      for (int a = 0; a < nkd; ++a) {
        if (g[a] < 0) continue;
        for (int j = 0; j < nt; ++j)
          for (int b = 0; b < nkd; ++b) {
            if (g[b] < 0) continue;
            double v = hp.A_hat[i * nt + j] * e.mass[(size_t)a * nkd + b];
            if (i == j) v += hp.tau * hp.B_hat[i * nt + i] * K[(size_t)a * nkd + b];
            C[(size_t)(i * nin + g[a]) * N + j * nin + g[b]] += v;
          }
      }
  }
  out.swap(C);
}

// 1D interpolation table of one direction between a fine and a coarse level.
void transfer_1d(const HostProblem& fine, const HostProblem& coarse, int d, std::vector<int>& pptr,
                 std::vector<int>& pidx, std::vector<double>& pwl, std::vector<int>& rptr, std::vector<int>& ridx,
                 std::vector<double>& rw) {
  std::vector<int> pc;
  std::vector<double> pw;
  const int K = fine.k, n = K + 1;
  const std::vector<double> gll = lobatto_nodes(K);
  const int nf = fine.nn[d], nc = coarse.nn[d];
  pc.assign(nf, 0);
  pw.assign((size_t)nf * n, 0.0);
  std::vector<std::vector<std::pair<int, double>>> cols(nc);
  for (int i = 0; i < nf; ++i) {
    const int cf = std::min(i / K, fine.cells[d] - 1);
    const double pos = cf + gll[i - cf * K];
    const double cpos = 0.5 * pos;
    const int ccell = std::min((int)std::floor(cpos), coarse.cells[d] - 1);
    const double s = cpos - ccell;
    pc[i] = ccell;
    const bool fine_bd = i == 0 || i == nf - 1;
    for (int a = 0; a < n; ++a) {
      const int j = ccell * K + a;
      const bool coarse_bd = j == 0 || j == nc - 1;
      double w = (fine_bd || coarse_bd) ? 0.0 : lagrange(gll, a, s);
      pw[(size_t)i * n + a] = w;
      if (w != 0.0) cols[j].push_back({i, w});
    }
  }
  rptr.assign(nc + 1, 0);
  ridx.clear();
  rw.clear();
  for (int j = 0; j < nc; ++j) {
    for (auto& t : cols[j]) {
      ridx.push_back(t.first);
      rw.push_back(t.second);
    }
    rptr[j + 1] = (int)ridx.size();
  }
  // interpolation lists: fine node i <- coarse nodes pc[i] K + a with nonzero weight
  pptr.assign(nf + 1, 0);
  pidx.clear();
  pwl.clear();
  for (int i = 0; i < nf; ++i) {
    for (int a = 0; a < n; ++a)
      if (pw[(size_t)i * n + a] != 0.0) {
        pidx.push_back(pc[i] * K + a);
        pwl.push_back(pw[(size_t)i * n + a]);
      }
    pptr[i + 1] = (int)pidx.size();
  }
}

template <typename T>
cudaError_t upload_vec(T** dst, const std::vector<T>& src) {
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(dst), std::max<size_t>(1, src.size()) * sizeof(T));
  if (e != cudaSuccess) return e;
  if (!src.empty()) e = cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
  return e;
}

cudaError_t upload_values(void** dst, const std::vector<double>& src, int precision) {
  if (precision == kPrecF32) {
    std::vector<float> f(src.begin(), src.end());
    return upload_vec(reinterpret_cast<float**>(dst), f);
  }
  return upload_vec(reinterpret_cast<double**>(dst), src);
}

// The diagonal (block-Jacobi) coupling table: row alpha keeps its own column.
void diagonal_table(const HostProblem& fine, GTable& g, std::vector<std::vector<double>>& diag_of_row) {
  diag_of_row.assign(fine.n_xi, std::vector<double>(fine.n_terms, 0.0));
  for (int a = 0; a < fine.n_xi; ++a)
    for (int e = fine.g.row[a]; e < fine.g.row[a + 1]; ++e)
      if (fine.g.col[e] == a) diag_of_row[a][fine.g.term[e]] += fine.g.val[e];
  g.row.assign(fine.n_xi + 1, 0);
  g.col.clear();
  g.term.clear();
  g.val.clear();
  for (int a = 0; a < fine.n_xi; ++a) {
    for (int t = 0; t < fine.n_terms; ++t)
      if (diag_of_row[a][t] != 0.0) {
        g.col.push_back(a);
        g.term.push_back(t);
        g.val.push_back(diag_of_row[a][t]);
      }
    g.row[a + 1] = (int)g.col.size();
  }
}

// Averages a per-cell scale over the 2^d children of every coarse cell.
std::vector<double> coarsen_scale(const std::vector<double>& s, const HostProblem& fine) {
  if (s.empty()) return s;
  const int cx = fine.cells[0] / 2, cy = fine.cells[1] / 2, cz = fine.dim == 3 ? fine.cells[2] / 2 : 1;
  std::vector<double> out((size_t)cx * cy * cz, 0.0);
  const int kz = fine.dim == 3 ? 2 : 1;
  const double inv = 1.0 / (4 * kz);
  for (int z = 0; z < cz; ++z)
    for (int y = 0; y < cy; ++y)
      for (int x = 0; x < cx; ++x) {
        double acc = 0.0;
        for (int dz = 0; dz < kz; ++dz)
          for (int dy = 0; dy < 2; ++dy)
            for (int dx = 0; dx < 2; ++dx)
              acc += s[((size_t)(kz * z + dz) * fine.cells[1] + 2 * y + dy) * fine.cells[0] + 2 * x + dx];
        out[((size_t)z * cy + y) * cx + x] = acc * inv;
      }
  return out;
}

template <typename T>
cudaError_t issue_vcycle(MG& mg, int l, cudaStream_t s, int trans);

// r -= A x inside by the row-diagonal apply (r holds b inside and 0 on the boundary)
cudaError_t diag_residual(MG& mg, MGLevel& L, cudaStream_t s, int trans) {
  DiagParams q;
  std::memset(&q, 0, sizeof(q));
  q.x = L.d_x;
  q.y = L.d_r;
  q.ctab = L.d_coef;
  q.wgt = mg.d_wused;
  q.amq = L.amq[trans ? 1 : 0].data();
  q.sign = -1.0;
  q.n_x = L.hp.n_x;
  q.n_cells = (int)L.hp.n_cells;
  q.rows = L.hp.n_xi;
  q.n_terms = (int)mg.used.size();
  for (int d = 0; d < 3; ++d) {
    q.nn[d] = L.hp.nn[d];
    q.cells[d] = L.hp.cells[d];
    q.ratio[d] = d < L.hp.dim ? (L.hp.h[0] * L.hp.h[0]) / (L.hp.h[d] * L.hp.h[d]) : 1.0;
  }
  for (int i = 0; i < L.hp.n_t; ++i) q.tb[i] = L.hp.tau * L.hp.B_hat[i * L.hp.n_t + i];
  return launch_diag_apply(mg.precision, L.hp.dim, L.hp.k, L.hp.n_t, q, s);
}

// r = b - A x in one apply (residual mode: the init kernel writes b minus the
// Dirichlet rows, the cell kernel subtracts).
// `preset`: r already holds b inside and 0 on the boundary.
template <typename T>
cudaError_t residual(MG& mg, int l, cudaStream_t s, int trans, bool preset) {
  MGLevel& L = mg.lv[l];
  if (L.use_diag) {
    // the level operator couples no two rows (block Jacobi): the row-diagonal
    // apply with the weights G_mu[alpha][alpha] (Psi_mu(xi_s) for samples).
    // x = b on the boundary, as on every level, so the Dirichlet rows are 0.
    if (!preset)
      launch_vec_start<T>(static_cast<const T*>(L.d_b), static_cast<const T*>(L.d_x), static_cast<T*>(L.d_r), 4,
                          L.hp.n_xi * L.hp.n_t, L.hp.n_x, L.hp.nn, L.hp.dim, s);
    return diag_residual(mg, L, s, trans);
  }
  ApplyParams p;
  fill_apply_params(L.hp, L.ls, L.d_ctab, L.d_grow, L.d_gcol, L.d_gterm, L.d_gval, L.d_perm, L.d_x, L.d_r, trans, p);
  p.b = L.d_b;
  p.mode = kApplyResidual;
  return launch_apply(L.hp, L.ls, p, s);
}

// Shared memory of a Vanka chunk: r and the corrections of the tile's slots,
// the staged inverses of one class, then the nodes' global indices and
// private flags, the slot modes and the patch-column offsets.
size_t vanka_smem(const MGLevel& L, int n_blk, int tile_slots, int chunk, size_t value_bytes, size_t inv_bytes) {
  const int N = L.hp.k + 1, lyz = L.hp.dim == 2 ? N : N * N;
  const size_t ln = (size_t)(chunk * L.hp.k + 1) * lyz;   // nodes of a chunk
  const int blocks = std::min(n_blk, std::max(1, tile_slots / kVankaVB));
  const size_t sl = (size_t)vanka_slots(blocks);
  const size_t row = (size_t)vanka_row_pieces(L.np, (int)inv_bytes) * 16;
  // the corrections and two stages of r, inverses and tables
  return 3 * (size_t)L.hp.n_t * ln * sl * value_bytes + 2 * (size_t)chunk * L.np * row +
         2 * (ln + sl) * sizeof(int);
}

// Bytes of one stored patch-inverse value.
size_t inv_value_bytes(const MG& mg) { return mg.bf16 ? 2 : (mg.precision == kPrecF32 ? 4 : 8); }

// Cells per Vanka chunk: up to 8, within the shared-memory budget.
int vanka_chunk(const MGLevel& L, int n_blk, int tile_slots, size_t value_bytes, size_t inv_bytes, size_t budget) {
  int best = 0;
  for (int c = 1; c <= std::min(8, L.hp.cells[0]); ++c)
    if (vanka_smem(L, n_blk, tile_slots, c, value_bytes, inv_bytes) <= budget) best = c;
  return best;
}

template <typename T, typename W, int DIM, int K, int NT>
cudaError_t launch_vanka_w(MG& mg, MGLevel& L, cudaStream_t s, int trans) {
  VankaParams<T> p;
  p.r = static_cast<const T*>(L.vanka_r ? L.vanka_r : L.d_r);
  p.x = static_cast<T*>(L.d_x);
  p.inv = L.d_inv;
  p.blk_cls = mg.d_blk_cls;
  p.blk_alpha = mg.d_blk_alpha;
  p.n_blk = mg.n_blk;
  const int tile = L.vanka_tile > 0 ? L.vanka_tile : mg.vanka_tile;
  p.chunk = L.vanka_chunk;
  p.tile_blocks = std::min(mg.n_blk, std::max(1, tile / kVankaVB));
  p.n_tiles = (mg.n_blk + p.tile_blocks - 1) / p.tile_blocks;
  p.npp = vanka_row_pitch(L.np);
  p.n_x = L.hp.n_x;
  p.n_cells = L.hp.n_cells;
  for (int d = 0; d < 3; ++d) {
    p.cells[d] = L.hp.cells[d];
    p.nn[d] = L.hp.nn[d];
  }
  p.omega = T(mg.omega);
  const size_t smem = vanka_smem(L, mg.n_blk, tile, L.vanka_chunk, sizeof(T), sizeof(W));
  p.n_vec_x = (long long)L.hp.n_xi * L.hp.n_t * L.hp.n_x;
  p.inv_count = (long long)mg.n_classes * L.hp.n_cells * L.np * p.npp;
  const int N = L.hp.k + 1, lyz = L.hp.dim == 2 ? N : N * N;
  {
    const size_t ln = (size_t)(L.vanka_chunk * L.hp.k + 1) * lyz;
    p.smem_values = 3 * (size_t)L.hp.n_t * ln * vanka_slots(p.tile_blocks) * sizeof(T) +
                    2 * (size_t)L.vanka_chunk * L.np * vanka_row_pieces(L.np, (int)sizeof(W)) * 16;
  }
  // threads: the row-group x slot-block items of a chunk (one class), whole warps
  const int nrg = (L.np + kVankaR - 1) / kVankaR;
  const int items = L.vanka_chunk * nrg * p.tile_blocks;
  const int threads = std::max(64, std::min(256, (items + 31) / 32 * 32));
  auto kern = trans ? &mg_vanka<T, W, DIM, K, NT, true> : &mg_vanka<T, W, DIM, K, NT, false>;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
  if (e != cudaSuccess) return e;
  const int cpr = (L.hp.cells[0] + L.vanka_chunk - 1) / L.vanka_chunk;
  const long long units = (long long)cpr * L.hp.cells[1] * L.hp.cells[2] * p.n_tiles;
  const int grid = (int)std::max<long long>(1, std::min<long long>(units, sg::sm_count() * std::max(1, per_sm)));
  kern<<<grid, threads, smem, s>>>(p);
  return cudaGetLastError();
}

// Allows the Vanka kernels of one shape the opt-in shared-memory maximum
// (called at set-up, outside any stream capture).
template <typename T, typename W, int DIM, int K, int NT>
cudaError_t prepare_vanka_w() {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaError_t e = cudaFuncSetAttribute(&mg_vanka<T, W, DIM, K, NT, false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(&mg_vanka<T, W, DIM, K, NT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  return e;
}

cudaError_t prepare_vanka(int dim, int k, int nt, bool f32, bool bf16) {
#define SG_PV(D, KK, TT)                                                           \
  if (dim == D && k == KK && nt == TT) {                                           \
    if (!f32) return prepare_vanka_w<double, double, D, KK, TT>();                 \
    if (bf16) return prepare_vanka_w<float, __nv_bfloat16, D, KK, TT>();           \
    return prepare_vanka_w<float, float, D, KK, TT>();                             \
  }
  SG_PV(2, 1, 1) SG_PV(2, 1, 2) SG_PV(2, 1, 3) SG_PV(2, 1, 4)
  SG_PV(2, 2, 1) SG_PV(2, 2, 2) SG_PV(2, 2, 3) SG_PV(2, 2, 4)
  SG_PV(2, 3, 1) SG_PV(2, 3, 2) SG_PV(2, 3, 3) SG_PV(2, 3, 4)
  SG_PV(3, 1, 1) SG_PV(3, 1, 2) SG_PV(3, 2, 1) SG_PV(3, 2, 2)
#undef SG_PV
  return cudaErrorInvalidValue;
}

template <typename T, int DIM, int K, int NT>
cudaError_t launch_vanka(MG& mg, MGLevel& L, cudaStream_t s, int trans) {
  if constexpr (std::is_same<T, float>::value) {
    if (L.vanka_kind == 2)
      return launch_vanka_reg(L.hp, static_cast<const float*>(L.vanka_r ? L.vanka_r : L.d_r), static_cast<float*>(L.d_x),
                              L.d_inv_col, mg.bf16, mg.d_blk_cls, mg.d_blk_alpha, mg.n_blk, mg.n_classes,
                              (float)mg.omega, trans, s);
    if (mg.bf16 && L.vanka_kind == 1 && !trans) {
      const int tile = L.vanka_tile > 0 ? L.vanka_tile : mg.vanka_tile;
      const float* r = static_cast<const float*>(L.vanka_r ? L.vanka_r : L.d_r);
      return launch_vanka_tc(L.hp, r, static_cast<float*>(L.d_x), L.d_inv, mg.d_blk_alpha, mg.n_blk, L.vanka_chunk,
                             tile, mg.d_status, (float)mg.omega, s);
    }
    if (mg.bf16) return launch_vanka_w<T, __nv_bfloat16, DIM, K, NT>(mg, L, s, trans);
  }
  return launch_vanka_w<T, T, DIM, K, NT>(mg, L, s, trans);
}

// The tensor-core sweep applies to this level: bf16 factors, one diagonal
// class, a patch of at most 64 unknowns, tiles of at most 80 slots.
bool tc_level_ok(const MG& mg, const MGLevel& L, int tile) {
  return mg.bf16 && mg.n_classes == 1 && !L.coarsest && vanka_tc_eligible(L.hp.dim, L.hp.k, L.hp.n_t, tile);
}

template <typename T>
bool vanka(MG& mg, MGLevel& L, cudaStream_t s, int trans) {
  const int d = L.hp.dim, k = L.hp.k, t = L.hp.n_t;
#define SG_V(D, KK, TT) \
  if (d == D && k == KK && t == TT) return launch_vanka<T, D, KK, TT>(mg, L, s, trans) == cudaSuccess;
  SG_V(2, 1, 1) SG_V(2, 1, 2) SG_V(2, 1, 3) SG_V(2, 1, 4)
  SG_V(2, 2, 1) SG_V(2, 2, 2) SG_V(2, 2, 3) SG_V(2, 2, 4)
  SG_V(2, 3, 1) SG_V(2, 3, 2) SG_V(2, 3, 3) SG_V(2, 3, 4)
  SG_V(3, 1, 1) SG_V(3, 1, 2) SG_V(3, 2, 1) SG_V(3, 2, 2)
#undef SG_V
  return false;
}

bool vk_launch(MG& mg, MGLevel& L, cudaStream_t s) {
  return mg.precision == kPrecF32 ? vanka<float>(mg, L, s, 0) : vanka<double>(mg, L, s, 0);
}

// the padded width of lists whose longest has n entries
int axis_width(int n) {
  for (int w : {2, 3, 4, 5, 8})
    if (n <= w) return w;
  return kAxisMax;
}

// CSR lists (ptr, idx, wt) -> width entries per output, entry-major
void pad_lists(const std::vector<int>& ptr, const std::vector<int>& idx, const std::vector<double>& wt, int width,
               std::vector<int>& pidx, std::vector<double>& pw) {
  const int n = (int)ptr.size() - 1;
  pidx.assign((size_t)width * n, 0);
  pw.assign((size_t)width * n, 0.0);
  for (int o = 0; o < n; ++o) {
    const int c = ptr[o + 1] - ptr[o];
    for (int k = 0; k < width; ++k) {
      pidx[(size_t)k * n + o] = k < c ? idx[ptr[o] + k] : (c > 0 ? idx[ptr[o]] : -1);
      pw[(size_t)k * n + o] = k < c ? wt[ptr[o] + k] : 0.0;
    }
  }
  // outputs without entries (Dirichlet nodes) point where their neighbour does
  for (int k = 0; k < width; ++k)
    for (int pass = 0; pass < 2; ++pass)
      for (int i = 1; i < n; ++i) {
        const int o = pass ? n - 1 - i : i, nb = pass ? o + 1 : o - 1;
        int& at = pidx[(size_t)k * n + o];
        if (at < 0) at = pidx[(size_t)k * n + nb];
      }
  for (int& at : pidx) at = std::max(at, 0);
}

// The tiles of `tile` outputs each of a padded list: first input and number of inputs, per tile.
int tile_ranges(const std::vector<int>& pidx, int width, int n, int tile, std::vector<int>& range) {
  int most = 0;
  range.clear();
  for (int o0 = 0; o0 < n; o0 += tile) {
    int lo = pidx[o0], hi = lo;
    for (int o = o0; o < std::min(n, o0 + tile); ++o)
      for (int k = 0; k < width; ++k) {
        lo = std::min(lo, pidx[(size_t)k * n + o]);
        hi = std::max(hi, pidx[(size_t)k * n + o]);
      }
    range.push_back(lo);
    range.push_back(hi - lo + 1);
    most = std::max(most, hi - lo + 1);
  }
  return most;
}

// Columns a pass takes at a time: as few parts of a row as keep three quarters
// of the threads busy (129 nodes: 65 x 3 rows instead of 129 x 1).
int column_block(int cols) {
  int best = std::min(cols, kTransferThreads);
  for (int m = 1; m <= 16; ++m) {
    const int cb = std::min((cols + m - 1) / m, kTransferThreads);
    const int busy = kTransferThreads / cb * cb, had = kTransferThreads / best * best;
    if (busy >= 3 * kTransferThreads / 4) return cb;
    if (busy > had) best = cb;
  }
  return best;
}

template <typename T>
void transfer_params(const MGLevel& I, const MGLevel& O, const MGLevel::Transfer& t, int V, TransferParams<T>& p) {
  for (int d = 0; d < 3; ++d) {
    p.idx[d] = t.idx[d];
    p.w[d] = static_cast<const T*>(t.w[d]);
    p.ni[d] = I.hp.nn[d];
    p.no[d] = O.hp.nn[d];
  }
  p.range = t.range;
  p.range_x = t.range_x;
  p.n_in = I.hp.n_x;
  p.n_out = O.hp.n_x;
  p.tile = t.tile;
  p.max_rows = t.max_rows;
  p.z = I.hp.dim == 3;
  p.tile_x = t.tile_x;
  p.max_cols = t.max_cols;
  p.n_vec = (unsigned)V;
  p.planes = (unsigned)p.no[2];
  p.tiles = (unsigned)((p.no[1] + t.tile - 1) / t.tile);
  p.cb_in = column_block(t.tile_x > 0 ? t.max_cols : p.ni[0]);
  p.cb_out = column_block(t.tile_x > 0 ? t.tile_x : p.no[0]);
  p.lim_in = (long long)V * I.hp.n_x;
  p.lim_out = (long long)V * O.hp.n_x;
}

// Bytes of shared memory of a transfer block: the input rows, and the rows
// between its passes (restriction: the input rows; interpolation: the tile,
// with coarse and then fine rows).
size_t transfer_smem(bool up, int max_rows, int tile, int nfx, int ncx, size_t vb) {
  return vb * (up ? (size_t)max_rows * ncx + (size_t)tile * (ncx + nfx) : (size_t)max_rows * (nfx + ncx));
}

// The launch grid of a transfer: vectors, planes and tiles of rows, or all of
// them and the tiles of columns on x.
template <typename T>
dim3 transfer_grid(const TransferParams<T>& p, const MGLevel::Transfer& t) {
  if (t.tile_x == 0) return dim3(p.n_vec, p.planes, p.tiles);
  return dim3((unsigned)((size_t)p.n_vec * p.planes * p.tiles * ((p.no[0] + t.tile_x - 1) / t.tile_x)));
}

#define SG_TRANSFER_WIDTHS(CALL) \
  switch (t.width) {             \
    case 2: CALL(2); break;      \
    case 3: CALL(3); break;      \
    case 4: CALL(4); break;      \
    case 5: CALL(5); break;      \
    case 8: CALL(8); break;      \
    default: CALL(kAxisMax); break; \
  }

// x_fine += P e_coarse; r_fine = b_fine inside, 0 on the boundary
template <typename T>
cudaError_t prolong(MGLevel& F, MGLevel& C, int V, cudaStream_t s) {
  const MGLevel::Transfer& t = F.up;
  TransferParams<T> p;
  transfer_params(C, F, t, V, p);
  p.in = static_cast<const T*>(C.d_x);
  p.b = static_cast<const T*>(F.d_b);
  p.out = static_cast<T*>(F.d_x);
  p.x = nullptr;
  p.r = static_cast<T*>(F.d_r);
  const dim3 grid = transfer_grid(p, t);
#define SG_CALL(W)                                                                  \
  if (t.tile_x > 0) mg_prolong<T, W, true><<<grid, kTransferThreads, t.smem, s>>>(p); \
  else mg_prolong<T, W, false><<<grid, kTransferThreads, t.smem, s>>>(p)
  SG_TRANSFER_WIDTHS(SG_CALL)
#undef SG_CALL
  return cudaGetLastError();
}

// b_coarse = P^T r_fine; x_coarse = 0, r_coarse = b_coarse
template <typename T>
cudaError_t restrict_to(MGLevel& F, MGLevel& C, int V, cudaStream_t s) {
  const MGLevel::Transfer& t = F.down;
  TransferParams<T> p;
  transfer_params(F, C, t, V, p);
  p.in = static_cast<const T*>(F.d_r);
  p.b = nullptr;
  p.out = static_cast<T*>(C.d_b);
  p.x = static_cast<T*>(C.d_x);
  p.r = static_cast<T*>(C.d_r);
  const dim3 grid = transfer_grid(p, t);
#define SG_CALL(W)                                                                  \
  if (t.tile_x > 0) mg_restrict<T, W, true><<<grid, kTransferThreads, t.smem, s>>>(p); \
  else mg_restrict<T, W, false><<<grid, kTransferThreads, t.smem, s>>>(p)
  SG_TRANSFER_WIDTHS(SG_CALL)
#undef SG_CALL
  return cudaGetLastError();
}

template <typename T>
cudaError_t issue_vcycle(MG& mg, int l, cudaStream_t s, int trans) {
  MGLevel& L = mg.lv[l];
  const int V = L.hp.n_xi * L.hp.n_t;
  if (L.coarsest) {   // x holds the boundary values and 0 inside (restriction, or the start of a one-level hierarchy)
    const size_t smem = (size_t)kCoarseModes * L.n_int * sizeof(T);
    mg_coarse<T><<<dim3((L.n_int + kCoarseRows - 1) / kCoarseRows, mg.n_blk), 32 * kCoarseRows, smem, s>>>(
        static_cast<const T*>(L.d_b), static_cast<T*>(L.d_x), static_cast<const T*>(L.d_inv), mg.d_blk_cls,
        mg.d_blk_alpha, reinterpret_cast<const long long*>(L.d_inner), L.n_int, L.hp.n_t, L.hp.n_x, trans,
        (long long)V * L.hp.n_x, (long long)mg.n_classes * L.n_int * L.n_int);
    return cudaGetLastError();
  }
  cudaError_t e;
  // the level arrives started: x = the boundary values of b and 0 inside,
  // r = b inside and 0 on the boundary.  The first sweep's residual b - A x is
  // b on the interior, where the sweep reads it; r is then the preset of the
  // residual that follows.
  for (int it = 0; it < mg.nu; ++it) {
    if (it > 0 && (e = residual<T>(mg, l, s, trans, it == 1)) != cudaSuccess) return e;
    L.vanka_r = it == 0 ? L.d_b : nullptr;
    const bool ok = vanka<T>(mg, L, s, trans);
    L.vanka_r = nullptr;
    if (!ok) return cudaErrorInvalidValue;
  }
  if ((e = residual<T>(mg, l, s, trans, mg.nu == 1)) != cudaSuccess) return e;
  MGLevel& C = mg.lv[l + 1];
  if (C.hp.n_xi * C.hp.n_t != V) return cudaErrorInvalidValue;   // level buffers hold V vectors
  if ((e = restrict_to<T>(L, C, V, s)) != cudaSuccess) return e;
  if ((e = issue_vcycle<T>(mg, l + 1, s, trans)) != cudaSuccess) return e;
  if ((e = prolong<T>(L, C, V, s)) != cudaSuccess) return e;
  for (int it = 0; it < mg.nu; ++it) {
    if ((e = residual<T>(mg, l, s, trans, it == 0)) != cudaSuccess) return e;
    if (!vanka<T>(mg, L, s, trans)) return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

// Device time of one launch of a set-up candidate: a single timed launch when
// it takes more than 2 ms (the large levels, where one launch is steady and
// repeating it costs seconds), else the mean of three launches after it.
template <class F>
static float time_candidate(F&& launch, cudaStream_t s, cudaEvent_t a, cudaEvent_t b, cudaError_t& e) {
  float ms = 0.0f;
  if (e == cudaSuccess) e = cudaEventRecord(a, s);
  if (e == cudaSuccess) e = launch();
  if (e == cudaSuccess) e = cudaEventRecord(b, s);
  if (e == cudaSuccess) e = cudaEventSynchronize(b);
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
  if (e != cudaSuccess || ms > 2.0f) return ms;
  if (e == cudaSuccess) e = cudaEventRecord(a, s);
  for (int r = 0; r < 3 && e == cudaSuccess; ++r) e = launch();
  if (e == cudaSuccess) e = cudaEventRecord(b, s);
  if (e == cudaSuccess) e = cudaEventSynchronize(b);
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
  return ms / 3.0f;
}

// The residual apply of the smoothed levels.  The row-diagonal apply wins
// wherever its values fit the registers with warps to spare (V-cycle with it
// and with the SG cell kernel on every level, ms: 32^3 Q2 FP32 1.40 / 2.11,
// FP64 17.1 / 17.7; 64^2 Q2 FP32 0.201 / 0.279, FP64 0.84 / 0.89; 64^2 Q3 dG(3)
// FP32 0.70 / 0.73), but not for FP64 Q3 (254 registers; 8.60 / 8.22): those
// levels of at least 256 cells are timed on their own buffers, against the SG
// cell kernel over (cells per chunk x 256 / 512 threads), then the staggered
// first chunk of its best shape.
static cudaError_t tune_level_applies(MG& mg) {
  if (mg.precision == kPrecF32 || mg.lv[0].hp.k < 3) return cudaSuccess;
  const size_t vb = sizeof(double);
  cudaEvent_t a = nullptr, b = nullptr;
  cudaError_t e = cudaEventCreate(&a);
  if (e == cudaSuccess) e = cudaEventCreate(&b);
  for (size_t l = 0; l < mg.lv.size() && e == cudaSuccess; ++l) {
    MGLevel& L = mg.lv[l];
    if (L.coarsest || L.hp.n_cells < 256) continue;
    auto res = [&]() { return residual<double>(mg, (int)l, mg.stream, 0, false); };
    const long long n = (long long)L.hp.n_xi * L.hp.n_t * L.hp.n_x;
    if ((e = cudaMemsetAsync(L.d_x, 0, n * vb, mg.stream)) != cudaSuccess) break;
    if ((e = cudaMemsetAsync(L.d_b, 0, n * vb, mg.stream)) != cudaSuccess) break;
    L.use_diag = true;
    float best_ms = time_candidate(res, mg.stream, a, b, e);
    bool best_diag = true;
    LaunchShape best_ls = L.ls;
    if (L.chunk_ok) {
      // the SG cell kernel over (cells per chunk x threads)
      int dev = 0, optin = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      const int max1 = max_apply_chunk(L.hp, (size_t)optin - 1024);
      std::vector<int> chunks;
      for (int c = max1; c >= 1; c = c > 1 ? (c + 1) / 2 - (c == 2) : 0) chunks.push_back(c);
      L.use_diag = false;
      const LaunchShape keep = L.ls;
      // (cells per chunk x threads), then the staggered first chunk of the best
      for (int c : chunks)
        for (int t : {256, 512}) {
          if (e != cudaSuccess) break;
          LaunchShape ls;
          std::string msg;
          if (plan_apply_shape(L.hp, c, t, ls, msg) != SG_OK) continue;
          ls.stagger = 0;
          L.ls = ls;
          const float ms = time_candidate(res, mg.stream, a, b, e);
          if (e == cudaSuccess && ms < best_ms) {
            best_ms = ms;
            best_diag = false;
            best_ls = ls;
          }
        }
      if (!best_diag && best_ls.chunk > 1 && e == cudaSuccess) {
        LaunchShape ls = best_ls;
        ls.stagger = (ls.chunk + 1) / 2;
        L.ls = ls;
        const float ms = time_candidate(res, mg.stream, a, b, e);
        if (e == cudaSuccess && ms < best_ms) {
          best_ms = ms;
          best_ls = ls;
        }
      }
      L.ls = best_diag ? keep : best_ls;
    }
    L.use_diag = best_diag;
  }
  if (a) cudaEventDestroy(a);
  if (b) cudaEventDestroy(b);
  return e;
}

// Picks the cells per Vanka chunk of every smoothed level, and with a single
// diagonal class on levels with few cells the modes per tile (the whole set,
// 16 or 8: smaller tiles give them more CTAs), by timing sweeps on the level's own buffers for
// every candidate within the shared-memory budget; keeps the fastest.
static cudaError_t tune_vanka(MG& mg) {
  const size_t vb = mg.precision == kPrecF32 ? 4 : 8;
  cudaEvent_t a = nullptr, b = nullptr;
  cudaError_t e = cudaEventCreate(&a);
  if (e == cudaSuccess) e = cudaEventCreate(&b);
  for (MGLevel& L : mg.lv) {
    if (L.coarsest || L.vanka_kind == 2 || e != cudaSuccess) continue;
    const long long n = (long long)L.hp.n_xi * L.hp.n_t * L.hp.n_x;
    if ((e = cudaMemsetAsync(L.d_r, 0, n * vb, mg.stream)) != cudaSuccess) break;
    if ((e = cudaMemsetAsync(L.d_x, 0, n * vb, mg.stream)) != cudaSuccess) break;
    std::vector<int> tiles = {mg.vanka_tile};
    // smaller tiles only where one-cell chunks of whole tiles leave the GPU short of CTAs
    const long long units1 = (long long)L.hp.n_cells * ((mg.n_blk * kVankaVB + mg.vanka_tile - 1) / mg.vanka_tile);
    if (units1 < sg::sm_count() * 16)
      for (int t : {16, 8})
        if (t < mg.vanka_tile && t % kVankaVB == 0) tiles.push_back(t);
    int best_c = L.vanka_chunk, best_t = 0;
    float best_ms = 1e30f;
    for (int tile : tiles) {
      const int max_c = vanka_chunk(L, mg.n_blk, tile, vb, inv_value_bytes(mg),
                                    tile == mg.vanka_tile
                                        ? std::max<size_t>(100 * 1024, vanka_smem(L, mg.n_blk, tile, L.vanka_chunk, vb,
                                                                                 inv_value_bytes(mg)))
                                        : 100 * 1024);
      if (max_c == 0) continue;
      std::vector<int> cand;
      for (int c = 1; c <= max_c; c *= 2) cand.push_back(c);
      if (cand.back() != max_c) cand.push_back(max_c);
      for (int c : cand) {
        if (e != cudaSuccess) break;
        L.vanka_chunk = c;
        L.vanka_tile = tile == mg.vanka_tile ? 0 : tile;
        const float ms = time_candidate(
            [&]() { return vk_launch(mg, L, mg.stream) ? cudaSuccess : cudaErrorInvalidValue; }, mg.stream, a, b, e);
        if (e == cudaSuccess && ms < best_ms) {
          best_ms = ms;
          best_c = c;
          best_t = L.vanka_tile;
        }
      }
    }
    L.vanka_chunk = L.ffma_chunk = best_c;
    L.vanka_tile = L.ffma_tile = best_t;
    L.vanka_kind = 0;
    // the tensor-core sweep over its chunk sizes, where it applies; kept if faster
    const int tile_all = mg.vanka_tile;
    if (e == cudaSuccess && tc_level_ok(mg, L, tile_all)) {
      int dev = 0, optin = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      int tc_c = 0;
      float tc_ms = 1e30f;
      for (int c : {1, 2}) {                     // one or two staging buffers
        if (e != cudaSuccess) break;
        if (vanka_tc_smem(L.hp.dim, L.hp.k, L.hp.n_t, c, std::min(tile_all, mg.n_blk * kVankaVB)) >
            (size_t)optin - 1024)
          break;
        L.vanka_chunk = c;
        L.vanka_tile = 0;
        L.vanka_kind = 1;
        const float ms = time_candidate(
            [&]() { return vk_launch(mg, L, mg.stream) ? cudaSuccess : cudaErrorInvalidValue; }, mg.stream, a, b, e);
        if (e == cudaSuccess && ms < tc_ms) {
          tc_ms = ms;
          tc_c = c;
        }
      }
      if (tc_c > 0 && tc_ms < best_ms) {
        L.vanka_chunk = tc_c;
        L.vanka_tile = 0;
        L.vanka_kind = 1;
      } else {
        L.vanka_chunk = best_c;
        L.vanka_tile = best_t;
        L.vanka_kind = 0;
      }
    }
  }
  if (a) cudaEventDestroy(a);
  if (b) cudaEventDestroy(b);
  return e;
}

void mg_free(MG& mg) {
  for (int t = 0; t < 2; ++t) {
    if (mg.exec_t[t]) cudaGraphExecDestroy(mg.exec_t[t]);
    if (mg.graph_t[t]) cudaGraphDestroy(mg.graph_t[t]);
    mg.exec_t[t] = nullptr;
    mg.graph_t[t] = nullptr;
  }
  if (mg.stream) cudaStreamDestroy(mg.stream);
  cudaFree(mg.d_blk_cls);
  cudaFree(mg.d_blk_alpha);
  cudaFree(mg.d_wused);
  cudaFree(mg.d_status);
  mg.d_wused = nullptr;
  mg.used.clear();
  mg.d_status = nullptr;
  mg.d_blk_cls = mg.d_blk_alpha = nullptr;
  for (MGLevel& L : mg.lv) {
    cudaFree(L.d_ctab); cudaFree(L.d_grow); cudaFree(L.d_gcol); cudaFree(L.d_gterm); cudaFree(L.d_gval);
    cudaFree(L.d_perm); cudaFree(L.d_inv); cudaFree(L.d_inv_col); cudaFree(L.d_inner); cudaFree(L.d_coef);
    cudaFree(L.d_x); cudaFree(L.d_b); cudaFree(L.d_r);
    for (MGLevel::Transfer* t : {&L.down, &L.up}) {
      for (int d = 0; d < 3; ++d) {
        cudaFree(t->idx[d]);
        cudaFree(t->w[d]);
      }
      cudaFree(t->range);
      cudaFree(t->range_x);
    }
  }
  mg.lv.clear();
  mg.stream = nullptr;
}

// Lets the coarse solve stage up to 2048 unknowns of four modes (64 KB in FP64).
static cudaError_t prepare_coarse(int precision) {
  const int most = kCoarseModes * 2048 * (int)sizeof(double);
  return precision == kPrecF32 ? cudaFuncSetAttribute(&mg_coarse<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, most)
                               : cudaFuncSetAttribute(&mg_coarse<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// Lets the transfer kernels use more than 48 KB of shared memory (rows of
// more than about 1000 nodes).
template <typename T, int W>
static cudaError_t prepare_transfers_w(int optin) {
  cudaError_t e = cudaFuncSetAttribute(&mg_restrict<T, W, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  return e == cudaSuccess ? cudaFuncSetAttribute(&mg_prolong<T, W, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin)
                          : e;
}
template <typename T>
static cudaError_t prepare_transfers_t() {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaError_t e = cudaSuccess;
  for (auto f : {&prepare_transfers_w<T, 2>, &prepare_transfers_w<T, 3>, &prepare_transfers_w<T, 4>,
                 &prepare_transfers_w<T, 5>, &prepare_transfers_w<T, 8>, &prepare_transfers_w<T, kAxisMax>})
    if (e == cudaSuccess) e = f(optin);
  return e;
}
static cudaError_t prepare_transfers(size_t vb) {
  return vb == 4 ? prepare_transfers_t<float>() : prepare_transfers_t<double>();
}

// The transfers between a level F and the next coarser one: the 1D lists of
// every direction padded to one width, and the tiles of the plane kernels.
// Rows per tile: halved from the whole plane until a block's rows fit in 48 KB
// of shared memory and the blocks cover the GPU four times, or 4 rows are left
// (64^2 Q2, 70 vectors: 8 rows, 630 blocks; 32^3 Q2: whole planes of 65 rows).
// Where a row does not fit at all (FP64 from 6456 cells of Q1 along x, 1384 of
// Q2 and 588 of Q3; twice that in FP32), or the grid has more than 65535 planes
// or tiles: tiles of 8 rows, and columns halved until a block takes 48 KB.
static cudaError_t build_transfers(MGLevel& F, const MGLevel& C, size_t vb) {
  std::vector<int> ptr[2][3], idx[2][3];
  std::vector<double> w[2][3];
  int longest[2] = {0, 0};
  for (int d = 0; d < F.hp.dim; ++d) {
    transfer_1d(F.hp, C.hp, d, ptr[1][d], idx[1][d], w[1][d], ptr[0][d], idx[0][d], w[0][d]);
    for (int u = 0; u < 2; ++u)
      for (size_t i = 0; i + 1 < ptr[u][d].size(); ++i) longest[u] = std::max(longest[u], ptr[u][d][i + 1] - ptr[u][d][i]);
  }
  cudaError_t e = cudaSuccess;
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int precision = vb == 4 ? kPrecF32 : SG_PREC_FP64;
  for (int u = 0; u < 2; ++u) {
    MGLevel::Transfer& t = u ? F.up : F.down;
    if (longest[u] > kAxisMax) return cudaErrorInvalidValue;
    t.width = axis_width(longest[u]);
    std::vector<int> pi, px, py;
    std::vector<double> pw;
    for (int d = 0; d < F.hp.dim; ++d) {
      pad_lists(ptr[u][d], idx[u][d], w[u][d], t.width, pi, pw);
      if (d == 0) px = pi;
      if (d == 1) py = pi;
      if ((e = upload_vec(&t.idx[d], pi)) != cudaSuccess) return e;
      if ((e = upload_values(&t.w[d], pw, precision)) != cudaSuccess) return e;
    }
    const HostProblem& out = u ? F.hp : C.hp;
    const long long planes = (long long)F.hp.n_xi * F.hp.n_t * (F.hp.dim == 3 ? out.nn[2] : 1);
    std::vector<int> range;
    t.tile = out.nn[1];
    while (true) {
      t.max_rows = tile_ranges(py, t.width, out.nn[1], t.tile, range);
      t.smem = transfer_smem(u == 1, t.max_rows, t.tile, F.hp.nn[0], C.hp.nn[0], vb);
      const long long blocks = planes * ((out.nn[1] + t.tile - 1) / t.tile);
      if (t.tile == 1 || (t.smem <= 48 * 1024 && (blocks >= 4 * sg::sm_count() || t.tile <= 4))) break;
      t.tile = (t.tile + 1) / 2;
    }
    if (t.smem > (size_t)optin || out.nn[2] > 65535 || (out.nn[1] + t.tile - 1) / t.tile > 65535) {
      std::vector<int> rx;
      t.tile = std::min(8, out.nn[1]);
      t.tile_x = out.nn[0];
      t.max_rows = tile_ranges(py, t.width, out.nn[1], t.tile, range);
      while (true) {
        t.max_cols = tile_ranges(px, t.width, out.nn[0], t.tile_x, rx);
        t.smem = transfer_smem(u == 1, t.max_rows, t.tile, u ? t.tile_x : t.max_cols, u ? t.max_cols : t.tile_x, vb);
        if (t.smem <= 48 * 1024 || t.tile_x == 1) break;
        t.tile_x = (t.tile_x + 1) / 2;
      }
      if ((e = upload_vec(&t.range_x, rx)) != cudaSuccess) return e;
    }
    if (t.smem > 48 * 1024 && (e = prepare_transfers(vb)) != cudaSuccess) return e;
    if ((e = upload_vec(&t.range, range)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

sg_status mg_build(const HostProblem& fine, int precision, int nu, double omega, MG& mg, std::string& msg,
                   bool single_class) {
  const auto t0 = std::chrono::steady_clock::now();
  mg.requested = precision;
  mg.bf16 = precision == SG_PREC_BF16;
  if (mg.bf16) precision = kPrecF32;          // FP32 vectors, bf16-stored patch inverses
  mg.precision = precision;
  mg.nu = nu;
  mg.omega = omega;
  // diagonal classes of the chaos rows
  GTable gdiag;
  std::vector<std::vector<double>> drow;
  diagonal_table(fine, gdiag, drow);
  std::map<std::vector<double>, int> key;
  std::vector<std::vector<double>> class_diag;
  mg.cls.assign(fine.n_xi, 0);
  for (int a = 0; a < fine.n_xi; ++a) {
    auto it = key.find(drow[a]);
    if (it == key.end()) {
      key[drow[a]] = (int)class_diag.size();
      mg.cls[a] = (int)class_diag.size();
      class_diag.push_back(drow[a]);
    } else {
      mg.cls[a] = it->second;
    }
  }
  if (single_class) {
    // the mean block: coefficient term with the zero chaos index, weight 1
    std::vector<double> mean_diag(fine.n_terms, 0.0);
    for (int t = 0; t < fine.n_terms; ++t)
      if (std::all_of(fine.mus[t].begin(), fine.mus[t].end(), [](int v) { return v == 0; })) mean_diag[t] = 1.0;
    class_diag.assign(1, mean_diag);
    std::fill(mg.cls.begin(), mg.cls.end(), 0);
  }
  mg.n_classes = (int)class_diag.size();
  // Vanka mode blocks: the modes of one class, kVankaVB at a time
  std::vector<int> blk_cls, blk_alpha;
  for (int c = 0; c < mg.n_classes; ++c) {
    std::vector<int> modes;
    for (int a = 0; a < fine.n_xi; ++a)
      if (mg.cls[a] == c) modes.push_back(a);
    for (size_t i = 0; i < modes.size(); i += kVankaVB) {
      blk_cls.push_back(c);
      for (int u = 0; u < kVankaVB; ++u) blk_alpha.push_back(i + u < modes.size() ? modes[i + u] : -1);
    }
  }
  mg.n_blk = (int)blk_cls.size();
  // slots per Vanka tile: every block, or (Monte-Carlo batches) the requested
  // number of samples
  if (mg.vanka_tile <= 0 || !mg.mc || mg.vanka_tile > mg.n_blk * kVankaVB) mg.vanka_tile = mg.n_blk * kVankaVB;
  // level problems
  std::vector<HostProblem> hps;
  hps.push_back(fine);
  while (true) {
    const HostProblem& f = hps.back();
    bool ok = true;
    for (int d = 0; d < f.dim; ++d) ok = ok && f.cells[d] % 2 == 0 && f.cells[d] > 2;
    if (!ok) break;
    // a level small enough for the dense coarse solve ends the hierarchy
    long long inner = f.n_t;
    for (int d = 0; d < f.dim; ++d) inner *= std::max(0, f.nn[d] - 2);
    if (mg.coarse_dofs > 0 && inner <= mg.coarse_dofs) break;
    sg_mesh m;
    std::memset(&m, 0, sizeof(m));
    m.dim = f.dim;
    for (int d = 0; d < 3; ++d) {
      m.cells[d] = d < f.dim ? f.cells[d] / 2 : 1;
      m.lo[d] = f.lo[d];
      m.hi[d] = f.lo[d] + f.h[d] * f.cells[d];
    }
    std::vector<Piece> pieces = f.pieces;
    for (Piece& pc : pieces) pc.scale = coarsen_scale(pc.scale, f);
    HostProblem c;
    sg_status st = build_host_problem_pieces(&m, f.k, f.r, f.n_slabs, f.T, f.M, f.p, pieces, c, msg);
    if (st != SG_OK) return st;
    // every level carries the rows of the fine problem (chaos modes, or the
    // samples of a Monte-Carlo batch): same count, same coupling table
    c.n_xi = fine.n_xi;
    c.idx = fine.idx;
    hps.push_back(std::move(c));
  }
  for (const HostProblem& h : hps)
    if (h.n_xi != fine.n_xi || h.n_t != fine.n_t || h.n_terms != fine.n_terms) {
      msg = "multigrid levels disagree in rows, time nodes or coefficient terms";
      return SG_ERR_ARG;
    }
  mg.lv.resize(hps.size());
  cudaError_t e = cudaSuccess;
  {
    // per-row weights of the row-diagonal apply, G_mu[alpha][alpha], of the terms any row uses
    for (int t = 0; t < fine.n_terms; ++t)
      for (int a = 0; a < fine.n_xi; ++a)
        if (drow[a][t] != 0.0) {
          mg.used.push_back(t);
          break;
        }
    std::vector<double> w;
    for (int a = 0; a < fine.n_xi; ++a)
      for (int t : mg.used) w.push_back(drow[a][t]);
    if ((e = upload_values(&mg.d_wused, w, precision)) != cudaSuccess) {
      msg = std::string("multigrid set-up: ") + cudaGetErrorString(e);
      return e == cudaErrorMemoryAllocation ? SG_ERR_OOM : SG_ERR_CUDA;
    }
  }
  for (size_t l = 0; l < hps.size(); ++l) {
    MGLevel& L = mg.lv[l];
    L.hp = std::move(hps[l]);
    L.hp.g = gdiag;
    L.hp.perm.resize(L.hp.n_xi);
    for (int a = 0; a < L.hp.n_xi; ++a) L.hp.perm[a] = a;
    L.hp.precision = precision;
    L.coarsest = l + 1 == mg.lv.size();
    {
      // the level residual is the diagonal apply: time-mass tables of A_t and A_t^T
      std::vector<double> At((size_t)L.hp.n_t * L.hp.n_t);
      for (int i = 0; i < L.hp.n_t; ++i)
        for (int j = 0; j < L.hp.n_t; ++j) At[(size_t)i * L.hp.n_t + j] = L.hp.A_hat[(size_t)j * L.hp.n_t + i];
      mc_amq(L.hp, L.hp.A_hat, L.amq[0]);
      mc_amq(L.hp, At, L.amq[1]);
      // the SG cell kernel with the diagonal coupling table, where it applies
      std::string m2;
      L.chunk_ok = !mg.mc && plan_apply(L.hp, L.ls, m2) == SG_OK;
      if (L.chunk_ok && (e = prepare_apply_kernel(precision, L.hp.dim, L.hp.k, L.hp.n_t, L.ls.smem)) != cudaSuccess) break;
      L.use_diag = true;
    }
    const int n = L.hp.k + 1;
    const int nkd = L.hp.dim == 2 ? n * n : n * n * n;
    L.np = L.hp.n_t * nkd;
    if (L.coarsest) {
      const ElementData ed = element_data(L.hp);
      std::vector<long long> node_of;
      for (long long m = 0; m < L.hp.n_x; ++m) {
        const int g[3] = {(int)(m % L.hp.nn[0]), (int)((m / L.hp.nn[0]) % L.hp.nn[1]),
                          (int)(m / ((long long)L.hp.nn[0] * L.hp.nn[1]))};
        if (node_interior(L.hp, g)) node_of.push_back(m);
      }
      L.n_int = L.hp.n_t * (int)node_of.size();
      if (L.n_int > 2048 || L.n_int * sizeof(double) > 48 * 1024) {
        msg = "coarsest multigrid level too large (mesh cannot be coarsened enough)";
        return SG_ERR_UNSUPPORTED;
      }
      std::vector<long long> inner_dofs;
      for (int i = 0; i < L.hp.n_t; ++i)
        for (long long m : node_of) inner_dofs.push_back((long long)i * L.hp.n_x + m);
      const size_t vb_c = precision == kPrecF32 ? 4 : 8, n2 = (size_t)L.n_int * L.n_int;
      if ((e = cudaMalloc(&L.d_inv, mg.n_classes * n2 * vb_c)) != cudaSuccess) break;
      for (int c = 0; c < mg.n_classes && e == cudaSuccess; ++c) {
        std::vector<double> ci;
        void* dst = static_cast<char*>(L.d_inv) + c * n2 * vb_c;
        bool ok = false;
        coarse_matrix(L.hp, ed, class_diag[c], node_of, ci);
        e = coarse_inverse_device(ci, L.n_int, precision, dst, ok);
        if (ok || e != cudaSuccess) continue;
        // pivoting elimination on the host
        if (!invert(ci, L.n_int)) { msg = "singular coarse operator"; return SG_ERR_ARG; }
        if (precision == kPrecF32) {
          const std::vector<float> f(ci.begin(), ci.end());
          e = cudaMemcpy(dst, f.data(), n2 * vb_c, cudaMemcpyHostToDevice);
        } else {
          e = cudaMemcpy(dst, ci.data(), n2 * vb_c, cudaMemcpyHostToDevice);
        }
      }
      if (e != cudaSuccess) break;
      if ((e = upload_vec(reinterpret_cast<long long**>(&L.d_inner), inner_dofs)) != cudaSuccess) break;
      if ((e = prepare_coarse(precision)) != cudaSuccess) break;
    }
    // level apply tables (coefficient stays double; vectors use the MG precision)
    if ((e = upload_vec(reinterpret_cast<double**>(&L.d_ctab), L.hp.ctab)) != cudaSuccess) break;
    if (!L.coarsest &&
        (e = diag_coefficients(precision, L.hp, static_cast<const double*>(L.d_ctab), mg.used, &L.d_coef, 0)) != cudaSuccess)
      break;
    if (!L.coarsest) {
      // Vanka patch inverses, assembled and factored on the device
      const int npp = vanka_row_pitch(L.np);
      const int kind = mg.bf16 ? 2 : precision == kPrecF32 ? 1 : 0;
      const size_t wb = kind == 2 ? sizeof(__nv_bfloat16) : kind == 1 ? sizeof(float) : sizeof(double);
      if ((e = cudaMalloc(&L.d_inv, (size_t)mg.n_classes * L.hp.n_cells * L.np * npp * wb)) != cudaSuccess) break;
      bool singular = false;
      const auto tf = std::chrono::steady_clock::now();
      if ((e = vanka_factor(L.hp, static_cast<const double*>(L.d_ctab), class_diag, kind, L.d_inv, npp, singular,
                            0)) != cudaSuccess)
        break;
      mg.factor_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - tf).count();
      if (singular) {
        msg = "singular Vanka patch";
        return SG_ERR_ARG;
      }
      int dev = 0, optin = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      const size_t vb = precision == kPrecF32 ? 4 : 8;
      L.vanka_chunk = vanka_chunk(L, mg.n_blk, mg.vanka_tile, vb, inv_value_bytes(mg), 100 * 1024);
      if (L.vanka_chunk == 0)
        L.vanka_chunk = vanka_chunk(L, mg.n_blk, mg.vanka_tile, vb, inv_value_bytes(mg), (size_t)optin - 1024);
      if (L.vanka_chunk == 0) {
        msg = "Vanka smoother: one cell with all rows does not fit in shared memory (fewer samples per batch)";
        return SG_ERR_UNSUPPORTED;
      }
      L.ffma_chunk = L.vanka_chunk;
      if ((e = prepare_vanka(L.hp.dim, L.hp.k, L.hp.n_t, precision == kPrecF32, mg.bf16)) != cudaSuccess) break;
      if (mg.bf16 && (e = prepare_vanka_tc(L.hp.dim, L.hp.k, L.hp.n_t)) != cudaSuccess) break;
      // FP32 vectors and small 2D patches: the register sweep, untimed.  V-cycle with it
      // and with the best of the other sweeps over their chunks, ms: 32^2 Q2 dG(1), 35 rows
      // 0.064 / 0.078; 64^2, 165 rows 0.289 / 0.478; 256^2, 35 rows FP32 0.970 / 1.288, bf16
      // 0.946 / 1.133 (tensor cores), of 35 diagonal classes 2.24 / 17.7; 512^2, 35 rows 3.48 /
      // 4.74; 1024^2, 2 rows 1.69 / 2.78; Q1 dG(0) 1024^2, 35 rows 1.90 / 3.27; Q1 dG(3)
      // 512^2, 35 rows 2.30 / 3.38: faster on each of the 40 shapes measured in that range.
      if (precision == kPrecF32 && vanka_reg_eligible(L.hp.dim, L.hp.k, L.hp.n_t)) {
        // its order takes the place of the order by cell; without room for both at once the
        // level keeps that one, and its sweep is timed like the others
        e = vanka_reg_reorder(true, L.d_inv, mg.bf16, L.np, npp, mg.n_classes, L.hp.n_cells, &L.d_inv_col);
        if (e == cudaSuccess) {
          cudaFree(L.d_inv);
          L.d_inv = nullptr;
          L.vanka_kind = 2;
        } else if (e == cudaErrorMemoryAllocation) {
          cudaGetLastError();
          e = cudaSuccess;
        }
        if (e != cudaSuccess) break;
      }
    }
    if ((e = upload_vec(&L.d_grow, L.hp.g.row)) != cudaSuccess) break;
    if ((e = upload_vec(&L.d_gcol, L.hp.g.col)) != cudaSuccess) break;
    if ((e = upload_vec(&L.d_gterm, L.hp.g.term)) != cudaSuccess) break;
    if ((e = upload_vec(&L.d_gval, L.hp.g.val)) != cudaSuccess) break;
    if ((e = upload_vec(&L.d_perm, L.hp.perm)) != cudaSuccess) break;
    const size_t vb = precision == kPrecF32 ? 4 : 8;
    const size_t bytes = (size_t)L.hp.n_xi * L.hp.n_t * L.hp.n_x * vb;
    if ((e = cudaMalloc(&L.d_x, bytes)) != cudaSuccess) break;
    if ((e = cudaMalloc(&L.d_b, bytes)) != cudaSuccess) break;
    if ((e = cudaMalloc(&L.d_r, bytes)) != cudaSuccess) break;
    if (l > 0) {
      MGLevel& F = mg.lv[l - 1];
      if ((e = build_transfers(F, L, vb)) != cudaSuccess) break;
    }
  }
  if (e == cudaSuccess) e = upload_vec(&mg.d_blk_cls, blk_cls);
  if (e == cudaSuccess) e = upload_vec(&mg.d_blk_alpha, blk_alpha);
  if (e == cudaSuccess) e = cudaMalloc(&mg.d_status, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(mg.d_status, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&mg.stream, cudaStreamNonBlocking);
  const auto tt = std::chrono::steady_clock::now();
  if (e == cudaSuccess) e = tune_level_applies(mg);
  if (e == cudaSuccess) e = tune_vanka(mg);
  mg.tune_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - tt).count();
  if (e == cudaSuccess) {
    int status = 0;
    e = cudaMemcpy(&status, mg.d_status, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && status != 0) {
      msg = "multigrid set-up: a tensor-core Vanka sweep timed out waiting for its MMAs";
      return SG_ERR_TIMEOUT;
    }
  }
  if (e != cudaSuccess) {
    msg = std::string("multigrid set-up: ") + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? SG_ERR_OOM : SG_ERR_CUDA;
  }
  mg.setup_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  return SG_OK;
}

sg_status mg_build_mc(const HostProblem& fine, int precision, int nu, double omega, MG& mg, std::string& msg) {
  mg.mc = true;
  // Vanka tiles: a multiple of 8 samples whose patch data fit beside each other
  mg.vanka_tile = std::min(fine.n_xi, 64);
  if (mg.vanka_tile < fine.n_xi) mg.vanka_tile = 64;
  return mg_build(fine, precision, nu, omega, mg, msg, true);
}

sg_status mg_level_info(const MG& mg, int level, int info[10], std::string& msg) {
  if (level < 0 || level >= (int)mg.lv.size()) {
    msg = "level out of range";
    return SG_ERR_ARG;
  }
  const MGLevel& L = mg.lv[level];
  info[0] = (int)mg.lv.size();
  info[1] = (int)L.hp.n_cells;
  info[2] = L.coarsest ? 1 : 0;
  info[3] = L.coarsest ? -1 : (L.use_diag ? 1 : 0);
  info[4] = L.coarsest ? 0 : L.vanka_chunk;
  info[5] = L.coarsest ? 0 : (L.vanka_tile > 0 ? L.vanka_tile : mg.vanka_tile);
  info[6] = L.np;
  info[7] = mg.n_classes;
  info[8] = L.coarsest ? 0 : L.vanka_kind;
  info[9] = 0;
  return SG_OK;
}

sg_status mg_force_variant(MG& mg, int level, int residual_kind, int chunk, int tile, int kind, std::string& msg) {
  if (level < -1 || level >= (int)mg.lv.size()) {
    msg = "level out of range";
    return SG_ERR_ARG;
  }
  if (residual_kind < -1 || residual_kind > 1 || chunk < 0 || chunk > 8 || tile < -1 || kind < -1 || kind > 1) {
    msg = "variant out of range";
    return SG_ERR_ARG;
  }
  const size_t vb = mg.precision == kPrecF32 ? 4 : 8;
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // check every level first, then change them
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 1) {
      // levels that leave the register sweep need their inverses by cell
      std::vector<std::pair<MGLevel*, void*>> rows;
      cudaError_t e = cudaSuccess;
      for (int l = 0; l < (int)mg.lv.size() && e == cudaSuccess; ++l) {
        MGLevel& L = mg.lv[l];
        if ((level >= 0 && l != level) || L.coarsest || L.vanka_kind != 2 || (kind < 0 && chunk == 0 && tile < 0)) continue;
        rows.emplace_back(&L, nullptr);
        e = vanka_reg_reorder(false, L.d_inv_col, mg.bf16, L.np, vanka_row_pitch(L.np), mg.n_classes, L.hp.n_cells,
                              &rows.back().second);
      }
      for (auto& [L, d] : rows) {
        if (e != cudaSuccess) {
          cudaFree(d);
          continue;
        }
        L->d_inv = d;
        cudaFree(L->d_inv_col);
        L->d_inv_col = nullptr;
      }
      if (e != cudaSuccess) {
        cudaGetLastError();
        msg = std::string("inverses by cell: ") + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? SG_ERR_OOM : SG_ERR_CUDA;
      }
    }
    for (int l = 0; l < (int)mg.lv.size(); ++l) {
      if (level >= 0 && l != level) continue;
      MGLevel& L = mg.lv[l];
      if (L.coarsest) {
        if (level >= 0) {
          msg = "the coarsest level has no smoother";
          return SG_ERR_ARG;
        }
        continue;
      }
      if (residual_kind == 0 && !L.chunk_ok) {
        msg = "the SG cell kernel has no launch shape on this level";
        return SG_ERR_UNSUPPORTED;
      }
      // the register sweep has no chunk or tile: asking for one asks for the FFMA sweep
      const int kd = kind >= 0 ? kind : (L.vanka_kind == 2 && (chunk > 0 || tile >= 0) ? 0 : L.vanka_kind);
      if (kd == 2) {
        if (pass == 1 && residual_kind >= 0) L.use_diag = residual_kind == 1;
        continue;
      }
      // "keep" of a sweep that is not running: the FFMA sweep's last chunk and
      // tile, two staging buffers and all modes for the tensor-core sweep
      const int keep = kd == L.vanka_kind ? L.vanka_chunk : (kd == 0 ? L.ffma_chunk : 2);
      const int keep_tile = kd == L.vanka_kind ? L.vanka_tile : (kd == 0 ? L.ffma_tile : 0);
      const int t = tile < 0 ? (keep_tile > 0 ? keep_tile : mg.vanka_tile) : (tile == 0 ? mg.vanka_tile : tile);
      if (t != mg.vanka_tile && (t % kVankaVB != 0 || t > mg.vanka_tile)) {
        msg = "mode tiles are multiples of 4 slots, at most all of them";
        return SG_ERR_ARG;
      }
      int c = chunk > 0 ? std::min(chunk, L.hp.cells[0]) : keep;
      if (kd == 1) c = std::max(1, std::min(chunk > 0 ? chunk : c, 2));   // staging buffers of the tensor-core sweep
      if (c <= 0) c = 1;
      if (kd == 1) {
        if (!tc_level_ok(mg, L, t)) {
          msg = "the tensor-core Vanka sweep needs bf16 factors, one diagonal class, a patch of at most 64 and "
                "at most 80 slots per tile";
          return SG_ERR_UNSUPPORTED;
        }
        if (vanka_tc_smem(L.hp.dim, L.hp.k, L.hp.n_t, c, std::min(t, mg.n_blk * kVankaVB)) > (size_t)optin - 1024) {
          msg = "Vanka chunk does not fit in shared memory";
          return SG_ERR_UNSUPPORTED;
        }
      } else if (vanka_smem(L, mg.n_blk, t, c, vb, inv_value_bytes(mg)) > (size_t)optin - 1024) {
        msg = "Vanka chunk does not fit in shared memory";
        return SG_ERR_UNSUPPORTED;
      }
      if (pass == 1) {
        if (residual_kind >= 0) L.use_diag = residual_kind == 1;
        L.vanka_chunk = c;
        L.vanka_tile = t == mg.vanka_tile ? 0 : t;
        L.vanka_kind = kd;
        if (kd == 0) {
          L.ffma_chunk = c;
          L.ffma_tile = L.vanka_tile;
        }
      }
    }
  }
  // the captured V-cycles hold the old launches
  for (int t = 0; t < 2; ++t) {
    if (mg.exec_t[t]) cudaGraphExecDestroy(mg.exec_t[t]);
    if (mg.graph_t[t]) cudaGraphDestroy(mg.graph_t[t]);
    mg.exec_t[t] = nullptr;
    mg.graph_t[t] = nullptr;
  }
  return SG_OK;
}

sg_status mg_patch_inverse(const MG& mg, int level, int alpha, long long cell, double* out, std::string& msg) {
  if (level < 0 || level >= (int)mg.lv.size() || mg.lv[level].coarsest) {
    msg = "level out of range (or the coarsest level)";
    return SG_ERR_ARG;
  }
  const MGLevel& L = mg.lv[level];
  if (alpha < 0 || alpha >= (int)mg.cls.size() || cell < 0 || cell >= L.hp.n_cells) {
    msg = "mode or cell out of range";
    return SG_ERR_ARG;
  }
  const int np = L.np, npp = vanka_row_pitch(np);
  const size_t wb = inv_value_bytes(mg);
  // the patch's entries: contiguous rows, or one value of every column
  const bool by_cell = L.d_inv != nullptr;
  const int pitch = by_cell ? npp : np;
  const size_t cnt = (size_t)np * pitch;
  std::vector<unsigned char> raw(cnt * wb);
  cudaError_t e;
  if (by_cell) {
    const size_t off = ((size_t)mg.cls[alpha] * L.hp.n_cells + (size_t)cell) * cnt;
    e = cudaMemcpy(raw.data(), static_cast<const char*>(L.d_inv) + off * wb, cnt * wb, cudaMemcpyDeviceToHost);
  } else {
    const size_t off = (size_t)mg.cls[alpha] * cnt * L.hp.n_cells + (size_t)cell;
    e = cudaMemcpy2D(raw.data(), wb, static_cast<const char*>(L.d_inv_col) + off * wb, L.hp.n_cells * wb, wb, cnt,
                     cudaMemcpyDeviceToHost);
  }
  if (e != cudaSuccess) {
    msg = cudaGetErrorString(e);
    return SG_ERR_CUDA;
  }
  for (int r = 0; r < np; ++r)
    for (int c = 0; c < np; ++c) {
      const unsigned char* v = raw.data() + ((size_t)r * pitch + c) * wb;
      out[(size_t)r * np + c] = mg.bf16 ? (double)__bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(v))
                                : mg.precision == kPrecF32 ? (double)*reinterpret_cast<const float*>(v)
                                                           : *reinterpret_cast<const double*>(v);
    }
  return SG_OK;
}

// b = r in the MG precision, and the start of the finest level (x, r)
static cudaError_t mg_enter(MG& mg, const double* r, cudaStream_t s) {
  MGLevel& L = mg.lv[0];
  const int V = L.hp.n_xi * L.hp.n_t;
  if (mg.precision == kPrecF32)
    launch_vec_enter<float>(r, static_cast<float*>(L.d_b), static_cast<float*>(L.d_x), static_cast<float*>(L.d_r), V,
                            L.hp.n_x, L.hp.nn, L.hp.dim, s);
  else
    launch_vec_enter<double>(r, static_cast<double*>(L.d_b), static_cast<double*>(L.d_x), static_cast<double*>(L.d_r), V,
                             L.hp.n_x, L.hp.nn, L.hp.dim, s);
  return cudaGetLastError();
}

static cudaError_t mg_leave(MG& mg, double* z, cudaStream_t s) {
  MGLevel& L = mg.lv[0];
  const long long n = (long long)L.hp.n_xi * L.hp.n_t * L.hp.n_x;
  if (mg.precision == kPrecF32)
    mg_convert<float, double><<<grid_for(n, 256), 256, 0, s>>>(static_cast<const float*>(L.d_x), z, n);
  else
    mg_convert<double, double><<<grid_for(n, 256), 256, 0, s>>>(static_cast<const double*>(L.d_x), z, n);
  return cudaGetLastError();
}

cudaError_t mg_issue(MG& mg, const double* r, double* z, cudaStream_t stream, int trans) {
  const int t = trans ? 1 : 0;
  cudaError_t e = mg_enter(mg, r, stream);
  if (e == cudaSuccess)
    e = mg.precision == kPrecF32 ? issue_vcycle<float>(mg, 0, stream, t) : issue_vcycle<double>(mg, 0, stream, t);
  return e == cudaSuccess ? mg_leave(mg, z, stream) : e;
}

cudaError_t mg_apply(MG& mg, const double* r, double* z, cudaStream_t stream, int trans) {
  const bool f32 = mg.precision == kPrecF32;
  const int t = trans ? 1 : 0;
  cudaError_t e;
  if (!mg.exec_t[t]) {
    if ((e = cudaStreamBeginCapture(mg.stream, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) return e;
    cudaError_t ei = f32 ? issue_vcycle<float>(mg, 0, mg.stream, t) : issue_vcycle<double>(mg, 0, mg.stream, t);
    e = cudaStreamEndCapture(mg.stream, &mg.graph_t[t]);
    if (ei != cudaSuccess) return ei;
    if (e != cudaSuccess) return e;
    if ((e = cudaGraphInstantiate(&mg.exec_t[t], mg.graph_t[t], 0)) != cudaSuccess) return e;
  }
  if ((e = mg_enter(mg, r, stream)) != cudaSuccess) return e;
  if ((e = cudaGraphLaunch(mg.exec_t[t], stream)) != cudaSuccess) return e;
  return mg_leave(mg, z, stream);
}

}  // namespace sg

SG_BOUNDS_FETCH(bounds_fetch_mg)
