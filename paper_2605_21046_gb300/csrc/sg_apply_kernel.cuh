// The SG slab-operator apply kernel, generic over the arithmetic policy
// (sg_arith.h).  See sg_apply.cu for the design; this header holds the device
// code that both precisions instantiate.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "sg_arith.h"
#include "sg_bounds.h"
#include "sg_internal.h"
#include "sg_shape_tables.h"

namespace sg {

template <int DIM, int K>
struct Shape {
  static constexpr int N = K + 1;                       // nodes = Gauss points per direction
  static constexpr int NKD = DIM == 2 ? N * N : N * N * N;
  static constexpr int NQD = NKD;
  static constexpr int NC = 1 + DIM;                    // value + gradient per point
};

template <int K>
__device__ __forceinline__ constexpr Cf cS(int a, int b) {
  return {RefShape<K>::S(a, b), RefShape<K>::Sh(a, b), RefShape<K>::Sl(a, b)};
}
template <int K>
__device__ __forceinline__ constexpr Cf cD(int a, int b) {
  return {RefShape<K>::D(a, b), RefShape<K>::Dh(a, b), RefShape<K>::Dl(a, b)};
}

// sum_j c(j) x(j) over J compile-time terms; exact zeros are skipped, a lone
// +-1 term is an exact copy, every other result is normalised once.
template <class A, int J, class CF, class XF>
__device__ __forceinline__ typename A::T cdot(CF cf, XF xf) {
  typename A::T s = A::zero();
  int nt = 0;
  bool unit = true;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const Cf c = cf(j);
    if (c.c == 0.0) continue;
    if (nt == 0) s = A::cmul(c, xf(j));
    else A::cfma(c, xf(j), s);
    ++nt;
    if (!(c.c == 1.0 || c.c == -1.0)) unit = false;
  }
  if (nt == 1 && unit) return s;
  return A::fin(s);
}

// --------------------------------------------------------------- 1D lines
// The passes of the sum factorisation along one line of N = K + 1 values.
//
// Derivatives are taken in units of a unit of their own: with the Gauss points'
// symmetry the collocation derivative needs few multiplies, and the remaining
// common factor of every gradient is left out here and put back, squared, into
// the coefficient (grad_weight<K>()), which multiplies each gradient once on
// its way there and back.  FP64 instructions per line, dense tables against
// this form: Q2 interpolation 6 / 6, derivative 8 / 4, their transposes 7 / 6
// and 8 / 7, and 9 and 12 where one line needs value and derivative (15 and
// 15); Q3 interpolation 16 / 14, derivative 16 / 12, transposes 16 / 14 and 16 / 18, both
// at once 24 and 26 (32); Q1 derivative 4 / 2.  Double-word sums cost more than products (8 against
// 4 instructions), so that arithmetic keeps the dense interpolation.  The
// constants of the parts are rounded once from 40 digits (RefShape::L): formed
// from the rounded tables they cost Q3 65 % more error.  Measured inside the
// domain against an 80-bit reference, FP64 Q2 0.86e-15 (dense tables 1.02e-15),
// Q3 3.5e-16 (3.7e-16), Q1 the same.
// That weight is 1 for Q1 (which has one multiply to lose, and loses accuracy
// with a rounded 3 a), 5/3 for Q2, and the square of Q3's unit.
template <int K>
__host__ __device__ constexpr double grad_weight() {
  return RefShape<K>::W;
}
inline double grad_weight(int k) {
  return k == 1 ? RefShape<1>::W : (k == 2 ? RefShape<2>::W : RefShape<3>::W);
}
__host__ __device__ constexpr Cf cf_of(double c) {
  return {c, (float)c, (float)(c - (double)(float)c)};
}

// FP64 constants.  A GB300 SM takes 16.9 cycles per warp for a DFMA of three
// registers but 20.0 for a DADD, a DMUL, or a DFMA with a literal or
// constant-bank operand (measured; the kernels here sat at 82 % of the FP64
// pipe at any occupancy).  So sums and products are written as fma(x, 1, y)
// and fma(x, y, -0), which round the same, and every constant is read from a
// shared-memory array, which forces it into a register.  64^2 Q2 165 -> 149 us,
// 32^3 Q2 3.02 -> 2.73 ms, 128^2 Q3 dG(3) 1.62 -> 1.47 ms.
enum { kOne, kNegZero, kTwo, kFour, kLineOwn };   // constants of every degree; then the degree's own
// Q2: half the difference of the end functions at the outer Gauss point
// (sqrt(3/5) / 2); their mean there is 0.3, the middle function 0.4.
enum { kA2 = kLineOwn, kM2, kB2, kG2 };
// Q3: even (E) and odd (C) parts of the end (0) and inner (1) basis functions
// at the outer (o) and inner (i) Gauss points, ratios of the odd parts, and
// the derivative's weights on (v3 - v0), (v2 - v1), (v0 + v3) - (v1 + v2).
enum { kEo0 = kLineOwn, kEo1, kEi0, kEi1, kCo, kCi, kRo, kRi, kTo, kTi, kAi, kBo, kBi, kQo, kQi, kQo2, kQi2, kAi2, kBo2, kBi2 };

template <int K>
__host__ __device__ constexpr double line_const(int i) {
  return i == kOne ? 1.0 : i == kNegZero ? -0.0 : i == kTwo ? 2.0 : i == kFour ? 4.0 : RefShape<K>::L(i - kLineOwn);
}
// The line constants of a degree as a kernel parameter (kLineConsts values).
inline void fill_line_consts(int k, double* out) {
  constexpr int n[4] = {0, kLineOwn, kG2 + 1, kBi2 + 1};
  for (int i = 0; i < kLineConsts; ++i)
    out[i] = i >= n[k] ? 0.0 : (k == 1 ? line_const<1>(i) : (k == 2 ? line_const<2>(i) : line_const<3>(i)));
}

template <class A, int K>
struct Line {
  using T = typename A::T;
  static constexpr int N = K + 1;
  static constexpr bool kF64 = std::is_same<A, F64>::value;
  const double* k;   // the constants in shared memory
  __device__ __forceinline__ explicit Line(const double* lk) : k(lk) {}

  __device__ __forceinline__ double reg(int i) const { return k[i]; }
  __device__ __forceinline__ T add(T a, T b) const {
    if constexpr (kF64) return ::fma(a, reg(kOne), b);
    else return A::add(a, b);
  }
  __device__ __forceinline__ T sub(T a, T b) const {
    if constexpr (kF64) return ::fma(b, -reg(kOne), a);
    else return A::add(a, A::neg(b));
  }
  __device__ __forceinline__ T mul(T a, T b) const {
    if constexpr (kF64) return ::fma(a, b, reg(kNegZero));
    else return A::mul(a, b);
  }
  // c x + y, -c x + y and c x for the constant I, as sums still to be finished (A::fin)
  template <int I>
  __device__ __forceinline__ T axpy(T x, T y) const {
    if constexpr (kF64) {
      return ::fma(reg(I), x, y);
    } else {
      A::cfma(cf_of(line_const<K>(I)), x, y);
      return y;
    }
  }
  template <int I>
  __device__ __forceinline__ T axmy(T x, T y) const {
    if constexpr (kF64) {
      return ::fma(-reg(I), x, y);
    } else {
      A::cfma(cf_of(-line_const<K>(I)), x, y);
      return y;
    }
  }
  template <int I>
  __device__ __forceinline__ T scale(T x) const {
    if constexpr (kF64) return ::fma(reg(I), x, reg(kNegZero));
    else return A::cmul(cf_of(line_const<K>(I)), x);
  }
  template <class F>
  static __device__ __forceinline__ void dense(F c, const T* x, T* y) {
#pragma unroll
    for (int a = 0; a < N; ++a)
      y[a] = cdot<A, N>([&](int j) { return c(a, j); }, [&](int j) { return x[j]; });
  }
  static __device__ __forceinline__ T lit_axpy(Cf c, T x, T y) {
    A::cfma(c, x, y);
    return y;
  }

  // nodal values -> values at the Gauss points
  __device__ __forceinline__ void interp(const T (&u)[N], T (&v)[N]) const {
    if constexpr (A::kDW || K == 1) {
      dense([](int a, int j) { return cS<K>(a, j); }, u, v);
    } else if constexpr (K == 2) {
      const T s = add(u[0], u[2]), d = sub(u[2], u[0]);
      const T e = axpy<kA2>(s, scale<kM2>(u[1]));
      v[0] = axmy<kB2>(d, e);
      v[1] = u[1];
      v[2] = axpy<kB2>(d, e);
    } else {
      T eo, ei;
      cubic(u, v, eo, ei);
    }
  }
  // values at the Gauss points -> derivatives there, in the scaled unit
  __device__ __forceinline__ void deriv(const T (&v)[N], T (&g)[N]) const {
    if constexpr (K == 1) {
      g[0] = g[1] = A::fin(lit_axpy(cD<1>(1, 1), v[1], A::cmul(cD<1>(1, 0), v[0])));
    } else if constexpr (K == 2) {
      const T m = sub(v[2], v[0]), a = sub(v[2], v[1]);
      const T p = axpy<kFour>(a, A::neg(m));
      g[0] = A::fin(axpy<kTwo>(m, A::neg(p)));
      g[1] = A::fin(m);
      g[2] = A::fin(p);
    } else {
      const T q = sub(add(v[0], v[3]), add(v[1], v[2]));
      cubic_deriv(sub(v[3], v[0]), sub(v[2], v[1]), q, g);
    }
  }
  // both at once (v as interp, g as deriv of v)
  __device__ __forceinline__ void interp_deriv(const T (&u)[N], T (&v)[N], T (&g)[N]) const {
    if constexpr (!A::kDW && K == 2) {
      const T s = add(u[0], u[2]), d = sub(u[2], u[0]);
      const T t = axmy<kTwo>(u[1], s);
      const T e = axpy<kA2>(t, u[1]);
      v[0] = axmy<kB2>(d, e);
      v[1] = u[1];
      v[2] = axpy<kB2>(d, e);
      const T m = sub(v[2], v[0]);
      g[0] = axmy<kG2>(t, m);
      g[1] = m;
      g[2] = axpy<kG2>(t, m);
    } else if constexpr (!A::kDW && K == 3) {
      T eo, ei;
      cubic(u, v, eo, ei);
      const T q = sub(eo, ei);
      cubic_deriv(sub(v[3], v[0]), sub(v[2], v[1]), add(q, q), g);
    } else {
      interp(u, v);
      deriv(v, g);
    }
  }
  // r += transpose of deriv applied to g (sums still to be finished)
  __device__ __forceinline__ void deriv_t(const T (&g)[N], T (&r)[N]) const {
    if constexpr (K == 1) {
      const T G = add(g[0], g[1]);
      r[0] = lit_axpy(cD<1>(0, 0), G, r[0]);
      r[1] = lit_axpy(cD<1>(0, 1), G, r[1]);
    } else if constexpr (K == 2) {
      const T P = sub(g[2], g[0]);
      const T B = sub(axpy<kTwo>(g[0], g[1]), P);   // the odd part: -B on one end, B + 4 P on the other
      r[0] = sub(r[0], B);
      r[1] = axmy<kFour>(P, r[1]);
      r[2] = axpy<kFour>(P, add(r[2], B));
    } else if constexpr (A::kDW) {
#pragma unroll
      for (int a = 0; a < N; ++a)
#pragma unroll
        for (int j = 0; j < N; ++j) r[a] = lit_axpy(cf_of(deriv_const(j, a)), g[j], r[a]);
    } else {
      const T Go = add(g[0], g[3]), Gi = add(g[1], g[2]), Ho = sub(g[3], g[0]), Hi = sub(g[2], g[1]);
      const T Q = axpy<kQo>(Ho, scale<kQi>(Hi));
      const T X = axpy<kAi>(Gi, Go), Y = axpy<kBi>(Gi, scale<kBo>(Go));
      r[0] = sub(add(r[0], Q), X);
      r[1] = sub(sub(r[1], Q), Y);
      r[2] = add(sub(r[2], Q), Y);
      r[3] = add(add(r[3], Q), X);
    }
  }
  // transpose of interp
  __device__ __forceinline__ void interp_t(const T (&r)[N], T (&n)[N]) const {
    if constexpr (A::kDW || K == 1) {
      dense([](int a, int j) { return cS<K>(j, a); }, r, n);
    } else if constexpr (K == 2) {
      quad_t(add(r[0], r[2]), sub(r[2], r[0]), r[1], n);
    } else {
      cubic_t(add(r[0], r[3]), add(r[1], r[2]), sub(r[3], r[0]), sub(r[2], r[1]), n);
    }
  }
  // n = transpose of interp applied to (r + transpose of deriv applied to g)
  __device__ __forceinline__ void interp_deriv_t(T (&r)[N], const T (&g)[N], T (&n)[N]) const {
    if constexpr (!A::kDW && K == 2) {
      const T P = sub(g[2], g[0]), S = add(add(g[0], g[2]), g[1]);
      quad_t(axpy<kFour>(P, add(r[0], r[2])), axpy<kTwo>(S, sub(r[2], r[0])), axmy<kFour>(P, r[1]), n);
    } else if constexpr (!A::kDW && K == 3) {
      const T Go = add(g[0], g[3]), Gi = add(g[1], g[2]), Ho = sub(g[3], g[0]), Hi = sub(g[2], g[1]);
      const T Q = axpy<kQo2>(Ho, scale<kQi2>(Hi));
      const T so = add(add(r[0], r[3]), Q), si = sub(add(r[1], r[2]), Q);
      const T dO = axpy<kAi2>(Gi, axpy<kTwo>(Go, sub(r[3], r[0])));
      const T dI = axpy<kBi2>(Gi, axpy<kBo2>(Go, sub(r[2], r[1])));
      cubic_t(so, si, dO, dI, n);
    } else {
      deriv_t(g, r);
#pragma unroll
      for (int a = 0; a < N; ++a) r[a] = A::fin(r[a]);
      interp_t(r, n);
    }
  }

 private:
  // Q3: weight of value a in the derivative at point j, from the parts
  static __host__ __device__ constexpr double deriv_const(int j, int a) {
    const bool inner = j == 1 || j == 2, in_a = a == 1 || a == 2;
    const double odd = inner ? line_const<3>(in_a ? kBi : kAi) : (in_a ? line_const<3>(kBo) : 1.0);
    const double even = line_const<3>(inner ? kQi : kQo);
    return (a >= 2 ? odd : -odd) + ((j >= 2) != in_a ? even : -even);
  }
  __device__ __forceinline__ void quad_t(T s, T o, T r1, T (&n)[N]) const {
    const T t = scale<kA2>(s);
    n[0] = axmy<kB2>(o, t);
    n[1] = axpy<kM2>(s, r1);
    n[2] = axpy<kB2>(o, t);
  }
  __device__ __forceinline__ void cubic(const T (&u)[N], T (&v)[N], T& eo, T& ei) const {
    const T s0 = add(u[0], u[3]), s1 = add(u[1], u[2]), d0 = sub(u[3], u[0]), d1 = sub(u[2], u[1]);
    eo = axpy<kEo1>(s1, scale<kEo0>(s0));
    ei = axpy<kEi1>(s1, scale<kEi0>(s0));
    const T wo = axpy<kRo>(d1, d0), wi = axpy<kRi>(d0, d1);
    v[0] = axmy<kCo>(wo, eo);
    v[1] = axmy<kCi>(wi, ei);
    v[2] = axpy<kCi>(wi, ei);
    v[3] = axpy<kCo>(wo, eo);
  }
  __device__ __forceinline__ void cubic_deriv(T d0, T d1, T q, T (&g)[N]) const {
    const T eo = axpy<kBo>(d1, d0), ei = axpy<kBi>(d1, scale<kAi>(d0));
    g[0] = A::fin(axmy<kQo>(q, eo));
    g[1] = A::fin(axmy<kQi>(q, ei));
    g[2] = A::fin(axpy<kQi>(q, ei));
    g[3] = A::fin(axpy<kQo>(q, eo));
  }
  __device__ __forceinline__ void cubic_t(T so, T si, T dO, T dI, T (&n)[N]) const {
    const T n0 = axpy<kEi0>(si, scale<kEo0>(so)), n1 = axpy<kEi1>(si, scale<kEo1>(so));
    const T x0 = axpy<kTo>(dI, dO), x1 = axpy<kTi>(dO, dI);
    n[0] = axmy<kCo>(x0, n0);
    n[1] = axmy<kCi>(x1, n1);
    n[2] = axpy<kCi>(x1, n1);
    n[3] = axpy<kCo>(x0, n0);
  }
};

// Line i (of the others, counted in order) along direction d of an N^DIM
// array, x fastest: its first entry and its stride.
template <int N>
__host__ __device__ constexpr int line_stride(int d) {
  return d == 0 ? 1 : (d == 1 ? N : N * N);
}
template <int N>
__host__ __device__ constexpr int line_first(int d, int i) {
  return d == 0 ? i * N : (d == 1 ? (i / N) * N * N + i % N : i);
}

// --------------------------------------------------------------- phase 1
// Nodal values u (lexicographic, x fastest) -> values and reference gradients
// (in that unit) at the tensor Gauss points: x, then y (, then z)
// interpolation in place, the last direction with its derivative; the other
// derivatives by collocation.  put(comp * NQD + point, value) stores them.
template <class A, int DIM, int K, class Put>
__device__ __forceinline__ void forward_cell(const Line<A, K>& L, typename A::T* u, Put put) {
  using T = typename A::T;
  constexpr int N = K + 1, NQD = Shape<DIM, K>::NQD, NL = NQD / N;
  T in[N], v[N], g[N];
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const int st = line_stride<N>(d);
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int o = line_first<N>(d, i);
#pragma unroll
      for (int j = 0; j < N; ++j) in[j] = u[o + j * st];
      if (d + 1 < DIM) {
        L.interp(in, v);
      } else {
        L.interp_deriv(in, v, g);
#pragma unroll
        for (int j = 0; j < N; ++j) put((1 + d) * NQD + o + j * st, g[j]);
      }
#pragma unroll
      for (int j = 0; j < N; ++j) {
        u[o + j * st] = v[j];
        if (d + 1 == DIM) put(o + j * st, v[j]);
      }
    }
  }
#pragma unroll
  for (int d = 0; d + 1 < DIM; ++d) {
    const int st = line_stride<N>(d);
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int o = line_first<N>(d, i);
#pragma unroll
      for (int j = 0; j < N; ++j) in[j] = u[o + j * st];
      L.deriv(in, g);
#pragma unroll
      for (int j = 0; j < N; ++j) put((1 + d) * NQD + o + j * st, g[j]);
    }
  }
}

// --------------------------------------------------------------- phase 3
// Point values and reference-gradient coefficients (get(comp * NQD + point))
// -> nodal contributions r: the transpose of forward_cell.
template <class A, int DIM, int K, class Get>
__device__ __forceinline__ void backward_cell(const Line<A, K>& L, Get get, typename A::T* r) {
  using T = typename A::T;
  constexpr int N = K + 1, NQD = Shape<DIM, K>::NQD, NL = NQD / N;
  T in[N], g[N], out[N];
#pragma unroll
  for (int q = 0; q < NQD; ++q) r[q] = get(q);
#pragma unroll
  for (int d = 0; d + 1 < DIM; ++d) {
    const int st = line_stride<N>(d);
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int o = line_first<N>(d, i);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        in[j] = r[o + j * st];
        g[j] = get((1 + d) * NQD + o + j * st);
      }
      L.deriv_t(g, in);
#pragma unroll
      for (int j = 0; j < N; ++j) r[o + j * st] = in[j];
    }
  }
#pragma unroll
  for (int d = DIM - 1; d >= 0; --d) {
    const int st = line_stride<N>(d);
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int o = line_first<N>(d, i);
#pragma unroll
      for (int j = 0; j < N; ++j) in[j] = r[o + j * st];
      if (d + 1 == DIM) {
#pragma unroll
        for (int j = 0; j < N; ++j) g[j] = get((1 + d) * NQD + o + j * st);
        L.interp_deriv_t(in, g, out);
      } else {
        L.interp_t(in, out);
      }
#pragma unroll
      for (int j = 0; j < N; ++j) r[o + j * st] = out[j];
    }
  }
}

// One coupling entry of a chaos row, packed for a single 8-byte shared load:
// the offset of column beta's vectors in a cell's value block and the offset
// of the entry's coefficient row in a cell's coefficient block (its (term, G)
// pair with pre-multiplied rows, else its term; -1 - e for an entry e whose
// pair is missing from the pair list, which then reads its tables globally).
struct alignas(8) CoupleEntry {
  int off;
  int tq;
};

// Phase-2 items held per thread (their results live in registers until the
// round's barrier), and the launch bounds: the 2D shapes with at most two
// time nodes and degree <= 2 run two 384-thread CTAs per SM within 80
// registers.
__host__ __device__ constexpr int chunk_kmax(int dim, int nt) {
  return 18 / (nt * (1 + dim)) < 1 ? 1 : (18 / (nt * (1 + dim)) > 3 ? 3 : 18 / (nt * (1 + dim)));
}
template <int DIM, int K, int NT>
struct ChunkBounds {
  static constexpr bool tight = DIM == 2 && K <= 2 && NT <= 2;
  static constexpr int threads = tight ? 384 : 512;
  static constexpr int blocks = tight ? 2 : 1;
};

// The persistent chunk kernel (design notes in sg_apply.cu).
template <class A, int DIM, int K, int NT>
__global__ void __launch_bounds__(ChunkBounds<DIM, K, NT>::threads, ChunkBounds<DIM, K, NT>::blocks)
    sg_apply_chunk_kernel(const __grid_constant__ ApplyParams p) {
  using T = typename A::T;
  using Sh = Shape<DIM, K>;
  constexpr int NQD = Sh::NQD, NKD = Sh::NKD, NC = Sh::NC, N = Sh::N;
  constexpr int SLOT = (NC * NQD) | 1;           // values per (cell, vector), odd pitch: no bank conflicts
                                                 // between the vectors of phases 1 and 3
  using IO = typename A::IO;
  const IO* __restrict__ xin = reinterpret_cast<const IO*>(p.x);
  IO* __restrict__ yout = reinterpret_cast<IO*>(p.y);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int n_xi = p.n_xi, V = n_xi * NT, C = p.chunk;
  __shared__ double s_lk[kLineConsts];   // an array of its own: stores to the values cannot alias it
  if (std::is_same<A, F64>::value && tid < kLineConsts) s_lk[tid] = p.lk[tid];   // visible after the first barrier
  const Line<A, K> L(s_lk);

  const bool premul = p.premul != 0;
  const int rows = premul ? p.n_pairs : p.n_terms;              // coefficient rows per cell
  T* Qs = reinterpret_cast<T*>(smem_raw);                       // [C][V][NC][NQD]
  T* Cs = Qs + (size_t)C * V * SLOT;                            // [C][rows][NQD]
  T* Amq = Cs + (size_t)C * rows * NQD;                         // [NQD][NT][NT]
  T* Tb = Amq + NQD * NT * NT;                                  // [NT]
  T* Rt = Tb + NT;                                              // [3] (h_0/h_d)^2
  T* Gv = Rt + 3;                                               // G per entry (unused with premul)
  // the packed coupling entries follow at a 16-byte boundary
  CoupleEntry* Ge = reinterpret_cast<CoupleEntry*>(
      (reinterpret_cast<uintptr_t>(Gv + (premul ? p.n_pairs : p.nnz)) + 15) & ~static_cast<uintptr_t>(15));
  int* Gr = reinterpret_cast<int*>(Ge + p.nnz);                 // [n_xi+1]
  int* Pm = Gr + n_xi + 1;                                      // [n_xi]
  int* Pt = Pm + n_xi;                                          // [n_pairs] term of each pair
  int* Nd = Pt + (premul ? p.n_pairs : 0);                      // [C][NKD] node of y / x, -1 on the boundary

  if (premul) {
    for (int k = tid; k < p.n_pairs; k += nthr) Pt[k] = p.pair_term[k];
  } else {
    for (int e = tid; e < p.nnz; e += nthr) Gv[e] = A::in(p.g_val[e]);
  }
  for (int e = tid; e < p.nnz; e += nthr) {
    CoupleEntry ce;
    ce.off = SG_IN(p.g_col[e], n_xi, 105) ? p.g_col[e] * NT * SLOT : 0;
    const int t = p.g_term[e];
    if (premul) {
      const double v = p.g_val[e];
      int k = 0;
      while (k < p.n_pairs && !(p.pair_term[k] == t && p.pair_val[k] == v)) ++k;
      ce.tq = k < p.n_pairs ? k * NQD : -1 - e;
    } else {
      ce.tq = SG_IN(t, p.n_terms, 106) ? t * NQD : 0;
    }
    Ge[e] = ce;
  }
  for (int e = tid; e <= n_xi; e += nthr) Gr[e] = p.g_row[e];
  for (int e = tid; e < n_xi; e += nthr) Pm[e] = p.perm[e];
  for (int e = tid; e < NQD * NT * NT; e += nthr) Amq[e] = A::in(p.amq[e]);
  if (tid < NT) Tb[tid] = A::in(p.mode == kApplyResidual ? -p.tb[tid] : p.tb[tid]);
  if (tid < 3) Rt[tid] = A::in(p.ratio[tid]);

  const long long c_begin = (long long)blockIdx.x * p.n_cells / gridDim.x;
  const long long c_end = (long long)(blockIdx.x + 1) * p.n_cells / gridDim.x;
  const int nnx = p.nn[0], nny = p.nn[1], nnz_ = p.nn[2];

  // the upper half of the CTAs may start with a shorter chunk, so that CTAs
  // sharing an SM do not reach their gather and scatter phases together
  const int first = (p.stagger > 0 && blockIdx.x >= gridDim.x / 2) ? min(C, p.stagger) : C;
  int nc = 0;
  for (long long c0 = c_begin; c0 < c_end; c0 += nc) {
    nc = (int)min((long long)(c0 == c_begin ? first : C), c_end - c0);
    __syncthreads();   // previous chunk done with Qs / Cs; tables visible
    // ---------------------------------------------------------- phase 0
    {
      const int per_cell = p.n_terms * NQD;
      if (premul) {
        // G value x a_term(x_q) per (cell, pair, point), multiplied in FP64
        // and converted once; pair_w carries the gradients' weight
        const int per_row = rows * NQD;
        for (int idx = tid; idx < nc * per_row; idx += nthr) {
          const int c = idx / per_row, r = idx - c * per_row;
          const int k = r / NQD, q = r - k * NQD;
          const long long at = (c0 + c) * per_cell + Pt[k] * NQD + q;
          if (SG_IN(at, p.n_cells * per_cell, 101)) Cs[idx] = A::in(p.pair_w[k] * p.ctab[at]);
        }
      } else {
        for (int idx = tid; idx < nc * per_cell; idx += nthr)
          if (SG_IN(c0 * per_cell + idx, p.n_cells * per_cell, 101))
            Cs[idx] = A::in(grad_weight<K>() * p.ctab[c0 * per_cell + idx]);
      }
    }
    // the global node of every (cell, local node) of the chunk, once per
    // chunk instead of once per vector (the integer divisions by the mesh
    // extents would otherwise dominate the gather and scatter)
    for (int i = tid; i < nc * NKD; i += nthr) {
      const int c = i / NKD, a = i - c * NKD;
      const unsigned int gc = (unsigned int)(c0 + c);       // cells < 2^31: 32-bit divisions
      const int cx = (int)(gc % (unsigned int)p.cells[0]);
      const int cy = (int)((gc / (unsigned int)p.cells[0]) % (unsigned int)p.cells[1]);
      const int cz = (int)(gc / ((unsigned int)p.cells[0] * (unsigned int)p.cells[1]));
      const int gx = cx * K + a % N, gy = cy * K + (a / N) % N, gz = DIM == 3 ? cz * K + a / (N * N) : 0;
      bool interior = gx > 0 && gx < nnx - 1 && gy > 0 && gy < nny - 1;
      if (DIM == 3) interior = interior && gz > 0 && gz < nnz_ - 1;
      const long long node = ((long long)gz * nny + gy) * nnx + gx;
      Nd[i] = interior && SG_IN(node, p.n_x, 102) ? (int)node : -1;
    }
    __syncthreads();
    // FP64 and FP32: the thread of a (cell, vector) loads its nodal values
    // itself in phase 1.  Double-word, which converts every value it loads,
    // stages them, spread over all threads.
    if constexpr (A::kDW) {
      // GU values per thread in flight: a batch's loads all issue before its
      // shared-memory stores
      constexpr int GU = 4;
      for (int c = 0; c < nc; ++c) {
        const int* nd = Nd + c * NKD;
        T* qc = Qs + (size_t)c * V * SLOT;
        for (int j0 = tid; j0 < V * NKD; j0 += GU * nthr) {
          T val[GU];
          int dst[GU];
#pragma unroll
          for (int g = 0; g < GU; ++g) {
            const int j = j0 + g * nthr;
            const int v = j / NKD, a = j - v * NKD;
            val[g] = A::zero();
            dst[g] = j < V * NKD ? v * SLOT + a : -1;
            const int node = j < V * NKD ? nd[a] : -1;
            if (node >= 0 && SG_IN((long long)v * p.n_x + node, (long long)V * p.n_x, 103))
              val[g] = A::in(xin[(long long)v * p.n_x + node]);
          }
#pragma unroll
          for (int g = 0; g < GU; ++g)
            if (dst[g] >= 0 && SG_IN((size_t)c * V * SLOT + dst[g], (size_t)C * V * SLOT, 104)) qc[dst[g]] = val[g];
        }
      }
      __syncthreads();
    }
    // ---------------------------------------------------------- phase 1
    for (int it = tid; it < nc * V; it += nthr) {
      T* q = Qs + (size_t)it * SLOT;
      T u[NKD];
      if constexpr (A::kDW) {
#pragma unroll
        for (int a = 0; a < NKD; ++a) u[a] = q[a];
      } else {
        const int c = it / V, v = it - c * V;
        const int* nd = Nd + c * NKD;
        const IO* src = xin + (long long)v * p.n_x;
#pragma unroll
        for (int a = 0; a < NKD; ++a) {
          const int node = nd[a];
          u[a] = node >= 0 && SG_IN((long long)v * p.n_x + node, (long long)V * p.n_x, 103) ? A::in(src[node]) : A::zero();
        }
      }
      forward_cell<A, DIM, K>(L, u, [&](int o, T val) { q[o] = val; });
    }
    __syncthreads();
    // ---------------------------------------------------------- phase 2
    // Rounds of PB Gauss points: the items of a round are (chaos row, point)
    // pairs, consecutive threads taking consecutive points of one row, so a
    // warp follows a single row (no divergence in the coupling loop, one
    // broadcast load per entry).  A thread holds up to KMAX items' results in
    // registers; every read of a round's points precedes its writes (one
    // barrier), and rounds touch disjoint points.
    {
      constexpr int KMAX = chunk_kmax(DIM, NT);
      const int PB = min(32, max(1, (KMAX * nthr) / n_xi));
      const int npts = nc * NQD;
      for (int p0 = 0; p0 < npts; p0 += PB) {
        const int pb = min(PB, npts - p0);
        const int items = n_xi * pb;
        T out[KMAX][NT][NC];
        int a_of[KMAX], c_of[KMAX], q_of[KMAX];
#pragma unroll
        for (int kk = 0; kk < KMAX; ++kk) {
          const int it = tid + kk * nthr;
          a_of[kk] = -1;
          c_of[kk] = q_of[kk] = 0;
          if (it < items) {
            const int slot = it / pb, pt = p0 + (it - slot * pb);
            const int a = Pm[slot];
            const int c = pt / NQD, q = pt - c * NQD;
            a_of[kk] = a;
            c_of[kk] = c;
            q_of[kk] = q;
            const T* base = Qs + (size_t)c * V * SLOT + q;
            T uv[NT];
#pragma unroll
            for (int j = 0; j < NT; ++j) uv[j] = base[(size_t)(a * NT + j) * SLOT];
            const T* am = Amq + q * NT * NT;
#pragma unroll
            for (int i = 0; i < NT; ++i) {
              T s = L.mul(am[i * NT], uv[0]);
#pragma unroll
              for (int j = 1; j < NT; ++j) A::fma(am[i * NT + j], uv[j], s);
              out[kk][i][0] = A::fin(s);
#pragma unroll
              for (int d = 0; d < DIM; ++d) out[kk][i][1 + d] = A::zero();
            }
            const T* cq = Cs + (size_t)c * rows * NQD + q;
            const int e_beg = Gr[a], e_end = Gr[a + 1];
            if constexpr (A::kDW) {
              // The first entry starts the sums (a sum costs twice a product) and
              // the others go two at a time, with the loads of both ahead of their
              // long arithmetic (128^2 Q2 M=4 P=4 649 -> 626 us).  FP64 takes them
              // one by one: in pairs, or with the values of one loaded ahead,
              // 32^3 Q2 went from 2.73 to 2.90 and 3.01 ms.
              // An entry's weight: the staged product, or G times the staged a_term
              // (-1 - e marks a pair missing from the pair list: tables from memory).
              auto weight = [&](int e, const CoupleEntry ce) -> T {
                if (premul) {
                  if (ce.tq >= 0) return cq[ce.tq];
                  const long long at = (c0 + c) * p.n_terms * NQD + p.g_term[e] * NQD + q;
                  const double a_q = SG_IN(at, p.n_cells * p.n_terms * NQD, 108) ? p.ctab[at] : 0.0;
                  return A::fin(A::mul(A::in(p.g_val[e]), A::in(grad_weight<K>() * a_q)));
                }
                return A::fin(A::mul(Gv[e], cq[ce.tq]));
              };
              auto load = [&](const CoupleEntry ce, T (&g)[NT][DIM]) {
                const T* gb = base + ce.off;
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                  for (int d = 0; d < DIM; ++d) g[i][d] = gb[(size_t)i * SLOT + (1 + d) * NQD];
              };
              auto couple = [&](const T w, const T (&g)[NT][DIM]) {
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                  for (int d = 0; d < DIM; ++d) A::fma(w, g[i][d], out[kk][i][1 + d]);
              };
              int e = e_beg;
              if (e < e_end) {
                const CoupleEntry ce = Ge[e];
                const T w = weight(e, ce);
                T g[NT][DIM];
                load(ce, g);
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                  for (int d = 0; d < DIM; ++d) out[kk][i][1 + d] = A::mul(w, g[i][d]);
                ++e;
              }
              for (; e + 1 < e_end; e += 2) {
                const CoupleEntry ce0 = Ge[e], ce1 = Ge[e + 1];
                const T w0 = weight(e, ce0), w1 = weight(e + 1, ce1);
                T g0[NT][DIM], g1[NT][DIM];
                load(ce0, g0);
                load(ce1, g1);
                couple(w0, g0);
                couple(w1, g1);
              }
              if (e < e_end) {
                const CoupleEntry ce = Ge[e];
                const T w = weight(e, ce);
                T g[NT][DIM];
                load(ce, g);
                couple(w, g);
              }
            } else {
              auto couple = [&](const T w, const int off) {
                const T* gb = base + off;
#pragma unroll
                for (int i = 0; i < NT; ++i)
#pragma unroll
                  for (int d = 0; d < DIM; ++d) A::fma(w, gb[(size_t)i * SLOT + (1 + d) * NQD], out[kk][i][1 + d]);
              };
              if (premul) {
                for (int e = e_beg; e < e_end; ++e) {
                  const CoupleEntry ce = Ge[e];
                  if (ce.tq >= 0) {
                    couple(cq[ce.tq], ce.off);
                  } else {
                    const int ee = -1 - ce.tq;
                    const long long at = (c0 + c) * p.n_terms * NQD + p.g_term[ee] * NQD + q;
                    const double a_q = SG_IN(at, p.n_cells * p.n_terms * NQD, 108) ? p.ctab[at] : 0.0;
                    couple(A::fin(A::mul(A::in(p.g_val[ee]), A::in(grad_weight<K>() * a_q))), ce.off);
                  }
                }
              } else {
                for (int e = e_beg; e < e_end; ++e) {
                  const CoupleEntry ce = Ge[e];
                  couple(A::fin(A::mul(Gv[e], cq[ce.tq])), ce.off);
                }
              }
            }
#pragma unroll
            for (int i = 0; i < NT; ++i)
#pragma unroll
              for (int d = 0; d < DIM; ++d) {
                if (p.aniso && d > 0) out[kk][i][1 + d] = L.mul(A::fin(out[kk][i][1 + d]), Rt[d]);
                out[kk][i][1 + d] = A::fin(out[kk][i][1 + d]);
              }
          }
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < KMAX; ++kk) {
          if (a_of[kk] < 0) continue;
          T* base = Qs + (size_t)c_of[kk] * V * SLOT + q_of[kk];
#pragma unroll
          for (int i = 0; i < NT; ++i)
#pragma unroll
            for (int cc = 0; cc < NC; ++cc) base[(size_t)(a_of[kk] * NT + i) * SLOT + cc * NQD] = out[kk][i][cc];
        }
      }
    }
    __syncthreads();
    // ---------------------------------------------------------- phase 3
    for (int it = tid; it < nc * V; it += nthr) {
      T* q = Qs + (size_t)it * SLOT;
      T r[NKD];
      backward_cell<A, DIM, K>(L, [&](int o) { return q[o]; }, r);
#pragma unroll
      for (int a = 0; a < NKD; ++a) q[a] = r[a];
    }
    __syncthreads();
    // ---------------------------------------------------------- phase 4
    // y's start pass may still be running (launch_apply): wait for it before
    // the first reduction
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int c = 0; c < nc; ++c) {
      const int* nd = Nd + c * NKD;
      const T* qc = Qs + (size_t)c * V * SLOT;
      for (int j = tid; j < V * NKD; j += nthr) {
        const int v = j / NKD, a = j - v * NKD;
        const int node = nd[a];
        if (node >= 0 && SG_IN((long long)v * p.n_x + node, (long long)V * p.n_x, 107)) {
          T val = L.mul(Tb[v % NT], qc[(size_t)v * SLOT + a]);
          A::add_out(yout + (long long)v * p.n_x + node, val);
        }
      }
    }
  }
}

}  // namespace sg
