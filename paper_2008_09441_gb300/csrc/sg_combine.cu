// Signed combination of the component fields on the regular nodes:
//   E_comb(x_j) = sum_i c_i (P_i E_i)(x_j)
// (eq. sparse_filter's c_i and P_i of eq. restriction, applied to the
// fields).  P_i is a product of one prolongation per axis, so the sum is taken
// axis by axis, the last axis first:
//   3D: k_combine_planes prolongs every grid along z, to 2^l_1 x 2^l_2 x N
//       nodes; where sums run in double, the grids that share (l_1, l_2) -- at
//       most three, of coefficients +1, -2, +1 -- collapse into one array.
//   2D, and every z plane of a 3D run: k_combine_line interpolates each grid
//       between the two coarse lines that bracket a regular line, and prolongs
//       along x by Horner's scheme (prolong level l to l + 1, add the grids of
//       x level l + 1, ...), exact for nested node-centred grids.
// A regular line reads two brackets of every grid instead of four.  In FP32 the
// collapse (28 arrays instead of 64 at n = 7, tau = 1) would round partial sums
// to floats between the kernels, or pass them as float pairs, whose
// interpolation costs as much as the grids' own (3D n = 7 80 us, the grids 77).
//
// The fields are stored node-interleaved, from the solve's output to the
// combined field, so one load brings all components of a node and one thread
// carries them through the same operations two at a time (f32x2
// instructions; 3D pads the third component with a zero fourth).
#include <algorithm>
#include <type_traits>

#include "sg_kernels.cuh"

namespace sg {

// ---------------------------------------------------------------- accumulators
//
// Values of W components at one node, and their sums.
//
// FP32 path: the sums are float pairs hi + lo carried without
// renormalisation: every hi addition is an error-free two_sum whose error
// goes to lo, so lo collects the exact rounding errors of hi and the pair
// stays accurate to ~2^-48 of the largest intermediate, whatever the
// cancellation; one final two_sum renormalises before the hi / lo planes
// are stored.  FP64 path: plain double.
//
// FP32 fields combined with FP64 accumulation (sg_params.combine =
// SG_COMBINE_FP64): each grid's term c_i w E_i is formed in double, which
// is exact (c_i and the transverse weights w are dyadic, E_i a float), and
// the alternating-sign sum and the Horner prolongation run in double.  The
// result is split into hi + lo floats for the same output planes.  GB300
// issues double arithmetic at a small fraction of the float rate, so this
// variant is the slower one.

// Two floats in one 64-bit register pair, operated on by one instruction.
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_pack(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void f2_unpack(f2 a, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a)); }
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) { return f2_fma(b, f2_pack(-1.f, -1.f), a); }  // one rounding
__device__ __forceinline__ f2 f2_two_sum(f2 a, f2 b, f2& err) {
  const f2 s = f2_add(a, b);
  const f2 bb = f2_sub(s, a);
  err = f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb));
  return s;
}

// One node's W values: T float in pairs (W even), else plain.
template <typename T, int W>
struct Term {
  static constexpr bool packed = sizeof(T) == 4 && W % 2 == 0;
  static constexpr int P = packed ? W / 2 : W;
  using E = typename std::conditional<packed, f2, T>::type;
  E v[P];
  static __device__ __forceinline__ E splat(T x) {
    if constexpr (packed) return f2_pack(x, x);
    else return x;
  }
  // w0 * a + w1 * b, the second product fused (weights are exact)
  static __device__ __forceinline__ Term lerp(T w0, const Term& a, T w1, const Term& b) {
    Term r;
    const E s0 = splat(w0), s1 = splat(w1);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      if constexpr (packed) r.v[p] = f2_fma(s1, b.v[p], f2_mul(s0, a.v[p]));
      else r.v[p] = fma(s1, b.v[p], s0 * a.v[p]);
    }
    return r;
  }
};

// Loads node i of an array stored with DP values per node.
template <typename T, int W, int DP, typename GT>
__device__ __forceinline__ Term<T, W> load_node(const GT* __restrict__ g, int i) {
  Term<T, W> t;
  const GT* p = g + (size_t)(unsigned)i * DP;
  if constexpr (Term<T, W>::packed) {
    if constexpr (W == 2) {
      t.v[0] = __ldg(reinterpret_cast<const f2*>(p));
    } else {
      const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2*>(p));
      t.v[0] = q.x;
      t.v[1] = q.y;
    }
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) t.v[w] = (T)__ldg(p + w);
  }
  return t;
}

template <typename T, int W>
struct Sum {  // FP64 accumulation
  using Tm = Term<T, W>;
  T v[W];
  static __device__ __forceinline__ Sum zero() {
    Sum r;
#pragma unroll
    for (int p = 0; p < W; ++p) r.v[p] = (T)0;
    return r;
  }
  static __device__ __forceinline__ Sum avg(const Sum& a, const Sum& b) {
    Sum r;
#pragma unroll
    for (int p = 0; p < W; ++p) r.v[p] = (a.v[p] + b.v[p]) * (T)0.5;
    return r;
  }
  static __device__ __forceinline__ Sum add(const Sum& a, const Sum& b) {
    Sum r;
#pragma unroll
    for (int p = 0; p < W; ++p) r.v[p] = a.v[p] + b.v[p];
    return r;
  }
  __device__ __forceinline__ void add_term(const Tm& t) {
#pragma unroll
    for (int p = 0; p < W; ++p) v[p] += t.v[p];
  }
  __device__ __forceinline__ void add_mid(const Tm& a, const Tm& b) {  // (a + b) / 2
#pragma unroll
    for (int p = 0; p < W; ++p) v[p] += (T)0.5 * (a.v[p] + b.v[p]);
  }
};
template <int W>
struct __align__(16) Sum<float, W> {  // float pairs
  using Tm = Term<float, W>;
  static constexpr int P = Tm::P;
  using E = typename Tm::E;
  E hi[P], lo[P];
  static __device__ __forceinline__ E two_sum_e(E a, E b, E& err) {
    if constexpr (Tm::packed) {
      return f2_two_sum(a, b, err);
    } else {
      const ff s = two_sum(a, b);
      err = s.lo;
      return s.hi;
    }
  }
  static __device__ __forceinline__ E add_e(E a, E b) {
    if constexpr (Tm::packed) return f2_add(a, b);
    else return a + b;
  }
  static __device__ __forceinline__ Sum zero() {
    Sum r;
#pragma unroll
    for (int p = 0; p < P; ++p) r.hi[p] = r.lo[p] = Tm::splat(0.f);
    return r;
  }
  static __device__ __forceinline__ Sum avg(const Sum& a, const Sum& b) {
    Sum r;
    const E h = Tm::splat(0.5f);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      E err;
      const E s = two_sum_e(a.hi[p], b.hi[p], err);
      const E l = add_e(add_e(a.lo[p], b.lo[p]), err);
      if constexpr (Tm::packed) {
        r.hi[p] = f2_mul(s, h);
        r.lo[p] = f2_mul(l, h);
      } else {
        r.hi[p] = s * h;
        r.lo[p] = l * h;
      }
    }
    return r;
  }
  static __device__ __forceinline__ Sum add(const Sum& a, const Sum& b) {
    Sum r;
#pragma unroll
    for (int p = 0; p < P; ++p) {
      E err;
      r.hi[p] = two_sum_e(a.hi[p], b.hi[p], err);
      r.lo[p] = add_e(add_e(a.lo[p], b.lo[p]), err);
    }
    return r;
  }
  __device__ __forceinline__ void add_term(const Tm& t) {
#pragma unroll
    for (int p = 0; p < P; ++p) {
      E err;
      hi[p] = two_sum_e(hi[p], t.v[p], err);
      lo[p] = add_e(lo[p], err);
    }
  }
  // (a + b) / 2 without rounding it: the sum and its error go into the pair
  __device__ __forceinline__ void add_mid(const Tm& a, const Tm& b) {
    const E h = Tm::splat(0.5f);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      E e1, e2;
      const E s = two_sum_e(a.v[p], b.v[p], e1);
      if constexpr (Tm::packed) {
        hi[p] = f2_two_sum(hi[p], f2_mul(h, s), e2);
        lo[p] = f2_fma(h, e1, f2_add(lo[p], e2));
      } else {
        hi[p] = two_sum_e(hi[p], h * s, e2);
        lo[p] = fmaf(h, e1, lo[p] + e2);
      }
    }
  }
  // the normalised hi and lo parts, by component; the hi parts also as they are
  __device__ __forceinline__ void split(float* h, float* l, E* s) const {
#pragma unroll
    for (int p = 0; p < P; ++p) {
      E err;
      s[p] = two_sum_e(hi[p], lo[p], err);
      if constexpr (Tm::packed) {
        f2_unpack(s[p], h[2 * p], h[2 * p + 1]);
        f2_unpack(err, l[2 * p], l[2 * p + 1]);
      } else {
        h[p] = s[p];
        l[p] = err;
      }
    }
  }
};

// The two level-lev nodes that bracket regular node y along one axis and
// the weight of the second: node-centred, y / 2^r in coarse units (r = n -
// lev); cell-centred, (y + 1/2) / 2^r - 1/2 = (2y + 1 - 2^r) / 2^(r+1), whose
// floor may be -1 (wrapped).  Both weights are dyadic: exact.
template <typename real, bool CELL>
__device__ __forceinline__ void bracket(int y, int n, int lev, int& k0, int& k1, real& f) {
  const int r = n - lev;
  const int nl = 1 << lev;
  if (!CELL) {
    k0 = y >> r;
    f = (real)(y & ((1 << r) - 1)) * ((real)1 / (real)(1 << r));
  } else {
    const int num = 2 * y + 1 - (1 << r);
    const int fl = num >> (r + 1);  // arithmetic shift: floor
    f = (real)(num - fl * (2 << r)) * ((real)1 / (real)(2 << r));
    k0 = fl & (nl - 1);
  }
  k1 = (k0 + 1) & (nl - 1);
}

// Values per node of an array of NC components: 2D fields 2, 3D fields 4
// (one pad), a density 1.
template <int NC>
constexpr int node_stride() { return NC == 1 ? 1 : NC == 2 ? 2 : 4; }
// Components a thread of the line kernel carries: floats all of them, in
// whole pairs; doubles one (their latency is long, more threads hide it).
template <typename T, int NC>
constexpr int carried() { return sizeof(T) == 4 ? node_stride<NC>() : 1; }

// ---------------------------------------------------------------- 3D: prolongation along z
//
// out[z][off + e] = sum over an array's grids of c_i times the linear
// interpolation along z of in-plane node e.  One thread per in-plane node walks
// PL_Z planes; loads are consecutive in e.  Bound: latency (7 us at n = 7, tau =
// 1: 624 K nodes from 64 grids).
constexpr int PL_Z = 4;
constexpr int PL_LEVELS = 9;  // 3D levels 0..8
template <typename T>
struct __align__(16) PlaneBracket {
  int k0, k1;
  T w0, w1;
};
template <typename real, typename T, int NC, bool CELL>
__global__ void __launch_bounds__(256) k_combine_planes(const PlaneArray* __restrict__ arrays, int narrays,
                                                        const real* __restrict__ E, int S2, int n, int z0, int nz,
                                                        T* __restrict__ out) {
  constexpr int DP = node_stride<NC>(), W = sizeof(T) == 4 ? DP : NC;
  __shared__ PlaneArray sp[CB_MAX_GRIDS];
  __shared__ PlaneBracket<T> sb[PL_LEVELS][PL_Z];
  pdl_trigger();
  const int zb = blockIdx.y * PL_Z;
  {
    const int* src = reinterpret_cast<const int*>(arrays);
    int* dst = reinterpret_cast<int*>(sp);
    for (int i = threadIdx.x; i < narrays * (int)(sizeof(PlaneArray) / 4); i += blockDim.x) dst[i] = src[i];
    if (threadIdx.x < (n + 1) * PL_Z) {
      const int l = threadIdx.x / PL_Z, z = threadIdx.x % PL_Z;
      PlaneBracket<T> t;
      bracket<T, CELL>(z0 + zb + z, n, l, t.k0, t.k1, t.w1);
      t.w0 = (T)1 - t.w1;
      sb[l][z] = t;
    }
  }
  __syncthreads();
  pdl_wait(E);  // the solve's fields
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= S2) return;
  int lo = 0, hi = narrays;  // the last array with off <= e
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (sp[mid].off <= e) lo = mid;
    else hi = mid;
  }
  const PlaneArray P = sp[lo];
  const int le = e - P.off;
  const int x = le & ((1 << P.lx) - 1);
  const int at = e - x + line_pos(x, P.lx, n);
#pragma unroll
  for (int z = 0; z < PL_Z; ++z) {
    if (zb + z >= nz) break;
    auto term = [&](int q) {
      const PlaneBracket<T> t = sb[P.lz[q]][z];
      const T c = (T)P.coeff[q];
      const int g = P.goff[q] + le;
      return Term<T, W>::lerp(c * t.w0, load_node<T, W, DP>(E, g + (t.k0 << P.logs)), c * t.w1,
                              load_node<T, W, DP>(E, g + (t.k1 << P.logs)));
    };
    Term<T, W> v = term(0);
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int q = 1; q < 3; ++q)
        if (q < P.ng) {
          const Term<T, W> t = term(q);
#pragma unroll
          for (int w = 0; w < W; ++w) v.v[w] += t.v[w];
        }
    }
    T* d = out + ((size_t)(zb + z) * S2 + at) * DP;
    if constexpr (sizeof(T) == 4 && W == 4) {
      *reinterpret_cast<ulonglong2*>(d) = make_ulonglong2(v.v[0], v.v[1]);
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) d[w] = v.v[w];
    }
  }
}

// ---------------------------------------------------------------- lines
//
// Levels up to n - log2 K: the block's threads hold one node each of every
// line in shared memory (all arrays that enter at any of these levels are
// interpolated at once, then the prolongation runs level by level), so no
// value is computed twice and every load is consecutive.  Above, a thread
// computes K consecutive nodes: it needs 2 nodes of the shared level, then
// 3, 5, ..., K + 1, and prolongs that cone by itself, which spares the
// barriers of the widest levels for a few values computed twice.  Bound:
// 3D, L1 (62% busy), issue slots (40%) and latency at 31% of the warps (four
// loads in flight instead of two: 88 -> 84 us); 2D, the latency of the block's
// phases (36% of issue slots).  With profiling events, before (one warp per
// line, four brackets) -> now, planes included: 3D n = 7 151 -> 78 us, tau = 2
// 137 -> 75, n = 6 cell-centred 64 -> 31; 2D n = 11 134 -> 53, n = 10 27 ->
// 22.5, n = 8 14.3 -> 12.3 us.

// Transverse interpolation of one array at regular line y: the two coarse
// lines that bracket it, each weight times the coefficient (dyadic: exact).
template <typename T>
struct __align__(16) RowTerm {
  int off[2];
  T w[2];
};

template <typename T, int W, int DP, typename GT>
__device__ __forceinline__ Term<T, W> row_node(const GT* __restrict__ G, const RowTerm<T>& rt, int x) {
  return Term<T, W>::lerp(rt.w[0], load_node<T, W, DP>(G, rt.off[0] + x), rt.w[1],
                          load_node<T, W, DP>(G, rt.off[1] + x));
}

// R consecutive nodes of an array of x level l at line y, from node a (a
// multiple of R), X of them past the run's end, periodically (X = 1).  PERM:
// the array is stored in line_pos order.
template <typename T, int W, int DP, int R, int X, bool PERM, typename GT>
__device__ __forceinline__ void row_run(const GT* __restrict__ G, const RowTerm<T>& rt, int a, int l, Term<T, W>* t) {
  constexpr int LR = R == 4 ? 2 : R == 2 ? 1 : 0;
  const int mask = (1 << l) - 1;
  if constexpr (!PERM && W == 1 && sizeof(GT) == 4 && R > 1) {  // a plain density: vector loads
    GT x[2][R];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const GT* p = G + rt.off[k] + a;
      if constexpr (R == 4) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(p));
        x[k][0] = q.x;
        x[k][1] = q.y;
        x[k][2] = q.z;
        x[k][3] = q.w;
      } else {
        const float2 q = __ldg(reinterpret_cast<const float2*>(p));
        x[k][0] = q.x;
        x[k][1] = q.y;
      }
    }
#pragma unroll
    for (int j = 0; j < R; ++j) t[j].v[0] = fma(rt.w[1], (T)x[1][j], rt.w[0] * (T)x[0][j]);
  } else {
#pragma unroll
    for (int j = 0; j < R; ++j)
      t[j] = row_node<T, W, DP>(G, rt, PERM ? (j << (l - LR)) + (a >> LR) : a + j);
  }
  if constexpr (X) {
    const int b = (a + R) & mask;
    t[R] = row_node<T, W, DP>(G, rt, PERM ? b >> LR : b);
  }
}

// Cell-centred grids.  Linear interpolation through the centres of a
// level-l line is the node-centred interpolant of the level-(l+1) line
// whose odd nodes are the centres (g[2k+1] = E[k]) and whose even nodes are
// the midpoints (g[2k] = (E[k-1] + E[k]) / 2); the regular centres are the
// midpoints of the level-n nodes.  So the same Horner scheme runs with each
// array entering one level higher as g, and the regular-centre values are
// (T[j] + T[j+1]) / 2 of its level-n result, plus the arrays of x level n
// at their own centres.

// Sum, at node x of `level`, of the arrays that enter there.
template <typename T, int W, int DP, bool CELL, typename GT>
__device__ __forceinline__ Sum<T, W> entering(const GT* __restrict__ G, const RowTerm<T>* tab, const int* start,
                                              int level, int x) {
  Sum<T, W> acc = Sum<T, W>::zero();
  const int l = CELL ? level - 1 : level;
  if (CELL && l < 0) return acc;
  const int mask = (1 << l) - 1;
  const int i1 = CELL ? x >> 1 : x;
  const int end = start[l + 1];
#pragma unroll DP == 4 ? 4 : 2  // loads in flight (3D n = 7: two 88 us, four 84)
  for (int gi = start[l]; gi < end; ++gi) {
    const RowTerm<T> rt = tab[gi];
    const Term<T, W> t = row_node<T, W, DP>(G, rt, i1);
    if constexpr (CELL) {  // an even node: the midpoint of two centres
      const int i0 = (x & 1) ? i1 : (i1 - 1) & mask;
      const Term<T, W> t0 = row_node<T, W, DP>(G, rt, i0);
      acc.add_mid(t0, t);  // of a centre and itself: the centre
    } else {
      acc.add_term(t);
    }
  }
  return acc;
}

// Nodes a .. a + C of `level` (a a multiple of C) -> a' .. a' + 2C of the next
// one, with its arrays added; up to CB_RUN nodes of level n.  The node past
// the thread's last one is dropped at level n, unless the cell-centred
// midpoints need it.
template <typename T, int W, int DP, int C, bool CELL, bool PERM, typename GT>
__device__ __forceinline__ void expand(Sum<T, W>* v, const GT* __restrict__ G, const RowTerm<T>* tab,
                                       const int* start, int level, int j0, int n) {
  using S = Sum<T, W>;
  if constexpr (C < CB_RUN) {
    constexpr int C2 = 2 * C, X = (C2 < CB_RUN || CELL) ? 1 : 0;
    v[C2] = v[C];
#pragma unroll
    for (int i = C - 1; i >= 0; --i) {  // in place, high to low
      v[2 * i + 1] = S::avg(v[i], v[i + 1 < C ? 2 * (i + 1) : C2]);
      v[2 * i] = v[i];
    }
    ++level;
    const int l = CELL ? level - 1 : level;
    const int mask = (1 << l) - 1;
    const int a = (j0 >> (n - level)) >> (CELL ? 1 : 0);
    const int end = start[l + 1];
    for (int gi = start[l]; gi < end; ++gi) {
      const RowTerm<T> rt = tab[gi];
      if constexpr (CELL) {
        Term<T, W> t[C + 2];
        const int b = (a - 1) & mask;
        t[0] = row_node<T, W, DP>(G, rt, PERM && C == 2 ? ((b & 1) << (l - 1)) + (b >> 1) : b);
        row_run<T, W, DP, C, 1, PERM && C == 2>(G, rt, a, l, t + 1);
#pragma unroll
        for (int j = 0; j <= C; ++j) v[2 * j].add_mid(t[j], t[j + 1]);
#pragma unroll
        for (int j = 0; j < C; ++j) v[2 * j + 1].add_term(t[j + 1]);
      } else {
        Term<T, W> t[C2 + X];
        row_run<T, W, DP, C2, X, PERM>(G, rt, a, l, t);
#pragma unroll
        for (int j = 0; j < C2 + X; ++j) v[j].add_term(t[j]);
      }
    }
    expand<T, W, DP, C2, CELL, PERM>(v, G, tab, start, level, j0, n);
  }
}

// SquareSum of the combined field's high parts, W components at a time.
template <int W>
struct Energy {
  using Tm = Term<float, W>;
  using E = typename Tm::E;
  E hi, lo;
  __device__ __forceinline__ Energy() : hi(Tm::splat(0.f)), lo(Tm::splat(0.f)) {}
  __device__ __forceinline__ void add(const E* x) {
#pragma unroll
    for (int p = 0; p < Tm::P; ++p) {
      E err;
      if constexpr (Tm::packed) hi = f2_two_sum(hi, f2_mul(x[p], x[p]), err);
      else hi = Sum<float, W>::two_sum_e(hi, __fmul_rn(x[p], x[p]), err);
      lo = Sum<float, W>::add_e(lo, err);
    }
  }
  __device__ __forceinline__ double value() const {
    if constexpr (Tm::packed) {
      float h0, h1, l0, l1;
      f2_unpack(hi, h0, h1);
      f2_unpack(lo, l0, l1);
      const ff s = two_sum(h0, h1);
      return (double)s.hi + (double)(s.lo + (l0 + l1));
    } else {
      return (double)hi + (double)lo;
    }
  }
};

constexpr int CL_THREADS = 256;

// One block: `lpb` consecutive lines, N / CB_RUN threads per line and group of
// carried components.  zstride: values between the planes of G (2D: one
// plane).  row0: first line of the launch.
template <typename real, typename GT, typename T, int NC, bool CELL, bool PERM>
__global__ void __launch_bounds__(CL_THREADS, sizeof(T) == 8 ? 2 : NC == 3 ? 3 : 4)
    k_combine_line(const LineGrid* __restrict__ lg, const LevelStarts ls, int lmin, const GT* __restrict__ G,
                   size_t zstride, int n, int lpb, int row0, size_t nd, real* __restrict__ Ehi,
                   float* __restrict__ Elo, double* __restrict__ partials, int n_part, const CombineFinal fin) {
  constexpr int K = CB_RUN, LK = 2;
  constexpr int DP = node_stride<NC>(), W = carried<T, NC>();
  constexpr int MG = W >= NC ? 1 : NC;  // groups of components
  constexpr int WO = W < NC ? W : NC;   // components a thread writes
  using S = Sum<T, W>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  __shared__ int start[18];
  const int N = 1 << n;
  const int ipl = N >> LK;  // threads per line and group
  const int ngl = ls.start[17];
  RowTerm<T>* tab = reinterpret_cast<RowTerm<T>*>(smem_raw);  // [lpb][ngl]
  // node x of level l of line and group q at lat[q * 2 ipl + 2^l + x], q = line * MG + group
  S* lat = reinterpret_cast<S*>(tab + (size_t)lpb * ngl);
  const int brow = row0 + blockIdx.x * lpb;  // first line of the block
  pdl_trigger();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < 18; ++i) start[i] = ls.start[i];  // constant indices: no local copy
  }
  for (int e = threadIdx.x; e < lpb * ngl; e += blockDim.x) {
    const int r = e / ngl;
    const LineGrid g = lg[e - r * ngl];
    int k0, k1;
    T f;
    bracket<T, CELL>((brow + r) & (N - 1), n, g.ly, k0, k1, f);
    const T c = (T)g.coeff;
    RowTerm<T> rt;
    rt.off[0] = g.off + (k0 << g.lx);
    rt.off[1] = g.off + (k1 << g.lx);
    rt.w[0] = c * ((T)1 - f);
    rt.w[1] = c * f;
    tab[e] = rt;
  }
  __syncthreads();
  pdl_wait(G);  // the fields (3D: their planes)
  const int ntask = lpb * MG * ipl;
  const GT* Gz = G + (size_t)((brow - row0) >> n) * zstride;  // lpb <= N: the block's lines lie in one plane
  int level = min(CELL ? lmin + 1 : lmin, n - LK);
  for (int t = threadIdx.x; t < 2 * ntask; t += blockDim.x) {
    const int e = t & (2 * ipl - 1), q = t >> (n - LK + 1);
    const int l = 31 - __clz(e);
    if (l >= level) lat[t] = entering<T, W, DP, CELL>(Gz + q % MG, tab + q / MG * ngl, start, l, e - (1 << l));
  }
  __syncthreads();
  while (level < n - LK) {  // prolong level by level
    ++level;
    for (int t = threadIdx.x; t < (lpb * MG << level); t += blockDim.x) {
      const int x = t & ((1 << level) - 1);
      S* base = lat + (size_t)(t >> level) * 2 * ipl;
      const S* pl = base + (1 << (level - 1));
      S v = pl[x >> 1];
      if (x & 1) v = S::avg(v, pl[((x >> 1) + 1) & ((1 << (level - 1)) - 1)]);
      base[(1 << level) + x] = S::add(v, base[(1 << level) + x]);
    }
    __syncthreads();
  }
  Energy<W> energy;       // float pairs
  double energy_d = 0.0;  // double accumulation: the squares of the double results
  for (int task = threadIdx.x; task < ntask; task += blockDim.x) {
    const int item = task & (ipl - 1);
    const int q = task >> (n - LK), r = q / MG, m0 = q % MG;
    const int j0 = item << LK;
    const RowTerm<T>* rtab = tab + r * ngl;
    const GT* Gm = Gz + m0;
    const S* top = lat + (size_t)q * 2 * ipl + ipl;
    S v[K + 1];
    v[0] = top[item];
    v[1] = top[(item + 1) & (ipl - 1)];
    expand<T, W, DP, 1, CELL, PERM>(v, Gm, rtab, start, level, j0, n);
    if constexpr (CELL) {  // to the regular centres, then the arrays of x level n
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] = S::avg(v[k], v[k + 1]);
      const int end = start[n + 1];
      for (int gi = start[n]; gi < end; ++gi) {
        const RowTerm<T> rt = rtab[gi];
        Term<T, W> t[K];
        row_run<T, W, DP, K, 0, PERM>(Gm, rt, j0, n, t);
#pragma unroll
        for (int k = 0; k < K; ++k) v[k].add_term(t[k]);
      }
    }
    const size_t node = (size_t)(brow + r) * N + j0;
    real* dst = Ehi + node * DP + m0;
    if constexpr (sizeof(real) == 4) {
      float lo[WO][K];
      float hi[K][W];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        float l[W];
        if constexpr (sizeof(T) == 4) {
          typename Term<float, W>::E s[Term<float, W>::P];
          v[k].split(hi[k], l, s);
          energy.add(s);  // a padding component is zero
        } else {
          hi[k][0] = (float)v[k].v[0];
          l[0] = (float)(v[k].v[0] - (double)hi[k][0]);
          energy_d = fma(v[k].v[0], v[k].v[0], energy_d);
        }
#pragma unroll
        for (int m = 0; m < WO; ++m) lo[m][k] = l[m];
      }
      if constexpr (W == DP) {
        const float* h = &hi[0][0];
#pragma unroll
        for (int i = 0; i < K * DP; i += 4)
          *reinterpret_cast<float4*>(dst + i) = make_float4(h[i], h[i + 1], h[i + 2], h[i + 3]);
      } else {
#pragma unroll
        for (int k = 0; k < K; ++k) dst[k * DP] = hi[k][0];
      }
      if (Elo) {
#pragma unroll
        for (int m = 0; m < WO; ++m)
          *reinterpret_cast<float4*>(Elo + (size_t)(m0 + m) * nd + node) =
              make_float4(lo[m][0], lo[m][1], lo[m][2], lo[m][3]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        dst[k * DP] = v[k].v[0];
        energy_d = fma(v[k].v[0], v[k].v[0], energy_d);
      }
    }
  }
  const double tot = block_sum_double(sizeof(T) == 4 ? energy.value() : energy_d, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = tot;
  if (!fin.active) return;
  combine_finalize(partials - (n_part - (int)gridDim.x), n_part, fin, red);
}

template <typename real, typename GT, typename T, int NC, bool CELL, bool PERM>
static int launch_lines(const CombineTables& ct, const GT* G, size_t zstride, int n, int row0, int rows, size_t nd,
                        real* Ehi, float* Elo, double* partials, int* part0, const CombineFinal& fin,
                        cudaStream_t s) {
  const int N = 1 << n, ipl = N / CB_RUN;
  constexpr int W = carried<T, NC>(), MG = W >= NC ? 1 : NC;
  // Threads per block and tasks to share among them.  From 2^18 tasks on
  // (2D n = 10, 3D n = 7) a block takes 384 or more (3D fields 192, whose
  // tables are three times as long), two per thread, which spreads its tables
  // and barriers: 3D n = 7 77 us against 86 with 128 and 128, 84 with 384 (the
  // energy then summed in floats); 2D
  // n = 10 20.5 against 21.2.  Below, small blocks reach more SMs: 3D n = 6 25
  // against 43 us, 2D n = 8 12.3 against 14.5.  Doubles on tiny grids go smaller
  // still (2D n = 6: 13.5 against 14.3 us).
  const size_t tasks = nd * MG / CB_RUN;
  const bool large = sizeof(T) == 4 && tasks >= ((size_t)1 << 18);
  const int ft = large ? (NC == 3 ? 192 : 384) : sizeof(T) == 8 && tasks < ((size_t)1 << 14) ? 64 : 128;
  const int fthr = large ? ft / 2 : ft;
  int lpb = 1;
  while (2 * lpb <= std::min(rows, N) && lpb * MG * ipl < ft) lpb *= 2;
  const int ngl = ct.ls.start[17];
  const unsigned blocks = (unsigned)(rows / lpb);  // both powers of two
  const unsigned threads = (unsigned)std::min(fthr, (lpb * MG * ipl + 31) / 32 * 32);
  const size_t smem = (size_t)lpb * ngl * sizeof(RowTerm<T>) + (size_t)2 * lpb * MG * ipl * sizeof(Sum<T, W>);
  static DeviceSet allowed{0};
  if (smem > 40 * 1024)  // with the static part the total may pass 48 KB
    SG_TRY(allow_smem(k_combine_line<real, GT, T, NC, CELL, PERM>, allowed, 200 * 1024));
  SG_CUDA(launch_pdl(k_combine_line<real, GT, T, NC, CELL, PERM>, dim3(blocks), dim3(threads), smem, s, ct.lines, ct.ls,
                     ct.lmin, G, zstride, n, lpb, row0, nd, Ehi, Elo, partials + *part0, *part0 + (int)blocks, fin));
  *part0 += (int)blocks;
  SG_CHECK_LAUNCH();
  return SG_OK;
}

template <typename real, int D, int NC, bool CELL, typename T>
static int launch_combine_nc(const CombineTables& ct, const real* E, int n, real* Ehi, float* Elo, double* partials,
                             const CombineFinal& fin, cudaStream_t s) {
  const int N = 1 << n;
  const size_t nd = (size_t)1 << (D * n);
  int part0 = 0;
  if constexpr (D == 2) {
    return launch_lines<real, real, T, NC, CELL, (NC > 1)>(ct, E, 0, n, 0, N, nd, Ehi, Elo, partials, &part0, fin, s);
  } else {
    // as many planes at a time as the scratch holds (a power of two, so
    // that every launch has whole blocks); the last launch closes the step
    constexpr int DP = node_stride<NC>();
    const size_t plane = (size_t)DP * ct.S2;
    int nz = N;
    while (nz > 1 && (size_t)nz * plane * sizeof(T) > ct.scratch_bytes) nz >>= 1;
    if ((size_t)nz * plane * sizeof(T) > ct.scratch_bytes) {
      set_error("combination: scratch smaller than one plane");
      return SG_ERR_SIZE;
    }
    T* G = static_cast<T*>(ct.scratch);
    for (int z0 = 0; z0 < N; z0 += nz) {
      SG_CUDA(launch_pdl(k_combine_planes<real, T, NC, CELL>,
                         dim3((unsigned)((ct.S2 + 255) / 256), (unsigned)((nz + PL_Z - 1) / PL_Z)), dim3(256), 0, s,
                         ct.planes, ct.ls.start[17], E, ct.S2, n, z0, nz, G));
      SG_CHECK_LAUNCH();
      CombineFinal f = fin;
      if (z0 + nz < N) f.active = 0;
      SG_TRY(launch_lines<real, T, T, NC, CELL, true>(ct, G, plane, n, z0 * N, nz * N, nd, Ehi, Elo, partials, &part0, f,
                                                      s));
    }
    return SG_OK;
  }
}

template <typename real, int D, typename T>
static int launch_combine_acc(const CombineTables& ct, const real* E, int n, real* Ehi, float* Elo, double* partials,
                              const CombineFinal& fin, cudaStream_t s, int ncomp, bool cell) {
  if (cell) {
    if (ncomp == 1) return launch_combine_nc<real, D, 1, true, T>(ct, E, n, Ehi, Elo, partials, fin, s);
    return launch_combine_nc<real, D, D, true, T>(ct, E, n, Ehi, Elo, partials, fin, s);
  }
  if (ncomp == 1) return launch_combine_nc<real, D, 1, false, T>(ct, E, n, Ehi, Elo, partials, fin, s);
  return launch_combine_nc<real, D, D, false, T>(ct, E, n, Ehi, Elo, partials, fin, s);
}

// fp64_acc selects FP64 accumulation of FP32 fields; the FP64 path always
// accumulates in double.
template <typename real, int D>
int launch_combine(const CombineTables& ct, const real* E, int n, real* Ehi, float* Elo, double* energy_partials,
                   const CombineFinal& fin, cudaStream_t s, int ncomp, bool cell, bool fp64_acc) {
  if constexpr (sizeof(real) == 4) {
    if (fp64_acc) return launch_combine_acc<real, D, double>(ct, E, n, Ehi, Elo, energy_partials, fin, s, ncomp, cell);
  }
  return launch_combine_acc<real, D, real>(ct, E, n, Ehi, Elo, energy_partials, fin, s, ncomp, cell);
}

#define SG_INST_COMB(real, D)                                                                                     \
  template int launch_combine<real, D>(const CombineTables&, const real*, int, real*, float*, double*,            \
                                       const CombineFinal&, cudaStream_t, int, bool, bool);
SG_INST_COMB(float, 2)
SG_INST_COMB(float, 3)
SG_INST_COMB(double, 2)
SG_INST_COMB(double, 3)

}  // namespace sg
