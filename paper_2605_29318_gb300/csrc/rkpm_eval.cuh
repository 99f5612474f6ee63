// Device routines of the corrected RKPM shape functions at one evaluation point
// (internal; shared by the cloud's own shape functions, the two-set
// construction and the skinning weights at query points).  Sec. 3.2,
// Eqs. 7, 9-10; the basis written about the evaluation point (see shape.cu).
#pragma once

#include <type_traits>

#include "dfloat.cuh"
#include "ff_internal.cuh"

namespace ff {
namespace rkpm {

// w(q) and w'(q) / q of the cubic B-spline, from q^2: its root has half the square's
// relative error, and the inner piece takes the square itself
template <class C>
__device__ __forceinline__ void bspline(C q2, C& w, C& dwq) {
  const C q = sqrt(q2);
  if (q <= C(0.5)) {
    w = C(2.0 / 3.0) - C(4) * (q2 * (C(1) - q));
    dwq = C(-8) + C(12) * q;
  } else if (q <= C(1)) {
    const C t = C(1) - q, t2 = t * t;
    w = C(4.0 / 3.0) * t * t2;
    dwq = C(-4) * t2 / q;
  } else {
    w = C(0);
    dwq = C(0);
  }
}

// a + b where the terms may cancel
template <class C>
__device__ __forceinline__ C sum2(C a, C b) {
  if constexpr (std::is_same_v<C, dfloat>)
    return df_add2(a, b);
  else
    return a + b;
}

// normalises an accumulator of mac between two terms: the tail of a dozen unnormalised
// terms grows, and with it the rounding of its own sum
template <class C>
__device__ __forceinline__ void settle(C& a) {
  if constexpr (std::is_same_v<C, dfloat>) fast_two_sum(a.h, a.l, a.h, a.l);
}

// Raw kernels varphi_k as functors: from the squared distance d2 = |X - p_k|^2
// they give w = varphi_k(X) and gs with grad_X varphi_k = gs (p_k - X).
// BSpline: the cubic B-spline of radius a_k = p.w (the nodal discretisation).
struct BSpline {
  static constexpr bool kStash = false;
  template <class C>
  __device__ __forceinline__ void eval(int, float4 p, C d2, C& w, C& gs) const {
    const C ak = (C)p.w, ak2 = ak * ak;
    C dwq;
    bspline<C>(d2 / ak2, w, dwq);
    gs = -dwq / ak2;
  }
};

__device__ __forceinline__ float gauss_exp(float x) { return expf(x); }
__device__ __forceinline__ double gauss_exp(double x) { return exp(x); }
__device__ __forceinline__ dfloat gauss_exp(dfloat x) { return df_exp(x); }

// Gauss: exp(-|X - p_k|^2 / r_k^2) (Sec. 3.2) with the FP64 radii r_k of the
// two-set construction; grad_X = (2 w / r_k^2)(p_k - X).  FP32 takes the square
// of the rounded radius (p.w), double-float 1 / r_k^2 rounded from FP64 (inv),
// once per centre: where the radius would cost two conversions from FP64 and more
// a pair.  In double-float the exponential is df_exp (reduction by ln 2 and a
// Taylor polynomial on the FP32 pipes).
struct Gauss {
  static constexpr bool kStash = true;
  const double* rad;
  const dfloat* inv;
  template <class C>
  __device__ __forceinline__ C slope(int k, float4 p, C w) const {
    if constexpr (sizeof(C) == 4) {
      return C(2) * w / p.w;
    } else if constexpr (std::is_same_v<C, dfloat>) {
      return C(2) * w * inv[k];
    } else {
      const double rk = rad[k];
      return 2.0 * w / (rk * rk);
    }
  }
  template <class C>
  __device__ __forceinline__ void eval(int k, float4 p, C d2, C& w, C& gs) const {
    if constexpr (sizeof(C) == 4) {
      w = gauss_exp(-(d2 / p.w));
    } else if constexpr (std::is_same_v<C, dfloat>) {
      w = gauss_exp(-(d2 * inv[k]));
    } else {
      const double rk = rad[k];
      w = gauss_exp(-(d2 / (rk * rk)));
    }
    gs = slope<C>(k, p, w);
  }
};

// sum over the L lanes of each aligned group of a warp
template <int L, class C>
__device__ __forceinline__ C group_sum(C v) {
#pragma unroll
  for (int o = L / 2; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// symmetric 4x4 packed upper triangle: (0,0)(0,1)(0,2)(0,3)(1,1)(1,2)(1,3)(2,2)(2,3)(3,3)
__device__ __forceinline__ constexpr int sidx(int r, int c) {
  const int lo = r < c ? r : c, hi = r < c ? c : r;
  return lo * 4 - lo * (lo - 1) / 2 + (hi - lo);
}

// A divisor d with its reciprocal r, rounded once: t / d as t r corrected by the
// remainder, as good as a division.  (t r by itself is a rounding more, which M's
// condition number amplifies: 7 to 12 % on a row's largest error, in FP32 and in
// double-float.)
template <class C>
struct Divisor {
  C d, r;
  __device__ __forceinline__ void set(C x) {
    d = x;
    r = C(1) / x;
  }
  __device__ __forceinline__ C into(C t) const {
    const C q = t * r;
    return fma(fma(-q, d, t), r, q);
  }
};
template <>
struct Divisor<dfloat> {
  dfloat d;
  float r;
  __device__ __forceinline__ void set(dfloat x) {
    d = x;
    r = __fdiv_rn(1.f, x.h);
  }
  __device__ __forceinline__ dfloat into(dfloat t) const { return df_div_by(t, d, r); }
};

// Cholesky factor of a 4x4 SPD matrix: the strict lower triangle and the diagonal
template <class C>
struct Chol4 {
  C l[4][4];
  Divisor<C> piv[4];
  // false if a pivot is not positive relative to the trace
  __device__ __forceinline__ bool factor(const C* m, C rel_tol) {
    const C tr = m[0] + m[4] + m[7] + m[9];
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      C s = m[sidx(j, j)];
#pragma unroll
      for (int p = 0; p < j; ++p) s -= l[j][p] * l[j][p];
      ok = ok && s > rel_tol * tr;
      piv[j].set(sqrt(s));
#pragma unroll
      for (int i = j + 1; i < 4; ++i) {
        C t = m[sidx(i, j)];
#pragma unroll
        for (int p = 0; p < j; ++p) t -= l[i][p] * l[j][p];
        l[i][j] = piv[j].into(t);
      }
    }
    return ok;
  }
  __device__ __forceinline__ void solve(const C* b, C* x) const {
    C y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      C t = b[i];
#pragma unroll
      for (int p = 0; p < i; ++p) t -= l[i][p] * y[p];
      y[i] = piv[i].into(t);
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
      C t = y[i];
#pragma unroll
      for (int p = i + 1; p < 4; ++p) t -= l[p][i] * x[p];
      x[i] = piv[i].into(t);
    }
  }
};

// Evaluate one row per group of L lanes in compute precision C, writing
// outputs of precision T (phi; with GRAD dphi too).  Every lane of the warp
// takes part (a group without a row passes s == e).  Returns 0 ok, 1 singular,
// 2 ill-conditioned (only when check_cond), the same in every lane of a group;
// no values are written then (where kernels are stashed, phi holds those).
//
// The row's pairs cost ~110 (values alone: ~50) instructions an entry of a
// lane, the moment solve ~900 a warp whatever the rows it holds; so a warp
// takes 32 / L rows at once.
template <class C, class T, int L, bool GRAD, class Kern = BSpline>
__device__ __forceinline__ int shape_rows(const float4* __restrict__ pos, long long s, long long e,
                                          const int* __restrict__ idx, float4 Xi,
                                          T* __restrict__ phi, T* __restrict__ dphi, long long n1,
                                          double cond_limit, bool check_cond,
                                          const Kern& kern = Kern()) {
  const int lane = threadIdx.x & (L - 1);
  const C xi = (C)Xi.x, yi = (C)Xi.y, zi = (C)Xi.z, si = (C)Xi.w;
  const C isi = C(1) / si;  // the basis scale's reciprocal, once per row
  // the raw kernel of a pair waits in its phi slot for the second pass where
  // it is costly and the slot holds it exactly (the Gaussian in double-float)
  constexpr bool stash = Kern::kStash && std::is_same_v<C, dfloat> && std::is_same_v<T, dfloat>;
  constexpr int ND = GRAD ? 3 : 0;
  C m[10], dm[GRAD ? 3 : 1][10];
#pragma unroll
  for (int q = 0; q < 10; ++q) {
    m[q] = C(0);
#pragma unroll
    for (int d = 0; d < ND; ++d) dm[d][q] = C(0);
  }
  for (long long t = s + lane; t < e; t += L) {
    const int k = idx[t];
    const float4 p = pos[k];
    const C r0 = (C)p.x - xi, r1 = (C)p.y - yi, r2 = (C)p.z - zi;
    C w, gs;  // grad_X varphi = gs * r
    kern.template eval<C>(k, p, r0 * r0 + r1 * r1 + r2 * r2, w, gs);
    if constexpr (stash) phi[t] = w;
    const C P[4] = {C(1), r0 * isi, r1 * isi, r2 * isi};
    const C g[3] = {gs * r0, gs * r1, gs * r2};
    int o = 0;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a; b < 4; ++b, ++o) {
        const C pp = P[a] * P[b];
        mac(m[o], w, pp);  // fused, finished below
        settle(m[o]);
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          mac(dm[d][o], g[d], pp);
          settle(dm[d][o]);
        }
      }
  }
#pragma unroll
  for (int q = 0; q < 10; ++q) {
    m[q] = group_sum<L>(finish(m[q]));
#pragma unroll
    for (int d = 0; d < ND; ++d) dm[d][q] = group_sum<L>(finish(dm[d][q]));
  }
  Chol4<C> ch;
  if (!ch.factor(m, C(1e-12))) return 1;
  C Cv[4], dC[GRAD ? 3 : 1][4];
  {
    const C e0[4] = {C(1), C(0), C(0), C(0)};
    ch.solve(e0, Cv);
  }
  if (check_cond) {
    // 1-norm condition number from the explicit inverse
    C inv_norm = C(0), m_norm = C(0);
#pragma unroll
    for (int col = 0; col < 4; ++col) {
      C x[4];
      if (col == 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = Cv[r];
      } else {
        const C ecol[4] = {C(0), C(col == 1), C(col == 2), C(col == 3)};
        ch.solve(ecol, x);
      }
      C a1 = C(0), a2 = C(0);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        a1 += fabs(x[r]);
        a2 += fabs(m[sidx(r, col)]);
      }
      inv_norm = fmax(inv_norm, a1);
      m_norm = fmax(m_norm, a2);
    }
    if (!((double)(inv_norm * m_norm) <= cond_limit)) return 2;
  }
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    C rhs[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      C t = C(0);
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) t = sum2(t, dm[d][sidx(r, cc)] * Cv[cc]);
      rhs[r] = -t;
    }
    rhs[1 + d] = sum2(rhs[1 + d], isi);
    ch.solve(rhs, dC[d]);
  }
  for (long long t = s + lane; t < e; t += L) {
    const int k = idx[t];
    const float4 p = pos[k];
    const C r0 = (C)p.x - xi, r1 = (C)p.y - yi, r2 = (C)p.z - zi;
    C w, gs;
    if constexpr (stash) {
      w = phi[t];
      gs = kern.template slope<C>(k, p, w);
    } else {
      kern.template eval<C>(k, p, r0 * r0 + r1 * r1 + r2 * r2, w, gs);
    }
    const C P[4] = {C(1), r0 * isi, r1 * isi, r2 * isi};
    C PC = Cv[0];
#pragma unroll
    for (int a = 1; a < 4; ++a) mac(PC, P[a], Cv[a]);
    PC = finish(PC);
    phi[t] = (T)(w * PC);
    const C g[3] = {gs * r0, gs * r1, gs * r2};
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      C PdC = dC[d][0];
#pragma unroll
      for (int a = 1; a < 4; ++a) mac(PdC, P[a], dC[d][a]);
      PdC = finish(PdC);
      dphi[d * n1 + t] = (T)sum2(g[d] * PC, w * PdC);
    }
  }
  return 0;
}

// Cholesky of a 4x4 SPD matrix (packed) with divisions; false if a pivot is not
// positive relative to the trace.  L dense row-major lower.
__device__ __forceinline__ bool chol4_div(const float* m, float* L, float rel_tol) {
  const float tr = m[0] + m[4] + m[7] + m[9];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float s = m[sidx(j, j)];
#pragma unroll
    for (int p = 0; p < j; ++p) s -= L[j * 4 + p] * L[j * 4 + p];
    if (!(s > rel_tol * tr)) return false;
    const float d = sqrtf(s);
    L[j * 4 + j] = d;
#pragma unroll
    for (int i = j + 1; i < 4; ++i) {
      float t = m[sidx(i, j)];
#pragma unroll
      for (int p = 0; p < j; ++p) t -= L[i * 4 + p] * L[j * 4 + p];
      L[i * 4 + j] = t / d;
    }
  }
  return true;
}

__device__ __forceinline__ void chol4_div_solve(const float* L, const float* b, float* x) {
  float y[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float t = b[i];
#pragma unroll
    for (int p = 0; p < i; ++p) t -= L[i * 4 + p] * y[p];
    y[i] = t / L[i * 4 + i];
  }
#pragma unroll
  for (int i = 3; i >= 0; --i) {
    float t = y[i];
#pragma unroll
    for (int p = i + 1; p < 4; ++p) t -= L[p * 4 + i] * x[p];
    x[i] = t / L[i * 4 + i];
  }
}

// The FP32 rows of a two-set build, eight lanes a row, in one fixed order of
// operations: entry 32 u + v of a row is summed in partial v, and the 32 partials
// in a binary tree (v with v + 16, then + 8, 4, 2, 1), whatever lanes hold them.
// A moment matrix's condition number (up to the redo's limit of 100) amplifies a
// change of rounding here, and the low modes of the matrices amplify it again
// (a tree over eight partials moved the modes of a million-point splat by 2e-5);
// so a faster split of the lanes keeps the bits.  A lane takes four partials,
// two at a time; the solves of a row are shared by its lanes.  phi holds the raw
// kernel of a pair between the passes.
template <class Kern>
__device__ __forceinline__ int shape_rows_ordered(const float4* __restrict__ pos, long long s,
                                                  long long e, const int* __restrict__ idx,
                                                  float4 Xi, float* __restrict__ phi,
                                                  float* __restrict__ dphi, long long n1,
                                                  double cond_limit, const Kern& kern) {
  constexpr int L = 8;
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & (L - 1);
  const float xi = Xi.x, yi = Xi.y, zi = Xi.z, si = Xi.w;
  const float isi = 1.f / si;
  // sums q < 10: M; 10 (1 + d) + q: dM / dx_d
  auto partial = [&](int v, float (&m)[40]) {
#pragma unroll
    for (int q = 0; q < 40; ++q) m[q] = 0.f;
    for (long long t = s + v; t < e; t += 32) {
      const int k = idx[t];
      const float4 p = pos[k];
      const float r0 = p.x - xi, r1 = p.y - yi, r2 = p.z - zi;
      float w, gs;  // grad_X varphi = gs * r
      kern.template eval<float>(k, p, r0 * r0 + r1 * r1 + r2 * r2, w, gs);
      phi[t] = w;
      const float P[4] = {1.f, r0 * isi, r1 * isi, r2 * isi};
      const float g[3] = {gs * r0, gs * r1, gs * r2};
      int o = 0;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a; b < 4; ++b, ++o) {
          const float pp = P[a] * P[b];
          m[o] = fmaf(w, pp, m[o]);
#pragma unroll
          for (int d = 0; d < 3; ++d) m[10 * (1 + d) + o] = fmaf(g[d], pp, m[10 * (1 + d) + o]);
        }
    }
  };
  float m[40];
  {
    float b[40];
    partial(lane, m);
    partial(lane + 16, b);
#pragma unroll
    for (int q = 0; q < 40; ++q) m[q] += b[q];
  }
  {
    float b[40], c[40];
    partial(lane + 8, b);
    partial(lane + 24, c);
#pragma unroll
    for (int q = 0; q < 40; ++q) m[q] += b[q] + c[q];
  }
#pragma unroll
  for (int q = 0; q < 40; ++q) m[q] = group_sum<L>(m[q]);
  float Lf[16];
  const bool spd = chol4_div(m, Lf, 1e-12f);
  if (!spd)
#pragma unroll
    for (int q = 0; q < 16; ++q) Lf[q] = 1.f;  // solved for nothing below
  // a lane a column of the inverse (twice): the 1-norm condition number, and
  // C, its first column
  const int col = lane & 3;
  float x[4];
  {
    const float ecol[4] = {(float)(col == 0), (float)(col == 1), (float)(col == 2),
                           (float)(col == 3)};
    chol4_div_solve(Lf, ecol, x);
  }
  float inv_norm = 0.f, m_norm = 0.f;
#pragma unroll
  for (int r = 0; r < 4; ++r) inv_norm += fabsf(x[r]);
  inv_norm = fmaxf(0.f, inv_norm);
#pragma unroll
  for (int o = 2; o; o >>= 1) inv_norm = fmaxf(inv_norm, __shfl_xor_sync(kAll, inv_norm, o));
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float a = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) a += fabsf(m[sidx(r, c)]);
    m_norm = fmaxf(m_norm, a);
  }
  float Cv[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) Cv[r] = __shfl_sync(kAll, x[r], 0, L);
  // a lane a direction (lanes past 2 repeat the last): dC
  float dC[3][4];
  {
    const int d = min(col, 2);
    float rhs[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float t = 0.f;
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const int q = 10 + sidx(r, cc);
        const float md = d == 0 ? m[q] : d == 1 ? m[q + 10] : m[q + 20];
        t += md * Cv[cc];
      }
      rhs[r] = -t;
    }
    if (d == 0) rhs[1] += isi;
    if (d == 1) rhs[2] += isi;
    if (d == 2) rhs[3] += isi;
    chol4_div_solve(Lf, rhs, x);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int r = 0; r < 4; ++r) dC[d][r] = __shfl_sync(kAll, x[r], d, L);
  if (!spd) return 1;
  if ((double)(inv_norm * m_norm) > cond_limit) return 2;
  for (long long t = s + lane; t < e; t += L) {
    const int k = idx[t];
    const float4 p = pos[k];
    const float r0 = p.x - xi, r1 = p.y - yi, r2 = p.z - zi;
    const float w = phi[t], gs = kern.template slope<float>(k, p, w);
    const float P[4] = {1.f, r0 * isi, r1 * isi, r2 * isi};
    float PC = Cv[0];
#pragma unroll
    for (int a = 1; a < 4; ++a) PC = fmaf(P[a], Cv[a], PC);
    phi[t] = w * PC;
    const float g[3] = {gs * r0, gs * r1, gs * r2};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float PdC = dC[d][0];
#pragma unroll
      for (int a = 1; a < 4; ++a) PdC = fmaf(P[a], dC[d][a], PdC);
      dphi[d * n1 + t] = g[d] * PC + w * PdC;
    }
  }
  return 0;
}

// Rows an FP32 pass leaves to FP64 (a moment matrix with a 1-norm condition
// number above its limit, or singular in FP32): list[0] counts them, their
// indexes follow.  A second pass takes them a warp a row, because an FP64
// instruction costs the same for one lane as for 32.
__device__ __forceinline__ void redo_later(int* __restrict__ list, long long i) {
  list[1 + atomicAdd(list, 1)] = (int)i;
}

// the list of a pass over n rows, emptied in stream order
inline int* redo_list(ff_ctx* c, long long n) {
  int* list = reinterpret_cast<int*>(c->redo.ensure(sizeof(int) * (n + 1)));
  FF_CUDA(cudaMemsetAsync(list, 0, sizeof(int), c->stream));
  return list;
}
inline unsigned redo_grid(long long n) {
  return (unsigned)(n < 8LL * 4 * sm_count() ? (n + 7) / 8 : 4LL * sm_count());
}

template <class T, bool GRAD, class Kern>
__global__ void __launch_bounds__(256)
    k_shape_redo(const float4* __restrict__ pos, const float4* __restrict__ at,
                 const float* __restrict__ Q, float scale, const long long* __restrict__ ptr,
                 const int* __restrict__ idx, long long n1, T* __restrict__ phi,
                 T* __restrict__ dphi, const int* __restrict__ list, DevFlags* __restrict__ flags,
                 Kern kern) {
  const int count = list[0];
  const int warps = gridDim.x * 8;
  for (int q = blockIdx.x * 8 + (threadIdx.x >> 5); q < count; q += warps) {
    const int i = list[1 + q];
    const float4 Xi = at ? at[i] : make_float4(Q[3LL * i], Q[3LL * i + 1], Q[3LL * i + 2], scale);
    const int st = shape_rows<double, T, 32, GRAD>(pos, ptr[i], ptr[i + 1], idx, Xi, phi, dphi, n1,
                                                   0.0, false, kern);
    if ((threadIdx.x & 31) == 0) {
      if (st == 0)
        atomicAdd(&flags->fallback, 1);
      else if (atomicCAS(&flags->code, 0, (int)FF_ERR_SINGULAR_MOMENT) == 0)
        flags->index = i;
    }
  }
}

}  // namespace rkpm
}  // namespace ff
