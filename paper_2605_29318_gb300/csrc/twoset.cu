// The paper's two-set RKPM discretisation (Supp. Sec. B "RKPM construction",
// with the Gaussian kernel of Sec. 3.2).
//
// Quadrature points X_i with volumes v_i (an inside grid of the object, or its
// own points); K kernel centres p_k chosen among them by farthest-point
// sampling; radius r_k = distance from p_k to its second-nearest other centre;
// raw kernel exp(-|X - p_k|^2 / r_k^2), cut at t r_k when t > 0; the corrected
// shape functions of Eqs. 7, 9-10 at the quadrature points.  The result is laid
// out like the nodal discretisation's (rows = quadrature points, columns =
// centres, plus the transposed lists), so the assembly of H_w (Prop. 1) and M
// (Eq. 14) and the eigensolver run unchanged on the K centres.
//
// Every decision taken in floating point is the FP64 one on the FP32-stored
// points, each operation rounded separately:
//   * squared distances ((dx*dx + dy*dy) + dz*dz);
//   * farthest-point sampling from `start`, ties to the lowest index;
//   * r_k = sqrt of the second-smallest squared distance to the other centres;
//   * centre k covers X iff d2 < (t*t) * (r_k*r_k).
// Each is first settled in FP32 with a relative margin of 1e-5 (FP32 and FP64
// squared distances differ by less than 4e-7 relative); only values within
// the margin are evaluated in FP64.  Distances are compared by their FP64 bit
// patterns where they are ordered (non-negative doubles order like integers).
//
// Kernels:
//   k_fps_rounds   up to one block per SM, each with its slice of the points;
//                  several centres a grid barrier
//   k_radii        one warp per centre: the two smallest squared distances
//   k_cover_bits, k_cover_fill
//                  each point's covering centres as bits, then as an ascending
//                  list (k_cover_rows, one thread per point, for many centres)
//   k_cover_cols   one warp per centre: the points it covers, ascending, and
//                  the centre's position in each point's row
//   k_shape_twoset eight lanes per quadrature point, Eqs. 7, 9-10 with the Gaussian
#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>
#include <vector>

#include "dfloat.cuh"
#include "ff_internal.cuh"
#include "rkpm_eval.cuh"

namespace ff {
namespace {

constexpr int kFpsT = 512;                   // threads per block
constexpr int kFpsSmemMax = 200 * 1024;      // dynamic shared memory per block
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ double d2_f64(float ax, float ay, float az, float bx, float by,
                                         float bz) {
  const double dx = __dsub_rn((double)ax, (double)bx);
  const double dy = __dsub_rn((double)ay, (double)by);
  const double dz = __dsub_rn((double)az, (double)bz);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__device__ __forceinline__ float d2_f32(float ax, float ay, float az, float bx, float by,
                                        float bz) {
  const float dx = __fsub_rn(ax, bx), dy = __fsub_rn(ay, by), dz = __fsub_rn(az, bz);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// the filter's form, within the same margin of the FP64 value
__device__ __forceinline__ float d2_fma(float ax, float ay, float az, float bx, float by,
                                        float bz) {
  const float dx = ax - bx, dy = ay - by, dz = az - bz;
  return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// centre (p, l32 = fl32(lim), lim = t^2 r^2 or +inf) covers the point (x, y, z)
__device__ __forceinline__ bool covers2(float x, float y, float z, float4 p, float l32,
                                        double lim) {
  if (l32 >= 1e-30f) {
    const float d32 = d2_f32(x, y, z, p.x, p.y, p.z);
    if (d32 < __fmul_rn(l32, 0.99999f)) return true;
    if (d32 > __fmul_rn(l32, 1.00001f)) return false;
  }
  return d2_f64(x, y, z, p.x, p.y, p.z) < lim;
}

// ------------------------------------------------------------------ validation
__global__ void k_validate_points(const float* __restrict__ X, const float* __restrict__ v,
                                  long long n, int* __restrict__ bad) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float x = X[3 * i], y = X[3 * i + 1], z = X[3 * i + 2], vi = v[i];
    const bool ok = isfinite(x) && isfinite(y) && isfinite(z) && fabsf(x) < 1e18f &&
                    fabsf(y) < 1e18f && fabsf(z) < 1e18f && isfinite(vi) && vi > 0.f;
    if (!ok) atomicMin(bad, (int)i);
  }
}

// ------------------------------------------------------------------ farthest-point sampling
// The grid barrier is a monotone arrival counter in global memory; its wait is
// bounded (about a second of clock cycles) and a block that gives up records
// FF_ERR_TIMEOUT in the flags and in `abort`, and every block leaves at the next
// barrier it sees it at.
constexpr long long kGridWaitCycles = 2000000000LL;

__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned target, int* abort,
                                             DevFlags* flags,
                                             long long limit = kGridWaitCycles) {
  __shared__ int s_abort;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const long long t0 = clock64();
    int ab = 0;
    while (*reinterpret_cast<volatile unsigned*>(bar) < target) {
      if (*reinterpret_cast<volatile int*>(abort)) {
        ab = 1;
        break;
      }
      if (clock64() - t0 > limit) {
        atomicExch(abort, 1);
        if (atomicCAS(&flags->code, 0, (int)FF_ERR_TIMEOUT) == 0) flags->index = -1;
        ab = 1;
        break;
      }
      __nanosleep(32);
    }
    __threadfence();
    s_abort = ab || *reinterpret_cast<volatile int*>(abort);
  }
  __syncthreads();
  return s_abort == 0;
}

// Farthest-point sampling in rounds, a cooperative launch of up to one block per
// SM.  Block b owns points [b S, min(n, (b + 1) S)) and keeps, in shared memory
// (global memory when the slice does not fit), each point's position, the FP32
// squared distance to its nearest chosen centre and that centre's index; the
// exact (FP64) distance is computed from the two only where it decides.
//
// A distance only falls as centres are added, so the largest distance known
// for a point bounds it for the rest of the run.  Each round
//   1. folds the centres chosen last into the slice (FP32; FP64 within the
//      margin of a near tie),
//   2. publishes the block's `top` farthest points in the exact order
//      (distance, then lowest index), and the next one as its bound,
//   3. one grid barrier,
//   4. every block chooses centres among the published points alone (two a
//      thread; 256 threads of four points took 1.3 times as long), folding each
//      into the others, while the farthest of them comes before every block's
//      bound in that order: no unpublished point can then come before it, so it
//      is the farthest of all points.  FP32 decides a choice unless two
//      distances, or one and the bound, lie within its margin.
// The first choice of a round always passes, so a round adds one centre at
// least; holes of the covering are many once some tens of centres stand, and a
// round adds up to kFpsNew.
//
// One centre a barrier was bound by the barrier and by FP64 updates (a warp
// instruction costs the same for one lane as for 32): 8.19 ms for 1M points and
// 1,000 centres, 6.45 ms for 228k grid points; 1.50 and 1.81 ms in 37
// and 51 rounds.  Up to 1,024 points one block takes them all as
// its published points and needs no round.
struct FpsCand {
  unsigned long long key;  // bit pattern of the squared distance (>= 0)
  int idx;
  float x, y, z;
  int near;                // its nearest chosen centre
  int pad;
};

constexpr int kFpsNew = 128;   // centres a round chooses at most
constexpr int kPool = 2 * kFpsT;  // published points: two a thread
constexpr unsigned long long kNoKey = ~0ull;

// whether (ka, ia) comes before (kb, ib): larger key, ties to the lower index
__device__ __forceinline__ bool fps_before(unsigned long long ka, int ia, unsigned long long kb,
                                           int ib) {
  return ka > kb || (ka == kb && ia < ib);
}

// the first of the warp's (key, idx) in every lane
__device__ __forceinline__ void fps_warp_first(unsigned long long& key, int& idx) {
  const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
  const unsigned mh = __reduce_max_sync(kFull, hi);
  const unsigned ml = __reduce_max_sync(kFull, hi == mh ? lo : 0u);
  idx = __reduce_min_sync(kFull, hi == mh && lo == ml ? idx : INT_MAX);
  key = (unsigned long long)mh << 32 | ml;
}

// the first (key, idx) of the block, with its position, in every thread; red
// alternates between two buffers, so one barrier a call also orders its reuse
__device__ __forceinline__ FpsCand fps_block_first(FpsCand c, FpsCand (*red)[kFpsT / 32],
                                                   int& buf) {
  const int lane = threadIdx.x & 31;
  FpsCand w = c;
  fps_warp_first(w.key, w.idx);
  const unsigned own = __ballot_sync(kFull, c.key == w.key && c.idx == w.idx);
  if (lane == __ffs(own) - 1) red[buf][threadIdx.x >> 5] = c;
  __syncthreads();
  c = red[buf][lane % (kFpsT / 32)];
  buf ^= 1;
  w = c;
  fps_warp_first(w.key, w.idx);
  const int src = __ffs(__ballot_sync(kFull, c.key == w.key && c.idx == w.idx)) - 1;
  w.x = __shfl_sync(kFull, c.x, src);
  w.y = __shfl_sync(kFull, c.y, src);
  w.z = __shfl_sync(kFull, c.z, src);
  return w;
}

// (called, not inlined: the deciding paths are rare and the FP32 ones short)
__device__ __noinline__ unsigned long long fps_key(float x, float y, float z,
                                                      const float* __restrict__ X, int centre) {
  return (unsigned long long)__double_as_longlong(
      d2_f64(x, y, z, X[3LL * centre], X[3LL * centre + 1], X[3LL * centre + 2]));
}

// the FP32 distance up to which a new centre may be nearer than d: the filter's
// margin above it, everything for tiny distances, nothing for d < 0
__device__ __forceinline__ float fps_near(float d) {
  return d >= 0.f && d < 1e-30f ? INFINITY : __fmul_rn(d, 1.00001f);
}

// the largest and second largest FP32 distance (bits) of a warp's published
// points, and the point of the largest
struct __align__(16) FpsPick {
  int m1, m2, idx, pad;
  float x, y, z, w;
};

__global__ void __launch_bounds__(kFpsT, 1)
    k_fps_rounds(const float* __restrict__ X, int n, int K, int start, int S, int top,
                 int in_smem, float* __restrict__ gslice, int* __restrict__ gnear,
                 long long* __restrict__ chosen, FpsCand* __restrict__ cand, unsigned* bar,
                 int* abort, DevFlags* __restrict__ flags) {
  const int G = gridDim.x, rank = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int p0 = (int)min((long long)rank * S, (long long)n);
  const int cnt = min(n - p0, S);
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ FpsCand red[2][kFpsT / 32];
  __shared__ float4 fresh[kFpsNew];  // the centres chosen last, w their index
  __shared__ unsigned s_max[kFpsT / 16];
  static_assert(kFpsT == 512, "the threshold takes 32 half-warps, one a lane");
  __shared__ FpsPick pick[2][kFpsT / 32];
  __shared__ FpsCand tie[2][kFpsT / 32];
  float *xs, *ys, *zs, *cur;
  int* near;
  if (in_smem) {
    xs = reinterpret_cast<float*>(sm_raw);
    near = reinterpret_cast<int*>(xs + 4 * (size_t)S);
  } else {
    xs = gslice + 4 * (size_t)S * rank;
    near = gnear + (size_t)S * rank;
  }
  ys = xs + S;
  zs = ys + S;
  cur = zs + S;
  for (int p = tid; p < cnt; p += kFpsT) {
    const long long g = 3LL * (p0 + p);
    xs[p] = X[g];
    ys[p] = X[g + 1];
    zs[p] = X[g + 2];
    cur[p] = __int_as_float(0x7f800000);
    near[p] = start;
  }
  if (tid == 0) {
    fresh[0] = make_float4(X[3LL * start], X[3LL * start + 1], X[3LL * start + 2],
                           __int_as_float(start));
    if (rank == 0) chosen[0] = start;
  }
  __syncthreads();
  int nnew = 1, j = 1, buf = 0, pbuf = 0, tbuf = 0;
  const bool whole = G == 1 && n <= kPool;  // every point is a published one
  const FpsCand* pool = nullptr;
  unsigned long long bkey = 0ull;
  int bidx = INT_MAX;
  for (int round = 1; j < K; ++round) {
    if (!whole) {
      // ---- 1. fold in the fresh centres (four points a thread at a time)
      unsigned fmax = 0;  // bits of the thread's largest FP32 distance
      for (int q = tid; q < cnt; q += 4 * kFpsT) {
        float x[4], y[4], z[4], d[4];
        int c[4];
  #pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = q + u * kFpsT;
          const bool in = p < cnt;
          x[u] = in ? xs[p] : 0.f;
          y[u] = in ? ys[p] : 0.f;
          z[u] = in ? zs[p] : 0.f;
          d[u] = in ? cur[p] : -1.f;  // -1: below every squared distance
          c[u] = in ? near[p] : 0;
        }
        float near_d[4];  // a distance up to this needs a closer look
#pragma unroll
        for (int u = 0; u < 4; ++u) near_d[u] = fps_near(d[u]);
        for (int b = 0; b < nnew; ++b) {
          const float4 f = fresh[b];
          float dn[4];
          bool look = false;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            dn[u] = d2_fma(x[u], y[u], z[u], f.x, f.y, f.z);
            look |= dn[u] <= near_d[u];
          }
          if (!look) continue;
          const int cn = __float_as_int(f.w);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (!(dn[u] <= near_d[u])) continue;
            if ((dn[u] < __fmul_rn(d[u], 0.99999f) && d[u] >= 1e-30f) ||
                fps_key(x[u], y[u], z[u], X, cn) < fps_key(x[u], y[u], z[u], X, c[u])) {
              d[u] = dn[u];
              c[u] = cn;
              // a point that coincides with a centre has nothing left to fold
              if (dn[u] < 1e-30f && fps_key(x[u], y[u], z[u], X, cn) == 0ull) d[u] = -1.f;
              near_d[u] = fps_near(d[u]);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = q + u * kFpsT;
          if (p < cnt) {
            cur[p] = d[u];
            near[p] = c[u];
            if (d[u] > 0.f) fmax = max(fmax, __float_as_uint(d[u]));
          }
        }
      }
      // ---- 2. a threshold that `top` half-warps' points reach (all when the
      // block has fewer), widened so that rounding hides no point
      {
        const unsigned hm = __reduce_max_sync(lane < 16 ? 0xffffu : 0xffff0000u, fmax);
        if (lane % 16 == 0) s_max[tid / 16] = hm;
      }
      __syncthreads();
      float tau;
      {
        unsigned v = s_max[lane], m = 0;
        for (int t = 0; t < min(top, 32); ++t) {
          m = __reduce_max_sync(kFull, v);
          const unsigned first = __ballot_sync(kFull, v == m);
          if (lane == __ffs(first) - 1) v = 0;
        }
        tau = __fmul_rn(__uint_as_float(m), 0.999997f);
        if (tau < 1e-30f) tau = -1.f;
      }
      // the thread's first two points at or above the threshold, exactly
      FpsCand a{0ull, INT_MAX, 0.f, 0.f, 0.f, 0, 0};
      unsigned long long k2 = 0ull;
      int i2 = INT_MAX;
      int left = 0;  // those beyond the two
      auto scan = [&](unsigned long long lk, int li) {  // those after (lk, li)
        left = -2;
        a.key = k2 = 0ull;
        a.idx = i2 = INT_MAX;
        for (int p = tid; p < cnt; p += kFpsT) {
          if (!(cur[p] >= tau)) continue;
          const unsigned long long k = fps_key(xs[p], ys[p], zs[p], X, near[p]);
          const int g = p0 + p;
          if (!fps_before(lk, li, k, g)) continue;
          ++left;
          if (fps_before(k, g, a.key, a.idx)) {
            k2 = a.key;
            i2 = a.idx;
            a.key = k;
            a.idx = g;
          } else if (fps_before(k, g, k2, i2)) {
            k2 = k;
            i2 = g;
          }
        }
      };
      if (__uint_as_float(fmax) >= tau && tid < cnt) scan(~0ull, -1);
      FpsCand* mine = cand + ((size_t)(round & 1) * G + rank) * (top + 1);
      int t = 0;
      FpsCand w = fps_block_first(a, red, buf);
      for (; t < top && w.idx != INT_MAX; ++t) {
        if (w.idx == a.idx) {  // the owner publishes it and offers its next
          const int p = a.idx - p0;
          mine[t] = FpsCand{a.key, a.idx, xs[p], ys[p], zs[p], near[p], 0};
          if (i2 != INT_MAX) {
            a.key = k2;
            a.idx = i2;
            i2 = INT_MAX;
          } else if (left > 0) {
            scan(w.key, w.idx);
          } else {
            a.key = 0ull;
            a.idx = INT_MAX;
          }
        }
        w = fps_block_first(a, red, buf);
      }
      if (tid == 0) {
        // the bound: the next point, or what a point below the threshold may reach
        FpsCand r{0ull, -1, 0.f, 0.f, 0.f, 0, 0};
        if (tau > 0.f) r.key = (unsigned long long)__double_as_longlong((double)tau * 1.000002);
        mine[top] = w.idx != INT_MAX && fps_before(w.key, w.idx, r.key, r.idx) ? w : r;
        for (; t < top; ++t) mine[t] = FpsCand{0ull, INT_MAX, 0.f, 0.f, 0.f, 0, 0};
      }
      // ---- 3.
      if (!grid_barrier(bar, (unsigned)round * (unsigned)G, abort, flags)) break;
      // the first of the bounds (L1 bypassed)
      pool = cand + (size_t)(round & 1) * G * (top + 1);
      FpsCand bound{0ull, INT_MAX, 0.f, 0.f, 0.f, 0, 0};
      for (int q = tid; q < G; q += kFpsT) {
        const FpsCand* c = pool + (size_t)q * (top + 1) + top;
        const unsigned long long k = __ldcg(&c->key);
        const int i = __ldcg(&c->idx);
        if (fps_before(k, i, bound.key, bound.idx)) {
          bound.key = k;
          bound.idx = i;
        }
      }
      bound = fps_block_first(bound, red, buf);
      bkey = bound.key;
      bidx = bound.idx;
    }
    // ---- 4. choose among the published points
    bool stop = false;
    int taken = 0;
    {
      float x[2], y[2], z[2], d[2];  // d < 0: none, or at a chosen centre
      int id[2], nr[2];
      unsigned long long ek[2];  // exact distances, computed when asked for
      auto exact = [&](int u) {
        if (ek[u] == kNoKey) ek[u] = fps_key(x[u], y[u], z[u], X, nr[u]);
        return ek[u];
      };
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int e = tid + u * kFpsT;
        id[u] = INT_MAX;
        nr[u] = start;
        d[u] = -1.f;
        ek[u] = kNoKey;
        x[u] = y[u] = z[u] = 0.f;
        if (whole && e < cnt) {
          id[u] = e;
          x[u] = xs[e];
          y[u] = ys[e];
          z[u] = zs[e];
          d[u] = d2_f32(x[u], y[u], z[u], fresh[0].x, fresh[0].y, fresh[0].z);
          if (d[u] < 1e-30f && exact(u) == 0ull) d[u] = -1.f;
        } else if (!whole && e < G * top) {
          const FpsCand* c = pool + e / top * (top + 1) + e % top;
          id[u] = __ldcg(&c->idx);
          if (id[u] != INT_MAX) {
            x[u] = __ldcg(&c->x);
            y[u] = __ldcg(&c->y);
            z[u] = __ldcg(&c->z);
            nr[u] = __ldcg(&c->near);
            ek[u] = __ldcg(&c->key);
            d[u] = ek[u] ? (float)__longlong_as_double((long long)ek[u]) : -1.f;
          }
        }
      }
      // an FP32 distance above this lies above the bound for certain
      const float over = (float)__longlong_as_double((long long)bkey) * 1.000002f;
      while (j < K && (whole || taken < kFpsNew)) {
        int b1 = -1, b2 = -1, bu = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int v = d[u] >= 0.f ? __float_as_int(d[u]) : -1;
          if (v > b1) {
            b2 = b1;
            b1 = v;
            bu = u;
          } else if (v > b2) {
            b2 = v;
          }
        }
        const int m1 = __reduce_max_sync(kFull, b1);
        const int own = __ffs(__ballot_sync(kFull, b1 == m1)) - 1;
        const int m2 = __reduce_max_sync(kFull, lane == own ? b2 : b1);
        if (lane == own) {
          FpsPick r{m1, m2, INT_MAX, 0, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (u == bu) {
              r.idx = id[u];
              r.x = x[u];
              r.y = y[u];
              r.z = z[u];
            }
          pick[pbuf][wid] = r;
        }
        __syncthreads();
        FpsPick r = pick[pbuf][lane % (kFpsT / 32)];
        pbuf ^= 1;
        const int M = __reduce_max_sync(kFull, r.m1);
        const int src = __ffs(__ballot_sync(kFull, r.m1 == M)) - 1;
        if (M < 0) {  // every published point is at a chosen centre: so is every
                      // other one when no bound is above zero
          stop = bkey == 0ull;
          break;
        }
        const float far = __int_as_float(M);
        float near_far = __fmul_rn(far, 0.999997f);
        if (far < 1e-30f) near_far = 0.f;
        const int other = lane == src ? r.m2 : lane < kFpsT / 32 ? r.m1 : -1;
        const bool close =
            __any_sync(kFull, other >= 0 && __int_as_float(other) >= near_far);
        int wi = __shfl_sync(kFull, r.idx, src);
        float wx = __shfl_sync(kFull, r.x, src);
        float wy = __shfl_sync(kFull, r.y, src);
        float wz = __shfl_sync(kFull, r.z, src);
        if (close || far < 1e-30f || (taken > 0 && !(far > over))) {
          // too close to call in FP32: the exact order of the points near the top
          FpsCand a{0ull, INT_MAX, 0.f, 0.f, 0.f, 0, 0};
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (d[u] >= near_far) {
              const unsigned long long k = exact(u);
              if (fps_before(k, id[u], a.key, a.idx)) a = FpsCand{k, id[u], x[u], y[u], z[u], 0, 0};
            }
          FpsCand w = a;
          fps_warp_first(w.key, w.idx);
          const unsigned has = __ballot_sync(kFull, a.key == w.key && a.idx == w.idx);
          if (lane == __ffs(has) - 1) tie[tbuf][wid] = a;
          __syncthreads();
          a = tie[tbuf][lane % (kFpsT / 32)];
          tbuf ^= 1;
          w = a;
          fps_warp_first(w.key, w.idx);
          const int from = __ffs(__ballot_sync(kFull, a.key == w.key && a.idx == w.idx)) - 1;
          wi = w.idx;
          wx = __shfl_sync(kFull, a.x, from);
          wy = __shfl_sync(kFull, a.y, from);
          wz = __shfl_sync(kFull, a.z, from);
          if (w.key == 0ull) {
            // every published point coincides with a chosen centre: so does
            // every other one when no bound is above zero
            stop = bkey == 0ull;
            break;
          }
          if (taken > 0 && !fps_before(w.key, w.idx, bkey, bidx)) break;
        }
        if (tid == 0) {
          if (!whole) fresh[taken] = make_float4(wx, wy, wz, __int_as_float(wi));
          if (rank == 0) chosen[j] = wi;
        }
        ++taken;
        ++j;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float dn = d2_fma(x[u], y[u], z[u], wx, wy, wz);
          if (id[u] == wi) {
            d[u] = -1.f;
          } else if (dn <= fps_near(d[u])) {
            if ((dn < __fmul_rn(d[u], 0.99999f) && d[u] >= 1e-30f) ||
                fps_key(x[u], y[u], z[u], X, wi) < exact(u)) {
              d[u] = dn;
              nr[u] = wi;
              ek[u] = kNoKey;
              if (dn < 1e-30f && exact(u) == 0ull) d[u] = -1.f;
            }
          }
        }
      }
    }
    nnew = taken;
    if (stop) {
      if (rank == 0 && tid == 0 && atomicCAS(&flags->code, 0, (int)FF_ERR_INVALID_ARG) == 0)
        flags->index = j;
      break;
    }
    __syncthreads();  // fresh is read by every thread next
  }
}

// Self-check of the bounded wait: every block arrives once at a barrier that
// waits for one arrival more than the grid has, so the wait can only end by
// running out (FF_ERR_TIMEOUT in the flags) or through the abort word.
__global__ void k_wait_check(unsigned* bar, int* abort, DevFlags* flags, long long limit) {
  grid_barrier(bar, gridDim.x + 1u, abort, flags, limit);
}

__global__ void k_gather_centres(const float* __restrict__ X, const long long* __restrict__ chosen,
                                 int K, float4* __restrict__ cpos) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  const long long i = chosen[k];
  cpos[k] = make_float4(X[3 * i], X[3 * i + 1], X[3 * i + 2], 0.f);
}

// ------------------------------------------------------------------ radii
// r_k = sqrt(second-smallest squared distance to the other centres); lim_k =
// (t*t) * (r_k*r_k) or +inf without a cut.
__global__ void k_radii(const float4* __restrict__ cpos, int K, double tt, double* __restrict__ rad,
                        double* __restrict__ lim, float* __restrict__ lim32,
                        DevFlags* __restrict__ flags) {
  const int k = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (k >= K) return;
  const int lane = threadIdx.x & 31;
  const float4 p = cpos[k];
  double m1 = INFINITY, m2 = INFINITY;
  for (int j = lane; j < K; j += 32) {
    if (j == k) continue;
    const float4 q = cpos[j];
    const double d = d2_f64(q.x, q.y, q.z, p.x, p.y, p.z);
    if (d < m1) {
      m2 = m1;
      m1 = d;
    } else if (d < m2) {
      m2 = d;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const double a1 = __shfl_xor_sync(kFull, m1, o);
    const double a2 = __shfl_xor_sync(kFull, m2, o);
    const double lo = fmin(m1, a1);
    const double hi = fmin(fmax(m1, a1), fmin(m2, a2));
    m1 = lo;
    m2 = hi;
  }
  if (lane == 0) {
    const double r = __dsqrt_rn(m2);
    rad[k] = r;
    const double L = tt > 0.0 ? __dmul_rn(tt, __dmul_rn(r, r)) : (double)INFINITY;
    lim[k] = L;
    lim32[k] = (float)L;
    if (!(r > 0.0) || !isfinite(r))
      if (atomicCAS(&flags->code, 0, (int)FF_ERR_INVALID_ARG) == 0) flags->index = k;
  }
}

// ------------------------------------------------------------------ covering lists
// MODE 0: count the centres covering each point; MODE 1: list them, ascending
template <int MODE>
__global__ void __launch_bounds__(256)
    k_cover_rows(const float* __restrict__ Xq, long long nq, const float4* __restrict__ cpos,
                 const float* __restrict__ lim32, const double* __restrict__ lim, int K,
                 int* __restrict__ cnt, const long long* __restrict__ rptr,
                 int* __restrict__ ridx) {
  __shared__ float4 sp[256];
  __shared__ float sl32[256];
  __shared__ double sl[256];
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  const bool live = i < nq;
  float x = 0.f, y = 0.f, z = 0.f;
  long long base = 0, end = 0;
  if (live) {
    x = Xq[3 * i];
    y = Xq[3 * i + 1];
    z = Xq[3 * i + 2];
    if (MODE) {
      base = rptr[i];
      end = rptr[i + 1];
    }
  }
  int c = 0;
  for (int k0 = 0; k0 < K; k0 += 256) {
    __syncthreads();
    if (k0 + (int)threadIdx.x < K) {
      sp[threadIdx.x] = cpos[k0 + threadIdx.x];
      sl32[threadIdx.x] = lim32[k0 + threadIdx.x];
      sl[threadIdx.x] = lim[k0 + threadIdx.x];
    }
    __syncthreads();
    const int kn = min(256, K - k0);
    if (live) {
      for (int q = 0; q < kn; ++q) {
        if (covers2(x, y, z, sp[q], sl32[q], sl[q])) {
          if (MODE && base + c < end) ridx[base + c] = k0 + q;
          ++c;
        }
      }
    }
  }
  if (!MODE && live) cnt[i] = c;
}

// The covering of kBitPts points a block as bits, word-major (bits[w][i]: centres
// 32 w .. 32 w + 31 of point i), and the count of each point.  Two points a thread
// share the reads of a staged centre; a pair inside the FP32 margin is settled in
// FP64 after its word.  Bound by the tests' issue: 14 instructions a pair.  With
// k_cover_fill it stands for two passes of k_cover_rows (0.67 + 0.97 ms for 1M
// points and 1,000 centres): 0.36 + 0.23 ms.
constexpr int kBitPts = 512;

__global__ void __launch_bounds__(kBitPts / 2)
    k_cover_bits(const float* __restrict__ Xq, long long nq, const float4* __restrict__ cpos,
                 const float* __restrict__ lim32, const double* __restrict__ lim, int K,
                 int* __restrict__ cnt, unsigned* __restrict__ bits) {
  constexpr int T = kBitPts / 2;
  __shared__ float4 sp[T];   // position, upper limit of the FP32 margin
  __shared__ float slo[T];   // lower limit
  const int tid = threadIdx.x;
  long long i[2];
  float x[2], y[2], z[2];
  int c[2] = {0, 0};
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    i[u] = (long long)blockIdx.x * kBitPts + u * T + tid;
    const long long r = min(i[u], nq - 1);
    x[u] = Xq[3 * r];
    y[u] = Xq[3 * r + 1];
    z[u] = Xq[3 * r + 2];
  }
  for (int k0 = 0; k0 < K; k0 += T) {
    __syncthreads();
    {
      const int k = k0 + tid;
      float4 p = make_float4(0.f, 0.f, 0.f, -1.f);  // covers nothing
      float lo = -1.f;
      if (k < K) {
        p = cpos[k];
        const float l32 = lim32[k];
        // tiny limits: every pair in FP64
        p.w = l32 >= 1e-30f ? __fmul_rn(l32, 1.00001f) : INFINITY;
        lo = l32 >= 1e-30f ? __fmul_rn(l32, 0.99999f) : -1.f;
      }
      sp[tid] = p;
      slo[tid] = lo;
    }
    __syncthreads();
    for (int w0 = 0; w0 < T && k0 + w0 < K; w0 += 32) {
      unsigned in[2] = {0u, 0u}, near[2] = {0u, 0u};
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        const float4 p = sp[w0 + q];
        const float lo = slo[w0 + q];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float d = d2_fma(x[u], y[u], z[u], p.x, p.y, p.z);
          if (d < lo) in[u] |= 1u << q;
          if (d <= p.w) near[u] |= 1u << q;
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        for (unsigned b = near[u] & ~in[u]; b; b &= b - 1) {
          const int q = __ffs(b) - 1;
          const float4 p = sp[w0 + q];
          if (d2_f64(x[u], y[u], z[u], p.x, p.y, p.z) < lim[k0 + w0 + q]) in[u] |= 1u << q;
        }
        c[u] += __popc(in[u]);
        if (i[u] < nq) bits[(long long)((k0 + w0) >> 5) * nq + i[u]] = in[u];
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (i[u] < nq) cnt[i[u]] = c[u];
}

// The lists of 32 points a block from their bits: the words staged transposed in
// shared memory, then a warp a point, a lane a word.
__global__ void __launch_bounds__(256)
    k_cover_fill(const unsigned* __restrict__ bits, long long nq, int words,
                 const long long* __restrict__ rptr, int* __restrict__ ridx) {
  __shared__ unsigned sb[32][33];
  const long long i0 = (long long)blockIdx.x * 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long at[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const long long i = i0 + wid + 8 * u;
    at[u] = i < nq ? rptr[i] : 0;
  }
  for (int w0 = 0; w0 < words; w0 += 32) {
    if (w0) __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int w = w0 + wid + 8 * u;
      sb[wid + 8 * u][lane] = w < words && i0 + lane < nq ? bits[(long long)w * nq + i0 + lane] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      unsigned b = sb[lane][wid + 8 * u];
      const int h = __popc(b);
      int off = h;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, off, o);
        if (lane >= o) off += t;
      }
      long long p = at[u] + off - h;
      at[u] += __shfl_sync(kFull, off, 31);
      for (; b; b &= b - 1) ridx[p++] = 32 * (w0 + lane) + __ffs(b) - 1;
    }
  }
}

// MODE 0: count the points each centre covers; MODE 1: list them (ascending)
// with the position of the centre in each point's (ascending) row
template <int MODE>
__global__ void k_cover_cols(const float* __restrict__ Xq, long long nq,
                             const float4* __restrict__ cpos, const float* __restrict__ lim32,
                             const double* __restrict__ lim, int K, int* __restrict__ cnt,
                             const long long* __restrict__ tptr, int* __restrict__ tidx,
                             long long* __restrict__ tpos, const long long* __restrict__ rptr,
                             const int* __restrict__ ridx, DevFlags* __restrict__ flags) {
  const int k = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (k >= K) return;
  const int lane = threadIdx.x & 31;
  const float4 p = cpos[k];
  const float l32 = lim32[k];
  const double l64 = lim[k];
  const long long base = MODE ? tptr[k] : 0, end = MODE ? tptr[k + 1] : 0;
  long long c = 0;
  for (long long i0 = 0; i0 < nq; i0 += 32) {
    const long long i = i0 + lane;
    bool cov = false;
    if (i < nq) cov = covers2(Xq[3 * i], Xq[3 * i + 1], Xq[3 * i + 2], p, l32, l64);
    const unsigned bal = __ballot_sync(kFull, cov);
    if (MODE && cov) {
      const long long slot = base + c + __popc(bal & ((1u << lane) - 1u));
      if (slot < end) {
        long long lo = rptr[i], hi = rptr[i + 1];
        const long long row_end = hi;
        while (lo < hi) {
          const long long mid = (lo + hi) >> 1;
          if (ridx[mid] < k)
            lo = mid + 1;
          else
            hi = mid;
        }
        tidx[slot] = (int)i;
        if (lo < row_end && ridx[lo] == k) {
          tpos[slot] = lo;
        } else {  // the two passes disagree: report, keep the position in range
          tpos[slot] = rptr[i];
          if (atomicCAS(&flags->code, 0, (int)FF_ERR_CUDA) == 0) flags->index = k;
        }
      }
    }
    c += __popc(bal);
  }
  if (!MODE && lane == 0) cnt[k] = (int)c;
}

// ------------------------------------------------------------------ shape functions
// what the Gaussian's FP32 and double-float forms take of a radius: the square of
// its FP32 rounding, and 1 / r_k^2 rounded from FP64 (kept finite: a pair at
// distance 0 has weight 1 whatever the radius)
__global__ void k_centre_inv(const double* __restrict__ rad, int K, float4* __restrict__ cpos,
                             dfloat* __restrict__ inv) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  const float r = (float)rad[k];
  cpos[k].w = r * r;
  inv[k] = dfloat(fmin(1.0 / (rad[k] * rad[k]), 3e38));
}

// lanes a row: a point has ~100 covering centres, so eight lanes take a dozen
// each and a warp's moment solve serves four points.  FP32, 1M points of 98
// centres: 3.17 ms with a warp a point, 1.61 ms in its
// order of operations (0.95 ms in a free one; values alone 0.6 ms); double-float,
// 228k points: 5.79 ms, 2.91 ms now, of which 0.73 for sums and quotients as exact
// as a warp a point has them.
constexpr int kShapeLanes = 8;

template <class T, bool GRAD>
__global__ void __launch_bounds__(256, 2)
    k_shape_twoset(const float4* __restrict__ cpos, const rkpm::Gauss kern,
                   const float* __restrict__ Xq, float scale, const long long* __restrict__ ptr,
                   const int* __restrict__ idx, long long nq, long long n1, T* __restrict__ phi,
                   T* __restrict__ dphi, double cond_limit, int* __restrict__ redo,
                   DevFlags* __restrict__ flags) {
  const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kShapeLanes;
  const bool live = i < nq, first = threadIdx.x % kShapeLanes == 0;
  const long long s = live ? ptr[i] : 0, e = live ? ptr[i + 1] : 0;
  const float4 Xi = live ? make_float4(Xq[3 * i], Xq[3 * i + 1], Xq[3 * i + 2], scale)
                         : make_float4(0.f, 0.f, 0.f, 1.f);
  if constexpr (sizeof(T) == 4) {
    int st;
    if constexpr (GRAD)
      st = rkpm::shape_rows_ordered(cpos, s, e, idx, Xi, phi, dphi, n1, cond_limit, kern);
    else
      st = rkpm::shape_rows<float, T, kShapeLanes, GRAD>(cpos, s, e, idx, Xi, phi, dphi, n1,
                                                        cond_limit, true, kern);
    if (live && st != 0 && first) rkpm::redo_later(redo, i);
  } else {
    const int st = rkpm::shape_rows<dfloat, T, kShapeLanes, GRAD>(
        cpos, s, e, idx, Xi, phi, dphi, n1, 0.0, false, kern);
    if (live && st != 0 && first &&
        atomicCAS(&flags->code, 0, (int)FF_ERR_SINGULAR_MOMENT) == 0)
      flags->index = (int)i;
  }
}

__global__ void k_iota(int* __restrict__ a, int* __restrict__ b, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    a[t] = t;
    b[t] = t;
  }
}

__global__ void k_copy_f32(const float* __restrict__ x, float* __restrict__ y, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) y[t] = x[t];
}

}  // namespace

// Covering lists of arbitrary points (the rows of a shape-function table over
// the two-set centres): count, scan, fill.  Returns the number of pairs.
long long twoset_cover(ff_ctx* c, const float* Q, long long nq, Buf& ptrb, Buf& idxb,
                       Buf& cntb) {
  cudaStream_t st = c->stream;
  const int K = (int)c->n;
  int* cnt = reinterpret_cast<int*>(cntb.ensure(sizeof(int) * (nq + 1)));
  // as bits between the two passes while they take less room than the lists
  // (K / 8 bytes a point against 4 a pair, ~100 pairs) and 1 GB at most; else, or
  // without that room, the tests run twice.  More than kKeptScratch is given back
  const int words = (K + 31) / 32;
  const size_t room = sizeof(unsigned) * (size_t)words * nq;
  unsigned* bits = nullptr;
  if (K <= 3200 && room <= (1ull << 30)) {
    try {
      bits = reinterpret_cast<unsigned*>(c->scratch[6].ensure(room));
    } catch (const Error&) {
    }
  }
  if (bits)
    (k_cover_bits<<<ceil_div(nq, kBitPts), kBitPts / 2, 0, st>>>(
         Q, nq, c->pos.as<float4>(), c->clim32.as<float>(), c->clim.as<double>(), K, cnt, bits),
     ::ff::note_launch());
  else
    (k_cover_rows<0><<<ceil_div(nq, 256), 256, 0, st>>>(
         Q, nq, c->pos.as<float4>(), c->clim32.as<float>(), c->clim.as<double>(), K, cnt, nullptr,
         nullptr),
     ::ff::note_launch());
  FF_LAUNCH_CHECK();
  long long* ptr = reinterpret_cast<long long*>(ptrb.ensure(sizeof(long long) * (nq + 1)));
  scan_counts(cnt, ptr, nq, c, c->scratch[3]);
  long long n1 = 0;
  FF_CUDA(cudaMemcpyAsync(&n1, ptr + nq, sizeof(long long), cudaMemcpyDeviceToHost, st));
  FF_CUDA(cudaStreamSynchronize(st));
  int* idx = reinterpret_cast<int*>(idxb.ensure(sizeof(int) * std::max(n1, 1LL)));
  if (bits)
    (k_cover_fill<<<ceil_div(nq, 32), 256, 0, st>>>(bits, nq, words, ptr, idx),
     ::ff::note_launch());
  else
    (k_cover_rows<1><<<ceil_div(nq, 256), 256, 0, st>>>(
         Q, nq, c->pos.as<float4>(), c->clim32.as<float>(), c->clim.as<double>(), K, nullptr, ptr,
         idx),
     ::ff::note_launch());
  FF_LAUNCH_CHECK();
  if (bits) give_back(c, c->scratch[6], room);
  return n1;
}

// Gaussian shape functions of the two-set centres at nq points, launched on the
// context's stream: float (with the FP64 redo) when f32, else double-float
// pairs; with the gradients when dphi is given.  The caller resets the flags
// before and reads them after (FF_ERR_SINGULAR_MOMENT with the point).
void twoset_shape(ff_ctx* c, const float* Q, long long nq, const long long* ptr, const int* idx,
                  long long n1, void* phi, void* dphi, bool f32) {
  cudaStream_t st = c->stream;
  const float4* cpos = c->pos.as<float4>();
  const rkpm::Gauss kern{c->crad.as<double>(), c->cinv.as<dfloat>()};
  DevFlags* flags = c->flags.as<DevFlags>();
  const unsigned grid = ceil_div(nq * kShapeLanes, 256);
  auto run = [&](auto tag, auto grad) {
    using T = decltype(tag);
    constexpr bool GRAD = decltype(grad)::value;
    int* redo = sizeof(T) == 4 ? rkpm::redo_list(c, nq) : nullptr;
    (k_shape_twoset<T, GRAD><<<grid, 256, 0, st>>>(cpos, kern, Q, c->qscale, ptr, idx, nq, n1,
                                                   static_cast<T*>(phi), static_cast<T*>(dphi),
                                                   1e2, redo, flags),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    if constexpr (sizeof(T) == 4) {
      (rkpm::k_shape_redo<T, GRAD, rkpm::Gauss><<<rkpm::redo_grid(nq), 256, 0, st>>>(
           cpos, nullptr, Q, c->qscale, ptr, idx, n1, static_cast<T*>(phi),
           static_cast<T*>(dphi), redo, flags, kern),
       ::ff::note_launch());
      FF_LAUNCH_CHECK();
    }
  };
  if (f32 && dphi)
    run(float{}, std::true_type{});
  else if (f32)
    run(float{}, std::false_type{});
  else if (dphi)
    run(dfloat{}, std::true_type{});
  else
    run(dfloat{}, std::false_type{});
}

// The transposed covering lists of a two-set cloud: for every centre the
// points it covers (ascending) and its position in each point's row; checked
// against the row lists built before.
void twoset_columns(ff_ctx* c, const float* Xq) {
  cudaStream_t st = c->stream;
  const int T = 256;
  const int K = (int)c->n;
  const long long nq = c->nq, n1 = c->n1;
  const float4* cpos = c->pos.as<float4>();
  const float* lim32 = c->clim32.as<float>();
  const double* lim = c->clim.as<double>();
  int* ccnt = reinterpret_cast<int*>(c->scratch[6].ensure(sizeof(int) * (K + 1)));
  (k_cover_cols<0><<<ceil_div((long long)K * 32, T), T, 0, st>>>(
       Xq, nq, cpos, lim32, lim, K, ccnt, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr),
   ::ff::note_launch());
  FF_LAUNCH_CHECK();
  long long* tptr = reinterpret_cast<long long*>(c->nbrT_ptr.ensure(sizeof(long long) * (K + 1)));
  scan_counts(ccnt, tptr, K, c, c->scratch[3]);
  long long n1t = 0;
  FF_CUDA(cudaMemcpyAsync(&n1t, tptr + K, sizeof(long long), cudaMemcpyDeviceToHost, st));
  FF_CUDA(cudaStreamSynchronize(st));
  FF_REQUIRE(n1t == n1, FF_ERR_CUDA, "covering lists disagree between the two passes");
  int* tidx = reinterpret_cast<int*>(c->nbrT_idx.ensure(sizeof(int) * std::max(n1, 1LL)));
  long long* tpos =
      reinterpret_cast<long long*>(c->nbrT_pos.ensure(sizeof(long long) * std::max(n1, 1LL)));
  reset_flags(c);
  (k_cover_cols<1><<<ceil_div((long long)K * 32, T), T, 0, st>>>(
       Xq, nq, cpos, lim32, lim, K, nullptr, tptr, tidx, tpos, c->nbr_ptr.as<long long>(),
       c->nbr_idx.as<int>(), c->flags.as<DevFlags>()),
   ::ff::note_launch());
  FF_LAUNCH_CHECK();
  const DevFlags f = read_flags(c);
  FF_REQUIRE(f.code == 0, FF_ERR_CUDA, "covering lists disagree between the two passes");
  c->has_cols = true;
}

// The grid barrier of the farthest-point sampling with one arrival missing:
// the status the host reads once the bounded wait has run out.
ff_status selftest_device_wait(int device, long long wait_cycles) {
  int coop = 0;
  FF_CUDA(cudaSetDevice(device));
  FF_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device));
  FF_REQUIRE(coop, FF_ERR_CUDA, "the device has no cooperative launch");
  unsigned char* mem = nullptr;
  FF_CUDA(cudaMalloc(&mem, 256));
  ff_status out = FF_ERR_CUDA;
  try {
    unsigned* bar = reinterpret_cast<unsigned*>(mem);
    int* abort = reinterpret_cast<int*>(mem + 16);
    DevFlags* flags = reinterpret_cast<DevFlags*>(mem + 64);
    FF_CUDA(cudaMemset(mem, 0, 256));
    long long limit = wait_cycles;
    void* args[] = {&bar, &abort, &flags, &limit};
    FF_CUDA(cudaLaunchCooperativeKernel((const void*)k_wait_check, dim3(sm_count()), dim3(32),
                                        args, 0, nullptr));
    ::ff::note_launch();
    FF_CUDA(cudaDeviceSynchronize());
    DevFlags h{};
    FF_CUDA(cudaMemcpy(&h, flags, sizeof(h), cudaMemcpyDeviceToHost));
    out = h.code == FF_ERR_TIMEOUT ? FF_ERR_TIMEOUT : h.code == 0 ? FF_OK : (ff_status)h.code;
  } catch (...) {
    cudaFree(mem);
    throw;
  }
  cudaFree(mem);
  return out;
}

void build_twoset(ff_ctx* c, const float* Xq, const float* vq, long long nq, int K, double trunc,
                  long long start) {
  cudaStream_t st = c->stream;
  const int T = 256;
  // ---- 1. validation
  int* bad = reinterpret_cast<int*>(c->scratch[0].ensure(64));
  const int imax = INT_MAX;
  FF_CUDA(cudaMemcpyAsync(bad, &imax, sizeof(int), cudaMemcpyHostToDevice, st));
  (k_validate_points<<<(int)std::min<long long>(ceil_div(nq, T), (long long)sm_count() * 8), T, 0, st>>>(Xq, vq, nq,
                                                                                      bad),
   ::ff::note_launch());
  FF_LAUNCH_CHECK();
  int badi = INT_MAX;
  FF_CUDA(cudaMemcpyAsync(&badi, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  FF_CUDA(cudaStreamSynchronize(st));
  FF_REQUIRE(badi == INT_MAX, FF_ERR_INVALID_ARG,
             "invalid quadrature point " + std::to_string(badi) +
                 ": positions must be finite (|x| < 1e18) and volumes > 0");
  c->n = K;
  c->nq = nq;
  c->twoset = true;
  c->trunc = trunc;

  // ---- 2. farthest-point sampling: one block per 1,024 points up to one per
  // SM; the points the blocks publish a round fill the 1,024 places that are
  // chosen among (at most 16 a block: each costs a block reduction)
  const int n = (int)nq;
  long long* chosen = reinterpret_cast<long long*>(c->centre_idx.ensure(sizeof(long long) * K));
  reset_flags(c);
  {
    ProfScope ps(kProfFps);
    int coop = 0;
    FF_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, c->device));
    FF_REQUIRE(coop, FF_ERR_CUDA, "the device has no cooperative launch");
    int G = std::min(std::min(sm_count(), kPool), (n + kPool - 1) / kPool);
    int S = (n + G - 1) / G, top = std::min(16, kPool / G);
    const size_t smem = 20 * (size_t)S;
    int in_smem = smem <= (size_t)kFpsSmemMax ? 1 : 0;
    if (in_smem) set_max_dyn_smem((const void*)k_fps_rounds, (int)smem);
    float* gslice = nullptr;
    int* gnear = nullptr;
    if (!in_smem) {
      gslice = reinterpret_cast<float*>(c->scratch[1].ensure(16 * (size_t)S * G));
      gnear = reinterpret_cast<int*>(c->scratch[2].ensure(sizeof(int) * (size_t)S * G));
    }
    // two buffers of published points, then the barrier counter and the abort word
    const size_t pool = 2 * sizeof(FpsCand) * (size_t)G * (top + 1);
    unsigned char* sync = reinterpret_cast<unsigned char*>(c->scratch[7].ensure(pool + 64));
    FpsCand* cand = reinterpret_cast<FpsCand*>(sync);
    unsigned* bar = reinterpret_cast<unsigned*>(sync + pool);
    int* abort = reinterpret_cast<int*>(bar + 4);
    FF_CUDA(cudaMemsetAsync(bar, 0, 32, st));
    int nn = n, KK = K, st0 = (int)start;
    DevFlags* fl = c->flags.as<DevFlags>();
    void* args[] = {(void*)&Xq, &nn,  &KK,     &st0,  &S,   &top,   &in_smem, &gslice,
                    &gnear,     &chosen, &cand, &bar, &abort, &fl};
    FF_CUDA(cudaLaunchCooperativeKernel((const void*)k_fps_rounds, dim3(G), dim3(kFpsT), args,
                                        in_smem ? smem : 0, st));
    ::ff::note_launch();
  }
  DevFlags f = read_flags(c);
  FF_REQUIRE(f.code != FF_ERR_TIMEOUT, FF_ERR_TIMEOUT,
             "farthest-point sampling: a grid barrier wait ran out");
  FF_REQUIRE(f.code == 0, FF_ERR_INVALID_ARG,
             "the quadrature points hold fewer than K = " + std::to_string(K) +
                 " distinct positions (farthest-point step " + std::to_string(f.index) + ")");

  // ---- 3. centres and radii
  float4* cpos = reinterpret_cast<float4*>(c->pos.ensure(sizeof(float4) * K));
  (k_gather_centres<<<ceil_div(K, T), T, 0, st>>>(Xq, chosen, K, cpos), ::ff::note_launch());
  double* rad = reinterpret_cast<double*>(c->crad.ensure(sizeof(double) * K));
  double* lim = reinterpret_cast<double*>(c->clim.ensure(sizeof(double) * K));
  float* lim32 = reinterpret_cast<float*>(c->clim32.ensure(sizeof(float) * K));
  reset_flags(c);
  (k_radii<<<ceil_div((long long)K * 32, T), T, 0, st>>>(cpos, K, trunc > 0 ? trunc * trunc : 0.0,
                                                         rad, lim, lim32, c->flags.as<DevFlags>()),
   ::ff::note_launch());
  FF_LAUNCH_CHECK();
  f = read_flags(c);
  FF_REQUIRE(f.code == 0, FF_ERR_INVALID_ARG,
             "centre " + std::to_string(f.index) + " has a zero radius");
  (k_centre_inv<<<ceil_div(K, T), T, 0, st>>>(
       rad, K, cpos, reinterpret_cast<dfloat*>(c->cinv.ensure(sizeof(dfloat) * K))),
   ::ff::note_launch());
  FF_LAUNCH_CHECK();
  std::vector<double> hr(K);
  FF_CUDA(cudaMemcpy(hr.data(), rad, sizeof(double) * K, cudaMemcpyDeviceToHost));
  // basis scale of the shape functions (any positive value gives the same
  // functions; the largest radius keeps the moment matrices well scaled)
  c->qscale = (float)*std::max_element(hr.begin(), hr.end());

  // ---- 4. covering lists: rows (point -> centres) and columns (centre -> points)
  ProfScope ps_cover(kProfCover);
  const long long n1 = twoset_cover(c, Xq, nq, c->nbr_ptr, c->nbr_idx, c->scratch[5]);
  c->n1 = n1;
  ps_cover.close();

  // ---- 5. quadrature volumes, identity order of the centres
  float* vol = reinterpret_cast<float*>(c->vol.ensure(sizeof(float) * nq));
  (k_copy_f32<<<ceil_div(nq, T), T, 0, st>>>(vq, vol, nq), ::ff::note_launch());
  float* qpts = reinterpret_cast<float*>(c->qpts.ensure(sizeof(float) * 3 * nq));
  (k_copy_f32<<<ceil_div(3 * nq, T), T, 0, st>>>(Xq, qpts, 3 * nq), ::ff::note_launch());
  // the transposed lists (centre -> the points it covers) serve the row-owner
  // assembly, which runs when K is too large for the dense tiles of the
  // two-set assembly, and the matrix-free operator (built on demand there)
  c->has_cols = false;
  if (!tset_assembly_fits(K)) twoset_columns(c, qpts);
  int* perm = reinterpret_cast<int*>(c->perm.ensure(sizeof(int) * K));
  int* iperm = reinterpret_cast<int*>(c->iperm.ensure(sizeof(int) * K));
  (k_iota<<<ceil_div(K, T), T, 0, st>>>(perm, iperm, K), ::ff::note_launch());
  FF_LAUNCH_CHECK();

  // ---- 6. shape functions at the quadrature points
  const size_t es = tables_f32(c) ? 4 : 8;
  c->phi.ensure(es * std::max(n1, 1LL));
  c->dphi.ensure(3 * es * std::max(n1, 1LL));
  reset_flags(c);
  {
    ProfScope ps(kProfShape);
    twoset_shape(c, Xq, nq, c->nbr_ptr.as<long long>(), c->nbr_idx.as<int>(), n1, c->phi.p,
                 c->dphi.p, tables_f32(c));
  }
  f = read_flags(c);
  c->hflags->fallback = f.fallback;
  if (f.code == FF_ERR_SINGULAR_MOMENT)
    throw Error(FF_ERR_SINGULAR_MOMENT,
                "moment matrix of quadrature point " + std::to_string(f.index) +
                    " is singular: fewer than four non-coplanar centres cover it");
}

}  // namespace ff
