// Skinning weight fields and linear blend skinning at query points.
//
// The reduced-order basis of the paper is the set of weight fields
// W^j(X) = sum_k phi_k(X) c_k^j (Sec. 3.2): the corrected RKPM shape functions
// of the built cloud (the same kernel, supports and linear basis as the
// cloud's own shape functions, Eqs. 6-11) evaluated at X, times the nodal
// values c (the eigenmodes).  The deformation is linear blend skinning,
// Eq. 1: x = X + sum_j W^j(X) Z_j [X; 1] with Z_j in R^{3x4}.
//
// Pipeline: a gather search (each query point scans the 27 cells around its
// cell -- the cell edge is at least the largest support, so those hold every
// node that covers it; points outside the box are clamped to the boundary
// cells, which still hold every node within one support of them), the moment
// solve and the values (no gradients) of the shape functions (eight lanes a
// point; double-float in FP64 contexts, FP32 with the FP64 redo of
// ill-conditioned points in FP32 ones), and the weights as one warp per point
// over the modes, from a row-major copy of the nodal values.  Clouds of the
// two-set discretisation take its own covering test over the K centres and its
// Gaussian shape functions (twoset.cu).
#include <cstdint>
#include <type_traits>

#include "grid.cuh"
#include "rkpm_eval.cuh"

namespace ff {

template <class T>
void gather_block(ff_ctx* c, const T* X0, int m, T* X, int ld);

namespace {

// A warp takes kQueries points, whose cells it finds at once, a lane a coordinate:
// the FP64 division of a cell coordinate costs a warp the same for one lane as for
// 32.
constexpr int kQueries = 8;

__device__ __forceinline__ int query_coords(const float* __restrict__ Q, long long q0,
                                            long long nq, const GridDev& g, int lane) {
  const int d = lane % 3;
  const long long q = q0 + lane / 3;
  if (lane >= 3 * kQueries || q >= nq) return 0;
  return cell_coord(Q[3 * q + d], d == 0 ? g.o0 : d == 1 ? g.o1 : g.o2, g.h,
                    d == 0 ? g.d0 : d == 1 ? g.d1 : g.d2);
}

// the cell this lane searches for point u of the warp: nodes [i, end)
__device__ __forceinline__ void query_cell(int coords, int u, const GridDev& g,
                                           const int* __restrict__ cstart, int lane, int& i,
                                           int& end) {
  const int x = __shfl_sync(0xffffffffu, coords, 3 * u) + lane % 3 - 1;
  const int y = __shfl_sync(0xffffffffu, coords, 3 * u + 1) + lane / 3 % 3 - 1;
  const int z = __shfl_sync(0xffffffffu, coords, 3 * u + 2) + lane / 9 - 1;
  i = end = 0;
  if (lane < 27 && x >= 0 && x < g.d0 && y >= 0 && y < g.d1 && z >= 0 && z < g.d2) {
    const long long key = cell_key(g, x, y, z);
    i = cstart[key];
    end = cstart[key + 1];
  }
}

// a round's hits to the list, in cell order then node order; base moves on
__device__ __forceinline__ void query_put(unsigned hit, int i, int lane, long long& base,
                                          int* __restrict__ qidx) {
  const int h = __popc(hit);
  int off = h;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, off, o);
    if (lane >= o) off += t;
  }
  long long at = base + off - h;
  base += __shfl_sync(0xffffffffu, off, 31);
  for (unsigned b = hit; b; b &= b - 1) qidx[at++] = i + __ffs(b) - 1;
}

// MODE 0: count the nodes covering each query point, and keep the hits of its
// first kMaskRounds rounds (masks, 32 words a round; the last word of a point's
// first round is the number of rounds); MODE 1: list them, from the masks where they
// hold all the rounds.  A lane a cell tests up to 32 of its nodes a round
// (deterministic: rounds, then cells, then nodes).  A cell's edge is the largest
// support, so 27 cells hold ~250 nodes, ~900 where supports are uneven; bound by a
// load's 27 sectors.  A thread a point took 306 us a pass for 50,000 points of the
// latter kind, this 126 + 36 us; half warps on consecutive nodes, two cells at a
// time, 127 + 70 us.
constexpr int kMaskRounds = 3;

template <int MODE>
__global__ void __launch_bounds__(256)
    k_query_search(const float* __restrict__ Q, long long nq, const float4* __restrict__ pos,
                   GridDev g, const int* __restrict__ cstart, int* __restrict__ cnt,
                   unsigned* __restrict__ masks, const long long* __restrict__ qptr,
                   int* __restrict__ qidx) {
  constexpr unsigned kAll = 0xffffffffu;
  const long long q0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kQueries;
  if (q0 >= nq) return;
  const int lane = threadIdx.x & 31;
  const int coords = query_coords(Q, q0, nq, g, lane);
  for (int v = 0; v < kQueries && q0 + v < nq; ++v) {
    const long long q = q0 + v;
    const float4 X = make_float4(Q[3 * q], Q[3 * q + 1], Q[3 * q + 2], 0.f);
    int i, end;
    query_cell(coords, v, g, cstart, lane, i, end);
    unsigned* mine = masks ? masks + 32LL * kMaskRounds * q : nullptr;
    long long base = MODE ? qptr[q] : 0;
    int c = 0, round = 0;
    if (MODE == 1 && masks) {
      const int rounds = (int)mine[31];
      if (rounds <= kMaskRounds) {
        for (; round < rounds; ++round) {
          const unsigned hit = mine[32 * round + lane];
          query_put(lane < 27 ? hit : 0u, i + 32 * round, lane, base, qidx);
        }
        continue;
      }
    }
    while (__any_sync(kAll, i < end)) {
      const int n = min(end - i, 32);
      unsigned hit = 0, near = 0;
      for (int u0 = 0; u0 < n; u0 += 4) {
        float4 p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) p[u] = pos[min(i + u0 + u, end - 1)];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          // the predicate of covers(): FP32 outside a margin, settled below inside
          const float dx = X.x - p[u].x, dy = X.y - p[u].y, dz = X.z - p[u].z;
          const float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx)), a2 = p[u].w * p[u].w;
          if (u0 + u < n) {
            if (d2 < a2 * 0.99999f) hit |= 1u << (u0 + u);
            if (d2 <= a2 * 1.00001f) near |= 1u << (u0 + u);
          }
        }
      }
      for (unsigned b = near & ~hit; b; b &= b - 1) {
        const int u = __ffs(b) - 1;
        if (covers(X, pos[i + u])) hit |= 1u << u;
      }
      if (MODE) {
        query_put(hit, i, lane, base, qidx);
      } else {
        c += __popc(hit);
        if (mine && round < kMaskRounds) mine[32 * round + lane] = hit;
      }
      ++round;
      i += max(n, 0);
    }
    if (!MODE) {
      if (mine && lane == 31) mine[31] = (unsigned)round;  // lane 31 has no cell
      c = __reduce_add_sync(kAll, c);
      if (lane == 0) cnt[q] = c;
    }
  }
}

// values of the shape functions at the query points, eight lanes each: FP64
// contexts in double-float, FP32 ones in FP32 (ill-conditioned points listed
// for the FP64 redo).  scale normalises the linear basis (any positive value
// gives the same functions; the support size keeps M well scaled).  The
// weights need no gradients: 30 of the 40 moment sums fall away.
constexpr int kQueryLanes = 8;

template <class S>
__global__ void __launch_bounds__(256)
    k_query_shape(const float4* __restrict__ pos, const float* __restrict__ Q,
                  const long long* __restrict__ qptr, const int* __restrict__ qidx, long long nq,
                  float scale, S* __restrict__ phi, double cond_limit, int* __restrict__ redo,
                  DevFlags* __restrict__ flags) {
  const long long q = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kQueryLanes;
  const bool live = q < nq, first = threadIdx.x % kQueryLanes == 0;
  const long long s = live ? qptr[q] : 0, e = live ? qptr[q + 1] : 0;
  const float4 Xq = live ? make_float4(Q[3 * q], Q[3 * q + 1], Q[3 * q + 2], scale)
                         : make_float4(0.f, 0.f, 0.f, 1.f);
  S* const none = nullptr;
  if constexpr (sizeof(S) == 4) {
    const int st = rkpm::shape_rows<float, S, kQueryLanes, false>(pos, s, e, qidx, Xq, phi, none,
                                                                  0, cond_limit, true);
    if (live && st != 0 && first) rkpm::redo_later(redo, q);
  } else {
    const int st = rkpm::shape_rows<dfloat, S, kQueryLanes, false>(pos, s, e, qidx, Xq, phi, none,
                                                                   0, 0.0, false);
    if (live && st != 0 && first &&
        atomicCAS(&flags->code, 0, (int)FF_ERR_SINGULAR_MOMENT) == 0)
      flags->index = (int)q;
  }
}

// W[q][j] = sum over the nodes k covering q of phi_k(X_q) C[k][j], C row-major
// with ldc (a multiple of 16 bytes) columns.  One warp a point: W lanes of 16
// bytes span a row of C, 32 / W rows at a time; the point's pairs are loaded 32
// at a time, one a lane, and handed round by shuffles.  Bound by the L1 reads of
// C's rows.  Read column by column from the caller's block (a sector a lane) it
// took 11.6 ms for 1M points x 98 pairs x 64 FP32 modes, 1.42 ms so.  Nothing is
// written when the shape functions failed.
template <class T, class S, int W>
__global__ void __launch_bounds__(256)
    k_query_weights(const long long* __restrict__ qptr, const int* __restrict__ qidx,
                    const S* __restrict__ phi, long long nq, const T* __restrict__ C, int ldc,
                    int m, T* __restrict__ out, const DevFlags* __restrict__ flags) {
  constexpr int VEC = 16 / (int)sizeof(T), SUB = 32 / W;
  using V = std::conditional_t<sizeof(T) == 4, float4, double2>;
  const long long q = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (q >= nq || flags->code != 0) return;
  const int lane = threadIdx.x & 31, sub = lane / W;
  const long long s = qptr[q], e = qptr[q + 1];
  for (int c0 = 0; c0 < m; c0 += W * VEC) {
    const int col = c0 + lane % W * VEC;
    const bool in = col < m;
    T acc[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = T(0);
    for (long long t = s; t < e; t += 32) {
      const int cnt = (int)min(32LL, e - t);
      int k = 0;
      T ph = T(0);
      if (lane < cnt) {
        k = qidx[t + lane];
        ph = (T)phi[t + lane];
      }
#pragma unroll 4
      for (int u = 0; u < cnt; u += SUB) {
        const int ku = __shfl_sync(0xffffffffu, k, u + sub);
        const T pu = __shfl_sync(0xffffffffu, ph, u + sub);
        if (in && u + sub < cnt) {
          const V x = *reinterpret_cast<const V*>(C + (long long)ku * ldc + col);
          const T* xv = reinterpret_cast<const T*>(&x);
#pragma unroll
          for (int v = 0; v < VEC; ++v) mac(acc[v], pu, xv[v]);
        }
      }
    }
#pragma unroll
    for (int o = 16; o >= W; o >>= 1)
#pragma unroll
      for (int v = 0; v < VEC; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], o);
    if (sub == 0)
#pragma unroll
      for (int v = 0; v < VEC; ++v)
        if (col + v < m) out[q * m + col + v] = acc[v];
  }
}

// x_q = X_q + sum_j W[q][j] Z_j [X_q; 1]  (Z row-major m x 3 x 4).  A block
// stages its rows of W and the transforms, kCols modes at a time, in shared
// memory: by 16-byte asynchronous copies (kCopy; W 16-byte aligned and its rows
// whole 16 bytes), else by plain loads, a warp 128 consecutive bytes (kLoad).
// The staged rows are 16 bytes longer than their columns, so that a thread a
// point reads its own row 16 bytes at a time without bank conflicts; with kCopy
// a thread takes PTS points, which share its reads of the transforms.  FP32 rows
// of up to 64 modes that are not whole 16 bytes come as one flat copy of the
// block's span of W (kFlat), which starts on a 16-byte boundary where W does;
// read at a stride of m words, m % 4 != 0, that is two lanes a bank at most.  Rows
// of at most 32 bytes are read where they lie (kDirect): a sector or two a thread
// either way.
// Bound by reading W: every thread walking its row in global memory (a sector a
// lane a load) took 326 us for 1M points x 64 FP32 modes, 58 us so; in FP64 by
// its arithmetic (1.64 ms so, 1.27 ms with the 12 multiply-adds a mode of the form
// below).
enum LbsRead { kDirect, kLoad, kCopy, kFlat };

constexpr int kLbsFlat = 64;

template <class T, int TB, int PTS, LbsRead READ>
__global__ void __launch_bounds__(TB, 1024 / (TB * PTS))
    k_lbs(const float* __restrict__ Q, long long nq, const T* __restrict__ W, int m,
          const T* __restrict__ Z, T* __restrict__ x) {
  constexpr int E = 16 / (int)sizeof(T);  // elements of 16 bytes
  constexpr int kCols = READ == kFlat ? kLbsFlat : 32;
  constexpr int kRows = READ == kDirect ? 1 : TB * PTS;
  __shared__ __align__(16) T sw[kRows][READ == kFlat ? kCols : kCols + E];
  T* const flat = &sw[0][0];
  __shared__ __align__(16) T sz[kCols][12];
  const long long q0 = (long long)blockIdx.x * TB * PTS;
  const int rows = (int)min((long long)TB * PTS, nq - q0);
  const int tid = threadIdx.x;
  T X[PTS][3], o[PTS][3];
  int row[PTS];
#pragma unroll
  for (int p = 0; p < PTS; ++p) {
    row[p] = min(tid + p * TB, rows - 1);
#pragma unroll
    for (int d = 0; d < 3; ++d) o[p][d] = X[p][d] = (T)Q[3 * (q0 + row[p]) + d];
  }
  for (int j0 = 0; j0 < m; j0 += kCols) {
    const int jn = min(kCols, m - j0);
    const T* w0 = W + q0 * m + j0;
    if (j0) __syncthreads();
    if constexpr (READ == kCopy) {
      constexpr int kVecs = kCols / E;
#pragma unroll 4
      for (int t = tid; t < TB * PTS * kVecs; t += TB) {
        const int r = t / kVecs, c = t % kVecs * E;
        if (r < rows && c < jn) {
          const unsigned dst = (unsigned)__cvta_generic_to_shared(&sw[r][c]);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst),
                       "l"(w0 + (long long)r * m + c)
                       : "memory");
        }
      }
    } else if constexpr (READ == kFlat) {  // m <= kCols: the one chunk
      const int total = rows * m;
#pragma unroll 4
      for (int t = tid * E; t < total; t += TB * E) {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(flat + t);
        if (t + E <= total)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(w0 + t)
                       : "memory");
        else
          for (int u = t; u < total; ++u) flat[u] = w0[u];
      }
    } else if constexpr (READ == kLoad) {
      const int lane = tid & 31;
      if (lane < jn)
#pragma unroll 4
        for (int r = tid >> 5; r < rows; r += TB / 32) sw[r][lane] = w0[(long long)r * m + lane];
    }
    for (int t = tid; t < 12 * jn; t += TB) (&sz[0][0])[t] = Z[12LL * j0 + t];
    if constexpr (READ == kCopy || READ == kFlat)
      asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    auto add = [&](int p, T wj, const T* z) {
#pragma unroll
      for (int d = 0; d < 3; ++d)
        mac(o[p][d], wj,
            fma(z[4 * d + 2], X[p][2],
                fma(z[4 * d + 1], X[p][1], fma(z[4 * d], X[p][0], z[4 * d + 3]))));
    };
    int j = 0;
    if constexpr (READ == kCopy || READ == kLoad) {
      for (; j + E <= jn; j += E) {
        T wv[PTS][E];
#pragma unroll
        for (int p = 0; p < PTS; ++p)
          *reinterpret_cast<uint4*>(wv[p]) = *reinterpret_cast<const uint4*>(&sw[row[p]][j]);
#pragma unroll
        for (int u = 0; u < E; ++u)
#pragma unroll
          for (int p = 0; p < PTS; ++p) add(p, wv[p][u], sz[j + u]);
      }
    }
    // (unrolled, the few modes of kDirect all run in the remainder: two modes in FP64 took
    // 95 us for 1M points, 71 so)
    constexpr int kModes = READ == kDirect ? 1 : 4;
#pragma unroll kModes
    for (; j < jn; ++j)
#pragma unroll
      for (int p = 0; p < PTS; ++p) {
        if constexpr (READ == kDirect)
          add(p, w0[(long long)row[p] * m + j], sz[j]);
        else if constexpr (READ == kFlat)
          add(p, flat[row[p] * m + j], sz[j]);
        else
          add(p, sw[row[p]][j], sz[j]);
      }
  }
#pragma unroll
  for (int p = 0; p < PTS; ++p)
    if (tid + p * TB < rows)
#pragma unroll
      for (int d = 0; d < 3; ++d) x[3 * (q0 + row[p]) + d] = o[p][d];
}

template <class T>
void lbs_t(ff_ctx* c, const float* Q, long long nq, const T* W, int m, const T* Z, T* x) {
  auto go = [&](auto tb, auto pts, auto read) {
    constexpr int TB = decltype(tb)::value, PTS = decltype(pts)::value;
    (k_lbs<T, TB, PTS, decltype(read)::value>
     <<<ceil_div(nq, TB * PTS), TB, 0, c->stream>>>(Q, nq, W, m, Z, x),
     ::ff::note_launch());
  };
  // blocks of 128 threads where those fill the chip twice over, two points a
  // thread for FP32 copies; fewer points are spread thinner, 32 a block (1,000
  // points in 8 blocks of 128 would leave 144 SMs idle)
  auto pick = [&](auto read) {
    using One = std::integral_constant<int, 1>;
    using Pts = std::integral_constant<int, sizeof(T) == 4 && decltype(read)::value == kCopy ? 2 : 1>;
    if (nq >= 2LL * 128 * Pts::value * sm_count())
      go(std::integral_constant<int, 128>{}, Pts{}, read);
    else
      go(std::integral_constant<int, 32>{}, One{}, read);
  };
  const bool aligned = reinterpret_cast<uintptr_t>(W) % 16 == 0;
  if (m * sizeof(T) <= 32)
    pick(std::integral_constant<LbsRead, kDirect>{});
  else if (aligned && m * sizeof(T) % 16 == 0)
    pick(std::integral_constant<LbsRead, kCopy>{});
  else if (aligned && m <= kLbsFlat && sizeof(T) == 4)
    pick(std::integral_constant<LbsRead, sizeof(T) == 4 ? kFlat : kLoad>{});
  else
    pick(std::integral_constant<LbsRead, kLoad>{});
  FF_LAUNCH_CHECK();
  FF_CUDA(cudaStreamSynchronize(c->stream));
}

template <class T, class S>
void launch_weights(ff_ctx* c, const long long* qptr, const int* qidx, const S* phi, long long nq,
                    const T* C, int ldc, int m, T* W) {
  const unsigned grid = ceil_div(nq * 32, 256);
  const DevFlags* flags = c->flags.as<DevFlags>();
  auto go = [&](auto lanes) {
    (k_query_weights<T, S, decltype(lanes)::value><<<grid, 256, 0, c->stream>>>(
         qptr, qidx, phi, nq, C, ldc, m, W, flags),
     ::ff::note_launch());
  };
  const int need = (m * (int)sizeof(T) + 15) / 16;  // lanes of 16 bytes a row of C
  if (need <= 4)
    go(std::integral_constant<int, 4>{});
  else if (need <= 8)
    go(std::integral_constant<int, 8>{});
  else if (need <= 16)
    go(std::integral_constant<int, 16>{});
  else
    go(std::integral_constant<int, 32>{});
  FF_LAUNCH_CHECK();
}

template <class T>
void weights_t(ff_ctx* c, const float* Q, long long nq, const T* C, int m, T* W) {
  using S = std::conditional_t<sizeof(T) == 4, float, dfloat>;  // the shape values
  constexpr bool f32 = sizeof(T) == 4;
  cudaStream_t st = c->stream;
  const int TB = 256;
  long long nq1 = 0;
  const long long* qptr = nullptr;
  const int* qidx = nullptr;
  S* phi = nullptr;
  const char* what = "nodes";
  // the nodal values row-major in the internal order, rows of whole 16 bytes
  const int ldc = (m * (int)sizeof(T) + 15) / 16 * 16 / (int)sizeof(T);
  T* Ct = reinterpret_cast<T*>(c->sk_c.ensure(sizeof(T) * (size_t)c->n * ldc));
  gather_block<T>(c, C, m, Ct, ldc);
  if (c->twoset) {
    nq1 = twoset_cover(c, Q, nq, c->sk_ptr, c->sk_idx, c->sk_cnt);
    qptr = c->sk_ptr.as<long long>();
    qidx = c->sk_idx.as<int>();
    phi = reinterpret_cast<S*>(c->sk_phi.ensure(sizeof(S) * std::max(nq1, 1LL)));
    reset_flags(c);
    twoset_shape(c, Q, nq, qptr, qidx, nq1, phi, nullptr, f32);
    what = "centres";
  } else {
    const Grid& g = c->grid;
    const GridDev gd{g.origin[0], g.origin[1], g.origin[2], g.h, g.dims[0], g.dims[1], g.dims[2],
                     g.bdims[0], g.bdims[1], g.bdims[2]};
    int* cnt = reinterpret_cast<int*>(c->sk_cnt.ensure(sizeof(int) * (nq + 1)));
    long long* ptr = reinterpret_cast<long long*>(c->sk_ptr.ensure(sizeof(long long) * (nq + 1)));
    // the hits kept between the passes while they are small (2.8 million points; more
    // than kKeptScratch is given back); without them the second pass searches again
    unsigned* masks = nullptr;
    const size_t room = sizeof(unsigned) * 32 * kMaskRounds * (size_t)nq;
    if (room <= (1ull << 30)) {
      try {
        masks = reinterpret_cast<unsigned*>(c->scratch[6].ensure(room));
      } catch (const Error&) {
      }
    }
    (k_query_search<0><<<ceil_div(nq * 32, TB * kQueries), TB, 0, st>>>(
         Q, nq, c->pos.as<float4>(), gd, c->cell_start.as<int>(), cnt, masks, nullptr, nullptr),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    scan_counts(cnt, ptr, nq, c, c->scratch[3]);
    FF_CUDA(cudaMemcpyAsync(&nq1, ptr + nq, sizeof(long long), cudaMemcpyDeviceToHost, st));
    FF_CUDA(cudaStreamSynchronize(st));
    int* idx = reinterpret_cast<int*>(c->sk_idx.ensure(sizeof(int) * std::max(nq1, 1LL)));
    (k_query_search<1><<<ceil_div(nq * 32, TB * kQueries), TB, 0, st>>>(
         Q, nq, c->pos.as<float4>(), gd, c->cell_start.as<int>(), nullptr, masks, ptr, idx),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    if (masks) give_back(c, c->scratch[6], room);
    qptr = ptr;
    qidx = idx;
    phi = reinterpret_cast<S*>(c->sk_phi.ensure(sizeof(S) * std::max(nq1, 1LL)));
    reset_flags(c);
    const float scale = (float)(g.h / 1.001);
    int* redo = f32 ? rkpm::redo_list(c, nq) : nullptr;
    (k_query_shape<S><<<ceil_div(nq * kQueryLanes, TB), TB, 0, st>>>(
         c->pos.as<float4>(), Q, qptr, qidx, nq, scale, phi, 1e2, redo, c->flags.as<DevFlags>()),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    if constexpr (f32) {
      (rkpm::k_shape_redo<S, false, rkpm::BSpline><<<rkpm::redo_grid(nq), 256, 0, st>>>(
           c->pos.as<float4>(), nullptr, Q, scale, qptr, qidx, 0, phi, nullptr, redo,
           c->flags.as<DevFlags>(), rkpm::BSpline()),
       ::ff::note_launch());
      FF_LAUNCH_CHECK();
    }
  }
  launch_weights<T, S>(c, qptr, qidx, phi, nq, Ct, ldc, m, W);
  const DevFlags f = read_flags(c);
  if (f.code == FF_ERR_SINGULAR_MOMENT)
    throw Error(FF_ERR_SINGULAR_MOMENT,
                "query point " + std::to_string(f.index) +
                    " is covered by fewer than four non-coplanar " + what);
}

}  // namespace

void skinning_weights(ff_ctx* c, const float* Q, long long nq, const void* C, int m, void* W) {
  if (nq == 0) return;
  if (c->prec == FF_PREC_FP64)
    weights_t<double>(c, Q, nq, static_cast<const double*>(C), m, static_cast<double*>(W));
  else
    weights_t<float>(c, Q, nq, static_cast<const float*>(C), m, static_cast<float*>(W));
}

void lbs_deform(ff_ctx* c, const float* Q, long long nq, const void* W, int m, const void* Z,
                void* x) {
  if (nq == 0) return;
  if (c->prec == FF_PREC_FP64)
    lbs_t<double>(c, Q, nq, static_cast<const double*>(W), m, static_cast<const double*>(Z),
                  static_cast<double*>(x));
  else
    lbs_t<float>(c, Q, nq, static_cast<const float*>(W), m, static_cast<const float*>(Z),
                 static_cast<float*>(x));
}

}  // namespace ff
