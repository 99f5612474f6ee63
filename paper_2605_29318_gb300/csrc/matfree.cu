// Matrix-free application of H_w and M (Prop. 1 and Eq. 14 without
// assembling either matrix).
//
// Prop. 1 writes H_w as a sum over the quadrature points of rank-3 terms:
//   H_w X = sum_s G_s^T D G_s X,   M X = Phi^T V Phi X,
// with (G_s)_ik = d_s phi_k(X_i), Phi_ik = phi_k(X_i), D = diag(v_i (lambda_i +
// 4 mu_i)) and V = diag(v_i).  Two passes over the shape-function tables:
//   k_mf_gather   one warp per quadrature point i: Y_i = [G_0 X, G_1 X, G_2 X,
//                 Phi X]_i (4 m values), scaled by the point's weights;
//   k_mf_scatter  one warp per node k, over the points that node covers (the
//                 transposed lists, ascending): (H X)_k = sum_i sum_s
//                 d_s phi_k(X_i) Y_i,s and (M X)_k = sum_i phi_k(X_i) Y_i,3 --
//                 fixed order, no atomics.
// It reads the tables (n1 pairs x 4 values) twice and the block once per pair,
// where an assembled product reads n2 matrix entries: the smaller of the two
// wherever n2 / n1 is large.  The sums are FP64 in FP64 contexts (the tables'
// double-float pairs rounded to FP64) and FP32 otherwise.
#include <type_traits>

#include "dfloat.cuh"
#include "ff_internal.cuh"

namespace ff {

template <class T>
void gather_block(ff_ctx* c, const T* X0, int m, T* X, int ld);
template <class T>
void scatter_blocks(ff_ctx* c, const T* A, const T* B, int ld, int m, T* outA, T* outB,
                    const DevFlags* flags = nullptr);

namespace {

// Rows of 16-byte lanes: W lanes span a row of the block (ld columns, whole 16
// bytes), so a warp takes 32 / W pairs of a list at once; wider rows in several
// passes.  Places and table values of 32 pairs are loaded (and in FP64 contexts
// converted) one pair a lane and handed round by shuffles, so that the block's rows
// can be fetched several at a time: what bounds both passes is the latency of L2.
// Small blocks and two fetches a lane measured best (blocks of 512 threads and
// four: 41 + 72 us at 30,011 points x 32 FP32 columns against 31 + 49).
constexpr int kMfT = 128;
constexpr int kFly = 2;  // 16-byte loads a lane keeps in flight (the scatter: twice that)

// table value (pair, comp) of this lane: comp 0..2 the gradient, 3 the value
template <class C, class S>
__device__ __forceinline__ C mf_table(const S* __restrict__ phi, const S* __restrict__ dphi,
                                      long long n1, long long e, int comp) {
  return (C)(double)(comp < 3 ? dphi[comp * n1 + e] : phi[e]);
}
template <>
__device__ __forceinline__ float mf_table<float, float>(const float* __restrict__ phi,
                                                        const float* __restrict__ dphi,
                                                        long long n1, long long e, int comp) {
  return comp < 3 ? dphi[comp * n1 + e] : phi[e];
}

template <class C>
struct MfVec {
  static constexpr int n = 16 / (int)sizeof(C);
  using type = std::conditional_t<sizeof(C) == 4, float4, double2>;
};

// Y_i = the point's weighted G_0 X, G_1 X, G_2 X and Phi X (4 ld values).  One
// warp a point: 40 us with a lane a column for 30,011 points x 32 FP32 columns,
// 31 so.
template <class C, class S, int W>
__global__ void __launch_bounds__(kMfT)
    k_mf_gather(const long long* __restrict__ ptr, const int* __restrict__ idx,
                const S* __restrict__ phi, const S* __restrict__ dphi, long long n1,
                const S* __restrict__ wh, const float* __restrict__ vol, long long nq,
                const C* __restrict__ X, int ld, C* __restrict__ Y) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int VEC = MfVec<C>::n, SUB = 32 / W;
  using V = typename MfVec<C>::type;
  const long long i = ((long long)blockIdx.x * kMfT + threadIdx.x) >> 5;
  if (i >= nq) return;
  const int lane = threadIdx.x & 31, sub = lane / W;
  const long long s = ptr[i], end = ptr[i + 1];
  for (int c0 = 0; c0 < ld; c0 += W * VEC) {
    const int col = c0 + lane % W * VEC;
    const bool in = col < ld;
    C acc[4][VEC];
#pragma unroll
    for (int d = 0; d < 4; ++d)
#pragma unroll
      for (int v = 0; v < VEC; ++v) acc[d][v] = C(0);
    for (long long e0 = s; e0 < end; e0 += 32) {
      const int cnt = (int)min(32LL, end - e0);
      int k = 0;
      C t[4] = {C(0), C(0), C(0), C(0)};
      if (lane < cnt) {
        k = idx[e0 + lane];
#pragma unroll
        for (int d = 0; d < 4; ++d) t[d] = mf_table<C, S>(phi, dphi, n1, e0 + lane, d);
      }
      // kFly rows of the block in flight
      for (int u0 = 0; u0 < cnt; u0 += kFly * SUB) {
        V x[kFly];
#pragma unroll
        for (int f = 0; f < kFly; ++f) {
          const int p = u0 + f * SUB + sub;
          const int kp = __shfl_sync(kAll, k, p % 32);
          if (in && p < cnt) x[f] = *reinterpret_cast<const V*>(X + (long long)kp * ld + col);
        }
#pragma unroll
        for (int f = 0; f < kFly; ++f) {
          const int p = u0 + f * SUB + sub;
          C tp[4];
#pragma unroll
          for (int d = 0; d < 4; ++d) tp[d] = __shfl_sync(kAll, t[d], p % 32);
          if (in && p < cnt) {
            const C* xv = reinterpret_cast<const C*>(&x[f]);
#pragma unroll
            for (int d = 0; d < 4; ++d)
#pragma unroll
              for (int v = 0; v < VEC; ++v) mac(acc[d][v], tp[d], xv[v]);
          }
        }
      }
    }
#pragma unroll
    for (int o = 16; o >= W; o >>= 1)
#pragma unroll
      for (int d = 0; d < 4; ++d)
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[d][v] += __shfl_xor_sync(kAll, acc[d][v], o);
    if (sub == 0 && in) {
      const C w = (C)(double)wh[i], vq = (C)vol[i];
      C* y = Y + i * 4LL * ld + col;
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        V o;
        C* ov = reinterpret_cast<C*>(&o);
#pragma unroll
        for (int v = 0; v < VEC; ++v) ov[v] = (d < 3 ? w : vq) * acc[d][v];
        *reinterpret_cast<V*>(y + (long long)d * ld) = o;
      }
    }
  }
}

// (H X)_k and (M X)_k over the points node k covers.  Bound by the reads of Y (4
// ld values a pair): 83 us for 30,011 nodes x 32 FP32 columns with a lane a
// column in blocks of 8 nodes, 49 so.
template <class C, class S, int W>
__global__ void __launch_bounds__(kMfT)
    k_mf_scatter(const long long* __restrict__ tptr, const int* __restrict__ tidx,
                 const long long* __restrict__ tpos, const S* __restrict__ phi,
                 const S* __restrict__ dphi, long long n1, long long n, const C* __restrict__ Y,
                 int ld, C* __restrict__ YH, C* __restrict__ YM) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int VEC = MfVec<C>::n, SUB = 32 / W;
  using V = typename MfVec<C>::type;
  const long long k = ((long long)blockIdx.x * kMfT + threadIdx.x) >> 5;
  if (k >= n) return;
  const int lane = threadIdx.x & 31, sub = lane / W;
  const long long s = tptr[k], end = tptr[k + 1];
  for (int c0 = 0; c0 < ld; c0 += W * VEC) {
    const int col = c0 + lane % W * VEC;
    const bool in = col < ld;
    C h[VEC], mm[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) h[v] = mm[v] = C(0);
    for (long long a0 = s; a0 < end; a0 += 32) {
      const int cnt = (int)min(32LL, end - a0);
      int i = 0;
      C t[4] = {C(0), C(0), C(0), C(0)};
      if (lane < cnt) {
        i = tidx[a0 + lane];
        const long long e = tpos[a0 + lane];
#pragma unroll
        for (int d = 0; d < 4; ++d) t[d] = mf_table<C, S>(phi, dphi, n1, e, d);
      }
      constexpr int kF = kFly / 2;  // points in flight, four rows each
      for (int u0 = 0; u0 < cnt; u0 += kF * SUB) {
        V q[kF][4];
#pragma unroll
        for (int f = 0; f < kF; ++f) {
          const int p = u0 + f * SUB + sub;
          const int ip = __shfl_sync(kAll, i, p % 32);
          if (in && p < cnt) {
            const C* y = Y + (long long)ip * 4 * ld + col;
#pragma unroll
            for (int d = 0; d < 4; ++d) q[f][d] = *reinterpret_cast<const V*>(y + (long long)d * ld);
          }
        }
#pragma unroll
        for (int f = 0; f < kF; ++f) {
          const int p = u0 + f * SUB + sub;
          C tp[4];
#pragma unroll
          for (int d = 0; d < 4; ++d) tp[d] = __shfl_sync(kAll, t[d], p % 32);
          if (in && p < cnt)
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
#pragma unroll
              for (int d = 0; d < 3; ++d) mac(h[v], tp[d], reinterpret_cast<const C*>(&q[f][d])[v]);
              mac(mm[v], tp[3], reinterpret_cast<const C*>(&q[f][3])[v]);
            }
        }
      }
    }
#pragma unroll
    for (int o = 16; o >= W; o >>= 1)
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        h[v] += __shfl_xor_sync(kAll, h[v], o);
        mm[v] += __shfl_xor_sync(kAll, mm[v], o);
      }
    if (sub == 0 && in) {
      *reinterpret_cast<V*>(YH + k * ld + col) = *reinterpret_cast<const V*>(h);
      *reinterpret_cast<V*>(YM + k * ld + col) = *reinterpret_cast<const V*>(mm);
    }
  }
}

template <class C, class S>
void run(ff_ctx* c, const C* Xp, int ld, C* YHp, C* YMp, const S* wh) {
  cudaStream_t st = c->stream;
  const long long n = c->n, nq = c->nq, n1 = c->n1;
  C* Y = reinterpret_cast<C*>(c->scratch[1].ensure(sizeof(C) * 4 * (size_t)nq * ld));
  auto go = [&](auto lanes) {
    constexpr int W = decltype(lanes)::value;
    (k_mf_gather<C, S, W><<<ceil_div(nq * 32, kMfT), kMfT, 0, st>>>(
         c->nbr_ptr.as<long long>(), c->nbr_idx.as<int>(), c->phi.as<S>(), c->dphi.as<S>(), n1, wh,
         c->vol.as<float>(), nq, Xp, ld, Y),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    (k_mf_scatter<C, S, W><<<ceil_div(n * 32, kMfT), kMfT, 0, st>>>(
         c->nbrT_ptr.as<long long>(), c->nbrT_idx.as<int>(), c->nbrT_pos.as<long long>(),
         c->phi.as<S>(), c->dphi.as<S>(), n1, n, Y, ld, YHp, YMp),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
  };
  const int need = ld / MfVec<C>::n;  // 16-byte lanes a row
  if (need <= 4)
    go(std::integral_constant<int, 4>{});
  else if (need <= 8)
    go(std::integral_constant<int, 8>{});
  else if (need <= 16)
    go(std::integral_constant<int, 16>{});
  else
    go(std::integral_constant<int, 32>{});
}

}  // namespace

void apply_matfree(ff_ctx* c, const float* E, const float* nu, double E0, double nu0,
                   const void* X, int m, void* YH, void* YM) {
  if (!c->has_cols) twoset_columns(c, c->qpts.as<float>());
  const long long n = c->n, nq = c->nq;
  const bool f64 = c->prec == FF_PREC_FP64;
  void* wh = c->scratch[0].ensure((tables_f32(c) ? 4 : 8) * (size_t)nq + 64);
  material_weights(c, E, nu, E0, nu0, wh);
  auto go = [&](auto tag) {
    using C = decltype(tag);
    constexpr int VEC = MfVec<C>::n;
    const int ld = (m + VEC - 1) / VEC * VEC;  // rows of whole 16 bytes
    C* in = reinterpret_cast<C*>(c->scratch[4].ensure(sizeof(C) * n * ld));
    C* oh = reinterpret_cast<C*>(c->scratch[6].ensure(sizeof(C) * n * ld));
    C* om = reinterpret_cast<C*>(c->scratch[7].ensure(sizeof(C) * n * ld));
    gather_block<C>(c, static_cast<const C*>(X), m, in, ld);
    if constexpr (std::is_same_v<C, double>) {
      if (tables_f32(c))
        run<double, float>(c, in, ld, oh, om, static_cast<const float*>(wh));
      else
        run<double, dfloat>(c, in, ld, oh, om, static_cast<const dfloat*>(wh));
    } else
      run<float, float>(c, in, ld, oh, om, static_cast<const float*>(wh));
    // a bad material is read back once, with everything launched
    scatter_blocks<C>(c, oh, om, ld, m, static_cast<C*>(YH), static_cast<C*>(YM),
                      c->flags.as<DevFlags>());
    check_material(read_flags(c));
  };
  if (f64)
    go(double{});
  else
    go(float{});
}

}  // namespace ff
