// Corrected RKPM shape functions and gradients, a group of lanes per evaluation point.
//
// Sec. 3.2, Eqs. 7, 9-10: phi_k(X) = varphi_k(X) P(p_k)^T C(X), M(X) C(X) = P(X),
// M(X) = sum_k varphi_k(X) P(p_k) P(p_k)^T with the linear basis.  The basis is
// written about the evaluation point, P_o(p) = [1, (p - X_i)/a_i] (an invertible
// affine change of [1, x, y, z], so phi is unchanged and M is well scaled).  The
// gradient follows from differentiating M C = P_o:
//   d_s C = M^{-1} (e_{1+s}/a_i - (d_s M) C),
//   d_s phi_k = d_s varphi_k P_k^T C + varphi_k P_k^T d_s C.
// Raw kernel: cubic B-spline w(q), q = |X - p_k| / a_k, grad = (w'(q)/q)(X - p_k)/a_k^2.
//
// A group of lanes strides over the row's neighbours and accumulates the 10
// distinct entries of M and the 30 of d M; a butterfly reduction gives every
// lane of the group the sums; each then solves the 4x4 system (Cholesky) and
// writes phi / grad phi for its own neighbours.  In FP32 mode a row whose moment
// matrix has a 1-norm condition number above `cond_limit` is recomputed entirely
// in FP64 (by a second kernel, or in place where rows are few).  FP64 mode computes
// and stores double-float pairs (FP32 head and tail, ~2^-47 relative).
#include <type_traits>

#include "dfloat.cuh"
#include "ff_internal.cuh"
#include "rkpm_eval.cuh"

namespace ff {
namespace {

using rkpm::shape_rows;

// lanes a row: a nodal row has ~30-45 nodes, so eight lanes take four to six
// of them each and a warp's moment solve serves four rows (FP32, 200k
// particles: 1.41 ms with a warp a row, 0.37 ms now with the FP64 redo; double-float,
// 50k particles: 1.33 ms, 0.51 ms now, of which 0.15 for sums and quotients as exact
// as a warp a row has them).  Few rows take a warp each, and an ill-conditioned FP32 row
// its FP64 redo at once: their time is one row's chain of operations, which is shorter so.
// With eight lanes and with a warp: FP32 300 particles 75 and 41 us, 8,000 75 and 58, 12,000
// 83 and 76 (no second launch); double-float 1,000 44 and 32 us, 2,432 (the warps that are
// resident) 48 both, 2,600 47 and 65.
constexpr int kLanes = 8;

template <class T, int L>
__global__ void __launch_bounds__(256, 2)
    k_shape(const float4* __restrict__ pos, const long long* __restrict__ ptr,
            const int* __restrict__ idx, long long n, long long n1, T* __restrict__ phi,
            T* __restrict__ dphi, double cond_limit, int* __restrict__ redo,
            DevFlags* __restrict__ flags) {
  const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / L;
  const bool live = i < n, first = threadIdx.x % L == 0;
  const long long s = live ? ptr[i] : 0, e = live ? ptr[i + 1] : 0;
  const float4 Xi = live ? pos[i] : make_float4(0.f, 0.f, 0.f, 1.f);
  int st;
  if constexpr (sizeof(T) == 4) {
    st = shape_rows<float, T, L, true>(pos, s, e, idx, Xi, phi, dphi, n1, cond_limit, true);
    if constexpr (L == 32) {
      if (live && st != 0) {
        st = shape_rows<double, T, L, true>(pos, s, e, idx, Xi, phi, dphi, n1, 0.0, false);
        if (st == 0 && first) atomicAdd(&flags->fallback, 1);
      }
    } else {
      if (live && st != 0 && first) rkpm::redo_later(redo, i);
      return;
    }
  } else {
    // FP64 outputs computed in double-float (~2^-47 relative; GB300's FP64
    // rate made this kernel FP64-bound)
    st = shape_rows<dfloat, T, L, true>(pos, s, e, idx, Xi, phi, dphi, n1, 0.0, false);
  }
  if (live && st != 0 && first && atomicCAS(&flags->code, 0, (int)FF_ERR_SINGULAR_MOMENT) == 0)
    flags->index = (int)i;
}

}  // namespace

void build_shape(ff_ctx* c) {
  const long long n = c->n, n1 = c->n1;
  const int T = 256;
  reset_flags(c);
  size_t es = c->prec == FF_PREC_FP64 ? 8 : 4;
  c->phi.ensure(es * n1);
  c->dphi.ensure(3 * es * n1);
  const double cond_limit = 1e2;
  ProfScope ps(kProfShape);
  const float4* pos = c->pos.as<float4>();
  const long long* ptr = c->nbr_ptr.as<long long>();
  const int* idx = c->nbr_idx.as<int>();
  DevFlags* flags = c->flags.as<DevFlags>();
  const bool few = n <= (c->prec == FF_PREC_FP64 ? 16 : 64) * (long long)sm_count();
  const unsigned grid = ceil_div(n * (few ? 32 : kLanes), T);
  auto run = [&](auto tag, auto lanes, int* redo) {
    using S = decltype(tag);
    (k_shape<S, decltype(lanes)::value><<<grid, T, 0, c->stream>>>(
         pos, ptr, idx, n, n1, c->phi.as<S>(), c->dphi.as<S>(), cond_limit, redo, flags),
     ::ff::note_launch());
  };
  using Warp = std::integral_constant<int, 32>;
  using Part = std::integral_constant<int, kLanes>;
  if (c->prec == FF_PREC_FP64) {  // stored as double-float pairs for the assembly
    if (few)
      run(dfloat{}, Warp{}, nullptr);
    else
      run(dfloat{}, Part{}, nullptr);
  } else if (few) {
    run(float{}, Warp{}, nullptr);
  } else {
    int* redo = rkpm::redo_list(c, n);
    run(float{}, Part{}, redo);
    FF_LAUNCH_CHECK();
    (rkpm::k_shape_redo<float, true, rkpm::BSpline><<<rkpm::redo_grid(n), 256, 0, c->stream>>>(
         pos, pos, nullptr, 0.f, ptr, idx, n1, c->phi.as<float>(), c->dphi.as<float>(), redo,
         flags, rkpm::BSpline()),
     ::ff::note_launch());
  }
  FF_LAUNCH_CHECK();
  ps.close();
  DevFlags f = read_flags(c);
  c->hflags->fallback = f.fallback;
  if (f.code == FF_ERR_SINGULAR_MOMENT) {
    int orig = -1;
    FF_CUDA(cudaMemcpy(&orig, c->perm.as<int>() + f.index, sizeof(int), cudaMemcpyDeviceToHost));
    throw Error(FF_ERR_SINGULAR_MOMENT,
                "moment matrix of particle " + std::to_string(orig) +
                    " is singular: fewer than four non-coplanar nodes cover it");
  }
}

}  // namespace ff
