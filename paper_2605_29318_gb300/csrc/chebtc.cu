// Tensor-core step of the Chebyshev preconditioner (internal).
//
// The preconditioner applies H (FP32 values) to 40-column blocks of BF16
// direction vectors several hundred times per solve; on CUDA cores that step
// is bound by instruction issue (a gathered row and a multiply-add per nonzero
// and column).  Rows in the internal (cell) order are spatially local, so 16
// consecutive rows share most of their columns: per block of 16 rows the H
// entries are laid out as a dense 16 x K BF16 tile over the sorted union of the
// block's columns (K rounded up to 16; on the 50k torus K averages ~450 and
// ~35% of the tile is nonzero), stored in the A-fragment order of
// mma.m16n8k16 so that a k-step is one 16-byte load per lane.  A step gathers the 16 union rows of the
// direction block into shared memory once (16-byte asynchronous copies),
// forms the B fragments with ldmatrix.trans and accumulates in FP32.
//
// The tile entries are the BF16 roundings of H's values; the row sums hs used
// by the step's difference form (H d)_k = sum_l h_kl d_l - (sum_l h_kl) d_k are
// sums of the same rounded values, so the rounded operator still maps the
// constant vector to zero.  The preconditioner is a polynomial in the rounded
// matrix, which is symmetric like H.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "linalg.cuh"

namespace ff {
namespace {

constexpr int kTcRows = 16;            // rows per block (the M of the MMA)
constexpr int kTcMaxWords = 8192;      // bitmap words: column spans up to 262144
constexpr unsigned kFullMask = 0xffffffffu;

// column span of each block and the number of k-steps its union needs
__global__ void __launch_bounds__(256)
    k_tc_count(const long long* __restrict__ ptr, const int* __restrict__ col, int n,
               int* __restrict__ nks, int* __restrict__ lo_out, int* __restrict__ words_out) {
  extern __shared__ unsigned bm[];
  __shared__ int s_min, s_max, s_cnt;
  const int b = blockIdx.x, tid = threadIdx.x;
  const int k0 = b * kTcRows, k1 = min(n, k0 + kTcRows);
  const long long e0 = ptr[k0], e1 = ptr[k1];
  if (tid == 0) {
    s_min = 0x7fffffff;
    s_max = -1;
    s_cnt = 0;
  }
  __syncthreads();
  int mn = 0x7fffffff, mx = -1;
  for (long long e = e0 + tid; e < e1; e += blockDim.x) {
    const int c = col[e];
    mn = min(mn, c);
    mx = max(mx, c);
  }
  atomicMin(&s_min, mn);
  atomicMax(&s_max, mx);
  __syncthreads();
  const int lo = s_min;
  const int words = s_max >= lo ? (s_max - lo) / 32 + 1 : 0;
  if (words > kTcMaxWords) {
    if (tid == 0) nks[b] = -1;
    return;
  }
  for (int wd = tid; wd < words; wd += blockDim.x) bm[wd] = 0u;
  __syncthreads();
  for (long long e = e0 + tid; e < e1; e += blockDim.x) {
    const int off = col[e] - lo;
    atomicOr(&bm[off >> 5], 1u << (off & 31));
  }
  __syncthreads();
  int cnt = 0;
  for (int wd = tid; wd < words; wd += blockDim.x) cnt += __popc(bm[wd]);
  atomicAdd(&s_cnt, cnt);
  __syncthreads();
  if (tid == 0) {
    nks[b] = (s_cnt + 15) / 16;
    lo_out[b] = lo;
    words_out[b] = words;
  }
}

// union columns, tile entries (fragment order) and rounded row sums
__global__ void __launch_bounds__(256)
    k_tc_fill(const long long* __restrict__ ptr, const int* __restrict__ col,
              const float* __restrict__ hv, int n, const int* __restrict__ kofs,
              const int* __restrict__ lo_in, const int* __restrict__ words_in,
              int* __restrict__ ucol, unsigned short* __restrict__ tile, float* __restrict__ hs) {
  extern __shared__ unsigned smw[];
  __shared__ int wsum[8];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int k0 = b * kTcRows, k1 = min(n, k0 + kTcRows);
  const long long e0 = ptr[k0], e1 = ptr[k1];
  const int lo = lo_in[b], words = words_in[b];
  const long long s0 = kofs[b];
  const int ns = kofs[b + 1] - kofs[b];
  unsigned* bm = smw;          // words
  unsigned* pre = smw + words; // words: union entries before each word
  for (int wd = tid; wd < words; wd += blockDim.x) bm[wd] = 0u;
  // this block's tile region to zero (16-byte units: 32 per k-step)
  uint4* t4 = reinterpret_cast<uint4*>(tile) + s0 * 32;
  for (int q = tid; q < ns * 32; q += blockDim.x) t4[q] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (long long e = e0 + tid; e < e1; e += blockDim.x) {
    const int off = col[e] - lo;
    atomicOr(&bm[off >> 5], 1u << (off & 31));
  }
  __syncthreads();
  // exclusive scan of the popcounts: each thread a contiguous run of words
  const int per = (words + blockDim.x - 1) / blockDim.x;
  const int w0 = min(words, tid * per), w1 = min(words, w0 + per);
  int run = 0;
  for (int wd = w0; wd < w1; ++wd) run += __popc(bm[wd]);
  int incl = run;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFullMask, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[wid] = incl;
  __syncthreads();
  int base = 0;
  for (int q = 0; q < wid; ++q) base += wsum[q];
  int acc = base + incl - run;
  for (int wd = w0; wd < w1; ++wd) {
    pre[wd] = acc;
    acc += __popc(bm[wd]);
  }
  int total = 0;
  for (int q = 0; q < (int)(blockDim.x >> 5); ++q) total += wsum[q];
  __syncthreads();
  // union columns in ascending order; padding repeats the first column
  int* uc = ucol + s0 * 16;
  for (int wd = tid; wd < words; wd += blockDim.x) {
    unsigned bits = bm[wd];
    int r = pre[wd];
    while (bits) {
      const int j = __ffs(bits) - 1;
      uc[r++] = lo + 32 * wd + j;
      bits &= bits - 1;
    }
  }
  for (int r = total + tid; r < ns * 16; r += blockDim.x) uc[r] = lo;
  // entries: warp wid takes rows wid and wid + 8 of the block
  for (int rr = wid; rr < kTcRows; rr += 8) {
    const int k = k0 + rr;
    if (k >= n) break;
    float sum = 0.f;
    for (long long e = ptr[k] + lane; e < ptr[k + 1]; e += 32) {
      const int off = col[e] - lo;
      const int rank = pre[off >> 5] + __popc(bm[off >> 5] & ((1u << (off & 31)) - 1u));
      const int s = rank >> 4, kk = rank & 15;
      const int fl = (rr & 7) * 4 + ((kk & 7) >> 1);  // fragment lane
      const int reg = (rr >> 3) + 2 * (kk >> 3);      // a0..a3
      const __nv_bfloat16 q = __float2bfloat16(hv[e]);
      tile[((s0 + s) * 32 + fl) * 8 + reg * 2 + (kk & 1)] = __bfloat16_as_ushort(q);
      sum += __bfloat162float(q);
    }
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(kFullMask, sum, o);
    if (lane == 0) hs[k] = sum;
  }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait2() { asm volatile("cp.async.wait_group 2;\n" ::: "memory"); }
// every copy of the thread, those it has committed to no group among them
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// One block of WB warps per 16-row block; warp w takes the block's k-steps
// w, w + WB, ...: three staging buffers per warp keep the union rows of two
// later steps in flight while a step is multiplied (their union columns and
// A fragments loaded earlier still).  The warps' partial 16 x m products are
// summed through the same shared memory, then res -= D^-1 (H d),
// d' = c1 d + c2 res (BF16), x += d'.
// WB = 4 where the row blocks fill the GPU; WB = 16 where they are few (a
// K x K pencil of a two-set cloud: 63 row blocks for K = 1,000), so that each
// warp's chain of k-steps is four times shorter.
// Bound by the latency of its chains (a warp has about seven k-steps): the block's
// own rows of res, x and d therefore come with the third step's group and are
// finished as the contiguous run they are, 64 registers let eight blocks share an
// SM, and a step's kernel starts while the one before drains, reading its tables
// before it waits for that one's vectors.  50,000 rows, 40 columns, launch lists (cold,
// serialised): 28.2 us a step without these, 23.3 so, and about 3 us less between steps.
// Slower, in a timing where this form took 27.2 us and the one before 31.7: gathers that
// keep lines in L1 (29.5), two (30.8) or four (33.1) row blocks in a block to share them.
__host__ __device__ constexpr size_t tc_rows_bytes(int NT) { return (size_t)kTcRows * (8 * NT * 10 + 8); }
__host__ __device__ constexpr int tc_red_ld(int NT) { return 8 * NT + (NT % 2 ? 0 : 8); }  // conflict-free for 8 rows

template <int WB>
constexpr size_t tc_step_smem(int NT) {
  return std::max<size_t>((size_t)WB * 3 * kTcRows * 8 * NT * 2,
                          (size_t)WB * kTcRows * tc_red_ld(NT) * 4) +
         tc_rows_bytes(NT);
}

template <int NT, int WB>
__global__ void __launch_bounds__(32 * WB, WB == 4 && NT <= 5 ? 8 : 1)
    k_cheb_step_tc(const int* __restrict__ kofs, const int* __restrict__ ucol,
                   const uint4* __restrict__ tile, const float* __restrict__ hs,
                   const float* __restrict__ hdiag, int n, const __nv_bfloat16* __restrict__ din,
                   __nv_bfloat16* __restrict__ dout, float* __restrict__ x,
                   float* __restrict__ res, float c1, float c2) {
  constexpr int kWB = WB;
  constexpr int m = 8 * NT, PIECES = kTcRows * NT, ITERS = (PIECES + 31) / 32, NB = 3;
  constexpr int P = tc_red_ld(NT);
  extern __shared__ __align__(16) unsigned char smem[];
  const int b = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the block's own rows of res, x and d, and 1 / diagonal and row sum of each row
  float* own_r = reinterpret_cast<float*>(smem);
  float* own_x = own_r + kTcRows * m;
  __nv_bfloat16* own_d = reinterpret_cast<__nv_bfloat16*>(own_x + kTcRows * m);
  float* own_h = reinterpret_cast<float*>(own_d + kTcRows * m);
  unsigned char* work = smem + tc_rows_bytes(NT);
  __nv_bfloat16* stage = reinterpret_cast<__nv_bfloat16*>(work) + w * NB * kTcRows * m;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int s0 = kofs[b], ns = kofs[b + 1] - s0;
  const int k0 = b * kTcRows, nrow = min(kTcRows, n - k0);
  float acc[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  auto ucol_of = [&](int s) {
    return (s < ns && lane < 16) ? __ldg(ucol + (long long)(s0 + s) * 16 + lane) : 0;
  };
  auto tile_of = [&](int s, const uint4& dflt) {
    return s < ns ? __ldg(tile + (long long)(s0 + s) * 32 + lane) : dflt;
  };
  auto stage_step = [&](int buf, int u) {  // u: lane r < 16 holds the step's union column r
    __nv_bfloat16* dst = stage + buf * kTcRows * m;
#pragma unroll
    for (int it = 0; it < ITERS; ++it) {
      const int p = it * 32 + lane;
      const int rr = min(p / NT, kTcRows - 1), pc = p % NT;
      const int row = __shfl_sync(kFullMask, u, rr);
      if (p < PIECES) cp_async16(dst + rr * m + pc * 8, din + (long long)row * m + pc * 8);
    }
  };
  // Registers rotate without moves (a move would wait for its load): A[p]
  // holds the fragments of the step multiplied in phase p, U[p] the union
  // columns of the step staged in phase p; each is reloaded right after use
  // for the step three phases on.
  int s = w;
  const int u0 = ucol_of(s), u1 = ucol_of(s + kWB);
  const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
  uint4 A[3] = {tile_of(s, zero4), tile_of(s + kWB, zero4), tile_of(s + 2 * kWB, zero4)};
  int U[3] = {ucol_of(s + 2 * kWB), ucol_of(s + 3 * kWB), ucol_of(s + 4 * kWB)};
  if (threadIdx.x < nrow) {
    own_h[threadIdx.x] = 1.0f / hdiag[k0 + threadIdx.x];
    own_h[kTcRows + threadIdx.x] = hs[k0 + threadIdx.x];
  }
  // only the vectors come from the step before
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (s < ns) stage_step(0, u0);
  cp_commit();
  if (s + kWB < ns) stage_step(1, u1);
  cp_commit();
  {  // in the group of the third step (in none where the warp has no k-step)
    const long long o = (long long)k0 * m;
    for (int q = threadIdx.x; q < nrow * (m / 4); q += 32 * kWB) {
      cp_async16(own_r + 4 * q, res + o + 4 * q);
      cp_async16(own_x + 4 * q, x + o + 4 * q);
    }
    for (int q = threadIdx.x; q < nrow * NT; q += 32 * kWB)
      cp_async16(own_d + 8 * q, din + o + 8 * q);
  }
  auto phase = [&](const int p) {
    if (s + 2 * kWB < ns) stage_step((p + 2) % 3, U[p]);
    cp_commit();
    U[p] = ucol_of(s + 5 * kWB);
    cp_wait2();
    __syncwarp();
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(stage + p * kTcRows * m);
    const int mat = lane >> 3, krow = (mat & 1) * 8 + (lane & 7);
#pragma unroll
    for (int j = 0; j + 1 < NT; j += 2) {
      unsigned r0, r1, r2, r3;
      const unsigned addr = sbase + (unsigned)(krow * m * 2 + (j + (mat >> 1)) * 16);
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                   : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                   : "r"(addr));
      mma_bf16(acc[j], A[p], r0, r1);
      mma_bf16(acc[j + 1], A[p], r2, r3);
    }
    if (NT & 1) {
      constexpr int j = NT - 1;
      unsigned r0, r1;
      const unsigned addr =
          sbase + (unsigned)(((lane >> 3) & 1) * 8 * m * 2 + (lane & 7) * m * 2 + j * 16);
      asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                   : "=r"(r0), "=r"(r1)
                   : "r"(addr));
      mma_bf16(acc[j], A[p], r0, r1);
    }
    __syncwarp();
    A[p] = tile_of(s + 3 * kWB, zero4);
    s += kWB;
  };
  while (s < ns) {
    phase(0);
    if (s >= ns) break;
    phase(1);
    if (s >= ns) break;
    phase(2);
  }
  cp_wait_all();
  __syncthreads();  // every warp's copies are there, and it is done with its staging buffers
  float* red = reinterpret_cast<float*>(work);  // [kWB][16][P]
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      *reinterpret_cast<float2*>(red + (w * kTcRows + g + 8 * h) * P + 8 * j + 2 * t) =
          make_float2(acc[j][2 * h], acc[j][2 * h + 1]);
  __syncthreads();
  // the block's rows are contiguous: a thread takes pairs of columns of them
  for (int e = threadIdx.x; e < nrow * (m / 2); e += 32 * kWB) {
    const int row = e / (m / 2), col = 2 * (e % (m / 2));
    float2 c = make_float2(0.f, 0.f);
    for (int v = 0; v < kWB; ++v) {
      const float2 p = *reinterpret_cast<const float2*>(red + (v * kTcRows + row) * P + col);
      c.x += p.x;
      c.y += p.y;
    }
    const float dinv = own_h[row], hsk = own_h[kTcRows + row];
    const float2 dk = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(own_d)[e]);
    float2 r = reinterpret_cast<const float2*>(own_r)[e];
    float2 xx = reinterpret_cast<const float2*>(own_x)[e];
    r.x -= (c.x - hsk * dk.x) * dinv;
    r.y -= (c.y - hsk * dk.y) * dinv;
    const __nv_bfloat16 q0 = __float2bfloat16(c1 * dk.x + c2 * r.x);
    const __nv_bfloat16 q1 = __float2bfloat16(c1 * dk.y + c2 * r.y);
    xx.x += __bfloat162float(q0);
    xx.y += __bfloat162float(q1);
    const long long o = (long long)k0 * m + 2 * e;
    *reinterpret_cast<float2*>(res + o) = r;
    *reinterpret_cast<float2*>(x + o) = xx;
    __nv_bfloat162 qq;
    qq.x = q0;
    qq.y = q1;
    *reinterpret_cast<__nv_bfloat162*>(dout + o) = qq;
  }
}

// All the steps of a polynomial in one cooperative launch, for matrices of few
// row blocks (one block of 16 warps each, all resident): a block keeps its A
// fragments, union columns, residual and x in registers for the whole polynomial
// and only the directions pass through memory, with a grid barrier between steps.
// The same sums in the same order as k_cheb_step_tc<NT, 16>, bit for bit.  A
// step by itself is a launch, the loads of tiles and columns, and a tail: for
// 3,001 rows and 24 columns 7.8 us, 3.5 so; for the 1,000 x 1,000 pencil of the
// splat and 72 columns 9.6 us, 5.0 so.  Not for solves beside others on the GPU (a
// batch): a cooperative launch waits until all its blocks fit, and four objects of
// 2,000 to 20,000 particles took 108 ms with it against 103 without.
// Each warp's k-steps must fit its registers (kPolyK of them).
constexpr int kPolyK = 4;        // k-steps of a warp: unions up to 1,024 columns
constexpr int kPolyMax = 64;     // steps a launch
struct PolyCoef {
  float c1[kPolyMax], c2[kPolyMax];
};

// Arrivals counted up to `target` (modulo 2^32); false when the wait ran out
// (about a second: a block of the grid was not running)
__device__ __forceinline__ bool poly_barrier(unsigned* bar, unsigned target) {
  __shared__ int s_late;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const long long t0 = clock64();
    int late = 0;
    unsigned v;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (clock64() - t0 > 2000000000LL) late = 1;
    } while ((int)(v - target) < 0 && !late);
    __threadfence();
    s_late = late;
  }
  __syncthreads();
  return s_late == 0;
}

constexpr size_t poly_smem(int NT, int ksteps) {
  return std::max<size_t>((size_t)16 * ksteps * kTcRows * 8 * NT * 2, (size_t)16 * 32 * 4 * NT * 4);
}

template <int NT>
__global__ void __launch_bounds__(512, NT <= 5 ? 2 : 1)
    k_cheb_poly_tc(const int* __restrict__ kofs, const int* __restrict__ ucol,
                   const uint4* __restrict__ tile, const float* __restrict__ hs,
                   const float* __restrict__ hdiag, int n, __nv_bfloat16* d0, __nv_bfloat16* d1,
                   float* __restrict__ x, const float* __restrict__ res, int steps, PolyCoef coef,
                   int ksteps, unsigned* bar, unsigned base) {
  constexpr int kWB = 16;
  constexpr int m = 8 * NT, PIECES = kTcRows * NT, ITERS = (PIECES + 31) / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int b = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __nv_bfloat16* stage = reinterpret_cast<__nv_bfloat16*>(smem) + (size_t)w * ksteps * kTcRows * m;
  float* red = reinterpret_cast<float*>(smem);  // [kWB][32][4 NT]
  const int s0 = kofs[b], ns = kofs[b + 1] - s0;
  uint4 A[kPolyK];
  int U[kPolyK];
#pragma unroll
  for (int p = 0; p < kPolyK; ++p) {
    const int s = w + p * kWB;
    A[p] = s < ns ? __ldg(tile + (long long)(s0 + s) * 32 + lane) : make_uint4(0u, 0u, 0u, 0u);
    U[p] = s < ns && lane < 16 ? __ldg(ucol + (long long)(s0 + s) * 16 + lane) : 0;
  }
  // warp j finishes column tile j: rows g and g + 8, columns 8 j + 2 t and the next
  const int g = lane >> 2, t = lane & 3;
  float2 r[2], xx[2], dk[2];
  float dinv[2] = {0.f, 0.f}, hsk[2] = {0.f, 0.f};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = b * kTcRows + g + 8 * h;
    r[h] = xx[h] = dk[h] = make_float2(0.f, 0.f);
    if (w < NT && k < n) {
      const long long o = (long long)k * m + 8 * w + 2 * t;
      dinv[h] = 1.0f / hdiag[k];
      hsk[h] = hs[k];
      r[h] = *reinterpret_cast<const float2*>(res + o);
      xx[h] = *reinterpret_cast<const float2*>(x + o);
      dk[h] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(d0 + o));
    }
  }
  bool ok = true;
  for (int it = 0; it < steps; ++it) {
    const __nv_bfloat16* din = it & 1 ? d1 : d0;
    __nv_bfloat16* dout = it & 1 ? d0 : d1;
#pragma unroll
    for (int p = 0; p < kPolyK; ++p) {
      if (w + p * kWB < ns) {
        __nv_bfloat16* dst = stage + p * kTcRows * m;
#pragma unroll
        for (int q = 0; q < ITERS; ++q) {
          const int e = q * 32 + lane;
          const int rr = min(e / NT, kTcRows - 1), pc = e % NT;
          const int row = __shfl_sync(kFullMask, U[p], rr);
          if (e < PIECES) cp_async16(dst + rr * m + pc * 8, din + (long long)row * m + pc * 8);
        }
      }
      cp_commit();
    }
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
    for (int p = 0; p < kPolyK; ++p) {
      if (p == 0) asm volatile("cp.async.wait_group %0;\n" ::"n"(kPolyK - 1) : "memory");
      if (p == 1) asm volatile("cp.async.wait_group %0;\n" ::"n"(kPolyK - 2) : "memory");
      if (p == 2) asm volatile("cp.async.wait_group %0;\n" ::"n"(kPolyK - 3) : "memory");
      if (p == 3) asm volatile("cp.async.wait_group %0;\n" ::"n"(0) : "memory");
      __syncwarp();
      if (w + p * kWB >= ns) continue;
      const unsigned sbase = (unsigned)__cvta_generic_to_shared(stage + p * kTcRows * m);
      const int mat = lane >> 3, krow = (mat & 1) * 8 + (lane & 7);
#pragma unroll
      for (int j = 0; j + 1 < NT; j += 2) {
        unsigned r0, r1, r2, r3;
        const unsigned addr = sbase + (unsigned)(krow * m * 2 + (j + (mat >> 1)) * 16);
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                     : "r"(addr));
        mma_bf16(acc[j], A[p], r0, r1);
        mma_bf16(acc[j + 1], A[p], r2, r3);
      }
      if (NT & 1) {
        constexpr int j = NT - 1;
        unsigned r0, r1;
        const unsigned addr =
            sbase + (unsigned)(((lane >> 3) & 1) * 8 * m * 2 + (lane & 7) * m * 2 + j * 16);
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                     : "=r"(r0), "=r"(r1)
                     : "r"(addr));
        mma_bf16(acc[j], A[p], r0, r1);
      }
    }
    __syncthreads();  // every warp is done with its staging buffers
#pragma unroll
    for (int j = 0; j < NT; ++j)
      *reinterpret_cast<float4*>(red + (w * 32 + lane) * 4 * NT + 4 * j) =
          make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
    __syncthreads();
    if (w < NT) {
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int v = 0; v < kWB; ++v) {
        const float4 y =
            *reinterpret_cast<const float4*>(red + (v * 32 + lane) * 4 * NT + 4 * w);
        c[0] += y.x;
        c[1] += y.y;
        c[2] += y.z;
        c[3] += y.w;
      }
      const float c1 = coef.c1[it], c2 = coef.c2[it];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = b * kTcRows + g + 8 * h;
        if (k >= n) continue;
        r[h].x -= (c[2 * h] - hsk[h] * dk[h].x) * dinv[h];
        r[h].y -= (c[2 * h + 1] - hsk[h] * dk[h].y) * dinv[h];
        const __nv_bfloat16 q0 = __float2bfloat16(c1 * dk[h].x + c2 * r[h].x);
        const __nv_bfloat16 q1 = __float2bfloat16(c1 * dk[h].y + c2 * r[h].y);
        dk[h] = make_float2(__bfloat162float(q0), __bfloat162float(q1));
        xx[h].x += dk[h].x;
        xx[h].y += dk[h].y;
        __nv_bfloat162 qq;
        qq.x = q0;
        qq.y = q1;
        *reinterpret_cast<__nv_bfloat162*>(dout + (long long)k * m + 8 * w + 2 * t) = qq;
      }
    }
    if (it + 1 < steps) ok = poly_barrier(bar, base + (unsigned)(it + 1) * gridDim.x);
    if (!ok) break;
  }
  if (w < NT)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = b * kTcRows + g + 8 * h;
      // a wait that ran out leaves NaN, which the solver reports
      if (!ok) xx[h] = make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
      if (k < n) *reinterpret_cast<float2*>(x + (long long)k * m + 8 * w + 2 * t) = xx[h];
    }
}

}  // namespace

bool cheb_tc_build(ff_ctx* c) {
  cudaStream_t st = c->stream;
  c->tc_ksteps = 0;
  const long long n = c->n;
  if (n <= 0 || n >= (1LL << 30)) return false;
  const int nblk = (int)((n + kTcRows - 1) / kTcRows);
  int* nks = reinterpret_cast<int*>(c->scratch[4].ensure(sizeof(int) * 3 * (size_t)nblk));
  int* lo = nks + nblk;
  int* words = lo + nblk;
  set_max_dyn_smem((const void*)k_tc_count, (int)(sizeof(unsigned) * kTcMaxWords));
  set_max_dyn_smem((const void*)k_tc_fill, (int)(2 * sizeof(unsigned) * kTcMaxWords));
  (k_tc_count<<<nblk, 256, sizeof(unsigned) * kTcMaxWords, st>>>(
       c->a_ptr.as<long long>(), c->a_col.as<int>(), (int)n, nks, lo, words),
   ::ff::note_launch());
  FF_LAUNCH_CHECK();
  std::vector<int> h(nblk);
  FF_CUDA(cudaMemcpyAsync(h.data(), nks, sizeof(int) * nblk, cudaMemcpyDeviceToHost, st));
  FF_CUDA(cudaStreamSynchronize(st));
  std::vector<int> ofs(nblk + 1, 0);
  for (int b = 0; b < nblk; ++b) {
    if (h[b] < 0) return false;  // a block's columns span too far: CUDA-core step
    ofs[b + 1] = ofs[b] + h[b];
    if (ofs[b + 1] >= (1 << 26)) return false;
  }
  const long long S = ofs[nblk];
  c->tc_kmax = *std::max_element(h.begin(), h.end());
  int* kofs = reinterpret_cast<int*>(c->tc_kofs.ensure(sizeof(int) * (nblk + 1)));
  FF_CUDA(cudaMemcpyAsync(kofs, ofs.data(), sizeof(int) * (nblk + 1), cudaMemcpyHostToDevice, st));
  int* uc = reinterpret_cast<int*>(c->tc_ucol.ensure(sizeof(int) * 16 * (size_t)std::max(S, 1LL)));
  auto* tl = reinterpret_cast<unsigned short*>(c->tc_tile.ensure(512 * (size_t)std::max(S, 1LL)));
  float* hs = reinterpret_cast<float*>(c->tc_hs.ensure(sizeof(float) * n));
  (k_tc_fill<<<nblk, 256, 2 * sizeof(unsigned) * kTcMaxWords, st>>>(
       c->a_ptr.as<long long>(), c->a_col.as<int>(), c->h_f32.as<float>(), (int)n, kofs, lo,
       words, uc, tl, hs),
   ::ff::note_launch());
  FF_LAUNCH_CHECK();
  FF_CUDA(cudaStreamSynchronize(st));
  c->tc_ksteps = S;
  return true;
}

bool cheb_step_tc(cudaStream_t st, const ff_ctx* c, int m, const void* din, void* dout, float* x,
                  float* res, float c1, float c2) {
  // widths 8..120 in steps of 8 (the staging buffers stay in static shared memory)
  if (c->tc_ksteps <= 0 || m % 8 != 0 || m < 8 || m > 120 || c->n * m >= (1LL << 31)) return false;
  ProfScope ps(kProfPrecond);
  const int nblk = (int)((c->n + kTcRows - 1) / kTcRows);
  const auto* bi = static_cast<const __nv_bfloat16*>(din);
  auto* bo = static_cast<__nv_bfloat16*>(dout);
  const bool few = nblk < 2 * sm_count();
  auto go = [&](auto nt) {
    constexpr int NT = decltype(nt)::value;
    // a step's tables are fetched while the step before it drains
    cudaLaunchAttribute early;
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nblk);
    cfg.stream = st;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    auto launch = [&](auto fn, int warps, size_t sm) {
      set_max_dyn_smem((const void*)fn, (int)sm);
      cfg.blockDim = dim3(32 * warps);
      cfg.dynamicSmemBytes = sm;
      FF_CUDA(cudaLaunchKernelEx(&cfg, fn, (const int*)c->tc_kofs.as<int>(),
                                 (const int*)c->tc_ucol.as<int>(),
                                 reinterpret_cast<const uint4*>(c->tc_tile.p),
                                 (const float*)c->tc_hs.as<float>(),
                                 (const float*)c->hdiag_f32.as<float>(), (int)c->n, bi, bo, x, res,
                                 c1, c2));
      ::ff::note_launch();
    };
    if (few)
      launch(k_cheb_step_tc<NT, 16>, 16, tc_step_smem<16>(NT));
    else
      launch(k_cheb_step_tc<NT, 4>, 4, tc_step_smem<4>(NT));
  };
#define FF_TC(NT) go(std::integral_constant<int, NT>{})
  switch (m / 8) {
    case 1: FF_TC(1); break;
    case 2: FF_TC(2); break;
    case 3: FF_TC(3); break;
    case 4: FF_TC(4); break;
    case 5: FF_TC(5); break;
    case 6: FF_TC(6); break;
    case 7: FF_TC(7); break;
    case 8: FF_TC(8); break;
    case 9: FF_TC(9); break;
    case 10: FF_TC(10); break;
    case 11: FF_TC(11); break;
    case 12: FF_TC(12); break;
    case 13: FF_TC(13); break;
    case 14: FF_TC(14); break;
    default: FF_TC(15); break;
  }
#undef FF_TC
  FF_LAUNCH_CHECK();
  return true;
}

// The steps c1[j], c2[j] (count of them) on d (bin first, bout its other buffer)
// in one launch each of up to kPolyMax; false (nothing launched) when the row
// blocks do not all fit the GPU at once or a block's union is too wide.
bool cheb_poly_tc(cudaStream_t st, ff_ctx* c, int m, void* din, void* dout, float* x, float* res,
                  const float* c1, const float* c2, int count) {
  const int nblk = (int)((c->n + kTcRows - 1) / kTcRows);
  const int ksteps = (c->tc_kmax + 15) / 16;
  if (c->beside_others || c->tc_ksteps <= 0 || m % 8 != 0 || m < 8 || m > 120 ||
      nblk >= 2 * sm_count() ||
      ksteps > kPolyK || count < 2 || count > kPolyMax)
    return false;
  bool done = false;
  auto go = [&](auto nt) {
    constexpr int NT = decltype(nt)::value;
    const size_t sm = poly_smem(NT, ksteps);
    if (sm > 200 * 1024) return;
    const void* fn = (const void*)k_cheb_poly_tc<NT>;
    set_max_dyn_smem(fn, (int)sm);
    int per_sm = 0;
    FF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cheb_poly_tc<NT>, 512, sm));
    if (per_sm * sm_count() < nblk) return;
    if (!c->poly_bar.p) {
      c->poly_bar.ensure(64);
      FF_CUDA(cudaMemsetAsync(c->poly_bar.p, 0, 64, st));
    }
    ProfScope ps(kProfPrecond);
    const int* kofs = c->tc_kofs.as<int>();
    const int* ucol = c->tc_ucol.as<int>();
    const uint4* tile = c->tc_tile.as<uint4>();
    const float *hs = c->tc_hs.as<float>(), *hdiag = c->hdiag_f32.as<float>();
    int n = (int)c->n, ks = ksteps, steps = count;
    PolyCoef coef;
    std::copy(c1, c1 + count, coef.c1);
    std::copy(c2, c2 + count, coef.c2);
    unsigned* bar = c->poly_bar.as<unsigned>();
    unsigned base = c->poly_base;
    void* args[] = {&kofs, &ucol, &tile, &hs,   &hdiag, &n,  &din, &dout,
                    &x,    &res,  &steps, &coef, &ks,    &bar, &base};
    FF_CUDA(cudaLaunchCooperativeKernel(fn, dim3(nblk), dim3(512), args, sm, st));
    ::ff::note_launch();
    c->poly_base += (unsigned)(count - 1) * (unsigned)nblk;
    done = true;
  };
#define FF_TC(NT) go(std::integral_constant<int, NT>{})
  switch (m / 8) {
    case 1: FF_TC(1); break;
    case 2: FF_TC(2); break;
    case 3: FF_TC(3); break;
    case 4: FF_TC(4); break;
    case 5: FF_TC(5); break;
    case 6: FF_TC(6); break;
    case 7: FF_TC(7); break;
    case 8: FF_TC(8); break;
    case 9: FF_TC(9); break;
    case 10: FF_TC(10); break;
    case 11: FF_TC(11); break;
    case 12: FF_TC(12); break;
    case 13: FF_TC(13); break;
    case 14: FF_TC(14); break;
    default: FF_TC(15); break;
  }
#undef FF_TC
  return done;
}

}  // namespace ff
