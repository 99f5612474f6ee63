// Assembly of the weight-space Hessian H_w (Prop. 1) and the RKPM mass matrix
// (Sec. 3.2, Eq. 14) in CSR, one warp per matrix row (in tiles of neighbouring
// rows where the cloud's lists fit, k_tile_rows).
//
//   (H_w)_kl = sum_i v_i (lambda_i + 4 mu_i) grad phi_k(X_i) . grad phi_l(X_i)
//   M_kl     = sum_i v_i phi_k(X_i) phi_l(X_i)
// over the quadrature points X_i covered by both nodes k and l.
//
// Row-owner gather: the warp of row k walks the points i that node k covers
// (transposed neighbour lists, ascending i), and for each i its lanes add the
// contribution of every node l of row i into a shared-memory accumulator slot.
// Within one i the lanes touch distinct slots and the walk over i is
// sequential, so every entry is summed in a fixed order (deterministic, no
// atomics).  Column slots come from a shared-memory hash set of the row's
// 2-hop pattern; pass 1 counts the unique columns, pass 2 sorts them and
// accumulates the values.  The diagonal of H_w is replaced by minus the sum of
// the off-diagonal entries of its row, which makes H_w 1 = 0 exact in storage
// (the constant mode of Supp. Sec. B is an exact null vector).
#include <climits>
#include <type_traits>

#include "ff_internal.cuh"
#include "linalg.cuh"

namespace ff {
namespace {

constexpr int kEmpty = -1;

__device__ __forceinline__ unsigned int hash32(unsigned int x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

// insert key into a warp-private table; returns the slot (or -1 when full)
__device__ __forceinline__ int hset_insert(int* tab, int tsize, int key, bool& fresh) {
  unsigned int h = hash32((unsigned int)key) & (tsize - 1);
  for (int probe = 0; probe < tsize; ++probe) {
    int prev = atomicCAS(&tab[h], kEmpty, key);
    if (prev == kEmpty) {
      fresh = true;
      return (int)h;
    }
    if (prev == key) {
      fresh = false;
      return (int)h;
    }
    h = (h + 1) & (tsize - 1);
  }
  fresh = false;
  return -1;
}

__device__ __forceinline__ int hset_find(const int* tab, int tsize, int key) {
  unsigned int h = hash32((unsigned int)key) & (tsize - 1);
  for (int probe = 0; probe < tsize; ++probe) {
    int v = tab[h];
    if (v == key) return (int)h;
    if (v == kEmpty) return -1;
    h = (h + 1) & (tsize - 1);
  }
  return -1;
}

template <class T>
__global__ void k_material(const int* __restrict__ perm, long long n, const float* __restrict__ vol,
                           const float* __restrict__ E, const float* __restrict__ nu, double E0,
                           double nu0, T* __restrict__ wh, DevFlags* flags) {
  long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  int i = perm ? perm[j] : (int)j;  // caller index of quadrature point j
  double e = E ? (double)E[i] : E0;
  double p = nu ? (double)nu[i] : nu0;
  if (!(e > 0.0) || !(p >= 0.0) || !(p < 0.5) || !isfinite(e)) {
    if (atomicCAS(&flags->code, 0, (int)FF_ERR_INVALID_ARG) == 0) flags->index = i;
    return;
  }
  double lam = e * p / ((1.0 + p) * (1.0 - 2.0 * p));
  double mu = e / (2.0 * (1.0 + p));
  wh[j] = (T)((double)vol[j] * (lam + 4.0 * mu));
}

// rows to a tile (k_tile_rows below); wide (if given) holds a byte a tile, and the
// row-owner passes take the rows of the tiles marked in it
constexpr int kTileRows = 16;

// pass 1: unique 2-hop columns per row
__global__ void k_pattern_count(const long long* __restrict__ ptr, const int* __restrict__ idx,
                                const long long* __restrict__ tptr, const int* __restrict__ tidx,
                                long long n, int tsize, int* __restrict__ cnt,
                                const unsigned char* __restrict__ wide,
                                DevFlags* __restrict__ flags) {
  extern __shared__ int sm_tab[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int* tab = sm_tab + wib * tsize;
  const long long rows_per_grid = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long k = (long long)blockIdx.x * (blockDim.x >> 5) + wib; k < n; k += rows_per_grid) {
    if (wide && !wide[k / kTileRows]) continue;
    for (int q = lane; q < tsize; q += 32) tab[q] = kEmpty;
    __syncwarp();
    int fresh_cnt = 0;
    bool overflow = false;
    for (long long a = tptr[k]; a < tptr[k + 1]; ++a) {
      int i = tidx[a];
      for (long long e = ptr[i] + lane; e < ptr[i + 1]; e += 32) {
        bool fresh;
        int slot = hset_insert(tab, tsize, idx[e], fresh);
        if (slot < 0) overflow = true;
        fresh_cnt += fresh;
      }
    }
    fresh_cnt = __reduce_add_sync(0xffffffffu, fresh_cnt);
    overflow = __any_sync(0xffffffffu, overflow);
    if (lane == 0) {
      cnt[k] = fresh_cnt;
      atomicMax(&flags->max_row, fresh_cnt);
      if (overflow || 2 * fresh_cnt > tsize) {
        if (atomicCAS(&flags->code, 0, (int)FF_ERR_INVALID_ARG) == 0) flags->index = (int)k;
      }
    }
    __syncwarp();
  }
}

// pass 2: sorted columns and values
// T: shape functions, material weights and sums (double-float for FP64
// contexts); TO: the stored matrix values
template <class T, class TO = T>
__global__ void k_assemble(const long long* __restrict__ ptr, const int* __restrict__ idx,
                           const long long* __restrict__ tptr, const int* __restrict__ tidx,
                           const long long* __restrict__ tpos, const T* __restrict__ phi,
                           const T* __restrict__ dphi, long long n1, const float* __restrict__ vol,
                           const T* __restrict__ wh, long long n, int tsize, int maxrow,
                           const long long* __restrict__ aptr, int* __restrict__ acol,
                           TO* __restrict__ aval, float* __restrict__ hf32,
                           float* __restrict__ hdiag, const unsigned char* __restrict__ wide) {
  extern __shared__ unsigned char sm_raw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  // per-warp layout: tab[tsize], rnk[tsize], keys[maxrow], skeys[maxrow] (int),
  // then vh[maxrow], vm[maxrow] (T)
  size_t per_warp = (size_t)tsize * 8 + (size_t)maxrow * 8;
  per_warp = (per_warp + 15) & ~size_t(15);
  size_t per_warp_T = per_warp + (size_t)maxrow * 2 * sizeof(T);
  per_warp_T = (per_warp_T + 15) & ~size_t(15);
  unsigned char* base = sm_raw + per_warp_T * wib;
  int* tab = reinterpret_cast<int*>(base);
  int* rnk = tab + tsize;
  int* keys = rnk + tsize;
  int* skeys = keys + maxrow;
  T* vh = reinterpret_cast<T*>(base + per_warp);
  T* vm = vh + maxrow;
  const long long rows_per_grid = (long long)gridDim.x * wpb;
  for (long long k = (long long)blockIdx.x * wpb + wib; k < n; k += rows_per_grid) {
    if (wide && !wide[k / kTileRows]) continue;
    for (int q = lane; q < tsize; q += 32) tab[q] = kEmpty;
    __syncwarp();
    for (long long a = tptr[k]; a < tptr[k + 1]; ++a) {
      int i = tidx[a];
      for (long long e = ptr[i] + lane; e < ptr[i + 1]; e += 32) {
        bool fresh;
        hset_insert(tab, tsize, idx[e], fresh);
      }
    }
    __syncwarp();
    // compact the keys
    int m = 0;
    for (int q0 = 0; q0 < tsize; q0 += 32) {
      int v = tab[q0 + lane];
      bool has = v != kEmpty;
      unsigned int bal = __ballot_sync(0xffffffffu, has);
      if (has) keys[m + __popc(bal & ((1u << lane) - 1))] = v;
      m += __popc(bal);
    }
    __syncwarp();
    // rank of every key (columns ascending), recorded at its hash slot
    for (int q = lane; q < m; q += 32) {
      int v = keys[q];
      int r = 0;
      for (int b = 0; b < m; ++b) r += keys[b] < v;
      rnk[hset_find(tab, tsize, v)] = r;
      vh[q] = T(0);
      vm[q] = T(0);
    }
    __syncwarp();
    // accumulate over the points i covered by node k, ascending i
    for (long long a = tptr[k]; a < tptr[k + 1]; ++a) {
      int i = tidx[a];
      long long eik = tpos[a];
      T fk = phi[eik];
      T gk0 = dphi[eik], gk1 = dphi[n1 + eik], gk2 = dphi[2 * n1 + eik];
      T wi = wh[i], vi = (T)vol[i];
      T cH0 = wi * gk0, cH1 = wi * gk1, cH2 = wi * gk2, cM = vi * fk;
      for (long long e = ptr[i] + lane; e < ptr[i + 1]; e += 32) {
        int r = rnk[hset_find(tab, tsize, idx[e])];
        if constexpr (std::is_same_v<T, dfloat>) {  // unnormalised sums, normalised below
          df_mac(vh[r], cH0, dphi[e]);
          df_mac(vh[r], cH1, dphi[n1 + e]);
          df_mac(vh[r], cH2, dphi[2 * n1 + e]);
          df_mac(vm[r], cM, phi[e]);
        } else {
          vh[r] += cH0 * dphi[e] + cH1 * dphi[n1 + e] + cH2 * dphi[2 * n1 + e];
          vm[r] += cM * phi[e];
        }
      }
      __syncwarp();
    }
    // keys in rank (ascending column) order; vh / vm are already indexed by rank
    for (int q = lane; q < m; q += 32) {
      int v = keys[q];
      skeys[rnk[hset_find(tab, tsize, v)]] = v;
    }
    __syncwarp();
    T off = T(0);
    for (int r = lane; r < m; r += 32)
      if (skeys[r] != (int)k) off += finish(vh[r]);
#pragma unroll
    for (int o = 16; o; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
    const long long row0 = aptr[k];
    for (int r = lane; r < m; r += 32) {
      int col = skeys[r];
      const TO h = (col == (int)k) ? (TO)(-off) : (TO)finish(vh[r]);
      acol[row0 + r] = col;
      aval[2 * (row0 + r)] = h;
      aval[2 * (row0 + r) + 1] = (TO)finish(vm[r]);
      hf32[row0 + r] = (float)h;
    }
    if (lane == 0) hdiag[k] = (float)(TO)(-off);
    __syncwarp();
  }
}

size_t assemble_smem_per_warp(int tsize, int maxrow, size_t tbytes) {
  size_t per_warp = (size_t)tsize * 8 + (size_t)maxrow * 8;
  per_warp = (per_warp + 15) & ~size_t(15);
  size_t t = per_warp + (size_t)maxrow * 2 * tbytes;
  return (t + 15) & ~size_t(15);
}

// ------------------------------------------------------------------ tiles of rows
// The same sums for the rows of a spatially sorted cloud, kTileRows consecutive
// rows a block.  Neighbouring rows share most of their points and columns, so
// the block first lists, once for all its rows,
//   * the union of the points its nodes cover (a hash table: point -> local
//     number), and
//   * the union of those points' nodes (a hash table, then sorted: the rank of
//     a column), with the rank of every entry of every point's list (`lr`);
// each warp then takes rows: the ranks its points' entries mark become places in
// the row, and it walks the points in ascending order as the row-owner pass does
// (the same sums), a pair costing two 16-bit reads for its place where that pass
// hashes the column twice.  The next point's table values are loaded
// while the current ones are added.  Bound by issue and the latency of the
// accumulators in shared memory, at two blocks an SM.  The row-owner pass took 1.81 +
// 14.4 ms (count, values) for 200k particles in FP32, this 1.11 + 3.39 ms; in
// double-float (50k) 0.48 + 4.07 ms, this 0.29 + 1.09 ms.
// MODE 0 counts the rows' columns, reports the largest tile and marks in `wide`
// those beyond the capacities (a wide support, a dense spot), whose rows are left to
// the row-owner passes; MODE 1 writes the other tiles' columns and values, its
// tables sized by the report.  100,000 particles in FP32 with supports of 2.2, 2.4, 2.6
// and 3.0 spacings, the whole call: 12.0, 17.7, 36.2 and 102.4 ms by the row-owner passes
// alone, 3.6, 6.9, 29.0 and 102.1 so (at 3.0 all tiles are wide).
constexpr int kTileT = 256, kTileWarps = kTileT / 32;

struct TileDims {
  int pts, cols, pairs, row;  // capacities: points, columns and list entries of a
                              // tile, columns of a row
  int ptab, ctab;             // hash slots
};
struct TileMax {
  int wide;                    // tiles beyond the capacities
  int pts, cols, pairs, row;   // the most of the others
};
// of a tile whose tables hold entries of tbytes: 1,200 columns are the most that eight
// warps' double-float rows leave room for (1,536 would take 280,592 bytes)
__host__ __device__ constexpr TileDims tile_cap(int tbytes) {
  return tbytes == 8 ? TileDims{512, 1200, 20480, 1200, 1024, 4096}
                     : TileDims{512, 1536, 20480, 1536, 1024, 4096};
}

// shared memory of a tile: what lasts (points, list entries, sorted columns),
// then the column table, later the warps' rows
struct TileSmem {
  int ptab, plist, poff, scols, pid, lr, ctab, cid, cols, warp, per_warp, loc, total;
  __host__ __device__ constexpr TileSmem(const TileDims& d, int mode, int tbytes)
      : ptab(0), plist(0), poff(0), scols(0), pid(0), lr(0), ctab(0), cid(0), cols(0), warp(0),
        per_warp(0), loc(0), total(0) {
    int at = 0;
    auto take = [&](int bytes) {
      const int o = at;
      at += (bytes + 15) & ~15;
      return o;
    };
    ptab = take(4 * d.ptab);
    plist = take(4 * d.pts);
    poff = take(4 * (d.pts + 1));
    int room = 2;  // the sort's, a power of two
    while (room < d.cols) room <<= 1;
    scols = take(mode ? 4 * room : 0);
    pid = take(2 * d.ptab);
    lr = take(2 * d.pairs);
    const int shared_from = at;
    ctab = take(4 * d.ctab);
    cid = take(2 * d.ctab);
    cols = take(mode ? 4 * d.cols : 0);
    const int tables = at;
    // a warp: loc (MODE 0: marks), then the sums of H and M
    loc = 0;
    per_warp = mode ? ((2 * d.cols + 15) & ~15) + ((2 * d.row * tbytes + 15) & ~15)
                    : (d.cols + 15) & ~15;
    // MODE 0 marks while its table is dead too
    warp = shared_from;
    total = shared_from + per_warp * kTileWarps;
    if (total < tables) total = tables;
  }
};
// whatever the caps let through fits a block (227 KB, beside the kernel's own words)
static_assert(TileSmem(tile_cap(4), 1, 4).total <= 227 * 1024 - 64 &&
                  TileSmem(tile_cap(8), 1, 8).total <= 227 * 1024 - 64,
              "a tile within the caps does not fit a block");

template <int MODE, class T, class TO>
__global__ void __launch_bounds__(kTileT, 2)
    k_tile_rows(const long long* __restrict__ ptr, const int* __restrict__ idx,
                const long long* __restrict__ tptr, const int* __restrict__ tidx,
                const long long* __restrict__ tpos, const T* __restrict__ phi,
                const T* __restrict__ dphi, long long n1, const float* __restrict__ vol,
                const T* __restrict__ wh, long long n, TileDims dims, int* __restrict__ cnt,
                TileMax* __restrict__ tmax, const long long* __restrict__ aptr,
                int* __restrict__ acol, TO* __restrict__ aval, float* __restrict__ hf32,
                float* __restrict__ hdiag, unsigned char* __restrict__ wide) {
  constexpr unsigned kAll = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  if (MODE && wide[blockIdx.x]) return;
  __shared__ int s_np, s_nc, s_tot, s_over;
  const TileSmem L(dims, MODE, (int)sizeof(T));
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const unsigned below = (1u << lane) - 1;
  const long long k0 = (long long)blockIdx.x * kTileRows;
  const long long k1 = min(k0 + kTileRows, n);
  int* ptab = reinterpret_cast<int*>(sm_raw + L.ptab);
  int* plist = reinterpret_cast<int*>(sm_raw + L.plist);
  int* poff = reinterpret_cast<int*>(sm_raw + L.poff);
  int* scols = reinterpret_cast<int*>(sm_raw + L.scols);
  unsigned short* pid = reinterpret_cast<unsigned short*>(sm_raw + L.pid);
  unsigned short* lr = reinterpret_cast<unsigned short*>(sm_raw + L.lr);
  int* ctab = reinterpret_cast<int*>(sm_raw + L.ctab);
  unsigned short* cid = reinterpret_cast<unsigned short*>(sm_raw + L.cid);
  int* cols = reinterpret_cast<int*>(sm_raw + L.cols);
  for (int q = tid; q < dims.ptab; q += kTileT) ptab[q] = kEmpty;
  for (int q = tid; q < dims.ctab; q += kTileT) ctab[q] = kEmpty;
  if (tid == 0) s_np = s_nc = s_tot = s_over = 0;
  __syncthreads();
  // ---- the tile's points, numbered as they are found
  const long long a_end = tptr[k1];
  for (long long a = tptr[k0] + tid; a < a_end; a += kTileT) {
    if (*(volatile int*)&s_np > dims.pts) break;
    bool fresh;
    const int i = tidx[a];
    const int slot = hset_insert(ptab, dims.ptab, i, fresh);
    if (fresh) {
      const int q = atomicAdd(&s_np, 1);
      if (q < dims.pts) {
        plist[q] = i;
        pid[slot] = (unsigned short)q;
      }
    }
  }
  __syncthreads();
  const int np = s_np;
  bool over = np > dims.pts;
  if (!over)
    for (int p = tid; p < np; p += kTileT) {
      const int i = plist[p];
      poff[p] = atomicAdd(&s_tot, (int)(ptr[i + 1] - ptr[i]));
    }
  __syncthreads();
  over = over || s_tot > dims.pairs;
  // ---- their nodes: every list entry's slot in the column table (a warp a
  // point; the entries of four points are loaded before they are inserted)
  if (!over) {
    for (int p0 = wid * 4; p0 < np; p0 += kTileWarps * 4) {
      if (__any_sync(kAll, *(volatile int*)&s_nc > dims.cols)) break;
      int key[4][2], len[4];
      long long s[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = p0 + u < np ? plist[p0 + u] : -1;
        s[u] = i >= 0 ? ptr[i] : 0;
        len[u] = i >= 0 ? (int)(ptr[i + 1] - s[u]) : 0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v)
          key[u][v] = lane + 32 * v < len[u] ? idx[s[u] + lane + 32 * v] : -1;
      auto put = [&](int c, int at) {  // every lane takes part
        bool fresh = false;
        int slot = 0;
        if (c >= 0) {
          slot = hset_insert(ctab, dims.ctab, c, fresh);
          if (slot < 0) s_over = 1;
          lr[at] = (unsigned short)slot;
        }
        const unsigned f = __ballot_sync(kAll, fresh);
        if (f) {
          int q = 0;
          if (lane == 0) q = atomicAdd(&s_nc, __popc(f));
          q = __shfl_sync(kAll, q, 0) + __popc(f & below);
          if (fresh && q < dims.cols) {
            cid[slot] = (unsigned short)q;
            if (MODE) cols[q] = c;
          }
        }
      };
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (p0 + u >= np || __any_sync(kAll, *(volatile int*)&s_nc > dims.cols)) break;
        const int o = poff[p0 + u];
#pragma unroll
        for (int v = 0; v < 2; ++v)
          if (32 * v < len[u]) put(key[u][v], o + lane + 32 * v);
        for (int t0 = 64; t0 < len[u] && !__any_sync(kAll, *(volatile int*)&s_nc > dims.cols);
             t0 += 32) {
          const int t = t0 + lane;
          put(t < len[u] ? idx[s[u] + t] : -1, o + t);
        }
      }
    }
  }
  __syncthreads();
  const int nc = s_nc, tot = s_tot;
  over = over || s_over || nc > dims.cols;
  if (MODE == 0 && tid == 0) {
    wide[blockIdx.x] = over;
    if (over) {
      atomicAdd(&tmax->wide, 1);
    } else {
      atomicMax(&tmax->pts, np);
      atomicMax(&tmax->cols, nc);
      atomicMax(&tmax->pairs, tot);
    }
  }
  if (over) return;
  if (MODE) {  // the columns in order (bitonic): a number becomes a rank
    const int pow2 = 1 << (32 - __clz(max(nc - 1, 1)));
    for (int q = tid; q < pow2; q += kTileT) scols[q] = q < nc ? cols[q] : INT_MAX;
    __syncthreads();
    for (int size = 2; size <= pow2; size <<= 1)
      for (int step = size >> 1; step; step >>= 1) {
        for (int q = tid; q < pow2 / 2; q += kTileT) {
          const int lo = 2 * q - (q & (step - 1)), hi = lo + step;
          const int x = scols[lo], y = scols[hi];
          if ((x > y) == ((lo & size) == 0)) {
            scols[lo] = y;
            scols[hi] = x;
          }
        }
        __syncthreads();
      }
    for (int r = tid; r < nc; r += kTileT)
      cid[hset_find(ctab, dims.ctab, scols[r])] = (unsigned short)r;
    __syncthreads();
  }
  for (int q = tid; q < tot; q += kTileT) lr[q] = cid[lr[q]];
  __syncthreads();
  // ---- the rows, a warp each
  unsigned char* mine = sm_raw + L.warp + (size_t)wid * L.per_warp;
  unsigned short* loc = reinterpret_cast<unsigned short*>(mine);
  struct __align__(2 * sizeof(T)) Sums {
    T h, m;
  };
  Sums* sums = reinterpret_cast<Sums*>(mine + (((size_t)2 * dims.cols + 15) & ~size_t(15)));
  const int words = MODE ? (nc + 1) / 2 : (nc + 3) / 4;  // of the marks
  for (long long k = k0 + wid; k < k1; k += kTileWarps) {
    for (int w = lane; w < words; w += 32) reinterpret_cast<unsigned*>(mine)[w] = 0u;
    __syncwarp();
    const long long as = tptr[k];
    const int np_row = (int)(tptr[k + 1] - as);
    // the row's columns: the entries of its points marked
    for (int a0 = 0; a0 < np_row; a0 += 32) {
      const int here = min(32, np_row - a0);
      int off = 0, len = 0;
      if (lane < here) {
        const int i = tidx[as + a0 + lane];
        off = poff[pid[hset_find(ptab, dims.ptab, i)]];
        len = (int)(ptr[i + 1] - ptr[i]);
      }
      for (int u = 0; u < here; ++u) {
        const int o = __shfl_sync(kAll, off, u), e = __shfl_sync(kAll, len, u);
        for (int t = lane; t < e; t += 32) {
          const int r = lr[o + t];
          if (MODE)
            loc[r] = 1;
          else
            mine[r] = 1;
        }
      }
    }
    __syncwarp();
    if constexpr (MODE == 0) {
      int c = 0;
      for (int w = lane; w < words; w += 32) c += __popc(reinterpret_cast<unsigned*>(mine)[w]);
      c = __reduce_add_sync(kAll, c);
      if (lane == 0) {
        cnt[k] = c;
        if (c > *(volatile int*)&tmax->row) atomicMax(&tmax->row, c);
      }
    } else {
      // a rank becomes a place in the row
      const long long at = aptr[k];
      int m = 0, diag = -1;
      for (int r0 = 0; r0 < nc; r0 += 32) {
        const int r = r0 + lane;
        const bool in = r < nc && loc[r];
        const unsigned bal = __ballot_sync(kAll, in);
        if (in) {
          const int q = m + __popc(bal & below);
          const int c = scols[r];
          loc[r] = (unsigned short)q;
          acol[at + q] = c;
          if (c == (int)k) diag = q;
        }
        m += __popc(bal);
      }
      diag = __reduce_max_sync(kAll, diag);
      for (int q = lane; q < m; q += 32) sums[q] = Sums{T(0), T(0)};
      __syncwarp();
      // the sums over the row's points, ascending
      for (int a0 = 0; a0 < np_row; a0 += 32) {
        const int here = min(32, np_row - a0);
        // a lane a point: its list and the row's weighted values there
        int off = 0, len = 0;
        long long s = 0;
        T h0(0), h1(0), h2(0), hm(0);
        if (lane < here) {
          const int i = tidx[as + a0 + lane];
          off = poff[pid[hset_find(ptab, dims.ptab, i)]];
          s = ptr[i];
          len = (int)(ptr[i + 1] - s);
          const long long e = tpos[as + a0 + lane];
          const T w = wh[i];
          h0 = w * dphi[e];
          h1 = w * dphi[n1 + e];
          h2 = w * dphi[2 * n1 + e];
          hm = (T)vol[i] * phi[e];
        }
        // two entries a lane of the next point are in flight; longer lists take
        // the rest in a loop
        T g[2][4];
        int rk[2], nlen = 0, noff = 0;
        long long ns = 0;
        auto load = [&](int u) {
          nlen = __shfl_sync(kAll, len, u);
          ns = __shfl_sync(kAll, s, u);
          noff = __shfl_sync(kAll, off, u);
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            const int t = lane + 32 * v;
            rk[v] = -1;
            if (t < nlen) {
              const long long e = ns + t;
              rk[v] = loc[lr[noff + t]];
              g[v][0] = dphi[e];
              g[v][1] = dphi[n1 + e];
              g[v][2] = dphi[2 * n1 + e];
              g[v][3] = phi[e];
            }
          }
        };
        load(0);
        for (int u = 0; u < here; ++u) {
          const T c0 = __shfl_sync(kAll, h0, u), c1 = __shfl_sync(kAll, h1, u),
                  c2 = __shfl_sync(kAll, h2, u), cm = __shfl_sync(kAll, hm, u);
          const int mylen = nlen, myoff = noff;
          const long long mys = ns;
          T q[2][4];
          int r2[2];
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            r2[v] = rk[v];
#pragma unroll
            for (int d = 0; d < 4; ++d) q[v][d] = g[v][d];
          }
          if (u + 1 < here) load(u + 1);
          auto add = [&](int r, T x0, T x1, T x2, T xm) {
            Sums z = sums[r];
            if constexpr (std::is_same_v<T, dfloat>) {  // unnormalised, finished below
              df_mac(z.h, c0, x0);
              df_mac(z.h, c1, x1);
              df_mac(z.h, c2, x2);
              df_mac(z.m, cm, xm);
            } else {
              z.h += c0 * x0 + c1 * x1 + c2 * x2;
              z.m += cm * xm;
            }
            sums[r] = z;
          };
#pragma unroll
          for (int v = 0; v < 2; ++v)
            if (r2[v] >= 0) add(r2[v], q[v][0], q[v][1], q[v][2], q[v][3]);
          for (int t = lane + 64; t < mylen; t += 32) {
            const long long e = mys + t;
            add(loc[lr[myoff + t]], dphi[e], dphi[n1 + e], dphi[2 * n1 + e], phi[e]);
          }
          __syncwarp();
        }
      }
      T sum(0);
      for (int q = lane; q < m; q += 32)
        if (q != diag) sum += finish(sums[q].h);
#pragma unroll
      for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(kAll, sum, o);
      for (int q = lane; q < m; q += 32) {
        const TO h = q == diag ? (TO)(-sum) : (TO)finish(sums[q].h);
        aval[2 * (at + q)] = h;
        aval[2 * (at + q) + 1] = (TO)finish(sums[q].m);
        hf32[at + q] = (float)h;
      }
      if (lane == 0) hdiag[k] = (float)(TO)(-sum);
    }
    __syncwarp();
  }
}

__global__ void k_round_f32(const double* __restrict__ x, float* __restrict__ y, long long m) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < m) y[t] = (float)x[t];
}

// x = h + l with h = fl32(x), l = fl32(x - h): the double-float split
__global__ void k_split_df(const double* __restrict__ x, float2* __restrict__ y, long long m) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < m) {
    const float h = (float)x[t];
    y[t] = make_float2(h, (float)(x[t] - (double)h));
  }
}

}  // namespace

void finish_matrices(ff_ctx* c);

void check_material(const DevFlags& f) {
  if (f.code == FF_ERR_INVALID_ARG)
    throw Error(FF_ERR_INVALID_ARG, "invalid material (need E > 0, 0 <= nu < 0.5) at point " +
                                        std::to_string(f.index));
}

// v_i (lambda_i + 4 mu_i) per quadrature point into wh (double-float pairs in
// FP64 contexts, FP32 otherwise)
void material_weights(ff_ctx* c, const float* E, const float* nu, double E0, double nu0,
                      void* wh) {
  cudaStream_t st = c->stream;
  const long long nq = c->nq;
  const int T = 256;
  const int* qperm = c->twoset ? nullptr : c->perm.as<int>();
  reset_flags(c);
  if (!tables_f32(c))
    (k_material<dfloat><<<ceil_div(nq, T), T, 0, st>>>(qperm, nq, c->vol.as<float>(), E, nu, E0,
                                                     nu0, static_cast<dfloat*>(wh),
                                                     c->flags.as<DevFlags>()),
     ::ff::note_launch());
  else
    (k_material<float><<<ceil_div(nq, T), T, 0, st>>>(qperm, nq, c->vol.as<float>(), E, nu, E0,
                                                    nu0, static_cast<float*>(wh),
                                                    c->flags.as<DevFlags>()),
     ::ff::note_launch());
  FF_LAUNCH_CHECK();
}

void build_matrices(ff_ctx* c, const float* E, const float* nu, double E0, double nu0) {
  cudaStream_t st = c->stream;
  const long long n = c->n, n1 = c->n1, nq = c->nq;
  const int T = 256;
  const bool f64 = c->prec == FF_PREC_FP64;
  const bool tdf = !tables_f32(c);  // double-float tables, weights and sums
  const size_t tb = f64 ? 8 : 4;
  DevFlags f{};
  // material weights per quadrature point (the nodal points are in cell
  // order, the two-set quadrature points in the caller's)
  material_weights(c, E, nu, E0, nu0, c->wh.ensure((tdf ? 8 : 4) * nq));
  if (c->twoset && tset_assembly_fits(n)) {
    // two-set clouds: dense tiles of points grouped by their nearest centre
    f = read_flags(c);
    check_material(f);
    tset_assemble(c);
    finish_matrices(c);
    return;
  }
  int* cnt = reinterpret_cast<int*>(c->scratch[5].ensure(sizeof(int) * (n + 1)));
  const long long* ptr = c->nbr_ptr.as<long long>();
  const int* idx = c->nbr_idx.as<int>();
  const long long* tptr = c->nbrT_ptr.as<long long>();
  const int* tidx = c->nbrT_idx.as<int>();
  const long long* tpos = c->nbrT_pos.as<long long>();
  const float* vol = c->vol.as<float>();
  ProfScope ps_pattern(kProfPattern);
  // nodal clouds in tiles of rows; the rows of tiles beyond tile_cap (wide supports,
  // clouds of very uneven density) take the row-owner passes below
  const int ntiles = c->twoset ? 0 : (int)ceil_div(n, kTileRows);
  TileMax tmax{};
  unsigned char* wide = nullptr;  // null: every row is the row-owner passes'
  if (ntiles > 0) {
    TileMax* dmax = reinterpret_cast<TileMax*>(c->scratch[6].ensure(sizeof(TileMax) + ntiles));
    wide = reinterpret_cast<unsigned char*>(dmax + 1);
    FF_CUDA(cudaMemsetAsync(dmax, 0, sizeof(TileMax), st));
    const TileDims cap = tile_cap(tdf ? 8 : 4);
    const int smem = TileSmem(cap, 0, 4).total;
    set_max_dyn_smem((const void*)k_tile_rows<0, float, float>, smem);
    (k_tile_rows<0, float, float><<<ntiles, kTileT, smem, st>>>(
         ptr, idx, tptr, tidx, tpos, nullptr, nullptr, n1, vol, nullptr, n, cap, cnt, dmax,
         nullptr, nullptr, nullptr, nullptr, nullptr, wide),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    FF_CUDA(cudaMemcpyAsync(&tmax, dmax, sizeof(TileMax), cudaMemcpyDeviceToHost, st));
    f = read_flags(c);
    check_material(f);
  }
  const bool tiles = tmax.wide < ntiles, owners = tmax.wide > 0 || !wide;
  // row-owner pass 1: unique columns per row, in a table of 2048 slots per warp
  // (4 warps per block); clouds of uneven density (wide supports reaching into
  // dense regions) retry with 16384 slots per warp (2 warps per block)
  for (int attempt = 0; owners && attempt < 2; ++attempt) {
    const int tsize1 = attempt == 0 ? 2048 : 16384;
    const int wpb1 = attempt == 0 ? 4 : 2;
    const size_t smem1 = sizeof(int) * tsize1 * wpb1;
    if (smem1 > 48 * 1024) set_max_dyn_smem((const void*)k_pattern_count, (int)smem1);
    if (attempt > 0) reset_flags(c);
    int grid1 = (int)std::min<long long>(ceil_div(n, wpb1), (long long)sm_count() * 16);
    (k_pattern_count<<<grid1, 32 * wpb1, smem1, st>>>(ptr, idx, tptr, tidx, n, tsize1, cnt, wide,
                                                     c->flags.as<DevFlags>()),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    f = read_flags(c);
    const bool overflow =
        f.code == FF_ERR_INVALID_ARG && f.max_row > 0 && f.max_row * 2 > tsize1;
    if (!overflow) break;
    if (attempt == 1)
      throw Error(FF_ERR_INVALID_ARG, "a Hessian row has more than " + std::to_string(tsize1 / 2) +
                                          " distinct columns (support too large)");
  }
  ps_pattern.close();
  check_material(f);
  long long* aptr = reinterpret_cast<long long*>(c->a_ptr.ensure(sizeof(long long) * (n + 1)));
  scan_counts(cnt, aptr, n, c, c->scratch[3]);
  long long n2 = 0;
  FF_CUDA(cudaMemcpyAsync(&n2, aptr + n, sizeof(long long), cudaMemcpyDeviceToHost, st));
  FF_CUDA(cudaStreamSynchronize(st));
  c->n2 = n2;
  int* acol = reinterpret_cast<int*>(c->a_col.ensure(sizeof(int) * n2));
  c->a_val.ensure(2 * tb * n2);
  float* hf32 = reinterpret_cast<float*>(c->h_f32.ensure(sizeof(float) * n2));
  float* hdiag = reinterpret_cast<float*>(c->hdiag_f32.ensure(sizeof(float) * n));
  ProfScope ps_values(kProfAsmValues);
  auto values = [&](auto ttag, auto totag) {
    using TT = decltype(ttag);
    using TO = decltype(totag);
    const TT *phi = c->phi.as<TT>(), *dphi = c->dphi.as<TT>(), *wh = c->wh.as<TT>();
    TO* aval = c->a_val.as<TO>();
    if (tiles) {
      auto slots = [](int m) {
        int t = 64;
        while (t < 2 * m) t <<= 1;
        return t;
      };
      auto up = [](int m) { return (m + 7) & ~7; };
      const TileDims d{up(tmax.pts), up(tmax.cols), up(tmax.pairs), up(tmax.row),
                       slots(tmax.pts), slots(tmax.cols)};
      const int smem = TileSmem(d, 1, (int)sizeof(TT)).total;
      set_max_dyn_smem((const void*)k_tile_rows<1, TT, TO>, smem);
      (k_tile_rows<1, TT, TO><<<ntiles, kTileT, smem, st>>>(
           ptr, idx, tptr, tidx, tpos, phi, dphi, n1, vol, wh, n, d, nullptr, nullptr, aptr, acol,
           aval, hf32, hdiag, wide),
       ::ff::note_launch());
      FF_LAUNCH_CHECK();
    }
    if (!owners) return;
    const int maxrow = std::max(f.max_row, 1);
    int tsize2 = 64;
    while (tsize2 < 2 * maxrow) tsize2 <<= 1;
    const size_t pw = assemble_smem_per_warp(tsize2, maxrow, sizeof(TT));
    const int wpb2 = (int)std::max<size_t>(1, std::min<size_t>(8, (96 * 1024) / pw));
    const size_t smem = pw * wpb2;
    const int grid2 = (int)std::min<long long>(ceil_div(n, wpb2), (long long)sm_count() * 32);
    set_max_dyn_smem((const void*)k_assemble<TT, TO>, (int)std::max<size_t>(smem, 48 * 1024));
    (k_assemble<TT, TO><<<grid2, 32 * wpb2, smem, st>>>(ptr, idx, tptr, tidx, tpos, phi, dphi, n1,
                                                       vol, wh, n, tsize2, maxrow, aptr, acol,
                                                       aval, hf32, hdiag, wide),
     ::ff::note_launch());
  };
  if (f64 && !tdf)  // FP32 tables and sums, FP64 storage
    values(float{}, double{});
  else if (f64)
    values(dfloat{}, double{});
  else
    values(float{}, float{});
  FF_LAUNCH_CHECK();
  ps_values.close();
  finish_matrices(c);
}

// the copies of (H, M) the eigensolver reads besides the stored values, and
// the preconditioner's tensor-core tiles
void finish_matrices(ff_ctx* c) {
  cudaStream_t st = c->stream;
  const long long n2 = c->n2;
  const bool f64 = c->prec == FF_PREC_FP64;
  if (f64) {  // FP32 rounding of (H, M) for the FP32 phase of the eigensolver
    float* v32 = reinterpret_cast<float*>(c->a_val32.ensure(2 * sizeof(float) * n2));
    const long long m = 2 * n2;
    (k_round_f32<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(c->a_val.as<double>(), v32, m),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
    // and the double-float split for its second phase
    float2* vdf = reinterpret_cast<float2*>(c->a_valdf.ensure(2 * sizeof(float2) * n2));
    (k_split_df<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(c->a_val.as<double>(), vdf, m),
     ::ff::note_launch());
    FF_LAUNCH_CHECK();
  }
  cheb_tc_build(c);
  FF_CUDA(cudaStreamSynchronize(st));
}

}  // namespace ff
