// Batched dense kernels: the ragged GEMV that carries every local and coarse solve of the
// preconditioner apply (arXiv 2606.01433, Section 2.1/2.2: the A_i^{-1} terms, applied as
// block-LDU sweeps with explicit inverse diagonal blocks), and the set-up kernels that
// build those factors: a batched GEMM and a batched blocked Gauss-Jordan inverse with
// partial pivoting.
#include <cooperative_groups.h>

#include <cfloat>

#include "common.h"
#include "kernels.h"

namespace gdsw {

// ------------------------------------------------------------------ load helpers
template <typename T> struct Vec16;
template <> struct Vec16<double> { static constexpr int N = 2; };
template <> struct Vec16<float> { static constexpr int N = 4; };
template <> struct Vec16<__nv_bfloat16> { static constexpr int N = 8; };

__device__ __forceinline__ void load16(const double* p, double* v) {
  double2 t = __ldg(reinterpret_cast<const double2*>(p));
  v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void load16(const float* p, float* v) {
  float4 t = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load16(const __nv_bfloat16* p, float* v) {
  uint4 t = __ldg(reinterpret_cast<const uint4*>(p));
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&t);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float2 f = __bfloat1622float2(h[q]);
    v[2 * q] = f.x; v[2 * q + 1] = f.y;
  }
}
// streaming (evict-first) variant for matrices read once per apply
__device__ __forceinline__ void load16s(const double* p, double* v) {
  double2 t = __ldcs(reinterpret_cast<const double2*>(p));
  v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void load16s(const float* p, float* v) {
  float4 t = __ldcs(reinterpret_cast<const float4*>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load16s(const __nv_bfloat16* p, float* v) {
  uint4 t = __ldcs(reinterpret_cast<const uint4*>(p));
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&t);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float2 f = __bfloat1622float2(h[q]);
    v[2 * q] = f.x; v[2 * q + 1] = f.y;
  }
}

// ------------------------------------------------------------------ overlapped launch chain
// The local sweeps are chains of launches: each slab step reads the vectors the previous one
// wrote.  Each launch of the chain is a programmatic dependent launch (common.h): its CTAs may
// become resident while the previous launch drains its last wave, prefetch the start of their
// factor rows into L2 (the factors do not depend on the previous launch), and wait for the
// previous grid before reading a vector.
bool g_launch_overlap = true;

// raw 16-byte streaming load, unpacked only at the multiply (keeps BF16 tiles at half the
// registers of unpacked floats)
__device__ __forceinline__ uint4 ldraw(const void* p) { return __ldcs(reinterpret_cast<const uint4*>(p)); }
template <typename TM> struct Unpack;
template <> struct Unpack<double> {
  static __device__ __forceinline__ void run(const uint4& r, double* v) {
    v[0] = __hiloint2double(int(r.y), int(r.x));
    v[1] = __hiloint2double(int(r.w), int(r.z));
  }
};
template <> struct Unpack<float> {
  static __device__ __forceinline__ void run(const uint4& r, float* v) {
    v[0] = __uint_as_float(r.x); v[1] = __uint_as_float(r.y); v[2] = __uint_as_float(r.z); v[3] = __uint_as_float(r.w);
  }
};
template <> struct Unpack<__nv_bfloat16> {
  static __device__ __forceinline__ void run(const uint4& r, float* v) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float2 f = __bfloat1622float2(h[q]);
      v[2 * q] = f.x; v[2 * q + 1] = f.y;
    }
  }
};

// ------------------------------------------------------------------ sums over a warp
// Sums N (a power of two) values per lane over the warp, N of them at once: in each of the first log2 N
// steps a lane hands half of its values to its partner and keeps the other half, then one value is
// left per lane.  Lane l returns the sum of value N l / 32.  N + 4 - log2 N additions instead of 5 N --
// FP64 rows of 600 entries spent a fifth of their instructions there -- and every sum is formed in the
// order of a butterfly over lane distances 16, 8, 4, 2, 1, whatever N.  With tiles of 16 rows: FP64 apply
// of an 8^3 box in 8 parts 163 -> 135 us, with discontinuous pressure on a larger one 510 -> 446 us.
template <int N, typename T>
__device__ __forceinline__ T warp_sums(T (&a)[N], int lane) {
  int o = 16;
#pragma unroll
  for (int h = N / 2; h > 0; h /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < h; ++k) a[k] = (up ? a[k + h] : a[k]) + __shfl_xor_sync(0xffffffffu, up ? a[k] : a[k + h], o);
  }
#pragma unroll
  for (; o > 0; o /= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
  return a[0];
}

// ------------------------------------------------------------------ ragged batched GEMV
// One CTA = 8 warps = ROWS rows of one task; each warp owns ROWS/8 rows and streams them
// with 16-byte loads (four rows in flight per warp).  The task's input vector is staged in
// shared memory once per CTA.  y[r] = base[r] + alpha * sum_c M[r][c] x[c].
// Symmetric block stored as its upper-triangle tiles (T x T, T = 32 lanes x one 16-byte load,
// tiles (I, J >= I) in row-major order, zero padded): one CTA reads tile (I, J) once and
// produces both S_IJ x_J (rows of block I) and, off the diagonal, S_IJ^T x_I (rows of block
// J) as partial sums; k_sym_reduce adds the partials of each row in a fixed order.
template <typename TM, typename TV>
__device__ __forceinline__ void sym_tile(const TM* __restrict__ M, const TV* xbase, TV* part, const GemvTask& t,
                                         int I, int J, TV* smem) {
  constexpr int V = Vec16<TM>::N, T = 32 * V, RW = T / 8;
  TV* xi = smem;
  TV* xj = smem + T;
  TV* prow = smem + 2 * T;
  TV* pcol = smem + 3 * T;  // 8 x T
  const int s = t.rows, nt = t.ld;
  for (int e = threadIdx.x; e < T; e += blockDim.x) {
    xi[e] = I * T + e < s ? __ldcg(xbase + t.x + I * T + e) : TV(0);
    xj[e] = J * T + e < s ? __ldcg(xbase + t.x + J * T + e) : TV(0);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tidx = int64_t(I) * nt - int64_t(I) * (I - 1) / 2 + (J - I);
  const TM* tp = M + t.mat + tidx * T * T + int64_t(warp * RW) * T + lane * V;
  TV colacc[V], rowacc[RW];
#pragma unroll
  for (int u = 0; u < V; ++u) colacc[u] = TV(0);
#pragma unroll
  for (int rr = 0; rr < RW; rr += 4) {
    TV v[4][V];
#pragma unroll
    for (int q = 0; q < 4; ++q) load16s(tp + int64_t(rr + q) * T, v[q]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const TV xr = xi[warp * RW + rr + q];
      TV d = TV(0);
#pragma unroll
      for (int u = 0; u < V; ++u) {
        d = fma(v[q][u], xj[lane * V + u], d);
        colacc[u] = fma(v[q][u], xr, colacc[u]);
      }
      rowacc[rr + q] = d;
    }
  }
#pragma unroll
  for (int rr = 0; rr < RW; rr += 8) {
    TV part8[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) part8[q] = rowacc[rr + q];
    const TV d = warp_sums<8>(part8, lane);
    if (lane % 4 == 0) prow[warp * RW + rr + lane / 4] = d;
  }
#pragma unroll
  for (int u = 0; u < V; ++u) pcol[warp * T + lane * V + u] = colacc[u];
  __syncthreads();
  for (int e = threadIdx.x; e < T; e += blockDim.x) {
    part[t.part + (int64_t(I) * nt + J) * T + e] = prow[e];
    if (I != J) {
      TV cs = pcol[e];
#pragma unroll
      for (int w = 1; w < 8; ++w) cs += pcol[w * T + e];
      part[t.part + (int64_t(J) * nt + I) * T + e] = cs;
    }
  }
}

// Rows [row0, row0 + 8 RPW G) of one task: G consecutive groups of 8 RPW rows share one
// staging of the input vector, and every row is one warp's dot product in the same order
// whatever G is.  Vector reads go through L2 (ld.global.cg): in the persistent sweep other
// CTAs write the local vectors while this one runs.
template <typename TM, typename TV, int RPW, int G>
__device__ __forceinline__ void rows_tile(const TM* __restrict__ M, const TV* xbase, TV* ybase, const TV* bbase,
                                          const GemvTask& t, int row0, TV* xs) {
  const int ld = t.ld;
  for (int c = threadIdx.x; c < ld; c += blockDim.x) xs[c] = c < t.cols ? __ldcg(xbase + t.x + c) : TV(0);
  __syncthreads();
  constexpr int V = Vec16<TM>::N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int g = 0; g < G; ++g) {  // G is a compile-time constant: a runtime count here slows the loads
    const int rbeg = row0 + g * 8 * RPW + warp * RPW;
    if (rbeg - warp * RPW >= t.rows) break;
    TV acc[RPW];
    const TM* rowp[RPW];
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
      acc[q] = TV(0);
      int r = rbeg + q;
      rowp[q] = M + t.mat + int64_t(r < t.rows ? r : 0) * ld;
    }
    int c = lane * V;
    for (; c + 32 * V < ld; c += 64 * V) {  // two column chunks per row in flight
      uint4 m0[RPW], m1[RPW];
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        if (rbeg + q < t.rows) {
          m0[q] = ldraw(rowp[q] + c);
          m1[q] = ldraw(rowp[q] + c + 32 * V);
        }
      }
      TV xv0[V], xv1[V];
#pragma unroll
      for (int u = 0; u < V; ++u) {
        xv0[u] = xs[c + u];
        xv1[u] = xs[c + 32 * V + u];
      }
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        if (rbeg + q < t.rows) {
          TV mv0[V], mv1[V];
          Unpack<TM>::run(m0[q], mv0);
          Unpack<TM>::run(m1[q], mv1);
#pragma unroll
          for (int u = 0; u < V; ++u) acc[q] = fma(mv1[u], xv1[u], fma(mv0[u], xv0[u], acc[q]));
        }
      }
    }
    if (c < ld) {
      TV xv[V];
#pragma unroll
      for (int u = 0; u < V; ++u) xv[u] = xs[c + u];
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        if (rbeg + q < t.rows) {
          TV mv[V];
          load16s(rowp[q] + c, mv);
#pragma unroll
          for (int u = 0; u < V; ++u) acc[q] = fma(mv[u], xv[u], acc[q]);
        }
      }
    }
    const TV a = warp_sums<RPW>(acc, lane);
    if (lane % (32 / RPW) == 0) {
      const int r = rbeg + lane / (32 / RPW);
      if (r < t.rows) {
        TV v = TV(t.alpha) * a;
        if (t.base >= 0) v += __ldcg(bbase + t.base + r);
        ybase[t.y + r] = v;
      }
    }
  }
}

template <typename TM, typename TV, int RPW, int G>
__global__ void __launch_bounds__(256) k_gemv(const TM* __restrict__ M, const TV* xbase, TV* ybase,
                                              const TV* bbase, const GemvTask* __restrict__ tasks,
                                              const GemvTile* __restrict__ tiles) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TV* xs = reinterpret_cast<TV*>(smem_raw);
  const GemvTile tl = tiles[blockIdx.x];
  const GemvTask t = tasks[tl.task];
  dep_release();
  {  // factor prefetch before the dependency wait: the first 2 KB of the warp's first rows, or
     // the first eight rows of the warp's part of a symmetric tile
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (t.kind == 1) {
      constexpr int T = 32 * Vec16<TM>::N, RW = T / 8;
      const int I = tl.row0 >> 16, J = tl.row0 & 0xffff;
      const int64_t tidx = int64_t(I) * t.ld - int64_t(I) * (I - 1) / 2 + (J - I);
      prefetch_l2(M + t.mat + tidx * T * T + int64_t(warp * RW + (lane >> 2)) * T + (lane & 3) * (128 / sizeof(TM)));
    } else {
      for (int q = lane >> 4; q < RPW; q += 2) {
        const int r = tl.row0 + warp * RPW + q;
        const int off = (lane & 15) * int(128 / sizeof(TM));
        if (r < t.rows && off < t.ld) prefetch_l2(M + t.mat + int64_t(r) * t.ld + off);
      }
    }
  }
  dep_wait();
  if (t.kind == 1)  // packed symmetric tile; partial sums go to ybase + t.part
    sym_tile<TM, TV>(M, xbase, ybase, t, tl.row0 >> 16, tl.row0 & 0xffff, xs);
  else
    rows_tile<TM, TV, RPW, G>(M, xbase, ybase, bbase, t, tl.row0, xs);
}

// ------------------------------------------------------------------ ragged batched GEMV, transposed
// y[c] = base[c] + alpha * sum_r M[r][c] x[r] for the columns [col0, col0 + LW V) of a task
// (used with the sub-diagonal blocks G of a symmetric LDL^T factorisation, whose
// transposes are the super-diagonal blocks).  A group of LW lanes reads one row of the tile
// (a lane owns V consecutive columns, one 16-byte load); the 256 / LW groups split the rows,
// four rows in flight each; the partial sums of a column are combined in shared memory in a
// fixed order.  Narrow tiles (LW V columns) give many CTAs per task, so the ragged launch
// (tasks of different heights) spreads evenly over the SMs.
// lanes per tile row of the transposed GEMV: half warps
template <typename TM> struct ColsLanes { static constexpr int LW = 16; };

template <typename TM, typename TV>
__device__ __forceinline__ void cols_tile(const TM* __restrict__ M, const TV* xbase, TV* ybase, const TV* bbase,
                                          const GemvTask& t, int col0, TV* xs, TV* part) {
  constexpr int V = Vec16<TM>::N, LW = ColsLanes<TM>::LW, C = LW * V, NG = 256 / LW;
  for (int r = threadIdx.x; r < t.rows; r += blockDim.x) xs[r] = __ldcg(xbase + t.x + r);
  __syncthreads();
  const int ll = threadIdx.x % LW, grp = threadIdx.x / LW;  // NG row groups of LW lanes
  const int c0 = col0 + ll * V;  // tile column start + this lane's V columns
  TV acc[V];
#pragma unroll
  for (int u = 0; u < V; ++u) acc[u] = TV(0);
  if (c0 < t.ld) {
    const TM* p = M + t.mat + c0;
    int r = grp;
    for (; r + 3 * NG < t.rows; r += 4 * NG) {
      TV v[4][V];
#pragma unroll
      for (int q = 0; q < 4; ++q) load16s(p + int64_t(r + NG * q) * t.ld, v[q]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const TV xq = xs[r + NG * q];
#pragma unroll
        for (int u = 0; u < V; ++u) acc[u] = fma(v[q][u], xq, acc[u]);
      }
    }
    for (; r < t.rows; r += NG) {
      TV v0[V];
      load16s(p + int64_t(r) * t.ld, v0);
      const TV x0 = xs[r];
#pragma unroll
      for (int u = 0; u < V; ++u) acc[u] = fma(v0[u], x0, acc[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < V; ++u) part[grp * (C + 1) + ll * V + u] = acc[u];
  __syncthreads();
  for (int cc = threadIdx.x; cc < C; cc += blockDim.x) {
    const int c = col0 + cc;
    if (c < t.cols) {
      TV s = part[cc];
#pragma unroll
      for (int g = 1; g < NG; ++g) s += part[g * (C + 1) + cc];
      TV v = TV(t.alpha) * s;
      if (t.base >= 0) v += __ldcg(bbase + t.base + c);
      ybase[t.y + c] = v;
    }
  }
}

template <typename TM, typename TV>
__global__ void __launch_bounds__(256) k_gemvt(const TM* __restrict__ M, const TV* xbase, TV* ybase,
                                               const TV* bbase, const GemvTask* __restrict__ tasks,
                                               const GemvTile* __restrict__ tiles) {
  constexpr int LW = ColsLanes<TM>::LW, C = LW * Vec16<TM>::N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ TV part[(256 / LW) * (C + 1)];
  const GemvTile tl = tiles[blockIdx.x];
  const GemvTask t = tasks[tl.task];
  dep_release();
  {  // factor prefetch before the dependency wait: the tile's first 128 rows (two lines each)
    const int r = threadIdx.x >> 1, off = tl.row0 + (threadIdx.x & 1) * int(128 / sizeof(TM));
    if (r < t.rows && off < t.ld) prefetch_l2(M + t.mat + int64_t(r) * t.ld + off);
  }
  dep_wait();
  cols_tile<TM, TV>(M, xbase, ybase, bbase, t, tl.row0, reinterpret_cast<TV*>(smem_raw), part);
}

template <typename TM, typename TV>
void launch_gemv(const TM* M, const TV* x, TV* y, const TV* b, const GemvPlan& P, int launch, int max_ld,
                 cudaStream_t s) {
  int t0 = P.launch_tile_off[launch], t1 = P.launch_tile_off[launch + 1];
  if (t1 <= t0) return;
  size_t smem = size_t(max_ld) * sizeof(TV);
  const unsigned nb = unsigned(t1 - t0);
  const GemvTile* tl = P.d_tiles + t0;
  if (P.transposed) {
    launch_chained(k_gemvt<TM, TV>, dim3(nb), dim3(256), smem, s, M, x, y, b, P.d_tasks, tl);
    check_launch("k_gemvt");
  } else {
    if (P.rows_per_tile == 16)
      launch_chained(k_gemv<TM, TV, 2, 1>, dim3(nb), dim3(256), smem, s, M, x, y, b, P.d_tasks, tl);
    else if (P.rows_per_tile == 128)
      launch_chained(k_gemv<TM, TV, 4, 4>, dim3(nb), dim3(256), smem, s, M, x, y, b, P.d_tasks, tl);
    else if (P.rows_per_tile == 64)
      launch_chained(k_gemv<TM, TV, 4, 2>, dim3(nb), dim3(256), smem, s, M, x, y, b, P.d_tasks, tl);
    else
      launch_chained(k_gemv<TM, TV, 4, 1>, dim3(nb), dim3(256), smem, s, M, x, y, b, P.d_tasks, tl);
    check_launch("k_gemv");
  }
}

// y[r] = alpha * sum over the nt source blocks of the partials of row r (fixed order);
// one CTA per 256 rows of one symmetric task.
template <typename TV>
__device__ __forceinline__ void reduce_tile(const TV* vec, TV* ybase, const GemvTask& t, int row0, int T) {
  const int r = row0 + threadIdx.x;
  if (r >= t.rows) return;
  const int R = r / T, e = r - R * T;
  const TV* p = vec + t.part + int64_t(R) * t.ld * T + e;
  TV s = TV(0);
  for (int S = 0; S < t.ld; ++S) s += __ldcg(p + int64_t(S) * T);
  ybase[t.y + r] = TV(t.alpha) * s;
}

template <typename TV>
__global__ void k_sym_reduce(const TV* __restrict__ vec, TV* ybase, const GemvTask* __restrict__ tasks,
                             const GemvTile* __restrict__ tiles, int T) {
  const GemvTile tl = tiles[blockIdx.x];
  const GemvTask t = tasks[tl.task];
  dep_release();
  dep_wait();
  reduce_tile<TV>(vec, ybase, t, tl.row0, T);
}

template <typename TV>
void launch_sym_reduce(const TV* vec, TV* y, const GemvPlan& P, int T, cudaStream_t s) {
  int t0 = P.launch_tile_off[0], t1 = P.launch_tile_off[1];
  if (t1 <= t0) return;
  launch_chained(k_sym_reduce<TV>, dim3(unsigned(t1 - t0)), dim3(256), 0, s, vec, y, P.d_tasks, P.d_tiles + t0, T);
  check_launch("k_sym_reduce");
}
template void launch_sym_reduce<double>(const double*, double*, const GemvPlan&, int, cudaStream_t);
template void launch_sym_reduce<float>(const float*, float*, const GemvPlan&, int, cudaStream_t);

// ------------------------------------------------------------------ couplings of a condensed set
// y[rows] -= C w for the couplings between mid layers and slabs (y, w: the two local vectors): eight
// lanes per block of rows, whose rows share their columns (5.3 bytes an entry instead of 8).  A
// block has about 110 columns: whole warps spent as long on the butterflies as on the products in
// FP64, and eight lanes still read whole 32-byte sectors in FP32.  FP32: 24 us on a 20^3 box in 64 parts
// (70 MB), 28 us on the die, 60 us on the 32^3 channel; FP64: 29 us on 135 thousand local dofs.
template <typename TV>
__global__ void __launch_bounds__(256) k_coupling(int nblk, const int32_t* __restrict__ row,
                                                  const int32_t* __restrict__ nrow, const int64_t* __restrict__ off,
                                                  const int64_t* __restrict__ voff, const int32_t* __restrict__ col,
                                                  const TV* __restrict__ val, TV* y, const TV* w) {
  const int64_t b = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) / 8;
  const int lane = threadIdx.x & 7;
  dep_release();
  const bool in = b < nblk;
  const int64_t o = in ? off[b] : 0;
  const int n = in ? int(off[b + 1] - o) : 0, nr = in ? nrow[b] : 0, r0 = in ? row[b] : 0;
  const TV* v = val + (in ? voff[b] : 0);
  dep_wait();
  TV acc[3] = {TV(0), TV(0), TV(0)};
  if (nr == 3) {
#pragma unroll 4
    for (int j = lane; j < n; j += 8) {
      const TV x = __ldcg(w + col[o + j]);
#pragma unroll
      for (int r = 0; r < 3; ++r) acc[r] = fma(v[r * n + j], x, acc[r]);
    }
  } else {
#pragma unroll 4
    for (int j = lane; j < n; j += 8) acc[0] = fma(v[j], __ldcg(w + col[o + j]), acc[0]);
  }
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], d);
  if (lane < nr) y[r0 + lane] -= lane == 0 ? acc[0] : (lane == 1 ? acc[1] : acc[2]);
}

template <typename TV>
void launch_coupling(const Coupling& C, TV* vec, int64_t nvec, cudaStream_t s) {
  if (C.nblk == 0) return;
  launch_chained(k_coupling<TV>, dim3(unsigned((int64_t(C.nblk) * 8 + 255) / 256)), dim3(256), 0, s, C.nblk, C.row,
                 C.nrow, C.off, C.voff, C.col, static_cast<const TV*>(C.val), vec, vec + nvec);
  check_launch("k_coupling");
}
template void launch_coupling<double>(const Coupling&, double*, int64_t, cudaStream_t);
template void launch_coupling<float>(const Coupling&, float*, int64_t, cudaStream_t);

// ------------------------------------------------------------------ persistent level sweep
// One launch runs every tile of a level's local solves -- forward row tiles and packed
// symmetric tiles, the partial-sum reductions, the transposed backward tiles -- from a work
// list in dependency order.  CTAs claim items with an atomic counter (the next claim is made
// before the current item runs).  An item first waits until the per-slab counters of the
// tiles it reads from are complete (y_k written, partials written, w_k written, x_k
// written), runs, then adds one to its own counter.  Claims follow list order and every
// producer precedes its consumers in the list, so the lowest unfinished claimed item always
// has its producers finished: the sweep cannot deadlock, whatever the number of resident
// CTAs.  A wait longer than limit_ns sets *flag and every CTA returns; the host reports it.
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool wait_count(const unsigned* cnt, unsigned need, unsigned* flag,
                                           unsigned long long limit_ns) {
  const volatile unsigned* c = cnt;
  if (*c >= need) return true;
  const unsigned long long t_end = global_ns() + limit_ns;
  while (*c < need) {
    if (*reinterpret_cast<volatile unsigned*>(flag)) return false;
    if (global_ns() > t_end) {
      atomicExch(flag, 1u);
      return false;
    }
    __nanosleep(64);
  }
  return true;
}

template <typename TM, typename TV, int RPW, int G>
__global__ void __launch_bounds__(256, 3) k_sweep(const TM* __restrict__ M, TV* vec, const GemvTask* __restrict__ tasks,
                                               const SweepItem* __restrict__ items, int nitems, unsigned* ctr,
                                               unsigned* flag, int T, int xs_elems, unsigned long long limit_ns) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TV* xs = reinterpret_cast<TV*>(smem_raw);
  TV* cpart = xs + xs_elems;  // column partials of the transposed tiles
  __shared__ int s_item[2];
  __shared__ int s_ok;
  if (threadIdx.x == 0) s_item[0] = int(atomicAdd(ctr, 1u));
  __syncthreads();
  int cur = 0;
  while (true) {
    const int it = s_item[cur];
    if (it >= nitems) break;
    const SweepItem w = items[it];
    if (threadIdx.x == 0) {
      s_item[cur ^ 1] = int(atomicAdd(ctr, 1u));
      bool ok = true;
      if (w.wait0 >= 0) ok = wait_count(ctr + w.wait0, unsigned(w.need0), flag, limit_ns);
      if (ok && w.wait1 >= 0) ok = wait_count(ctr + w.wait1, unsigned(w.need1), flag, limit_ns);
      __threadfence();
      s_ok = ok ? 1 : 0;
    }
    __syncthreads();
    if (!s_ok) break;
    const GemvTask t = tasks[w.task];
    if (w.op == SWEEP_ROWS)
      rows_tile<TM, TV, RPW, G>(M, vec, vec, vec, t, w.arg, xs);
    else if (w.op == SWEEP_SYM)
      sym_tile<TM, TV>(M, vec, vec, t, w.arg >> 16, w.arg & 0xffff, xs);
    else if (w.op == SWEEP_REDUCE)
      reduce_tile<TV>(vec, vec, t, w.arg, T);
    else
      cols_tile<TM, TV>(M, vec, vec, vec, t, w.arg, xs, cpart);
    __syncthreads();  // every write of this item is issued; the shared staging is free again
    if (threadIdx.x == 0 && w.signal >= 0) {
      __threadfence();
      atomicAdd(ctr + w.signal, 1u);
    }
    cur ^= 1;
  }
}

// the persistent sweep with `rows` rows per forward tile
template <typename TM, typename TV, typename F>
static void sweep_form(int rows, F f) {
  if (rows == 16)
    f(k_sweep<TM, TV, 2, 1>);
  else if (rows == 64)
    f(k_sweep<TM, TV, 4, 2>);
  else if (rows == 128)
    f(k_sweep<TM, TV, 4, 4>);
  else
    f(k_sweep<TM, TV, 4, 1>);
}

template <typename TM, typename TV>
void size_sweep(SweepPlan& P) {
  constexpr int LW = ColsLanes<TM>::LW, C = LW * Vec16<TM>::N;
  P.smem = (size_t(P.xs_elems) + (256 / LW) * (C + 1)) * sizeof(TV);
  GDSW_CHECK(P.smem <= size_t(200) * 1024, GDSW_ERR_INVALID_ARG, "persistent sweep: staging exceeds shared memory");
  // one limit for every level's launch of this instantiation (the attribute is per kernel)
  int per_sm = 0, dev = 0, nsm = 0;
  sweep_form<TM, TV>(P.rows, [&](auto kernel) {
    GDSW_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    GDSW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, P.smem));
  });
  GDSW_CUDA(cudaGetDevice(&dev));
  GDSW_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  GDSW_CHECK(per_sm > 0, GDSW_ERR_CUDA, "persistent sweep: no CTA fits on an SM");
  P.max_per_sm = per_sm;
  const int want = P.ctas_per_sm > 0 ? std::min(P.ctas_per_sm, per_sm) : per_sm;
  P.grid = int(std::min<int64_t>(int64_t(want) * nsm, P.nitems));
}

template <typename TM, typename TV>
void launch_sweep(const TM* M, TV* vec, const SweepPlan& P, unsigned* flag, int T, cudaStream_t s) {
  if (P.nitems == 0) return;
  GDSW_CUDA(cudaMemsetAsync(P.d_ctr, 0, sizeof(unsigned) * P.nctr, s));
  sweep_form<TM, TV>(P.rows, [&](auto kernel) {
    kernel<<<P.grid, 256, P.smem, s>>>(M, vec, P.d_tasks, P.d_items, P.nitems, P.d_ctr, flag, T, P.xs_elems,
                                       kSweepWaitLimitNs);
  });
  check_launch("k_sweep");
}
template void size_sweep<double, double>(SweepPlan&);
template void size_sweep<float, float>(SweepPlan&);
template void size_sweep<__nv_bfloat16, float>(SweepPlan&);
template void launch_sweep<double, double>(const double*, double*, const SweepPlan&, unsigned*, int, cudaStream_t);
template void launch_sweep<float, float>(const float*, float*, const SweepPlan&, unsigned*, int, cudaStream_t);
template void launch_sweep<__nv_bfloat16, float>(const __nv_bfloat16*, float*, const SweepPlan&, unsigned*, int,
                                                 cudaStream_t);

// copy of T x T tiles out of full row-major blocks, zero padded (packing of the upper triangle)
template <typename T>
__global__ void k_pack_tiles(const T* __restrict__ src, T* __restrict__ dst, const PackTile* __restrict__ tiles,
                             int TT) {
  const PackTile p = tiles[blockIdx.x];
  for (int e = threadIdx.x; e < TT * TT; e += blockDim.x) {
    int r = e / TT, c = e - r * TT;
    dst[p.dst + e] = (r < p.rows && c < p.cols) ? src[p.src + int64_t(r) * p.ld + c] : T(0);
  }
}

template <typename T>
void pack_tiles(DevArena& tmp, const T* src, T* dst, const std::vector<PackTile>& tiles, int TT, cudaStream_t s) {
  if (tiles.empty()) return;
  PackTile* d = tmp.upload(tiles, s);
  for (size_t off = 0; off < tiles.size(); off += (size_t(1) << 30)) {
    int nb = int(std::min<size_t>(tiles.size() - off, size_t(1) << 30));
    k_pack_tiles<T><<<nb, 256, 0, s>>>(src, dst, d + off, TT);
    check_launch("k_pack_tiles");
  }
}
template void pack_tiles<double>(DevArena&, const double*, double*, const std::vector<PackTile>&, int, cudaStream_t);
template void pack_tiles<float>(DevArena&, const float*, float*, const std::vector<PackTile>&, int, cudaStream_t);

template void launch_gemv<double, double>(const double*, const double*, double*, const double*, const GemvPlan&,
                                          int, int, cudaStream_t);
template void launch_gemv<float, float>(const float*, const float*, float*, const float*, const GemvPlan&, int,
                                        int, cudaStream_t);
template void launch_gemv<__nv_bfloat16, float>(const __nv_bfloat16*, const float*, float*, const float*,
                                                const GemvPlan&, int, int, cudaStream_t);

void set_gemv_smem_limits() {
  cudaFuncSetAttribute(k_gemv<double, double, 2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<float, float, 2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<__nv_bfloat16, float, 2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<double, double, 4, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<float, float, 4, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<__nv_bfloat16, float, 4, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<double, double, 4, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<float, float, 4, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<__nv_bfloat16, float, 4, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<double, double, 4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<float, float, 4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemv<__nv_bfloat16, float, 4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_gemvt<double, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 180 * 1024);
  cudaFuncSetAttribute(k_gemvt<float, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 180 * 1024);
  cudaFuncSetAttribute(k_gemvt<__nv_bfloat16, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 180 * 1024);
}

// ------------------------------------------------------------------ batched GEMM (set-up)
// 64x64 output tile per CTA, 256 threads computing 4x4 each, K staged 16 at a time.  Few tiles with
// a long K (the Galerkin products X^T Y: a hundred columns, ten thousand rows) would leave most SMs
// idle -- 8 CTAs took 13.8 ms -- so run_gemm_engine cuts K into gridDim.y slices: raw products go to
// `part` and k_gemm_slices adds them in slice order.
template <typename T>
__global__ void __launch_bounds__(256) k_gemm(const GemmTaskP* __restrict__ tasks, const int32_t* __restrict__ tile_task,
                                              const int32_t* __restrict__ tile_id, T* __restrict__ part) {
  __shared__ T As[16][64 + 1];
  __shared__ T Bs[16][64 + 1];
  const GemmTaskP t = tasks[tile_task[blockIdx.x]];
  const int tiles_n = (t.N + 63) / 64;
  const int tm = tile_id[blockIdx.x] / tiles_n, tn = tile_id[blockIdx.x] % tiles_n;
  const T* A = static_cast<const T*>(t.a);
  const T* B = static_cast<const T*>(t.b);
  T* C = static_cast<T*>(t.c);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int steps = (t.K + 15) / 16, S = gridDim.y;
  const int kbeg = int(int64_t(steps) * blockIdx.y / S) * 16, kend = min(t.K, int(int64_t(steps) * (blockIdx.y + 1) / S) * 16);
  T acc[4][4] = {};
  for (int k0 = kbeg; k0 < kend; k0 += 16) {
    for (int e = threadIdx.x; e < 16 * 64; e += 256) {
      int kk = e / 64, mm = e % 64;
      int gm = tm * 64 + mm, gk = k0 + kk;
      T v = T(0);
      if (gm < t.M && gk < t.K) v = t.ta ? A[int64_t(gk) * t.lda + gm] : A[int64_t(gm) * t.lda + gk];
      As[kk][mm] = v;
      int gn = tn * 64 + mm;
      T w = T(0);
      if (gn < t.N && gk < t.K) w = t.tb ? B[int64_t(gn) * t.ldb + gk] : B[int64_t(gk) * t.ldb + gn];
      Bs[kk][mm] = w;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (S > 1) {
    T* out = part + (int64_t(blockIdx.y) * gridDim.x + blockIdx.x) * 4096;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) out[(ty * 4 + i) * 64 + tx * 4 + j] = acc[i][j];
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int gm = tm * 64 + ty * 4 + i;
    if (gm >= t.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int gn = tn * 64 + tx * 4 + j;
      if (gn >= t.N) continue;
      T* cp = C + int64_t(gm) * t.ldc + gn;
      T v = T(t.alpha) * acc[i][j];
      if (t.beta != 0.0) v += T(t.beta) * *cp;
      *cp = v;
    }
  }
}

// C = alpha (sum of the slices' products) + beta C for the tiles of a sliced k_gemm
template <typename T>
__global__ void __launch_bounds__(256) k_gemm_slices(const GemmTaskP* __restrict__ tasks,
                                                     const int32_t* __restrict__ tile_task,
                                                     const int32_t* __restrict__ tile_id, int S,
                                                     const T* __restrict__ part) {
  const GemmTaskP t = tasks[tile_task[blockIdx.x]];
  const int tiles_n = (t.N + 63) / 64;
  const int tm = tile_id[blockIdx.x] / tiles_n, tn = tile_id[blockIdx.x] % tiles_n;
  const int e = blockIdx.y * 256 + threadIdx.x, gm = tm * 64 + e / 64, gn = tn * 64 + e % 64;
  if (gm >= t.M || gn >= t.N) return;
  T s = T(0);
  for (int k = 0; k < S; ++k) s += part[(int64_t(k) * gridDim.x + blockIdx.x) * 4096 + e];
  T* cp = static_cast<T*>(t.c) + int64_t(gm) * t.ldc + gn;
  T v = T(t.alpha) * s;
  if (t.beta != 0.0) v += T(t.beta) * *cp;
  *cp = v;
}

// ------------------------------------------------------------------ FP32 GEMM tiles
// 128 x 128 outputs per CTA of 256 threads, 8 x 8 per thread (rows ty*4 + {0..3} and
// 64 + ty*4 + {0..3}, columns likewise with tx), K in steps of 16 staged transposed in
// shared memory; the next step's global loads are held in registers while the current
// step is multiplied (one barrier per step).  op(A)(r, k) = ta ? A[k*lda + r] : A[r*lda + k],
// op(B)(k, c) = tb ? B[c*ldb + k] : B[k*ldb + c].
struct GemmOp {
  const float* p;
  int ld, trans;
};

__device__ __forceinline__ void gemm_fetch(const GemmOp& A, const GemmOp& B, int M, int N, int K, int m0, int n0,
                                           int k0, float (&ra)[8], float (&rb)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int e = threadIdx.x + 256 * i;
    int m, k;
    if (A.trans) { k = e >> 7; m = e & 127; } else { m = e >> 4; k = e & 15; }
    const int gm = m0 + m, gk = k0 + k;
    ra[i] = (gm < M && gk < K) ? (A.trans ? A.p[int64_t(gk) * A.ld + gm] : A.p[int64_t(gm) * A.ld + gk]) : 0.f;
    int c, kk;
    if (B.trans) { c = e >> 4; kk = e & 15; } else { kk = e >> 7; c = e & 127; }
    const int gc = n0 + c, gk2 = k0 + kk;
    rb[i] = (gc < N && gk2 < K) ? (B.trans ? B.p[int64_t(gc) * B.ld + gk2] : B.p[int64_t(gk2) * B.ld + gc]) : 0.f;
  }
}

__device__ __forceinline__ void gemm_stash(const GemmOp& A, const GemmOp& B, const float (&ra)[8],
                                           const float (&rb)[8], float (*As)[132], float (*Bs)[132]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int e = threadIdx.x + 256 * i;
    if (A.trans) As[e >> 7][e & 127] = ra[i]; else As[e & 15][e >> 4] = ra[i];
    if (B.trans) Bs[e & 15][e >> 4] = rb[i]; else Bs[e >> 7][e & 127] = rb[i];
  }
}

// acc = op(A)[m0:, :K] op(B)[:K, n0:] for the CTA's 128 x 128 tile
__device__ __forceinline__ void gemm_tile_f32(const GemmOp& A, const GemmOp& B, int M, int N, int K, int m0, int n0,
                                              float (*As)[16][132], float (*Bs)[16][132], float (&acc)[8][8]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  float ra[8], rb[8];
  gemm_fetch(A, B, M, N, K, m0, n0, 0, ra, rb);
  gemm_stash(A, B, ra, rb, As[0], Bs[0]);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += 16) {
    const bool more = k0 + 16 < K;
    if (more) gemm_fetch(A, B, M, N, K, m0, n0, k0 + 16, ra, rb);
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[buf][kk][64 + tx * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) gemm_stash(A, B, ra, rb, As[buf ^ 1], Bs[buf ^ 1]);
    __syncthreads();
    buf ^= 1;
  }
}

__device__ __forceinline__ int gemm_row(int i) { return i < 4 ? (threadIdx.x >> 4) * 4 + i : 64 + (threadIdx.x >> 4) * 4 + i - 4; }
__device__ __forceinline__ int gemm_col(int j) { return j < 4 ? (threadIdx.x & 15) * 4 + j : 64 + (threadIdx.x & 15) * 4 + j - 4; }

__global__ void __launch_bounds__(256, 2) k_gemm_f32(const GemmTaskP* __restrict__ tasks,
                                                  const int32_t* __restrict__ tile_task,
                                                  const int32_t* __restrict__ tile_id) {
  __shared__ __align__(16) float As[2][16][132];
  __shared__ __align__(16) float Bs[2][16][132];
  const GemmTaskP t = tasks[tile_task[blockIdx.x]];
  const int tiles_n = (t.N + 127) / 128;
  const int m0 = (tile_id[blockIdx.x] / tiles_n) * 128, n0 = (tile_id[blockIdx.x] % tiles_n) * 128;
  const GemmOp A{static_cast<const float*>(t.a), t.lda, t.ta};
  const GemmOp B{static_cast<const float*>(t.b), t.ldb, t.tb};
  float acc[8][8];
  gemm_tile_f32(A, B, t.M, t.N, t.K, m0, n0, As, Bs, acc);
  float* C = static_cast<float*>(t.c);
  const float alpha = float(t.alpha), beta = float(t.beta);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int gm = m0 + gemm_row(i);
    if (gm >= t.M) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int gn = n0 + gemm_col(j);
      if (gn >= t.N) continue;
      float* cp = C + int64_t(gm) * t.ldc + gn;
      float v = alpha * acc[i][j];
      if (beta != 0.f) v = fmaf(beta, *cp, v);
      *cp = v;
    }
  }
}

// Which kernel takes the FP32 tasks of 96 x 96 outputs and more: the tensor cores (3xTF32,
// tc_gemm.cu; the default) or the SIMT 128 x 128 tiles below.
static int g_gemm_engine = GDSW_GEMM_AUTO;
void set_gemm_engine(int e) { g_gemm_engine = e; }
int gemm_engine() { return g_gemm_engine; }

template <typename T>
void run_gemm(DevArena& tmp, const std::vector<GemmTaskP>& tasks, cudaStream_t s) {
  run_gemm_engine<T>(tmp, tasks, s, g_gemm_engine);
}

template <typename T>
void run_gemm_engine(DevArena& tmp, const std::vector<GemmTaskP>& tasks, cudaStream_t s, int engine) {
  if (tasks.empty()) return;
  std::vector<int32_t> tt, ti, bt, bi;  // 64-tiles (k_gemm), 128-tiles (k_gemm_f32)
  std::vector<GemmTaskP> tc;             // tasks for the tensor cores
  for (size_t q = 0; q < tasks.size(); ++q) {
    const auto& t = tasks[q];
    if (t.M <= 0 || t.N <= 0) continue;
    if (sizeof(T) == 4 && t.M >= 96 && t.N >= 96 && t.K >= 1 && engine != GDSW_GEMM_SIMT) {
      tc.push_back(t);
      continue;
    }
    if (sizeof(T) == 4 && t.M >= 96 && t.N >= 96) {
      int nt = ((t.M + 127) / 128) * ((t.N + 127) / 128);
      for (int i = 0; i < nt; ++i) {
        bt.push_back(int32_t(q));
        bi.push_back(i);
      }
      continue;
    }
    int nt = ((t.M + 63) / 64) * ((t.N + 63) / 64);
    for (int i = 0; i < nt; ++i) {
      tt.push_back(int32_t(q));
      ti.push_back(i);
    }
  }
  if (!tc.empty()) run_gemm_tc(tc, s);
  if (tt.empty() && bt.empty()) return;
  GemmTaskP* d_t = tmp.upload(tasks, s);
  if (!tt.empty()) {
    int32_t* d_tt = tmp.upload(tt, s);
    int32_t* d_ti = tmp.upload(ti, s);
    // slices of K: enough CTAs for two per SM, at least 256 products each
    int kmax = 0;
    for (const auto& t : tasks) kmax = std::max(kmax, t.K);
    const int ntl = int(tt.size()), S = std::max(1, std::min(304 / ntl, kmax / 256));
    T* part = S > 1 ? tmp.alloc<T>(size_t(S) * ntl * 4096) : nullptr;
    k_gemm<T><<<dim3(ntl, S), 256, 0, s>>>(d_t, d_tt, d_ti, part);
    check_launch("k_gemm");
    if (S > 1) {
      k_gemm_slices<T><<<dim3(ntl, 16), 256, 0, s>>>(d_t, d_tt, d_ti, S, part);
      check_launch("k_gemm_slices");
      tmp.release(part);
    }
  }
  if (!bt.empty()) {
    int32_t* d_bt = tmp.upload(bt, s);
    int32_t* d_bi = tmp.upload(bi, s);
    k_gemm_f32<<<int(bt.size()), 256, 0, s>>>(d_t, d_bt, d_bi);
    check_launch("k_gemm_f32");
  }
}
template void run_gemm<double>(DevArena&, const std::vector<GemmTaskP>&, cudaStream_t);
template void run_gemm<float>(DevArena&, const std::vector<GemmTaskP>&, cudaStream_t);
template void run_gemm_engine<float>(DevArena&, const std::vector<GemmTaskP>&, cudaStream_t, int);

// ------------------------------------------------------------------ batched Gauss-Jordan inverse
// In-place inversion of square blocks with partial pivoting, blocked by panels of NB
// columns: (1) LU with partial pivoting of the remaining rows of the panel chooses the
// pivot rows, (2) the NB x NB block D of their entries is inverted, (3) the rows are swapped into
// place and the block sweep A_PP <- D^-1, A_Pj <- D^-1 A_Pj, A_iP <- -A_iP D^-1,
// A_ij <- A_ij - A_iP D^-1 A_Pj is applied as a rank-NB update, and (4) at the end the
// columns are permuted back.
constexpr int GJ_NB = 32;
constexpr int kGjClusterRows = 8 * 512;  // rows of a panel that a cluster of 8 CTAs holds in registers

// What a panel leaves for the sweep, per task: the rows chosen (their position before the panel's
// swaps) and, per row at the panel's own positions, where it went if it was not chosen (else -1).
struct GjSwaps {
  int32_t from[GJ_NB], to[GJ_NB];
};

// A pivot candidate: larger magnitude first, then the smaller position.  The magnitude's bits + 1
// (0: no candidate; a NaN counts as zero), split in two words for 64-bit types.
struct GjBest {
  unsigned hi, lo, npos;  // npos = ~position
};
__device__ __forceinline__ GjBest gj_key(float v, int pos) {
  const float a = fabsf(v);
  return {(a >= 0.f ? __float_as_uint(a) : 0u) + 1u, 0u, ~unsigned(pos)};
}
__device__ __forceinline__ GjBest gj_key(double v, int pos) {
  const double a = fabs(v);
  const unsigned long long b = (a >= 0.0 ? (unsigned long long)__double_as_longlong(a) : 0ull) + 1ull;
  return {unsigned(b >> 32), unsigned(b), ~unsigned(pos)};
}
__device__ __forceinline__ double gj_magnitude(const GjBest& k, float) { return double(__uint_as_float(k.hi - 1u)); }
__device__ __forceinline__ double gj_magnitude(const GjBest& k, double) {
  return __longlong_as_double((long long)(((unsigned long long)k.hi << 32 | k.lo) - 1ull));
}
template <typename T>
__device__ __forceinline__ GjBest gj_warp_best(GjBest k) {
  GjBest b;
  b.hi = __reduce_max_sync(0xffffffffu, k.hi);
  bool in = k.hi == b.hi;
  if (sizeof(T) == 8) {
    b.lo = __reduce_max_sync(0xffffffffu, in ? k.lo : 0u);
    in = in && k.lo == b.lo;
  } else {
    b.lo = 0u;
  }
  b.npos = __reduce_max_sync(0xffffffffu, in ? k.npos : 0u);
  return b;
}

// D^-1 by Gauss-Jordan in one warp (pivot order fixed by the panel LU, so no further pivoting); lane =
// column, its entries in registers.  The rows rotate by one per step, so that the pivot row is always
// the first register and the loop stays rolled (32 steps bring them back; steps beyond the block's
// size meet the unit rows that pad it).
template <typename T>
__device__ __forceinline__ void gj_dinv_warp(T (&D)[GJ_NB], T* out) {
  const int c = threadIdx.x & 31;
#pragma unroll 1
  for (int k = 0; k < GJ_NB; ++k) {
    T p = __shfl_sync(0xffffffffu, D[0], k);
    if (p == T(0)) p = T(1);
    const T inv = T(1) / p;
    const T rk = D[0];
#pragma unroll
    for (int r = 1; r < GJ_NB; ++r) {
      const T ck = __shfl_sync(0xffffffffu, D[r], k);
      D[r - 1] = c == k ? -ck * inv : D[r] - ck * rk * inv;
    }
    D[GJ_NB - 1] = c == k ? inv : rk * inv;
  }
#pragma unroll
  for (int r = 0; r < GJ_NB; ++r) out[r * GJ_NB + c] = D[r];
}

// Pivot choice and D^-1 of one panel, R rows of the panel per thread in registers, a cluster of CTAs
// per matrix.  Per column: every warp finds its best row (two or three integer warp reductions),
// the CTA its best warp; that warp copies the row to every CTA of the cluster (distributed shared
// memory), and after one cluster barrier all threads know the pivot row and eliminate theirs.  Rows
// are not moved: a thread keeps the position its row has after the swaps so far.  The chain of a
// column is latency only -- one block and one cluster barrier, 1.3 us -- so the panel's time hardly
// depends on the matrix size; with the panel in one CTA's shared memory a column took 13 us at 2000
// rows (eight matrices: eight CTAs at work).  The loop over the columns stays rolled (a row shifts by
// one register per column): unrolled 32 times it was bound by instruction fetches, 3 us per column.
// Panel, pivot block, swaps and E, F of eight 2000-row matrices: 489 -> 57 us (five launches -> two).
template <typename T, int NT, int R>
__global__ void __launch_bounds__(NT) k_gj_panel_rows(const InvTaskP* __restrict__ tasks, int kb, int CL,
                                                      int32_t* __restrict__ rowid, int64_t rowid_stride,
                                                      GjSwaps* __restrict__ swaps, T* __restrict__ dinv,
                                                      double* __restrict__ minpiv) {
  constexpr int NW = NT / 32, V = 16 / sizeof(T), NCH = GJ_NB / V, CMAX = 8;
  __shared__ GjBest wbest[2][NW];
  __shared__ GjBest cbest[2][CMAX];
  __shared__ __align__(16) T stage[2][GJ_NB];
  __shared__ __align__(16) T prow[2][CMAX][GJ_NB];
  __shared__ int32_t s_from[GJ_NB];
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const InvTaskP t = tasks[blockIdx.x / CL];
  if (kb >= t.n) return;  // the whole cluster
  const int rank = int(blockIdx.x) % CL;
  const int w = min(GJ_NB, t.n - kb), rows = t.n - kb;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T* A = static_cast<const T*>(t.a);
  int32_t* id = rowid + int64_t(t.id) * rowid_stride + kb;
  T v[R][GJ_NB];
  int pos[R], myid[R];
  bool live[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = (rank * R + q) * NT + int(threadIdx.x);
    live[q] = r < rows;
    pos[q] = r;
    myid[q] = live[q] ? id[r] : 0;
    const T* p = A + int64_t(kb + r) * t.ld + kb;
#pragma unroll
    for (int c = 0; c < GJ_NB; c += V) {
      if (live[q] && c < w) {  // the padded row holds the whole vector
        const uint4 raw = *reinterpret_cast<const uint4*>(p + c);
        const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
        for (int u = 0; u < V; ++u) v[q][c + u] = e[u];
      } else {
#pragma unroll
        for (int u = 0; u < V; ++u) v[q][c + u] = T(0);
      }
    }
  }
  double least = DBL_MAX;
  if (CL > 1) cl.sync();  // every CTA of the cluster runs before its shared memory is written
#pragma unroll 1
  for (int j = 0; j < w; ++j) {  // v[q][0] is column j: eliminating a row shifts it by one column
    constexpr GjBest none = {0u, 0u, 0u};
    const int buf = j & 1;
    GjBest k = live[0] ? gj_key(v[0][0], pos[0]) : none;
#pragma unroll
    for (int q = 1; q < R; ++q)
      if (live[q]) {
        const GjBest o = gj_key(v[q][0], pos[q]);
        if (o.hi > k.hi || (o.hi == k.hi && (o.lo > k.lo || (o.lo == k.lo && o.npos > k.npos)))) k = o;
      }
    GjBest b = gj_warp_best<T>(k);
    if (lane == 0) wbest[buf][warp] = b;
    __syncthreads();
    b = gj_warp_best<T>(lane < NW ? wbest[buf][lane] : none);  // the CTA's
    // the owner's warp passes the row on (warp 0 if the CTA has no row left)
    const bool some = (b.hi | b.lo) != 0u;
    bool own = false;
#pragma unroll
    for (int q = 0; q < R; ++q) own = own || (some && live[q] && ~unsigned(pos[q]) == b.npos);
    const bool push = some ? __any_sync(0xffffffffu, own) : warp == 0;
    if (push) {
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (some && live[q] && ~unsigned(pos[q]) == b.npos)
#pragma unroll
          for (int c = 0; c < GJ_NB; c += V) {
            uint4 raw;
            T* e = reinterpret_cast<T*>(&raw);
#pragma unroll
            for (int u = 0; u < V; ++u) e[u] = v[q][c + u];
            *reinterpret_cast<uint4*>(&stage[buf][c]) = raw;
          }
      __syncwarp();
      for (int i = lane; i < CL * NCH; i += 32) {
        const uint4 raw = *reinterpret_cast<const uint4*>(&stage[buf][(i % NCH) * V]);
        *reinterpret_cast<uint4*>(cl.map_shared_rank(&prow[buf][rank][(i % NCH) * V], i / NCH)) = raw;
      }
      if (lane < CL) *cl.map_shared_rank(&cbest[buf][rank], lane) = b;
    }
    if (CL > 1)
      cl.sync();
    else
      __syncthreads();
    const GjBest mine = lane < CL ? cbest[buf][lane] : none;
    b = gj_warp_best<T>(mine);
    const int src = __ffs(__ballot_sync(0xffffffffu, mine.hi == b.hi && mine.lo == b.lo && mine.npos == b.npos)) - 1;
    const int p = int(~b.npos);
    least = fmin(least, gj_magnitude(b, T(0)));
    T pr[GJ_NB];
#pragma unroll
    for (int c = 0; c < GJ_NB; c += V) {
      const uint4 raw = *reinterpret_cast<const uint4*>(&prow[buf][src][c]);
      const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
      for (int u = 0; u < V; ++u) pr[c + u] = e[u];
    }
    T d = pr[0];
    if (d == T(0)) d = T(1);  // singular: recorded through minpiv, keep the numbers finite
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (!live[q]) continue;
      if (pos[q] == p) {  // chosen: its position before the swaps goes to the first CTA
        pos[q] = j;
        live[q] = false;
        *cl.map_shared_rank(&s_from[j], 0) = (rank * R + q) * NT + int(threadIdx.x);
        continue;
      }
      if (pos[q] == j) pos[q] = p;
      const T l = v[q][0] / d;
#pragma unroll
      for (int c = 1; c < GJ_NB; ++c) v[q][c - 1] = v[q][c] - l * pr[c];
    }
  }
  if (CL > 1)
    cl.sync();
  else
    __syncthreads();
  GjSwaps* S = swaps + t.id;
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = (rank * R + q) * NT + int(threadIdx.x);
    if (r >= rows) continue;
    if (pos[q] != r) id[pos[q]] = myid[q];
    if (r < w) S->to[r] = pos[q] >= w ? kb + pos[q] : -1;
  }
  if (rank != 0) return;
  if (int(threadIdx.x) < w) S->from[threadIdx.x] = kb + s_from[threadIdx.x];
  if (threadIdx.x == 0 && least < minpiv[t.id]) minpiv[t.id] = least;
  if (warp == 0) {
    T D[GJ_NB];
#pragma unroll
    for (int r = 0; r < GJ_NB; ++r)
      D[r] = (r < w && lane < w) ? A[int64_t(kb + s_from[r]) * t.ld + kb + lane] : T(r == lane ? 1 : 0);
    gj_dinv_warp<T>(D, dinv + int64_t(t.id) * GJ_NB * GJ_NB);
  }
}

// Pivot choice for a panel of more rows than a cluster's registers hold: one CTA of 1024 threads.  The first
// RS rows of the panel copy live in shared memory (row stride NB + 1), the rest in the global scratch; the
// column maximum is found with warp shuffles (largest magnitude, smallest row on ties, the pivots of
// k_gj_panel_rows), and the rank-1 elimination runs one warp per row, lane = column.  Only the pivot rows
// are used afterwards.
template <typename T>
__device__ __forceinline__ T& panel_at(T* Ps, T* Pg, int RS, int r, int c) {
  return r < RS ? Ps[r * (GJ_NB + 1) + c] : Pg[int64_t(r) * GJ_NB + c];
}

template <typename T>
__global__ void __launch_bounds__(1024) k_gj_panel_fast(const InvTaskP* tasks, int kb, T* scratch, int64_t scr_stride,
                                                       int32_t* piv, int64_t piv_stride, double* minpiv, int RS) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Ps = reinterpret_cast<T*>(smem_raw);
  __shared__ double wv[32];
  __shared__ int wi[32];
  __shared__ int s_p;
  __shared__ T prow[GJ_NB];
  const InvTaskP t = tasks[blockIdx.x];
  if (kb >= t.n) return;
  const T* A = static_cast<const T*>(t.a);
  const int w = min(GJ_NB, t.n - kb), rows = t.n - kb;
  T* Pg = scratch + int64_t(t.id) * scr_stride;
  int32_t* pv = piv + int64_t(t.id) * piv_stride;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < rows * w; e += blockDim.x) {
    const int r = e / w, c = e - r * w;
    panel_at(Ps, Pg, RS, r, c) = A[int64_t(kb + r) * t.ld + kb + c];
  }
  __syncthreads();
  for (int j = 0; j < w; ++j) {
    double best = -1.0;
    int bi = rows;
    for (int r = j + threadIdx.x; r < rows; r += blockDim.x) {
      const double a = fabs(double(panel_at(Ps, Pg, RS, r, j)));
      if (a > best) { best = a; bi = r; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (lane == 0) { wv[warp] = best; wi[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
      const int nw = int(blockDim.x >> 5);
      double b = lane < nw ? wv[lane] : -2.0;
      int i = lane < nw ? wi[lane] : rows;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, b, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ob > b || (ob == b && oi < i)) { b = ob; i = oi; }
      }
      if (lane == 0) {
        s_p = i;
        pv[kb + j] = kb + i;
        if (b < minpiv[t.id]) minpiv[t.id] = b;
      }
    }
    __syncthreads();
    const int p = s_p;
    if (p != j && threadIdx.x < w) {
      T& x = panel_at(Ps, Pg, RS, j, threadIdx.x);
      T& y = panel_at(Ps, Pg, RS, p, threadIdx.x);
      const T tmp = x;
      x = y;
      y = tmp;
    }
    __syncthreads();
    if (threadIdx.x < w) prow[threadIdx.x] = panel_at(Ps, Pg, RS, j, threadIdx.x);
    __syncthreads();
    T d = prow[j];
    if (d == T(0)) d = T(1);  // singular: recorded through minpiv, keep the numbers finite
    const int nw = int(blockDim.x >> 5);
    const T pl = lane < w ? prow[lane] : T(0);
    int r = j + 1 + warp;
    for (; r + 3 * nw < rows; r += 4 * nw) {  // four rows of this warp in flight
      T l[4], v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        l[q] = panel_at(Ps, Pg, RS, r + q * nw, j);
        v[q] = lane < w ? panel_at(Ps, Pg, RS, r + q * nw, lane) : T(0);
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const T lq = l[q] / d;
        if (lane == j)
          panel_at(Ps, Pg, RS, r + q * nw, j) = lq;
        else if (lane > j && lane < w)
          panel_at(Ps, Pg, RS, r + q * nw, lane) = v[q] - lq * pl;
      }
    }
    for (; r < rows; r += nw) {
      const T l = panel_at(Ps, Pg, RS, r, j) / d;
      __syncwarp();
      if (lane == j)
        panel_at(Ps, Pg, RS, r, j) = l;
      else if (lane > j && lane < w)
        panel_at(Ps, Pg, RS, r, lane) -= l * pl;
    }
    __syncthreads();
  }
}

// The swaps of a panel that k_gj_panel_fast chose (more rows than a cluster's registers hold): the same
// GjSwaps and row numbers from its sequence of transpositions, and D^-1.
template <typename T>
__global__ void __launch_bounds__(32) k_gj_maps(const InvTaskP* __restrict__ tasks, int kb,
                                                const int32_t* __restrict__ piv, int64_t piv_stride,
                                                int32_t* __restrict__ rowid, int64_t rowid_stride,
                                                GjSwaps* __restrict__ swaps, T* __restrict__ dinv) {
  const InvTaskP t = tasks[blockIdx.x];
  if (kb >= t.n) return;
  const int w = min(GJ_NB, t.n - kb), lane = threadIdx.x;
  const int32_t* pv = piv + int64_t(t.id) * piv_stride + kb;
  int32_t* id = rowid + int64_t(t.id) * rowid_stride;
  // positions touched: the panel's own and the pivots'; at[] = the row (by position before) now there
  __shared__ int32_t where[2 * GJ_NB], at[2 * GJ_NB], ids[2 * GJ_NB], n;
  if (lane == 0) {
    n = w;
    for (int j = 0; j < w; ++j) where[j] = at[j] = kb + j;
    for (int j = 0; j < w; ++j) {
      int e = 0;
      while (e < n && where[e] != pv[j]) ++e;
      if (e == n) {
        where[n] = at[n] = pv[j];
        ++n;
      }
      const int32_t a = at[j];
      at[j] = at[e];
      at[e] = a;
    }
  }
  __syncwarp();
  for (int e = lane; e < n; e += 32) ids[e] = id[at[e]];
  __syncwarp();
  for (int e = lane; e < n; e += 32) id[where[e]] = ids[e];
  GjSwaps* S = swaps + t.id;
  if (lane < w) {
    S->from[lane] = at[lane];
    int32_t to = -1;
    for (int e = w; e < n; ++e)
      if (at[e] == kb + lane) to = where[e];
    S->to[lane] = to;
  }
  T D[GJ_NB];
  const T* A = static_cast<const T*>(t.a);
#pragma unroll
  for (int r = 0; r < GJ_NB; ++r) D[r] = (r < w && lane < w) ? A[int64_t(at[r]) * t.ld + kb + lane] : T(r == lane ? 1 : 0);
  gj_dinv_warp<T>(D, dinv + int64_t(t.id) * GJ_NB * GJ_NB);
}

// F = D^-1 A[P, :] (w x n) from the chosen rows where they are, E = A[:, P] (n x w) of the swapped
// matrix, and the displaced rows moved to their new positions.  One thread per column for the first
// and the last (it has read its column of the chosen rows before it overwrites them), one per row for
// E; a displaced row is read at its old position, which nothing writes here.
template <typename T>
__global__ void __launch_bounds__(128) k_gj_fe(const InvTaskP* __restrict__ tasks, int kb,
                                               const GjSwaps* __restrict__ swaps, const T* __restrict__ dinv,
                                               T* __restrict__ Fp, T* __restrict__ E, int64_t stride) {
  constexpr int V = 16 / sizeof(T);
  const InvTaskP t = tasks[blockIdx.y];
  if (kb >= t.n || int(blockIdx.x) * 128 >= t.n) return;
  __shared__ __align__(16) T Ds[GJ_NB * GJ_NB];
  __shared__ GjSwaps S;
  T* A = static_cast<T*>(t.a);
  const int w = min(GJ_NB, t.n - kb);
  const T* Di = dinv + int64_t(t.id) * GJ_NB * GJ_NB;
  for (int e = threadIdx.x; e < GJ_NB * GJ_NB; e += 128) Ds[e] = Di[e];
  if (threadIdx.x < GJ_NB) {
    S.from[threadIdx.x] = int(threadIdx.x) < w ? swaps[t.id].from[threadIdx.x] : 0;
    S.to[threadIdx.x] = int(threadIdx.x) < w ? swaps[t.id].to[threadIdx.x] : -1;
  }
  __syncthreads();
  T* F = Fp + int64_t(t.id) * stride;
  T* Ee = E + int64_t(t.id) * stride;
  const int idx = blockIdx.x * 128 + threadIdx.x;
  if (idx >= t.n) return;
  {
    T col[GJ_NB];
#pragma unroll
    for (int q = 0; q < GJ_NB; ++q) col[q] = q < w ? A[int64_t(S.from[q]) * t.ld + idx] : T(0);
    for (int r = 0; r < w; ++r) {
      T s = T(0);
#pragma unroll
      for (int q = 0; q < GJ_NB; q += V) {
        T dv[V];
        *reinterpret_cast<uint4*>(dv) = *reinterpret_cast<const uint4*>(&Ds[r * GJ_NB + q]);
#pragma unroll
        for (int u = 0; u < V; ++u) s = fma(dv[u], col[q + u], s);
      }
      F[int64_t(r) * t.ld + idx] = s;
    }
#pragma unroll
    for (int r = 0; r < GJ_NB; ++r) col[r] = S.to[r] >= 0 ? A[int64_t(kb + r) * t.ld + idx] : T(0);
#pragma unroll
    for (int r = 0; r < GJ_NB; ++r)
      if (S.to[r] >= 0) A[int64_t(S.to[r]) * t.ld + idx] = col[r];
  }
  if (idx >= kb && idx < kb + w) return;  // pivot rows: not used by the sweep
  int src = idx;
#pragma unroll
  for (int r = 0; r < GJ_NB; ++r)
    if (S.to[r] == idx) src = kb + r;
  const T* p = A + int64_t(src) * t.ld + kb;
  // a row that is displaced by another thread's columns is not read here; the others do not change
  for (int q = 0; q < GJ_NB; q += V) {
    uint4 raw = make_uint4(0, 0, 0, 0);
    if (q < w) raw = *reinterpret_cast<const uint4*>(p + q);
    *reinterpret_cast<uint4*>(Ee + int64_t(idx) * GJ_NB + q) = raw;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_gj_update(const InvTaskP* tasks, const int32_t* tile_task,
                                                   const int32_t* tile_id, int kb, const T* dinv, const T* Fp,
                                                   const T* E, int64_t stride) {
  const InvTaskP t = tasks[tile_task[blockIdx.x]];
  if (kb >= t.n) return;
  T* A = static_cast<T*>(t.a);
  const int w = min(GJ_NB, t.n - kb);
  const int tiles = (t.n + 63) / 64;
  const int ti = tile_id[blockIdx.x] / tiles, tj = tile_id[blockIdx.x] % tiles;
  const T* Di = dinv + int64_t(t.id) * GJ_NB * GJ_NB;
  const T* F = Fp + int64_t(t.id) * stride;
  const T* Ee = E + int64_t(t.id) * stride;
  __shared__ T Es[64][GJ_NB + 1];
  __shared__ T Fs[GJ_NB][64 + 1];
  __shared__ T Ds[GJ_NB][GJ_NB + 1];
  for (int e = threadIdx.x; e < 64 * GJ_NB; e += 256) {
    int r = e / GJ_NB, q = e % GJ_NB;
    int gi = ti * 64 + r;
    Es[r][q] = (gi < t.n) ? Ee[int64_t(gi) * GJ_NB + q] : T(0);
    int q2 = e / 64, c = e % 64;
    int gj = tj * 64 + c;
    Fs[q2][c] = (gj < t.n && q2 < w) ? F[int64_t(q2) * t.ld + gj] : T(0);
  }
  for (int e = threadIdx.x; e < GJ_NB * GJ_NB; e += 256) Ds[e / GJ_NB][e % GJ_NB] = Di[e];
  __syncthreads();
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    int li = ty * 4 + a, gi = ti * 64 + li;
    if (gi >= t.n) continue;
    bool pi = gi >= kb && gi < kb + w;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int lj = tx * 4 + b, gj = tj * 64 + lj;
      if (gj >= t.n) continue;
      bool pj = gj >= kb && gj < kb + w;
      T* ap = A + int64_t(gi) * t.ld + gj;
      if (pi && pj) {
        *ap = Ds[gi - kb][gj - kb];
      } else if (pi) {
        *ap = Fs[gi - kb][lj];
      } else if (pj) {
        T s = T(0);
        for (int q = 0; q < w; ++q) s = fma(Es[li][q], Ds[q][gj - kb], s);
        *ap = -s;
      } else {
        T s = *ap;
        for (int q = 0; q < w; ++q) s = fma(-Es[li][q], Fs[q][lj], s);
        *ap = s;
      }
    }
  }
}

// FP32 rank-NB sweep on 128 x 128 tiles.  The sweep is bound by the read-modify-write of A,
// so every global load of a tile is issued at once: the A tile and F = D^-1 A[P, :] go to
// shared memory with cp.async, E = A[:, P] (taken before the sweep) is staged transposed; one
// barrier, then the 8 x 8 register-tiled product E F and the epilogue with the four cases of
// the block Gauss-Jordan step (pivot block D^-1, pivot rows F, pivot columns -E D^-1, the rest
// A - E F).  F has the leading dimension of the matrix, so every row starts 16-byte aligned.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int GJU_LD = 132;  // shared row stride (floats) of the update tiles
constexpr size_t GJU_SMEM = size_t(128 + 32 + 32) * GJU_LD * sizeof(float);

__global__ void __launch_bounds__(256, 2) k_gj_update_f32(const InvTaskP* __restrict__ tasks,
                                                          const int32_t* __restrict__ tile_task,
                                                          const int32_t* __restrict__ tile_id, int kb,
                                                          const float* __restrict__ dinv, const float* __restrict__ Fp,
                                                          const float* __restrict__ E, int64_t stride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* Cs = reinterpret_cast<float*>(smem_raw);  // 128 x GJU_LD
  float* Es = Cs + 128 * GJU_LD;                   // 32 x GJU_LD, Es[k][m] = E[m0 + m][k]
  float* Fs = Es + 32 * GJU_LD;                    // 32 x GJU_LD, Fs[k][c] = F[k][n0 + c]
  __shared__ float Ds[GJ_NB][GJ_NB + 1];
  const InvTaskP t = tasks[tile_task[blockIdx.x]];
  if (kb >= t.n) return;
  const int w = min(GJ_NB, t.n - kb);
  const int tiles = (t.n + 127) / 128;
  const int m0 = (tile_id[blockIdx.x] / tiles) * 128, n0 = (tile_id[blockIdx.x] % tiles) * 128;
  const float* Di = dinv + int64_t(t.id) * GJ_NB * GJ_NB;
  const float* F = Fp + int64_t(t.id) * stride;
  const float* Ee = E + int64_t(t.id) * stride;
  float* Am = static_cast<float*>(t.a);
  const int nch = min(32, (t.ld - n0) / 4);  // 16-byte chunks of a tile row inside the padded row
  for (int e = threadIdx.x; e < 128 * 32; e += 256) {  // A tile
    const int r = e >> 5, ch = e & 31;
    if (m0 + r < t.n && ch < nch) cp_async16(Cs + r * GJU_LD + ch * 4, Am + int64_t(m0 + r) * t.ld + n0 + ch * 4);
  }
  for (int e = threadIdx.x; e < 32 * 32; e += 256) {  // F tile
    const int k = e >> 5, ch = e & 31;
    if (k < w && ch < nch) cp_async16(Fs + k * GJU_LD + ch * 4, F + int64_t(k) * t.ld + n0 + ch * 4);
  }
  for (int e = threadIdx.x; e < 128 * 8; e += 256) {  // E tile, transposed
    const int r = e >> 3, q = (e & 7) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m0 + r < t.n) v = *reinterpret_cast<const float4*>(Ee + int64_t(m0 + r) * GJ_NB + q);
    Es[(q + 0) * GJU_LD + r] = v.x;
    Es[(q + 1) * GJU_LD + r] = v.y;
    Es[(q + 2) * GJU_LD + r] = v.z;
    Es[(q + 3) * GJU_LD + r] = v.w;
  }
  for (int e = threadIdx.x; e < GJ_NB * GJ_NB; e += 256) Ds[e / GJ_NB][e % GJ_NB] = Di[e];
  cp_async_wait_all();
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  for (int k = 0; k < w; ++k) {
    const float4 a0 = *reinterpret_cast<const float4*>(Es + k * GJU_LD + ty * 4);
    const float4 a1 = *reinterpret_cast<const float4*>(Es + k * GJU_LD + 64 + ty * 4);
    const float4 b0 = *reinterpret_cast<const float4*>(Fs + k * GJU_LD + tx * 4);
    const float4 b1 = *reinterpret_cast<const float4*>(Fs + k * GJU_LD + 64 + tx * 4);
    const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
  }
  if (m0 + 128 <= t.n && n0 + 128 <= t.n && (m0 >= kb + w || m0 + 128 <= kb) && (n0 >= kb + w || n0 + 128 <= kb)) {
    // a whole tile off the pivot rows and columns (most): 16-byte stores
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int li = gemm_row(i);
      float* row = Am + int64_t(m0 + li) * t.ld + n0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int lj = gemm_col(4 * h);
        const float4 c = *reinterpret_cast<const float4*>(Cs + li * GJU_LD + lj);
        *reinterpret_cast<float4*>(row + lj) = make_float4(c.x - acc[i][4 * h], c.y - acc[i][4 * h + 1],
                                                           c.z - acc[i][4 * h + 2], c.w - acc[i][4 * h + 3]);
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int li = gemm_row(i), gi = m0 + li;
    if (gi >= t.n) continue;
    const bool pi = gi >= kb && gi < kb + w;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int lj = gemm_col(j), gj = n0 + lj;
      if (gj >= t.n) continue;
      const bool pj = gj >= kb && gj < kb + w;
      float v;
      if (pi && pj) {
        v = Ds[gi - kb][gj - kb];
      } else if (pi) {
        v = Fs[(gi - kb) * GJU_LD + lj];
      } else if (pj) {
        float sum = 0.f;
        for (int q = 0; q < w; ++q) sum = fmaf(Es[q * GJU_LD + li], Ds[q][gj - kb], sum);
        v = -sum;
      } else {
        v = Cs[li * GJU_LD + lj] - acc[i][j];
      }
      Am[int64_t(gi) * t.ld + gj] = v;
    }
  }
}

// A^-1 = X P for the inverse X of the row-permuted matrix: column i of X belongs to the row that
// ended at position i.  A CTA permutes whole rows through shared memory.
template <typename T>
__global__ void __launch_bounds__(256) k_gj_colperm(const InvTaskP* __restrict__ tasks,
                                                    const int32_t* __restrict__ rowid, int64_t rowid_stride, int rows) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);
  const InvTaskP t = tasks[blockIdx.y];
  const int32_t* id = rowid + int64_t(t.id) * rowid_stride;
  const int r1 = min(t.n, (int(blockIdx.x) + 1) * rows);
  for (int r = blockIdx.x * rows; r < r1; ++r) {
    T* A = static_cast<T*>(t.a) + int64_t(r) * t.ld;
    for (int c = threadIdx.x; c < t.n; c += 256) buf[id[c]] = A[c];
    __syncthreads();
    for (int c = threadIdx.x; c < t.n; c += 256) A[c] = buf[c];
    __syncthreads();
  }
}

// The same for rows that do not fit in shared memory: GJ_NB rows at a time to the scratch and back
template <typename T>
__global__ void __launch_bounds__(256) k_gj_colperm_wide(const InvTaskP* __restrict__ tasks,
                                                         const int32_t* __restrict__ rowid, int64_t rowid_stride, int r0,
                                                         T* __restrict__ scratch, int64_t stride, int back) {
  const InvTaskP t = tasks[blockIdx.z];
  const int r = r0 + int(blockIdx.y), c = blockIdx.x * 256 + int(threadIdx.x);
  if (r >= t.n || c >= t.n) return;
  T* A = static_cast<T*>(t.a) + int64_t(r) * t.ld;
  T* S = scratch + int64_t(t.id) * stride + int64_t(blockIdx.y) * t.ld;
  if (back)
    A[c] = S[c];
  else
    S[rowid[int64_t(t.id) * rowid_stride + c]] = A[c];
}

__global__ void k_iota_rows(int32_t* p, int64_t stride, int64_t n) {
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) p[i] = int32_t(i % stride);
}

template <typename T, int NT, int R>
static void gj_panel_rows(const InvTaskP* tasks, int nt, int kb, int CL, int32_t* rowid, int64_t rowid_stride,
                          GjSwaps* swaps, T* dinv, double* minpiv, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(nt) * CL);
  cfg.blockDim = dim3(NT);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = unsigned(CL);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  GDSW_CUDA(cudaLaunchKernelEx(&cfg, k_gj_panel_rows<T, NT, R>, tasks, kb, CL, rowid, rowid_stride, swaps, dinv, minpiv));
}

__global__ void k_fill_d(double* p, double v, int64_t n) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) p[i] = v;
}

// Invert every task's matrix in place; returns the smallest pivot magnitude per task.
template <typename T>
void run_inverse(DevArena& tmp, const std::vector<InvTaskP>& tasks_in, std::vector<double>& minpiv,
                 cudaStream_t s) {
  minpiv.assign(tasks_in.size(), 0.0);
  std::vector<InvTaskP> tasks;
  int nmax = 0;
  for (size_t q = 0; q < tasks_in.size(); ++q) {
    InvTaskP t = tasks_in[q];
    t.id = int32_t(q);
    if (t.n > 0) {
      tasks.push_back(t);
      nmax = std::max(nmax, t.n);
    }
  }
  if (tasks.empty()) return;
  const int nt = int(tasks.size());
  const int64_t nq = int64_t(tasks_in.size());
  int ldmax = 8;
  for (const InvTaskP& t : tasks) ldmax = std::max(ldmax, t.ld);
  // F rows have the matrices' leading dimension
  const int64_t stride = std::max<int64_t>(pad8(nmax), ldmax) * GJ_NB;
  T* Fp = tmp.alloc<T>(size_t(nq) * stride);
  T* E = tmp.alloc<T>(size_t(nq) * stride);
  T* dinv = tmp.alloc<T>(size_t(nq) * GJ_NB * GJ_NB);
  int32_t* rowid = tmp.alloc<int32_t>(size_t(nq) * nmax);
  GjSwaps* swaps = tmp.alloc<GjSwaps>(size_t(nq));
  k_iota_rows<<<unsigned((nq * nmax + 255) / 256), 256, 0, s>>>(rowid, nmax, nq * nmax);
  // panels of more rows than a cluster's registers hold: one CTA per matrix, pivots in piv, scratch
  const bool wide = nmax > kGjClusterRows;
  T* scratch = wide ? tmp.alloc<T>(size_t(nq) * stride) : nullptr;
  int32_t* piv = wide ? tmp.alloc<int32_t>(size_t(nq) * nmax) : nullptr;
  double* d_min = tmp.alloc<double>(nq);
  k_fill_d<<<int((nq + 255) / 256), 256, 0, s>>>(d_min, DBL_MAX, nq);
  InvTaskP* d_tasks = tmp.upload(tasks, s);
  const int TE = sizeof(T) == 4 ? 128 : 64;  // update tile edge
  std::vector<int32_t> tt, ti;
  for (int q = 0; q < nt; ++q) {
    int tl = (tasks[q].n + TE - 1) / TE;
    for (int i = 0; i < tl * tl; ++i) {
      tt.push_back(q);
      ti.push_back(i);
    }
  }
  int32_t* d_tt = tmp.upload(tt, s);
  int32_t* d_ti = tmp.upload(ti, s);
  const dim3 gcol((nmax + 127) / 128, nt);
  const size_t panel_smem = size_t(200) * 1024;
  const int panel_rs = int(panel_smem / ((GJ_NB + 1) * sizeof(T)));
  if (wide)
    GDSW_CUDA(cudaFuncSetAttribute(k_gj_panel_fast<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(panel_smem)));
  GDSW_CUDA(cudaFuncSetAttribute(k_gj_update_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, int(GJU_SMEM)));
  for (int kb = 0; kb < nmax; kb += GJ_NB) {
    // one thread per row of the panel; matrices of a few warps take smaller CTAs
    const int rows = nmax - kb;
    auto cluster = [&](int per_cta) {
      int c = 1;
      while (c * per_cta < rows) c *= 2;
      return c;
    };
    if (rows <= 64)
      gj_panel_rows<T, 64, 1>(d_tasks, nt, kb, 1, rowid, nmax, swaps, dinv, d_min, s);
    else if (rows <= 128)
      gj_panel_rows<T, 128, 1>(d_tasks, nt, kb, 1, rowid, nmax, swaps, dinv, d_min, s);
    else if (rows <= 8 * 256)
      gj_panel_rows<T, 256, 1>(d_tasks, nt, kb, cluster(256), rowid, nmax, swaps, dinv, d_min, s);
    else if (rows <= kGjClusterRows)
      gj_panel_rows<T, 256, 2>(d_tasks, nt, kb, cluster(512), rowid, nmax, swaps, dinv, d_min, s);
    else {
      k_gj_panel_fast<T><<<nt, 1024, panel_smem, s>>>(d_tasks, kb, scratch, stride, piv, nmax, d_min, panel_rs);
      k_gj_maps<T><<<nt, 32, 0, s>>>(d_tasks, kb, piv, nmax, rowid, nmax, swaps, dinv);
    }
    k_gj_fe<T><<<gcol, 128, 0, s>>>(d_tasks, kb, swaps, dinv, Fp, E, stride);
    if (sizeof(T) == 4)
      k_gj_update_f32<<<int(tt.size()), 256, GJU_SMEM, s>>>(d_tasks, d_tt, d_ti, kb, reinterpret_cast<const float*>(dinv),
                                                     reinterpret_cast<const float*>(Fp),
                                                     reinterpret_cast<const float*>(E), stride);
    else
      k_gj_update<T><<<int(tt.size()), 256, 0, s>>>(d_tasks, d_tt, d_ti, kb, dinv, Fp, E, stride);
    check_launch("gauss-jordan panel");
  }
  const size_t row_bytes = size_t(nmax) * sizeof(T);
  if (row_bytes <= size_t(200) * 1024) {
    constexpr int kRows = 8;
    GDSW_CUDA(cudaFuncSetAttribute(k_gj_colperm<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    k_gj_colperm<T><<<dim3((nmax + kRows - 1) / kRows, nt), 256, row_bytes, s>>>(d_tasks, rowid, nmax, kRows);
    check_launch("k_gj_colperm");
  } else {
    for (int r0 = 0; r0 < nmax; r0 += GJ_NB)
      for (int back = 0; back < 2; ++back) {
        k_gj_colperm_wide<T><<<dim3((nmax + 255) / 256, GJ_NB, nt), 256, 0, s>>>(d_tasks, rowid, nmax, r0, Fp, stride,
                                                                                 back);
        check_launch("k_gj_colperm_wide");
      }
  }
  GDSW_CUDA(cudaMemcpyAsync(minpiv.data(), d_min, sizeof(double) * nq, cudaMemcpyDeviceToHost, s));
  GDSW_CUDA(cudaStreamSynchronize(s));
  for (size_t q = 0; q < tasks_in.size(); ++q)
    if (tasks_in[q].n == 0) minpiv[q] = 1.0;
  if (wide) {
    tmp.release(scratch);
    tmp.release(piv);
  }
  tmp.release(Fp); tmp.release(E); tmp.release(dinv); tmp.release(rowid); tmp.release(swaps);
  tmp.release(d_min); tmp.release(d_tasks); tmp.release(d_tt); tmp.release(d_ti);
}
template void run_inverse<double>(DevArena&, const std::vector<InvTaskP>&, std::vector<double>&, cudaStream_t);
template void run_inverse<float>(DevArena&, const std::vector<InvTaskP>&, std::vector<double>&, cudaStream_t);

// ------------------------------------------------------------------ conversions
__global__ void k_f64_to_f32(const double* a, float* b, int64_t n) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) b[i] = float(a[i]);
}
__global__ void k_f32_to_f64(const float* a, double* b, int64_t n) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) b[i] = double(a[i]);
}
__global__ void k_f32_to_bf16(const float* a, __nv_bfloat16* b, int64_t n) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) b[i] = __float2bfloat16_rn(a[i]);
}
__global__ void k_f64_to_bf16(const double* a, __nv_bfloat16* b, int64_t n) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) b[i] = __float2bfloat16_rn(float(a[i]));
}
void convert(const void* src, int sprec, void* dst, int dprec, int64_t n, cudaStream_t s) {
  if (n == 0) return;
  int blocks = int((n + 255) / 256);
  if (sprec == GDSW_FP64 && dprec == GDSW_FP32)
    k_f64_to_f32<<<blocks, 256, 0, s>>>(static_cast<const double*>(src), static_cast<float*>(dst), n);
  else if (sprec == GDSW_FP32 && dprec == GDSW_FP64)
    k_f32_to_f64<<<blocks, 256, 0, s>>>(static_cast<const float*>(src), static_cast<double*>(dst), n);
  else if (sprec == GDSW_FP32 && dprec == GDSW_BF16)
    k_f32_to_bf16<<<blocks, 256, 0, s>>>(static_cast<const float*>(src), static_cast<__nv_bfloat16*>(dst), n);
  else if (sprec == GDSW_FP64 && dprec == GDSW_BF16)
    k_f64_to_bf16<<<blocks, 256, 0, s>>>(static_cast<const double*>(src), static_cast<__nv_bfloat16*>(dst), n);
  else if (sprec == dprec)
    GDSW_CUDA(cudaMemcpyAsync(dst, src, n * elem_size(sprec), cudaMemcpyDeviceToDevice, s));
  else
    throw Error{GDSW_ERR_INVALID_ARG, "unsupported precision conversion"};
  check_launch("convert");
}

}  // namespace gdsw
