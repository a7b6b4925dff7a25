// Restarted flexible GMRES (right preconditioning) in FP64 on the device
// (arXiv 2606.01433, Section 3: the linearised system is solved by restarted FGMRES
// preconditioned by the multilevel monolithic Schwarz operator).
// Arnoldi with classical Gram-Schmidt applied twice (CGS2).  All reductions have a fixed
// order, so the iteration is bitwise reproducible.  The Hessenberg least-squares problem
// (Givens rotations, back substitution) stays on the device in FP64.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <vector>

#include "common.h"
#include "kernels.h"
#include "quotient.h"

namespace gdsw {

void apply_precond(gdsw_ctx* c, const double* r, double* z, cudaStream_t s);

constexpr int RB = 304;     // reduction blocks (2 per SM)
constexpr int RT = 256;

// ------------------------------------------------------------------ Arnoldi step
// CGS2 in four launches: dots; update and dots; update and norm; scaling and the Givens rotation.
// A warp owns up to EPL rows of 32 entries for all basis vectors, eight at a time, the next loads
// issued ahead of the products: EPL products per lane and vector, then one exchange-and-add tree for the eight sums
// (9 additions instead of 40).  The entries of w stay in registers between the update and the dots
// that follow it, and the CTA that finishes last adds the CTAs' partial sums in CTA order, so no
// launch does only that; every order of summation is fixed.
// Bound: the FP64 pipe -- 4 multiply-adds per basis entry and step, more than the time of reading the
// basis four times.  arnoldi_ctas balances the rows over the 152 SMs; small vectors take one
// entry per lane, where the step is bound by its launches.
// Measured per iteration beside apply and product, ~30 basis vectors, against eleven launches (dots,
// sum, update, dots, sum, update, sum, norm, norm sum, scaling, rotation): n = 11.5 thousand 82 ->
// 60 us, 180 thousand 115 -> 104 us, 656 thousand 276 -> 243, 798 thousand 310 -> 277, 876 thousand 335 -> 320
// (157 us of FP64 work at 751 thousand).  Above 934 thousand entries, in two waves or more, it is behind: 959
// thousand 351 -> 378, 1.8 million 573 -> 587; seven and eight entries a lane spill (-Xptxas -v: 48 to 268
// bytes).  One entry per lane in many CTAs (the form of the separate updates) is slower here: the end of a
// CTA, a fence and an atomic, is paid per wave (751 thousand: 79 us instead of 57 for update and norm).
constexpr int AT = 256, AW = AT / 32;  // threads, warps of a CTA
constexpr int AFLUSH = 64;             // basis vectors whose warp sums are staged at a time
constexpr int AGROUP = 32, AONE = 96;  // CTAs whose partial sums are added together; one group up to AONE
constexpr int AHMAX = 512;             // coefficients kept in shared memory (the rest through L2)

__device__ __forceinline__ double exchange_add(const double (&a)[8], int lane) {
  // lane l ends with the sum over the warp of a[l & 7]
  double b[4], c[2];
  const bool h4 = lane & 4, h2 = lane & 2, h1 = lane & 1;
#pragma unroll
  for (int k = 0; k < 4; ++k) b[k] = (h4 ? a[k + 4] : a[k]) + __shfl_xor_sync(0xffffffffu, h4 ? a[k] : a[k + 4], 4);
#pragma unroll
  for (int k = 0; k < 2; ++k) c[k] = (h2 ? b[k + 2] : b[k]) + __shfl_xor_sync(0xffffffffu, h2 ? b[k] : b[k + 2], 2);
  double d = (h1 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h1 ? c[0] : c[1], 1);
  d += __shfl_xor_sync(0xffffffffu, d, 8);
  d += __shfl_xor_sync(0xffffffffu, d, 16);
  return d;
}

// true in the CTA that arrives last of `of` (its threads then see the others' writes).  One thread
// fences for the CTA: the barrier before orders the other threads' writes ahead of it.
__device__ __forceinline__ bool last_cta(unsigned* count, unsigned of) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(count, 1u) == of - 1;
    if (s_last) *count = 0;  // for the next launch
    __threadfence();
  }
  __syncthreads();
  return s_last;
}

// out[t] = sum over k < m of rows[k * ldp + t], t < nvec, by one CTA: threads = (t, slice of the
// rows), sixteen loads of a thread in flight; rows in order within a slice, then the slices in order
__device__ __forceinline__ void sum_rows(const double* rows, int m, int ldp, int nvec, double* flat, double* out,
                                         double* acc) {
  for (int t0 = 0; t0 < nvec; t0 += AT) {
    const int w = min(nvec - t0, AT), T = (w + 31) & ~31, S = AT / T;
    const int t = int(threadIdx.x) % T, sl = int(threadIdx.x) / T;
    double s = 0.0;
    if (sl < S && t < w)
      for (int k0 = sl; k0 < m; k0 += 16 * S) {
        double x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) x[u] = k0 + u * S < m ? __ldcg(rows + int64_t(k0 + u * S) * ldp + t0 + t) : 0.0;
#pragma unroll
        for (int u = 0; u < 16; ++u) s += x[u];
      }
    flat[threadIdx.x] = s;
    __syncthreads();
    if (sl == 0 && t < w) {
      for (int k = 1; k < S; ++k) s += flat[k * T + t];
      out[t0 + t] = s;
      if (acc) acc[t0 + t] += s;
    }
    __syncthreads();
  }
}

enum { ARN_DOTS = 0, ARN_UPDATE_DOTS = 1, ARN_UPDATE_NORM = 2 };

// w -= sum_t hin[t] V[t] (but for ARN_DOTS), then hout[t] = (V[t], w) and hsum[t] += hout[t] (if
// given), or scal[1] = |w|.  part: gridDim x ldp partial sums.  Data that other launches wrote is
// read through L2 (the CTAs of a chained launch may start before the writer is done).
template <int EPL, int PHASE>
__global__ void __launch_bounds__(AT, 3) k_arnoldi(const double* V, int64_t n, int nvec, const double* hin, double* w,
                                                   double* part, int ldp, unsigned* count, double* hout,
                                                   double* hsum, double* scal) {
  __shared__ double red[AW][AFLUSH];
  __shared__ double hs[PHASE == ARN_DOTS ? 1 : AHMAX];
  dep_release();
  dep_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // rows of 32 entries [r0, r1) of the CTA, row r0 + warp + 8 i of the warp
  const int64_t rows = (n + 31) >> 5, r0 = rows * blockIdx.x / gridDim.x, r1 = rows * (blockIdx.x + 1) / gridDim.x;
  const int64_t e0 = 32 * (r0 + warp) + lane;
  constexpr int RS = 32 * AW;
  const int have = int((r1 - r0 - warp + AW - 1) / AW);  // rows of this warp (the same in all its lanes)
  bool in[EPL];
  double a[EPL];
#pragma unroll
  for (int i = 0; i < EPL; ++i) {
    in[i] = i < have && e0 + RS * i < n;
    a[i] = in[i] ? __ldcg(w + e0 + RS * i) : 0.0;
  }
  if (PHASE != ARN_DOTS) {
    for (int t = threadIdx.x; t < min(nvec, AHMAX); t += AT) hs[t] = __ldcg(hin + t);
    constexpr int U = EPL == 1 ? 8 : EPL == 2 ? 4 : EPL <= 4 ? 3 : 2;  // basis vectors per stage
    double x[U][EPL], y[U][EPL];
    auto load = [&](int t, double (&d)[U][EPL]) {
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int i = 0; i < EPL; ++i)
          d[u][i] = t + u < nvec && in[i] ? __ldcg(V + int64_t(t + u) * n + e0 + RS * i) : 0.0;
    };
    load(0, x);
    __syncthreads();
    for (int t = 0; t < nvec; t += U) {
      load(t + U, y);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const double h = t + u >= nvec ? 0.0 : t + u < AHMAX ? hs[t + u] : __ldcg(hin + t + u);
#pragma unroll
        for (int i = 0; i < EPL; ++i)
          if (i < have) a[i] = fma(-h, x[u][i], a[i]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int i = 0; i < EPL; ++i) x[u][i] = y[u][i];
    }
#pragma unroll
    for (int i = 0; i < EPL; ++i)
      if (in[i]) w[e0 + RS * i] = a[i];
  }
  if (PHASE == ARN_UPDATE_NORM) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < EPL; ++i) s = fma(a[i], a[i], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[0][warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double p = red[0][0];
#pragma unroll
      for (int k = 1; k < AW; ++k) p += red[0][k];
      part[blockIdx.x] = p;
    }
    if (!last_cta(count, gridDim.x)) return;
    double p = 0.0;
    for (int b = threadIdx.x; b < int(gridDim.x); b += AT) p += __ldcg(part + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    if (lane == 0) red[0][warp] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
      double q = red[0][0];
#pragma unroll
      for (int k = 1; k < AW; ++k) q += red[0][k];
      scal[1] = sqrt(q);
    }
    return;
  }
  {
    double x[8], y[8];
    auto load = [&](int t, int i, double (&d)[8]) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        d[u] = t + u < nvec && in[i] ? __ldcg(V + int64_t(t + u) * n + e0 + RS * i) : 0.0;
    };
    load(0, 0, x);
    for (int t0 = 0; t0 < nvec; t0 += AFLUSH) {
      const int t1 = min(nvec, t0 + AFLUSH);
      for (int t = t0; t < t1; t += 8) {
        double acc[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] = 0.0;
#pragma unroll
        for (int i = 0; i < EPL; ++i) {
          if (i + 1 < EPL)
            load(t, i + 1, y);
          else
            load(t + 8, 0, y);
          if (i < have)
#pragma unroll
            for (int u = 0; u < 8; ++u) acc[u] = fma(x[u], a[i], acc[u]);
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = y[u];
        }
        const double s = exchange_add(acc, lane);
        if (lane < 8) red[warp][t - t0 + lane] = s;
      }
      __syncthreads();
      for (int t = t0 + int(threadIdx.x); t < t1; t += AT) {
        double p = red[0][t - t0];
#pragma unroll
        for (int k = 1; k < AW; ++k) p += red[k][t - t0];
        part[int64_t(blockIdx.x) * ldp + t] = p;
      }
      __syncthreads();
    }
  }
  // the last CTA of every AGROUP adds their partial sums, the last group adds the groups'
  const unsigned gs = gridDim.x <= AONE ? gridDim.x : AGROUP;
  const unsigned ng = (gridDim.x + gs - 1) / gs, gr = blockIdx.x / gs;
  const unsigned in_group = min(gs, gridDim.x - gr * gs);
  if (!last_cta(count + 1 + gr, in_group)) return;
  const double* mine = part + int64_t(gr) * gs * ldp;
  double* flat = &red[0][0];
  static_assert(AW * AFLUSH >= AT, "one staged sum per thread");
  if (ng == 1) {
    sum_rows(mine, int(in_group), ldp, nvec, flat, hout, hsum);
    return;
  }
  double* groups = part + int64_t(gridDim.x) * ldp;
  sum_rows(mine, int(in_group), ldp, nvec, flat, groups + int64_t(gr) * ldp, nullptr);
  if (!last_cta(count, ng)) return;
  sum_rows(groups, int(ng), ldp, nvec, flat, hout, hsum);
}

// w <- w / scal[1] (0 if the norm vanished); CTA 0 meanwhile takes column j of H (column-major,
// leading dimension ldh): H[j+1][j] = scal[1], the previous rotations, a new rotation, and the
// updated right-hand side g.  scal[2] = |g[j+1]| (the residual estimate).
__global__ void __launch_bounds__(256) k_scale_givens(double* w, int64_t n, double* H, int ldh, int j, double* cs,
                                                      double* sn, double* g, double* scal) {
  dep_release();
  dep_wait();
  const double d = __ldcg(scal + 1);
  if (blockIdx.x > 0) {
    const double r = 1.0 / d;
    const bool ok = quotient_ok(d);
    for (int64_t e = (int64_t(blockIdx.x) - 1) * 1024 + threadIdx.x, k = 0; k < 4 && e < n; ++k, e += 256) {
      const double v = __ldcg(w + e);
      w[e] = ok ? quotient_by(v, d, r) : (d > 0.0 ? v / d : 0.0);
    }
    return;
  }
  // the rotations are a serial chain: their operands are staged in shared memory
  __shared__ double sc[256], ss[256], sh[257];
  double* col = H + int64_t(j) * ldh;
  double carry = __ldcg(col);  // entry i of the column after rotations 0 .. i - 1
  for (int i0 = 0; i0 < j; i0 += 256) {
    const int m = min(256, j - i0);
    if (int(threadIdx.x) < m) {
      sc[threadIdx.x] = __ldcg(cs + i0 + threadIdx.x);
      ss[threadIdx.x] = __ldcg(sn + i0 + threadIdx.x);
      sh[threadIdx.x] = __ldcg(col + i0 + threadIdx.x + 1);
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int i = 0; i < m; ++i) {
        const double c = sc[i], s = ss[i], hi = carry, lo = sh[i];
        sh[i] = c * hi + s * lo;
        carry = -s * hi + c * lo;
      }
    __syncthreads();
    if (int(threadIdx.x) < m) col[i0 + threadIdx.x] = sh[threadIdx.x];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double a = carry, b = d;
    const double den = hypot(a, b);
    const double c = den > 0.0 ? a / den : 1.0, s = den > 0.0 ? b / den : 0.0;
    cs[j] = c;
    sn[j] = s;
    col[j] = den;
    col[j + 1] = 0.0;
    const double gj = __ldcg(g + j);
    g[j + 1] = -s * gj;
    g[j] = c * gj;
    scal[2] = fabs(s * gj);
  }
}

// back substitution y = R^{-1} g for the first k columns: one CTA, column by column (the chain is
// one division and one update per column, not a sum over the columns)
__global__ void __launch_bounds__(256) k_backsolve(const double* __restrict__ H, int ldh, int k,
                                                   const double* __restrict__ g, double* __restrict__ y) {
  dep_release();
  dep_wait();
  __shared__ double yi;
  for (int i = threadIdx.x; i < k; i += 256) y[i] = g[i];
  for (int i = k - 1; i >= 0; --i) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const double d = H[int64_t(i) * ldh + i];
      yi = d != 0.0 ? y[i] / d : 0.0;
      y[i] = yi;
    }
    __syncthreads();
    const double v = yi;
    for (int q = threadIdx.x; q < i; q += 256) y[q] -= H[int64_t(i) * ldh + q] * v;
  }
}

// x += sum_t y[t] Z[t]
__global__ void k_xupdate(const double* __restrict__ Z, int64_t n, int nvec, const double* __restrict__ y,
                          double* __restrict__ x) {
  dep_release();
  dep_wait();
  extern __shared__ double ys[];
  for (int t = threadIdx.x; t < nvec; t += blockDim.x) ys[t] = y[t];
  __syncthreads();
  int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (e >= n) return;
  double a = x[e];
  for (int t = 0; t < nvec; ++t) a = fma(ys[t], Z[int64_t(t) * n + e], a);
  x[e] = a;
}

__global__ void k_norm_parts(const double* __restrict__ w, int64_t n, double* __restrict__ part) {
  dep_release();
  dep_wait();
  __shared__ double red[RT];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t e0 = blockIdx.x * chunk, e1 = min(n, e0 + chunk);
  double acc = 0.0;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += RT) acc = fma(w[e], w[e], acc);
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = RT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// scal[slot] = sqrt(sum of parts)
__global__ void k_norm_finish(const double* __restrict__ part, int nb, double* __restrict__ scal, int slot) {
  dep_release();
  dep_wait();
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  double s = 0.0;
  for (int b = threadIdx.x; b < nb; b += 32) s += part[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) scal[slot] = sqrt(s);
}

// v = w / scal[slot] (0 if the norm vanished)
__global__ void k_scale(const double* __restrict__ w, int64_t n, const double* __restrict__ scal, int slot,
                        double* __restrict__ v) {
  dep_release();
  dep_wait();
  int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (e >= n) return;
  double d = scal[slot];
  v[e] = d > 0.0 ? w[e] / d : 0.0;
}

// start of a cycle: V[0] = r / beta, g = (beta, 0, ...)
__global__ void k_cycle_start(double* __restrict__ g, int m1, const double* __restrict__ scal) {
  dep_release();
  dep_wait();
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < m1) g[t] = t == 0 ? scal[0] : 0.0;
}

// CTAs of the Arnoldi launches: a CTA per eight rows for small vectors, else the resident CTAs (three of
// 85 registers per SM), so that every SM gets the same rows to within one; a lane holds at most
// kArnoldiRows entries, so longer vectors take several such waves
constexpr int kArnoldiRows = 8;
static int arnoldi_ctas(int64_t n) {
  constexpr int64_t kWave = 3 * 152;
  const int64_t by8 = ((n + 31) / 32 + AW - 1) / AW;  // CTAs at one row per warp
  if (by8 <= kWave) return int(std::max<int64_t>(by8, 1));
  const int64_t waves = (by8 + kWave * kArnoldiRows - 1) / (kWave * kArnoldiRows);
  return int(waves * kWave);
}

// Pairs of estimates for the contexts of the process, in host memory that is page-locked once, by the first
// solve, and stays so: page-locking memory per context, and freeing it, would wait for the whole device
// (gdsw_destroy waited out a 0.4 s kernel on another stream).  Contexts beyond the pairs take pageable
// memory, where a copy holds the host until it is done: nothing runs ahead, and the results are the same.
// So it is if the page-locking fails, or after a reset of the device, which undoes it.
constexpr int kEstPairs = 4096;
alignas(65536) static double g_est[2 * kEstPairs];
static std::mutex g_est_mu;
static std::vector<int> g_est_free;
static bool g_est_ready = false;

static double* take_estimates() {
  {
    std::lock_guard<std::mutex> lock(g_est_mu);
    if (!g_est_ready) {
      g_est_free.resize(kEstPairs);
      for (int i = 0; i < kEstPairs; ++i) g_est_free[i] = kEstPairs - 1 - i;
      if (cudaHostRegister(g_est, sizeof(g_est), cudaHostRegisterPortable) != cudaSuccess) cudaGetLastError();
      g_est_ready = true;
    }
    if (!g_est_free.empty()) {
      const int i = g_est_free.back();
      g_est_free.pop_back();
      return g_est + 2 * i;
    }
  }
  return new double[2];
}

void give_estimates(double* p) {
  if (!p) return;
  if (p < g_est || p >= g_est + 2 * kEstPairs) {
    delete[] p;
    return;
  }
  std::lock_guard<std::mutex> lock(g_est_mu);
  g_est_free.push_back(int((p - g_est) / 2));
}

static void ensure_workspace(gdsw_ctx* c, int m) {
  if (c->m_alloc >= m) return;
  const int64_t n = c->mesh.n;
  c->d_V = c->arena.alloc<double>((m + 1) * n);
  c->d_Z = c->arena.alloc<double>(m * n);
  c->d_H = c->arena.alloc<double>((m + 1) * int64_t(m + 1));
  c->d_gvec = c->arena.alloc<double>(m + 1);
  c->d_cs = c->arena.alloc<double>(m + 1);
  c->d_sn = c->arena.alloc<double>(m + 1);
  c->d_y = c->arena.alloc<double>(m + 1);
  const int64_t ctas = arnoldi_ctas(n), groups = (ctas + AGROUP - 1) / AGROUP;
  c->d_part = c->arena.alloc<double>(std::max<int64_t>(RB, ctas + groups) * (m + 2));
  c->d_count = c->arena.alloc<unsigned>(1 + groups);
  GDSW_CUDA(cudaMemsetAsync(c->d_count, 0, sizeof(unsigned) * (1 + groups), c->stream));
  c->d_scal = c->arena.alloc<double>(8);
  if (!c->h_est) c->h_est = take_estimates();
  c->m_alloc = m;
}

template <int EPL>
static void arnoldi_as(gdsw_ctx* c, int j, double* w, cudaStream_t s) {
  const int64_t n = c->mesh.n;
  const int nvec = j + 1, ldp = c->m_alloc + 2;
  double* hcol = c->d_H + int64_t(j) * (c->m_alloc + 1);
  double* none = nullptr;
  const dim3 grid(unsigned(arnoldi_ctas(n)));
  launch_chained(k_arnoldi<EPL, ARN_DOTS>, grid, dim3(AT), 0, s, c->d_V, n, nvec, none, w, c->d_part, ldp,
                 c->d_count, hcol, none, c->d_scal);
  check_launch("k_arnoldi");
  launch_chained(k_arnoldi<EPL, ARN_UPDATE_DOTS>, grid, dim3(AT), 0, s, c->d_V, n, nvec, hcol, w, c->d_part, ldp,
                 c->d_count, c->d_y, hcol, c->d_scal);
  check_launch("k_arnoldi");
  launch_chained(k_arnoldi<EPL, ARN_UPDATE_NORM>, grid, dim3(AT), 0, s, c->d_V, n, nvec, c->d_y, w, c->d_part, ldp,
                 c->d_count, none, none, c->d_scal);
  check_launch("k_arnoldi");
}

// w <- w - V h twice (CGS2), scaled; H column j receives the summed coefficients and its rotation
static void arnoldi_step(gdsw_ctx* c, int j, double* w, cudaStream_t s) {
  const int64_t n = c->mesh.n;
  // four passes over the basis (two multi-dots, two multi-axpys) plus w traffic and the norm
  ProfScope ps(c, GDSW_K_ARNOLDI, 8.0 * n * (4.0 * (j + 1) + 7.0), s);
  const int64_t rows = (n + 31) / 32, ctas = arnoldi_ctas(n);
  switch (int(((rows + ctas - 1) / ctas + AW - 1) / AW)) {  // rows of a warp
    case 1: arnoldi_as<1>(c, j, w, s); break;
    case 2: arnoldi_as<2>(c, j, w, s); break;
    case 3: arnoldi_as<3>(c, j, w, s); break;
    case 4: arnoldi_as<4>(c, j, w, s); break;
    case 5: arnoldi_as<5>(c, j, w, s); break;
    case 6: arnoldi_as<6>(c, j, w, s); break;
    case 7: arnoldi_as<7>(c, j, w, s); break;
    default: arnoldi_as<kArnoldiRows>(c, j, w, s); break;
  }
  launch_chained(k_scale_givens, dim3(unsigned((n + 1023) / 1024 + 1)), dim3(256), 0, s, w, n, c->d_H,
                 c->m_alloc + 1, j, c->d_cs, c->d_sn, c->d_gvec, c->d_scal);
  check_launch("k_scale_givens");
}

// Two iterations may be in flight: the estimate of one is read while the next runs, so that the device
// does not wait for the host (10 us of the 117 us of an iteration on an 8^3 box).  An iteration whose
// predecessor turns out to have converged is dropped -- its column of H, its vectors and its
// entries of the rotated right-hand side are not read -- and the margin keeps that rare.
constexpr double kAheadMargin = 0.3;
struct EventPair {
  cudaEvent_t e[2] = {nullptr, nullptr};
  EventPair() {
    for (cudaEvent_t& v : e) GDSW_CUDA(cudaEventCreateWithFlags(&v, cudaEventDisableTiming));
  }
  ~EventPair() {
    for (cudaEvent_t v : e)
      if (v) cudaEventDestroy(v);
  }
};

void fgmres_solve(gdsw_ctx* c, const double* b, double* x, gdsw_solve_info* info) {
  cudaStream_t s = c->stream;
  const int64_t n = c->mesh.n;
  const int m = std::max(1, c->opt.restart);
  ensure_workspace(c, m);
  const int ldh = c->m_alloc + 1;
  const int ub = int((n + 255) / 256);
  cudaEvent_t e0, e1;
  GDSW_CUDA(cudaEventCreate(&e0));
  GDSW_CUDA(cudaEventCreate(&e1));
  GDSW_CUDA(cudaEventRecord(e0, s));
  // ||b||
  k_norm_parts<<<RB, RT, 0, s>>>(b, n, c->d_part);
  check_launch("k_norm_parts");
  k_norm_finish<<<1, 32, 0, s>>>(c->d_part, RB, c->d_scal, 3);
  check_launch("k_norm_finish");
  double bnorm = 0.0;
  GDSW_CUDA(cudaMemcpyAsync(&bnorm, c->d_scal + 3, 8, cudaMemcpyDeviceToHost, s));
  GDSW_CUDA(cudaStreamSynchronize(s));
  *info = gdsw_solve_info{};
  if (!(bnorm > 0.0)) {
    GDSW_CUDA(cudaMemsetAsync(x, 0, 8 * n, s));
    info->status = std::isfinite(bnorm) ? GDSW_OK : GDSW_ERR_NAN;
    GDSW_CUDA(cudaStreamSynchronize(s));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return;
  }
  const double tol = c->opt.tol;
  const bool may_run_ahead = !c->ext_precond;  // a V-cycle waits for its coarse solve anyway
  EventPair copied;
  int it = 0;
  double est = 0.0, beta = 0.0;
  const double spmv_b = c->spmv_bytes();
  auto true_residual = [&]() {
    {
      ProfScope ps(c, GDSW_K_SPMV, spmv_b + 8.0 * n, s);
      launch_spmv(c, x, c->d_V, b, s);  // V[0] = b - A x
    }
    k_norm_parts<<<RB, RT, 0, s>>>(c->d_V, n, c->d_part);
    check_launch("k_norm_parts");
    k_norm_finish<<<1, 32, 0, s>>>(c->d_part, RB, c->d_scal, 0);
    check_launch("k_norm_finish");
    GDSW_CUDA(cudaMemcpyAsync(&beta, c->d_scal, 8, cudaMemcpyDeviceToHost, s));
    GDSW_CUDA(cudaStreamSynchronize(s));
  };
  auto iteration = [&](int j) {
    double* zj = c->d_Z + int64_t(j) * n;
    double* w = c->d_V + int64_t(j + 1) * n;
    apply_precond(c, c->d_V + int64_t(j) * n, zj, s);
    {
      ProfScope ps(c, GDSW_K_SPMV, spmv_b, s);
      launch_spmv(c, zj, w, nullptr, s);
    }
    arnoldi_step(c, j, w, s);
    GDSW_CUDA(cudaMemcpyAsync(c->h_est + (j & 1), c->d_scal + 2, 8, cudaMemcpyDeviceToHost, s));
    GDSW_CUDA(cudaEventRecord(copied.e[j & 1], s));
  };
  true_residual();
  int status = GDSW_OK;
  while (true) {
    if (!std::isfinite(beta)) {
      status = GDSW_ERR_NAN;
      break;
    }
    if (beta / bnorm <= tol) break;
    if (it >= c->opt.max_it) {
      status = GDSW_ERR_NOT_CONVERGED;
      break;
    }
    k_scale<<<ub, 256, 0, s>>>(c->d_V, n, c->d_scal, 0, c->d_V);
    check_launch("k_scale");
    k_cycle_start<<<(m + 1 + 127) / 128, 128, 0, s>>>(c->d_gvec, m + 1, c->d_scal);
    check_launch("k_cycle_start");
    int jd = 0;
    bool ahead = false;
    double last = 0.0;  // the estimate before est
    est = beta;
    for (int j = 0; j < m && it < c->opt.max_it; ++j) {
      if (!ahead) iteration(j);
      // the next iteration is queued before this one's estimate is here, unless one more step at the
      // last rate could reach the tolerance
      ahead = may_run_ahead && j >= 2 && j + 1 < m && it + 1 < c->opt.max_it &&
              kAheadMargin * est * std::min(1.0, est / last) > tol * bnorm;
      if (ahead) iteration(j + 1);
      GDSW_CUDA(cudaEventSynchronize(copied.e[j & 1]));
      last = est;
      est = c->h_est[j & 1];
      ++it;
      jd = j + 1;
      if (!std::isfinite(est)) {
        status = GDSW_ERR_NAN;
        break;
      }
      if (est / bnorm <= tol) break;
    }
    if (status == GDSW_ERR_NAN) break;
    k_backsolve<<<1, 256, 0, s>>>(c->d_H, ldh, jd, c->d_gvec, c->d_y);
    check_launch("k_backsolve");
    k_xupdate<<<ub, 256, jd * sizeof(double), s>>>(c->d_Z, n, jd, c->d_y, x);
    check_launch("k_xupdate");
    true_residual();
  }
  GDSW_CUDA(cudaEventRecord(e1, s));
  GDSW_CUDA(cudaEventSynchronize(e1));
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (c->d_sweep_flag) {  // a persistent sweep gave up waiting: the preconditioner output is void
    unsigned flag = 0;
    GDSW_CUDA(cudaMemcpyAsync(&flag, c->d_sweep_flag, sizeof(flag), cudaMemcpyDeviceToHost, s));
    GDSW_CUDA(cudaStreamSynchronize(s));
    if (flag) {
      GDSW_CUDA(cudaMemsetAsync(c->d_sweep_flag, 0, sizeof(unsigned), s));
      status = GDSW_ERR_TIMEOUT;
      c->err = "persistent local sweep: a dependency wait exceeded its time limit";
    }
  }
  info->iterations = it;
  info->relres = beta / bnorm;
  info->est_relres = est / bnorm;
  info->status = status;
  info->time_ms = ms;
}

}  // namespace gdsw
