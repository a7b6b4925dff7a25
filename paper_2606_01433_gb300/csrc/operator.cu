// The saddle-point operator on the device: Carreau viscosity at the Gauss points, the
// assembly of A_cal = [[A, B^T], [B, 0]], the Dirichlet lifting and the FP64 SpMV.
//   arXiv 2606.01433, Section 2 (weak form, saddle-point equation), Section 3 (Carreau
//   law nu = nu0 (1 + (lambda gamma_dot)^2)^((n-1)/2), gamma_dot = sqrt(2 D:D), here with
//   an infinite-shear offset nu_inf; symmetric form 2 nu D(u):D(v)).
// Storage: 3x3 velocity blocks per (free velocity node, free velocity node) pair sharing
// a fluid element (row-major block, 72 bytes); pressure-velocity entries as 3-vectors in
// both row orientations (B rows per pressure node, B^T rows per velocity node).
#include "common.h"
#include "element.h"
#include "kernels.h"

namespace gdsw {

void host_tables(RefTables& T) {
  const double gx[3] = {-0.7745966692414834, 0.0, 0.7745966692414834};  // -sqrt(3/5), 0, sqrt(3/5)
  const double gw[3] = {5.0 / 9.0, 8.0 / 9.0, 5.0 / 9.0};
  auto q2 = [](int a, double x) { return a == 0 ? 0.5 * x * (x - 1.0) : (a == 1 ? 1.0 - x * x : 0.5 * x * (x + 1.0)); };
  auto dq2 = [](int a, double x) { return a == 0 ? x - 0.5 : (a == 1 ? -2.0 * x : x + 0.5); };
  auto q1 = [](int a, double x) { return a == 0 ? 0.5 * (1.0 - x) : 0.5 * (1.0 + x); };
  for (int qz = 0; qz < 3; ++qz)
    for (int qy = 0; qy < 3; ++qy)
      for (int qx = 0; qx < 3; ++qx) {
        int q = qx + 3 * qy + 9 * qz;
        double x = gx[qx], y = gx[qy], z = gx[qz];
        T.w[q] = gw[qx] * gw[qy] * gw[qz];
        T.p1[q][0] = 1.0;
        T.p1[q][1] = x;
        T.p1[q][2] = y;
        T.p1[q][3] = z;
        for (int az = 0; az < 3; ++az)
          for (int ay = 0; ay < 3; ++ay)
            for (int ax = 0; ax < 3; ++ax) {
              int a = ax + 3 * ay + 9 * az;
              T.dphi[q][a][0] = dq2(ax, x) * q2(ay, y) * q2(az, z);
              T.dphi[q][a][1] = q2(ax, x) * dq2(ay, y) * q2(az, z);
              T.dphi[q][a][2] = q2(ax, x) * q2(ay, y) * dq2(az, z);
            }
        for (int pz = 0; pz < 2; ++pz)
          for (int py = 0; py < 2; ++py)
            for (int px = 0; px < 2; ++px) T.psi[q][px + 2 * py + 4 * pz] = q1(px, x) * q1(py, y) * q1(pz, z);
      }
  for (int b = 0; b < 27; ++b)
    for (int d = 0; d < 3; ++d) {
      for (int k = 0; k < 8; ++k) {
        double s = 0.0;
        for (int q = 0; q < 27; ++q) s -= T.w[q] * T.psi[q][k] * T.dphi[q][b][d];
        T.div[k][b][d] = s;
      }
      for (int k = 0; k < 4; ++k) {
        double s = 0.0;
        for (int q = 0; q < 27; ++q) s -= T.w[q] * T.p1[q][k] * T.dphi[q][b][d];
        T.div1[k][b][d] = s;
      }
    }
}

struct Geo {
  int nx, ny, nz, NX, NY;
  double h;
};

__device__ __forceinline__ void node_ijk(int64_t v, const Geo& G, int& i, int& j, int& k) {
  i = int(v % G.NX);
  j = int((v / G.NX) % G.NY);
  k = int(v / (int64_t(G.NX) * G.NY));
}

// elements (per axis) containing both node coordinates a and b
__device__ __forceinline__ int shared_range(int a, int b, int n, int& e0) {
  int lo = max(a, b), hi = min(a, b);
  if (lo - hi > 2) return 0;
  e0 = lo < 2 ? 0 : (lo - 1) / 2;
  int e1 = min(n - 1, hi / 2);
  return e1 >= e0 ? e1 - e0 + 1 : 0;
}

// ------------------------------------------------------------------ a1: Carreau viscosity
// dn (optional, Newton linearisation of Section 3): per Gauss point D(u_k) (xx, yy, zz, xy, xz,
// yz) and N = 4 nu'(gamma_dot) / gamma_dot = 4 (nu0 - nu_inf)(n - 1) lambda^2
// (1 + (lambda gamma_dot)^2)^((n - 3)/2), the weight of the Newton term
// int N (D(u_k):D(w)) (D(u_k):D(v)) of the Carreau operator's derivative.
// Thread per Gauss point, eight elements per CTA (216 of 256 threads), the gradient by sum
// factorisation; the FP64 pipe bounds it (the power function is now most of the work): 0.55 -> 0.33
// ms on the 32^3 channel, 32 -> 16 us at 756 elements.
constexpr int kViscElems = 8;
__global__ void __launch_bounds__(256) k_viscosity(const int32_t* __restrict__ fluid, int64_t nfe,
                                                   const double* __restrict__ uk, Geo G, int form, int has_uk,
                                                   double nu0, double nu_inf, double lam, double ncar,
                                                   double* __restrict__ nu, double* __restrict__ dn) {
  __shared__ Grad1D B;
  __shared__ double u[kViscElems][3][27], s[kViscElems][2][3][27], w[kViscElems][3][3][27];
  dep_release();
  dep_wait();
  const int el = threadIdx.x / 27, q = threadIdx.x - 27 * el;
  const int64_t fe = int64_t(blockIdx.x) * kViscElems + el, t = fe * 27 + q;
  const bool active = el < kViscElems && fe < nfe;
  if (!has_uk || form == GDSW_FORM_GRADIENT) {
    if (!active) return;
    nu[t] = nu0;
    if (dn)
      for (int k = 0; k < 7; ++k) dn[t * 7 + k] = 0.0;
    return;
  }
  fill_grad1d(B, threadIdx.x);
  if (active) {
    const int e = fluid[fe];
    const int ex = e % G.nx, ey = (e / G.nx) % G.ny, ez = e / (G.nx * G.ny);
    const int64_t v = (2 * ex + q % 3) + int64_t(G.NX) * ((2 * ey + (q / 3) % 3) + int64_t(G.NY) * (2 * ez + q / 9));
#pragma unroll
    for (int c = 0; c < 3; ++c) u[el][c][q] = uk[3 * v + c];
  }
  __syncthreads();
  double gr[3][3];
  const int se = active ? el : 0;
  element_gradient(B, q, active, u[se], s[se], w[se], gr, [] { __syncthreads(); });
  if (!active) return;
  const double sc = 2.0 / G.h;
  double dd = 0.0;  // D : D
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      double d = 0.5 * sc * (gr[c][l] + gr[l][c]);
      dd = fma(d, d, dd);
    }
  double gdot = sqrt(2.0 * dd);
  double lg = lam * gdot;
  nu[t] = nu_inf + (nu0 - nu_inf) * pow(1.0 + lg * lg, 0.5 * (ncar - 1.0));
  if (dn) {
    double* o = dn + t * 7;
    o[0] = sc * gr[0][0];
    o[1] = sc * gr[1][1];
    o[2] = sc * gr[2][2];
    o[3] = 0.5 * sc * (gr[0][1] + gr[1][0]);
    o[4] = 0.5 * sc * (gr[0][2] + gr[2][0]);
    o[5] = 0.5 * sc * (gr[1][2] + gr[2][1]);
    o[6] = 4.0 * (nu0 - nu_inf) * (ncar - 1.0) * lam * lam * pow(1.0 + lg * lg, 0.5 * (ncar - 3.0));
  }
}

// pressure-velocity entry: -int psi_P d_d phi_J over shared fluid elements, d = 0..2 (the
// reference element's integrals are tabulated: they are the same on every cube of the mesh)
__device__ void divergence_entry(int64_t P, int64_t J, const Geo& G, const uint8_t* mask, const RefTables* T,
                                 double out[3]) {
  int pi, pj, pk, ji, jj, jk;
  node_ijk(P, G, pi, pj, pk);
  node_ijk(J, G, ji, jj, jk);
  out[0] = out[1] = out[2] = 0.0;
  int e0x, e0y, e0z;
  int nxr = shared_range(pi, ji, G.nx, e0x), nyr = shared_range(pj, jj, G.ny, e0y), nzr = shared_range(pk, jk, G.nz, e0z);
  const double sc = 0.25 * G.h * G.h;  // (h/2)^3 * (2/h)
  for (int cz = 0; cz < nzr; ++cz)
    for (int cy = 0; cy < nyr; ++cy)
      for (int cx = 0; cx < nxr; ++cx) {
        int ex = e0x + cx, ey = e0y + cy, ez = e0z + cz;
        int64_t e = ex + int64_t(G.nx) * (ey + int64_t(G.ny) * ez);
        if (!mask[e]) continue;
        int pl = ((pi - 2 * ex) >> 1) + 2 * ((pj - 2 * ey) >> 1) + 4 * ((pk - 2 * ez) >> 1);
        int b = (ji - 2 * ex) + 3 * (jj - 2 * ey) + 9 * (jk - 2 * ez);
#pragma unroll
        for (int d = 0; d < 3; ++d) out[d] = fma(sc, T->div[pl][b][d], out[d]);
      }
}

// The same entry for the P1-disc pressure (Section 2's element pair): row P = 4 f + k is the
// k-th basis function (1, xi, eta, zeta) of fluid element f, which alone carries it.
__device__ void divergence_entry_p1(int64_t P, int64_t J, const Geo& G, const int32_t* fluid, const RefTables* T,
                                    double out[3]) {
  const int64_t e = fluid[P >> 2];
  const int k = int(P & 3);
  const int ex = int(e % G.nx), ey = int((e / G.nx) % G.ny), ez = int(e / (int64_t(G.nx) * G.ny));
  int ji, jj, jk;
  node_ijk(J, G, ji, jj, jk);
  const int b = (ji - 2 * ex) + 3 * (jj - 2 * ey) + 9 * (jk - 2 * ez);
  const double sc = 0.25 * G.h * G.h;
#pragma unroll
  for (int d = 0; d < 3; ++d) out[d] = sc * T->div1[k][b][d];
}

// ------------------------------------------------------------------ a2: assembly
// Element blocks by sum factorisation, then a gather over the elements of every block.
//
// The Q2 basis and the Gauss rule are tensor products, so with f_q = nu_q w_q (h/2)^3 (2/h)^2
//   G_lm[a, b] = sum_q f_q d_l phi_a(q) d_m phi_b(q),   l, m = x, y, z,
// factors into three one-dimensional contractions: over q_x (X, per pair a_x, b_x and
// derivative pattern), over q_y (nine values per q_z for each pair of planar nodes A = (a_x, a_y),
// B = (b_x, b_y)), over q_z.  The block of nodes (a, b) is K_cd = G_dc + delta_cd tr G for the
// symmetric form 2 nu D:D (Section 3) and delta_cd tr G for the gradient form (Section 2).
// An element costs 14 thousand FP64 operations instead of the 133 thousand of a sum over the 27
// points per pair: the FP64 pipe (1.26 TFLOP/s, one warp instruction per 16 cycles and SM)
// bounds either form.  A thread owns one of the 45 planar pairs A <= B of an element (both
// forms of a block from its transpose) and runs its nine (a_z, b_z) with the one-dimensional
// values of the last contraction as compile-time constants, whose zeros (the middle Gauss point
// is the middle node) drop out.  Two elements per CTA of 96 threads: 94% of the lanes busy, and
// 512 elements (the smallest meshes) still give 256 CTAs.  Measured on the 32^3 channel (31
// thousand elements): 7.09 ms as a sum over the points per pair -> 0.83 ms here (FP64-bound) +
// 0.69 ms in k_gather_blocks (3 GB, 4.3 TB/s); 756 elements: 167 -> 29 + 25 us.
//
// Workspace: unit (a, b) of element e at ws[((a_z 3 + b_z) NT + 45 e + P(A, B)) 9 .. + 9], so a
// warp's 32 blocks are 2304 contiguous bytes.  It holds kAsmChunk elements (266 MB); larger
// meshes run chunk by chunk and the gather adds onto the blocks of the chunks before.  It lies in the
// buffer of the sliced copy, which is filled from the gathered blocks afterwards.
constexpr int kAsmPairs = 45;

// derivative pattern t of a one-dimensional pair: 0 value-value, 1 value-derivative (of b), 2
// derivative-derivative
__host__ __device__ constexpr double q2_pair(int t, int a, int b, int q) {
  return (t == 2 ? q2_d(a, q) : q2_v(a, q)) * (t == 0 ? q2_v(b, q) : q2_d(b, q));
}
// planar pair (A <= B) of an element: its rank and back
__host__ __device__ constexpr int planar_rank(int A, int B) { return A * 9 - A * (A - 1) / 2 + (B - A); }

// NEWTON adds sum_q f_N (D(u_k) grad phi_a)_c (D(u_k) grad phi_b)_d from the D, N values of k_viscosity.
template <bool SYM, bool NEWTON>
__global__ void __launch_bounds__(96) k_element_blocks(const double* __restrict__ nu, const RefTables* __restrict__ T,
                                                       double sc, const double* __restrict__ dn, int64_t f0,
                                                       int64_t nfe, double* __restrict__ ws) {
  constexpr int EPC = 2, NW = 3;
  __shared__ double t1[3][9][3];             // [pattern][a 3 + b][q]
  __shared__ double fq[EPC][27];
  __shared__ double X[EPC][3][9][9];         // [pattern][a_x 3 + b_x][q_y + 3 q_z]
  __shared__ double stage[NW][32 * 9];
  __shared__ double tg[NEWTON ? EPC * 27 * 27 * 3 : 1];  // [element][q][a][c]: (D grad phi_a)_c
  __shared__ double fn[EPC][27];
  dep_release();
  const int tid = threadIdx.x;
  if (tid < 81) {
    const int p = tid / 27, ab = (tid / 3) % 9, q = tid % 3, a = ab / 3, b = ab % 3;
    t1[p][ab][q] = (p == 2 ? q2_d(a, q) : q2_v(a, q)) * (p == 0 ? q2_v(b, q) : q2_d(b, q));
  }
  dep_wait();
  const int64_t e0 = int64_t(blockIdx.x) * EPC;
  const int ne = int(min(int64_t(EPC), nfe - e0));
  if (tid < EPC * 27) {
    const int el = tid / 27, q = tid - 27 * el;
    fq[el][q] = el < ne ? nu[(f0 + e0 + el) * 27 + q] * (T->w[q] * sc) : 0.0;
    if (NEWTON) fn[el][q] = el < ne ? dn[((f0 + e0 + el) * 27 + q) * 7 + 6] * (T->w[q] * sc) : 0.0;
  }
  if (NEWTON) {
    for (int i = tid; i < EPC * 729; i += 96) {
      const int el = i / 729, r = i - 729 * el, q = r / 27, a = r - 27 * q;
      const double* g = dn + ((f0 + e0 + min(el, ne - 1)) * 27 + q) * 7;
      const double d0 = T->dphi[q][a][0], d1 = T->dphi[q][a][1], d2 = T->dphi[q][a][2];
      double* o = tg + i * 3;
      o[0] = g[0] * d0 + g[3] * d1 + g[4] * d2;
      o[1] = g[3] * d0 + g[1] * d1 + g[5] * d2;
      o[2] = g[4] * d0 + g[5] * d1 + g[2] * d2;
    }
  }
  __syncthreads();
  for (int i = tid; i < EPC * 243; i += 96) {
    const int el = i / 243, r = i - 243 * el, p = r / 81, ab = (r / 9) % 9, q23 = r % 9;
    const double* f = fq[el] + 3 * q23;
    X[el][p][ab][q23] = fma(t1[p][ab][2], f[2], fma(t1[p][ab][1], f[1], t1[p][ab][0] * f[0]));
  }
  __syncthreads();
  const int el = tid >= kAsmPairs ? 1 : 0;
  int P = min(tid - kAsmPairs * el, kAsmPairs - 1);  // the last six lanes repeat a pair and store nothing
  int A = 0;
  while (P >= planar_rank(A + 1, A + 1)) ++A;
  const int B = A + (P - planar_rank(A, A));
  const int ax = A % 3, ay = A / 3, bx = B % 3, by = B / 3;
  // Y*[q_z]: names give the derivative of a, then of b, taken so far (0 = none)
  double Yxx[3], Yyy[3], Y00[3], Yxy[3], Yyx[3], Yx0[3], Y0x[3], Yy0[3], Y0y[3];
  {
    double s00[3], s01[3], s10[3], s11[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      s00[q] = t1[0][ay * 3 + by][q];
      s01[q] = t1[1][ay * 3 + by][q];
      s10[q] = t1[1][by * 3 + ay][q];
      s11[q] = t1[2][ay * 3 + by][q];
    }
    const double* x00 = X[el][0][ax * 3 + bx];
    const double* x01 = X[el][1][ax * 3 + bx];
    const double* x10 = X[el][1][bx * 3 + ax];
    const double* x11 = X[el][2][ax * 3 + bx];
#pragma unroll
    for (int z = 0; z < 3; ++z) {
      Yxx[z] = Yyy[z] = Y00[z] = Yxy[z] = Yyx[z] = Yx0[z] = Y0x[z] = Yy0[z] = Y0y[z] = 0.0;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double v00 = x00[q + 3 * z], v11 = x11[q + 3 * z];
        Yxx[z] = fma(v11, s00[q], Yxx[z]);
        Yyy[z] = fma(v00, s11[q], Yyy[z]);
        Y00[z] = fma(v00, s00[q], Y00[z]);
        if (SYM) {
          const double v01 = x01[q + 3 * z], v10 = x10[q + 3 * z];
          Yxy[z] = fma(v10, s01[q], Yxy[z]);
          Yyx[z] = fma(v01, s10[q], Yyx[z]);
          Yx0[z] = fma(v10, s00[q], Yx0[z]);
          Y0x[z] = fma(v01, s00[q], Y0x[z]);
          Yy0[z] = fma(v00, s10[q], Yy0[z]);
          Y0y[z] = fma(v00, s01[q], Y0y[z]);
        }
      }
    }
  }
  const int warp = tid >> 5, lane = tid & 31;
  const int nth = kAsmPairs * ne - 32 * warp;          // blocks of this warp (may be more than 32)
  const int cnt = 9 * max(0, min(32, nth));
  const int64_t NT = nfe * kAsmPairs;
  double* out = ws + (e0 * kAsmPairs + 32 * warp) * 9;
  double* st = stage[warp];
#pragma unroll
  for (int az = 0; az < 3; ++az)
#pragma unroll
    for (int bz = 0; bz < 3; ++bz) {
      double xx = 0, yy = 0, zz = 0, xy = 0, yx = 0, xz = 0, zx = 0, yz = 0, zy = 0;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double c00 = q2_pair(0, az, bz, q), c01 = q2_pair(1, az, bz, q), c10 = q2_pair(1, bz, az, q),
                     c11 = q2_pair(2, az, bz, q);
        if (c00 != 0.0) {
          xx = fma(Yxx[q], c00, xx);
          yy = fma(Yyy[q], c00, yy);
          if (SYM) {
            xy = fma(Yxy[q], c00, xy);
            yx = fma(Yyx[q], c00, yx);
          }
        }
        if (c11 != 0.0) zz = fma(Y00[q], c11, zz);
        if (SYM) {
          if (c01 != 0.0) {
            xz = fma(Yx0[q], c01, xz);
            yz = fma(Yy0[q], c01, yz);
          }
          if (c10 != 0.0) {
            zx = fma(Y0x[q], c10, zx);
            zy = fma(Y0y[q], c10, zy);
          }
        }
      }
      const double tr = (xx + yy) + zz;
      double K[9] = {tr, 0, 0, 0, tr, 0, 0, 0, tr};
      if (SYM) {
        K[0] += xx;
        K[1] = yx;
        K[2] = zx;
        K[3] = xy;
        K[4] += yy;
        K[5] = zy;
        K[6] = xz;
        K[7] = yz;
        K[8] += zz;
      }
      if (NEWTON) {
        const double* ta = tg + el * 2187 + (A + 9 * az) * 3;
        const double* tb = tg + el * 2187 + (B + 9 * bz) * 3;
        double N[9] = {};
        for (int q = 0; q < 27; ++q) {
          const double f = fn[el][q];
          const double b0 = tb[81 * q], b1 = tb[81 * q + 1], b2 = tb[81 * q + 2];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const double fa = f * ta[81 * q + c];
            N[3 * c] = fma(fa, b0, N[3 * c]);
            N[3 * c + 1] = fma(fa, b1, N[3 * c + 1]);
            N[3 * c + 2] = fma(fa, b2, N[3 * c + 2]);
          }
        }
#pragma unroll
        for (int m = 0; m < 9; ++m) K[m] += N[m];
      }
      __syncwarp();
#pragma unroll
      for (int m = 0; m < 9; ++m) st[lane * 9 + m] = K[m];
      __syncwarp();
      double* o = out + int64_t(az * 3 + bz) * NT * 9;
#pragma unroll
      for (int i = 0; i < 9; ++i)
        if (lane + 32 * i < cnt) o[lane + 32 * i] = st[lane + 32 * i];
    }
}

// Blocks of the CTAs [cta0, cta0 + gridDim): every upper block (I, J >= I) sums the units of the
// elements [f0, f1) in element order -- onto what the chunks before left, if its first unit lies
// in one of them -- and writes itself and, off the diagonal, its transpose (operator symmetric).
// A CTA holds the units of whole blocks (at most 256); its threads take single values, nine to a
// unit or block, so that loads and stores run along the 72-byte blocks.
__global__ void __launch_bounds__(256) k_gather_blocks(const int32_t* __restrict__ asm_cta, int cta0,
                                                       const int32_t* __restrict__ asm_uoff,
                                                       const uint32_t* __restrict__ asm_unit,
                                                       const int32_t* __restrict__ a_tpos,
                                                       const double* __restrict__ ws, int64_t f0, int64_t f1,
                                                       double* __restrict__ val) {
  __shared__ int64_t uaddr[256];   // workspace offset of the unit (transposed blocks: -1 - offset)
  __shared__ double part[256 * 9];
  __shared__ int32_t in[257];      // units of the chunk before unit u (its range is contiguous in a block)
  dep_release();
  const int blk0 = asm_cta[cta0 + blockIdx.x], blk1 = asm_cta[cta0 + blockIdx.x + 1];
  const int u0 = asm_uoff[blk0], nu = asm_uoff[blk1] - u0;
  const int64_t NT = (f1 - f0) * kAsmPairs;
  for (int u = threadIdx.x; u < nu; u += 256) {
    const uint32_t w = asm_unit[u0 + u];
    const int64_t fe = w >> 10;
    const int a = int((w >> 5) & 31u), b = int(w & 31u);
    const int A = a % 9, az = a / 9, B = b % 9, bz = b / 9;
    const bool tr = A > B;
    const int64_t z = tr ? bz * 3 + az : az * 3 + bz;
    const int64_t off = (z * NT + (fe - f0) * kAsmPairs + (tr ? planar_rank(B, A) : planar_rank(A, B))) * 9;
    uaddr[u] = tr ? -1 - off : off;
    in[u] = fe >= f0 && fe < f1;
  }
  __syncthreads();
  dep_wait();
  for (int i = threadIdx.x; i < nu * 9; i += 256) {
    const int u = i / 9, m = i - 9 * u;
    if (!in[u]) continue;
    const int64_t s = uaddr[u];
    part[i] = s >= 0 ? ws[s + m] : ws[-1 - s + (m % 3) * 3 + m / 3];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (blk1 - blk0) * 9; i += 256) {
    const int q = i / 9, m = i - 9 * q, blk = blk0 + q;
    const int v0 = asm_uoff[blk] - u0, v1 = asm_uoff[blk + 1] - u0;
    int v = v0;
    while (v < v1 && !in[v]) ++v;
    if (v == v1) continue;  // a lower block, or no unit in this chunk
    double* vp = val + int64_t(blk) * 9 + m;
    double s = v == v0 ? part[v * 9 + m] : *vp + part[v * 9 + m];
    for (++v; v < v1 && in[v]; ++v) s += part[v * 9 + m];
    *vp = s;
    const int tb = a_tpos[blk];
    if (tb != blk) val[int64_t(tb) * 9 + (m % 3) * 3 + m / 3] = s;
  }
}

// pfluid != nullptr: P1-disc rows (fluid element list), else Q1 rows (pressure node list)
__global__ void k_assemble_B(const int32_t* __restrict__ b_ptr, const int32_t* __restrict__ b_col,
                             const int32_t* __restrict__ pnode, const int32_t* __restrict__ pfluid,
                             const int32_t* __restrict__ vnode, int64_t np, Geo G, const uint8_t* mask,
                             const RefTables* T, double* __restrict__ bval) {
  int64_t P = blockIdx.x * int64_t(blockDim.x / 32) + threadIdx.x / 32;
  int lane = threadIdx.x & 31;
  if (P >= np) return;
  for (int e = b_ptr[P] + lane; e < b_ptr[P + 1]; e += 32) {
    double out[3];
    if (pfluid)
      divergence_entry_p1(P, vnode[b_col[e]], G, pfluid, T, out);
    else
      divergence_entry(pnode[P], vnode[b_col[e]], G, mask, T, out);
    bval[int64_t(e) * 3 + 0] = out[0];
    bval[int64_t(e) * 3 + 1] = out[1];
    bval[int64_t(e) * 3 + 2] = out[2];
  }
}

__global__ void k_copy_bt(const int32_t* __restrict__ bt2b, int64_t nbt, const double* __restrict__ bval,
                          double* __restrict__ btval) {
  int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (e >= nbt) return;
  int64_t s = bt2b[e];
  btval[e * 3 + 0] = bval[s * 3 + 0];
  btval[e * 3 + 1] = bval[s * 3 + 1];
  btval[e * 3 + 2] = bval[s * 3 + 2];
}

// b = -A_(free, D) g_D, element by element: the operator applied to the Dirichlet field on the
// elements that carry a nonzero datum (listed at set-up; every other entry of b is zero), then the
// sum over those elements per affected dof in element order.  One warp per element, lane = Gauss
// point / node; gradient, stress and test gradients by sum factorisation.  The block of every
// (row, Dirichlet node) pair, one lane each as before, was a serial chain of 27 points x 8
// elements: 147 us whatever the mesh and 0.80 ms on the 32^3 channel; now 14 + 5 and 18 + 7 us.
__global__ void __launch_bounds__(128) k_lift_elements(const int32_t* __restrict__ lift_elem,
                                                       const uint32_t* __restrict__ lift_mask, int64_t nle,
                                                       const int32_t* __restrict__ fluid, Geo G, int form, int pdisc,
                                                       const double* __restrict__ nu, const RefTables* __restrict__ T,
                                                       const double* __restrict__ g, double* __restrict__ lw) {
  __shared__ Grad1D B;
  __shared__ double su[4][3][27], ss[4][3][3][27], st[4][3][3][27];
  __shared__ double sdiv[4][27];
  dep_release();
  dep_wait();
  fill_grad1d(B, threadIdx.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, q = threadIdx.x & 31;
  const int64_t le = int64_t(blockIdx.x) * 4 + warp;
  if (le >= nle) return;
  const bool active = q < 27;
  const int64_t fe = lift_elem[le];
  double (*u)[27] = su[warp];
  double (*s)[3][27] = ss[warp];
  double (*t)[3][27] = st[warp];
  if (active) {
    const int e = fluid[fe];
    const int ex = e % G.nx, ey = (e / G.nx) % G.ny, ez = e / (G.nx * G.ny);
    const int64_t v = (2 * ex + q % 3) + int64_t(G.NX) * ((2 * ey + (q / 3) % 3) + int64_t(G.NY) * (2 * ez + q / 9));
    const bool dir = (lift_mask[le] >> q) & 1u;
#pragma unroll
    for (int c = 0; c < 3; ++c) u[c][q] = dir ? g[3 * v + c] : 0.0;
  }
  __syncwarp();
  double gr[3][3];
  element_gradient(B, q, active, u, s, t, gr, [] { __syncwarp(); });
  __syncwarp();
  const int x = q % 3, y = (q / 3) % 3, z = q / 9;
  if (active) {
    const double w = T->w[q], f = nu[fe * 27 + q] * w * (0.5 * G.h);
    sdiv[warp][q] = (gr[0][0] + gr[1][1] + gr[2][2]) * w * (0.25 * G.h * G.h);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int l = 0; l < 3; ++l) s[c][l][q] = f * (form == GDSW_FORM_SYMMETRIC ? gr[c][l] + gr[l][c] : gr[c][l]);
  }
  __syncwarp();
  double* o = lw + le * kLiftValues;
  double f[3];
  element_test(B, q, active, s, t, f, [] { __syncwarp(); });
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) o[3 * q + c] = -f[c];
  if (q < (pdisc ? 4 : 8)) {
    double a = 0.0;
    for (int k = 0; k < 27; ++k) a = fma(sdiv[warp][k], pdisc ? T->p1[k][q] : T->psi[k][q], a);
    o[81 + q] = a;
  }
}

__global__ void __launch_bounds__(256) k_lift_gather(const int32_t* __restrict__ dof, const int32_t* __restrict__ ptr,
                                                     const int32_t* __restrict__ src, int64_t ndof,
                                                     const double* __restrict__ lw, double* __restrict__ b) {
  dep_release();
  dep_wait();
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= ndof) return;
  double a = 0.0;
  for (int32_t e = ptr[i]; e < ptr[i + 1]; ++e) a += lw[src[e]];
  b[dof[i]] = a;
}

// ------------------------------------------------------------------ a3: SpMV
// Velocity rows from the sliced copy: slices of 32 rows, lane = row, every lane running the
// same number of blocks (the slice's longest row; shorter rows are zero padded),
// so each FP64 warp instruction has all 32 lanes busy.  Slot group g (32 slots, one per lane)
// keeps its 3x3 blocks component-major: value m of lane l at g * 288 + m * 32 + l (B^T: at
// g * 96 + m * 32 + l), so every value load is one coalesced 256-byte access.
// Pressure rows: LPR lanes per row, lane = entry (a contiguous 3-vector of B).  FP64 throughout;
// y = A x or y = b - A x.
__global__ void k_sell_fill(const int32_t* __restrict__ src, int64_t nslots, int m, const double* __restrict__ from,
                            double* __restrict__ to) {
  dep_release();
  dep_wait();
  const int64_t slot = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (slot >= nslots) return;
  const int64_t g = slot >> 5;
  const int lane = int(slot & 31);
  const int32_t e = src[slot];
  for (int c = 0; c < m; ++c) to[g * (32 * m) + c * 32 + lane] = e >= 0 ? from[int64_t(e) * m + c] : 0.0;
}

// operator values: evict-first when the operator is larger than L2, kept there otherwise
template <bool STREAM>
__device__ __forceinline__ double ldv(const double* p) {
  return STREAM ? __ldcs(p) : __ldg(p);
}

struct SpmvArgs {
  const int32_t* sell_row;
  const int64_t* aoff;
  const int32_t* acol;
  const double* aval;
  const int64_t* boff;
  const int32_t* bcol;
  const double* btval;
  int64_t nslices;
  const int32_t *b_ptr, *b_col;
  const double* bval;
  int64_t nv, np;
  const double* x;
  double* y;
  const double* rhs;
};

// W warps share a slice of C rows (32, or 8 with four lanes per row): warp w takes the slot groups
// w, w + W, ... (two in flight); the partial sums of a row are added over its lanes, then in warp
// order.  NWARP warps a CTA.  Slices are numbered by decreasing length (build_sell) and the
// pressure rows come last, so the launch ends on its shortest CTAs.
// Bounds: the FP64 pipe (one warp instruction per 16 cycles and SM) for large operators -- 152
// million multiply-adds, 241 us, on the 32^3 channel: 264 us, 286 before the numbering by length
// and the shared butterflies of the pressure rows.  For small ones the pipe of the one SM that
// holds a slice of the longest rows (125 blocks x 32 rows: 1200 warp instructions, 9 us) and the
// chain of dependent column and vector loads along a row: hence slices of 8 rows, four lanes and up
// to four warps a row, one slice a CTA, columns one pass ahead, values left in L2.
// Launched in plain stream order: with programmatic dependent launch the CTAs are placed beside the
// previous kernel's, unevenly, and the 8^3 product took 19 instead of 12 us.
template <int C, int W, int NWARP, int LPR>
__global__ void __launch_bounds__(32 * NWARP) k_spmv(const SpmvArgs a) {
  constexpr int SPC = NWARP / W, CW = 32 / C;
  constexpr bool STREAM = C == 32;
  __shared__ double red[NWARP][3][C];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nu = 3 * a.nv;
  const int64_t vblocks = (a.nslices + SPC - 1) / SPC;
  const double* __restrict__ x = a.x;
  dep_release();
  if (blockIdx.x < vblocks) {
    const int64_t sl = SPC * int64_t(blockIdx.x) + warp / W;
    const int sub = warp % W;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    if (sl < a.nslices) {
      const int64_t g0 = a.aoff[sl] >> 5, g1 = a.aoff[sl + 1] >> 5;
      const int64_t h0 = a.boff[sl] >> 5, h1 = a.boff[sl + 1] >> 5;
      // NG slot groups per pass, their loads independent of the accumulators (so all are in
      // flight at once) and their products chained into the same three sums: no extra FP64
      // adds to merge partial sums.  The columns run one pass ahead: a pass waits for one load
      // (its vector entries), not for two in a row.
      constexpr int NG = 2;
      int32_t j[NG];
      auto columns = [&](int64_t g) {
#pragma unroll
        for (int k = 0; k < NG; ++k) j[k] = g + k * W < g1 ? __ldg(a.acol + (g + k * W) * 32 + lane) : 0;
      };
      columns(g0 + sub);
      for (int64_t g = g0 + sub; g < g1; g += NG * W) {
        double v[NG][9], xv[NG][3];
#pragma unroll
        for (int k = 0; k < NG; ++k)
#pragma unroll
          for (int q = 0; q < 3; ++q) xv[k][q] = __ldg(x + 3 * int64_t(j[k]) + q);
#pragma unroll
        for (int k = 0; k < NG; ++k)
          if (k == 0 || g + k * W < g1)
#pragma unroll
            for (int q = 0; q < 9; ++q) v[k][q] = ldv<STREAM>(a.aval + (g + k * W) * 288 + lane + 32 * q);
        columns(g + NG * W);
#pragma unroll
        for (int k = 0; k < NG; ++k)
          if (k == 0 || g + k * W < g1) {
            a0 = fma(v[k][2], xv[k][2], fma(v[k][1], xv[k][1], fma(v[k][0], xv[k][0], a0)));
            a1 = fma(v[k][5], xv[k][2], fma(v[k][4], xv[k][1], fma(v[k][3], xv[k][0], a1)));
            a2 = fma(v[k][8], xv[k][2], fma(v[k][7], xv[k][1], fma(v[k][6], xv[k][0], a2)));
          }
      }
#pragma unroll 2
      for (int64_t h = h0 + sub; h < h1; h += W) {
        const double xp = __ldg(x + nu + __ldg(a.bcol + h * 32 + lane));
        const double* v = a.btval + h * 96 + lane;
        a0 = fma(ldv<STREAM>(v + 0), xp, a0);
        a1 = fma(ldv<STREAM>(v + 32), xp, a1);
        a2 = fma(ldv<STREAM>(v + 64), xp, a2);
      }
    }
#pragma unroll
    for (int o = CW / 2; o > 0; o >>= 1) {
      a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      a1 += __shfl_xor_sync(0xffffffffu, a1, o);
      a2 += __shfl_xor_sync(0xffffffffu, a2, o);
    }
    if (lane % CW == 0) {
      red[warp][0][lane / CW] = a0;
      red[warp][1][lane / CW] = a1;
      red[warp][2][lane / CW] = a2;
    }
    if (W > 1)
      __syncthreads();
    else
      __syncwarp();
    if (sub == 0 && sl < a.nslices) {
      for (int i = lane; i < 3 * C; i += 32) {
        const int r = i % C, c = i / C;
        const int32_t row = a.sell_row[sl * C + r];
        if (row < 0) continue;
        double t = red[warp][c][r];
#pragma unroll
        for (int k = 1; k < W; ++k) t += red[warp + k][c][r];
        const int64_t o = 3 * int64_t(row) + c;
        a.y[o] = a.rhs ? a.rhs[o] - t : t;
      }
    }
  } else {
    // LPR lanes per pressure row, four entries of a lane in flight; one butterfly over the LPR lanes
    // serves all rows of the warp
    constexpr int RPW = 32 / LPR;
    const int64_t P = ((int64_t(blockIdx.x) - vblocks) * NWARP + warp) * RPW + lane / LPR;
    const int sub = lane % LPR;
    const int32_t e0 = P < a.np ? a.b_ptr[P] : 0, e1 = P < a.np ? a.b_ptr[P + 1] : 0;
    double acc = 0.0;
#pragma unroll 4
    for (int32_t e = e0 + sub; e < e1; e += LPR) {
      const int64_t j = 3 * int64_t(__ldg(a.b_col + e));
      const double* v = a.bval + 3 * int64_t(e);
      acc = fma(ldv<STREAM>(v + 2), __ldg(x + j + 2),
                fma(ldv<STREAM>(v + 1), __ldg(x + j + 1), fma(ldv<STREAM>(v), __ldg(x + j), acc)));
    }
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (sub == 0 && P < a.np) a.y[nu + P] = a.rhs ? a.rhs[nu + P] - acc : acc;
  }
}

// ------------------------------------------------------------------ launchers
static Geo geo(const gdsw_ctx* c) {
  Geo G;
  G.nx = c->mesh.nx; G.ny = c->mesh.ny; G.nz = c->mesh.nz;
  G.NX = c->mesh.NX; G.NY = c->mesh.NY;
  G.h = c->mesh.h;
  return G;
}

void upload_tables(gdsw_ctx* c, cudaStream_t s) {
  RefTables T;
  host_tables(T);
  RefTables* d = c->arena.alloc<RefTables>(1);
  GDSW_CUDA(cudaMemcpyAsync(d, &T, sizeof(T), cudaMemcpyHostToDevice, s));
  GDSW_CUDA(cudaStreamSynchronize(s));
  c->d_tables = d;
}

// Picard update (Section 3): u_k at every free velocity node from the solution x (free dofs in
// solve order); the Dirichlet nodes keep their data g (copied before this kernel)
__global__ void k_picard_velocity(const int32_t* __restrict__ vnode, int64_t nv, const double* __restrict__ x,
                                  double* __restrict__ uk) {
  dep_release();
  dep_wait();
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= 3 * nv) return;
  const int64_t I = q / 3;
  uk[3 * int64_t(vnode[I]) + (q - 3 * I)] = x[q];
}

__global__ void k_axpy(double* __restrict__ x, const double* __restrict__ d, int64_t n) {
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) x[i] += d[i];
}

void launch_axpy(double* x, const double* d, int64_t n, cudaStream_t s) {
  if (n == 0) return;
  k_axpy<<<int((n + 255) / 256), 256, 0, s>>>(x, d, n);
  check_launch("k_axpy");
}

void launch_picard_velocity(gdsw_ctx* c, const double* x, cudaStream_t s) {
  const int64_t nv = c->mesh.nv;
  GDSW_CUDA(cudaMemcpyAsync(c->d_uk, c->d_gdir, sizeof(double) * 3 * c->mesh.nnodes, cudaMemcpyDeviceToDevice, s));
  if (nv > 0) {
    launch_chained(k_picard_velocity, dim3(unsigned((3 * nv + 255) / 256)), dim3(256), 0, s, c->d_vnode, nv, x,
                   c->d_uk);
    check_launch("k_picard_velocity");
  }
  c->has_uk = true;
}

void launch_viscosity(gdsw_ctx* c, cudaStream_t s) {
  const int64_t nfe = int64_t(c->mesh.fluid.size());
  launch_chained(k_viscosity, dim3(unsigned((nfe + kViscElems - 1) / kViscElems)), dim3(256), 0, s, c->d_fluid, nfe,
                 c->d_uk, geo(c), c->form, c->has_uk ? 1 : 0, c->nu0, c->nu_inf, c->lam, c->ncar, c->d_nu, c->d_dn);
  check_launch("k_viscosity");
}

void launch_assembly(gdsw_ctx* c, cudaStream_t s, bool newton) {
  c->jacobian = newton;
  const auto* T = static_cast<RefTables*>(c->d_tables);
  const int64_t np = c->mesh.np;
  double* aval = c->d_val;
  double* btval = c->d_val + 9 * c->nnzb;
  double* bval = btval + 3 * c->nbt;
  double* ws = c->d_sell_aval;  // of use again once launch_sell_fill has refreshed it below
  for (size_t q = 0; q + 1 < c->mesh.asm_chunk.size(); ++q) {
    const int64_t f0 = c->mesh.asm_chunk[q], f1 = c->mesh.asm_chunk[q + 1];
    const int cta0 = c->mesh.asm_chunk_cta[2 * q], cta1 = c->mesh.asm_chunk_cta[2 * q + 1];
    auto element = c->form != GDSW_FORM_SYMMETRIC ? k_element_blocks<false, false>
                   : newton                       ? k_element_blocks<true, true>
                                                  : k_element_blocks<true, false>;
    launch_chained(element, dim3(unsigned((f1 - f0 + 1) / 2)), dim3(96), 0, s, c->d_nu, T, 0.5 * c->mesh.h,
                   c->d_dn, f0, f1 - f0, ws);
    check_launch("k_element_blocks");
    if (cta1 > cta0) {
      launch_chained(k_gather_blocks, dim3(unsigned(cta1 - cta0)), dim3(256), 0, s, c->d_asm_cta, cta0,
                     c->d_asm_uoff, c->d_asm_unit, c->d_a_tpos, ws, f0, f1, aval);
      check_launch("k_gather_blocks");
    }
  }
  if (c->b_assembled) {  // B = -(q, div u) depends on the mesh only, not on the viscosity
    launch_sell_fill(c, false, s);
    return;
  }
  k_assemble_B<<<int((np + 7) / 8), 256, 0, s>>>(c->d_b_ptr, c->d_b_col, c->d_pnode,
                                                 c->mesh.pdisc ? c->d_fluid : nullptr, c->d_vnode, np, geo(c),
                                                 c->d_mask, T, bval);
  check_launch("k_assemble_B");
  if (c->nbt > 0) {
    k_copy_bt<<<int((c->nbt + 255) / 256), 256, 0, s>>>(c->d_bt2b, c->nbt, bval, btval);
    check_launch("k_copy_bt");
  }
  launch_sell_fill(c, true, s);
  c->b_assembled = true;
}

void launch_lift(gdsw_ctx* c, double* b, cudaStream_t s) {
  // every entry of b not written below (rows without a Dirichlet neighbour) is zero
  GDSW_CUDA(cudaMemsetAsync(b, 0, size_t(c->mesh.n) * sizeof(double), s));
  const int64_t nle = int64_t(c->mesh.lift_elem.size()), nd = int64_t(c->mesh.lift_dof.size());
  if (nle == 0 || nd == 0) return;
  launch_chained(k_lift_elements, dim3(unsigned((nle + 3) / 4)), dim3(128), 0, s, c->d_lift_elem, c->d_lift_mask, nle,
                 c->d_fluid, geo(c), c->form, c->mesh.pdisc ? 1 : 0, c->d_nu, static_cast<RefTables*>(c->d_tables),
                 c->d_gdir, c->d_lift_work);
  check_launch("k_lift_elements");
  launch_chained(k_lift_gather, dim3(unsigned((nd + 255) / 256)), dim3(256), 0, s, c->d_lift_dof, c->d_lift_ptr,
                 c->d_lift_src, nd, c->d_lift_work, b);
  check_launch("k_lift_gather");
}

template <int C, int W, int NWARP, int LPR>
static void spmv_as(const SpmvArgs& a, cudaStream_t s) {
  constexpr int SPC = NWARP / W, RPC = NWARP * (32 / LPR);
  const unsigned grid = unsigned((a.nslices + SPC - 1) / SPC + (a.np + RPC - 1) / RPC);
  k_spmv<C, W, NWARP, LPR><<<grid, 32 * NWARP, 0, s>>>(a);
  check_launch("k_spmv");
}

// The form of k_spmv by the operator's size; each line between two sizes is where the two forms
// beside it were equally fast (us per product, unit cubes of m^3 elements, m = 8 / 12 / 16 / 20 /
// 32): 8 rows 4 warps 12 / 23 / 49, 8 rows 2 warps 14 / 24 / 45, 32 rows 4 warps - / 46 / 43 / 72 /
// 286; before 25 / 50 / 62 / 102 / 306.  (32 rows with 2 warps: 283 at m = 32, but longer sums.)
void launch_spmv(gdsw_ctx* c, const double* x, double* y, const double* rhs, cudaStream_t s) {
  const int64_t nv = c->mesh.nv, np = c->mesh.np, ns = c->n_sell_slices;
  const double* bval = c->d_val + 9 * c->nnzb + 3 * c->nbt;
  const SpmvArgs a{c->d_sell_row, c->d_sell_aoff, c->d_sell_acol, c->d_sell_aval, c->d_sell_boff, c->d_sell_bcol,
                   c->d_sell_btval, ns, c->d_b_ptr, c->d_b_col, bval, nv, np, x, y, rhs};
  if (c->mesh.sell_c == 8) {
    if (nv <= 14000)
      spmv_as<8, 4, 4, 32>(a, s);
    else
      spmv_as<8, 2, 4, 16>(a, s);
  } else {
    spmv_as<32, 4, 4, 8>(a, s);
  }
}

// refresh the sliced copy of A (after every assembly) and of B^T (once B is assembled)
void launch_sell_fill(gdsw_ctx* c, bool with_bt, cudaStream_t s) {
  const MeshHost& M = c->mesh;
  const int64_t na = int64_t(M.sell_acol.size()), nb = int64_t(M.sell_bcol.size());
  if (na > 0) {
    launch_chained(k_sell_fill, dim3(unsigned((na + 255) / 256)), dim3(256), 0, s, c->d_sell_asrc, na, 9, c->d_val,
                   c->d_sell_aval);
    check_launch("k_sell_fill");
  }
  if (with_bt && nb > 0) {
    launch_chained(k_sell_fill, dim3(unsigned((nb + 255) / 256)), dim3(256), 0, s, c->d_sell_bsrc, nb, 3,
                   c->d_val + 9 * c->nnzb, c->d_sell_btval);
    check_launch("k_sell_fill");
  }
}

}  // namespace gdsw
