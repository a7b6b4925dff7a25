// One Q2 element: the one-dimensional basis at the Gauss points and sum-factorised gradients and test
// integrals (the basis and the 3 x 3 x 3 rule are tensor products; x runs fastest in nodes and points).
#pragma once

namespace gdsw {

// one-dimensional Q2 basis / derivative a at Gauss point q
__host__ __device__ constexpr double gauss_x(int q) { return q == 0 ? -0.7745966692414834 : (q == 1 ? 0.0 : 0.7745966692414834); }
__host__ __device__ constexpr double q2_v(int a, int q) {
  const double x = gauss_x(q);
  return a == 0 ? 0.5 * x * (x - 1.0) : (a == 1 ? 1.0 - x * x : 0.5 * x * (x + 1.0));
}
__host__ __device__ constexpr double q2_d(int a, int q) {
  const double x = gauss_x(q);
  return a == 0 ? x - 0.5 : (a == 1 ? -2.0 * x : x + 0.5);
}

// ------------------------------------------------------------------ sum factorisation on one element
// Values of the 27 nodes of an element -> reference gradients at its 27 Gauss points, one axis at a
// time (the Q2 basis is a tensor product: 72 multiply-adds per point and component triple instead
// of 243).  Thread q = 0..26 of the element owns node q, then the partial results of index q, then
// Gauss point q (x fastest throughout); u, s, t are the element's shared arrays [c][27], `sync` is
// a barrier over the element's threads.
struct Grad1D {
  double v[3][3], d[3][3];   // [basis][point]
};
__device__ __forceinline__ void fill_grad1d(Grad1D& B, int tid) {
  if (tid < 9) {
    B.v[tid / 3][tid % 3] = q2_v(tid / 3, tid % 3);
    B.d[tid / 3][tid % 3] = q2_d(tid / 3, tid % 3);
  }
}
// acc + sum over k of p[k step] times the values (DER: derivatives) of basis k at point i, or (TEST) of
// basis i at point k
template <bool DER, bool TEST>
__device__ __forceinline__ double line(const Grad1D& B, int i, const double* p, int step, double acc) {
  const double(*b)[3] = DER ? B.d : B.v;
  return fma(p[2 * step], TEST ? b[i][2] : b[2][i],
             fma(p[step], TEST ? b[i][1] : b[1][i], fma(p[0], TEST ? b[i][0] : b[0][i], acc)));
}
template <typename Sync>
__device__ __forceinline__ void element_gradient(const Grad1D& B, int q, bool active, const double (*u)[27],
                                                 double (*s)[3][27], double (*t)[3][27], double gr[3][3], Sync sync) {
  const int x = q % 3, y = (q / 3) % 3, z = q / 9;
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // along x: values s[0], derivatives s[1]
      s[0][c][q] = line<false, false>(B, x, u[c] + q - x, 1, 0.0);
      s[1][c][q] = line<true, false>(B, x, u[c] + q - x, 1, 0.0);
    }
  sync();
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // along y: dx t[0], dy t[1], no derivative t[2]
      t[0][c][q] = line<false, false>(B, y, s[1][c] + q - 3 * y, 3, 0.0);
      t[1][c][q] = line<true, false>(B, y, s[0][c] + q - 3 * y, 3, 0.0);
      t[2][c][q] = line<false, false>(B, y, s[0][c] + q - 3 * y, 3, 0.0);
    }
  sync();
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // along z
      gr[c][0] = line<false, false>(B, z, t[0][c] + q - 9 * z, 9, 0.0);
      gr[c][1] = line<false, false>(B, z, t[1][c] + q - 9 * z, 9, 0.0);
      gr[c][2] = line<true, false>(B, z, t[2][c] + q - 9 * z, 9, 0.0);
    }
}

// The transposed steps: with the stress s[c][l] (weights included) given at the Gauss points, f[c] =
// sum over points and l of s[c][l] d_l phi_q for node q.  s and t are overwritten.
template <typename Sync>
__device__ __forceinline__ void element_test(const Grad1D& B, int q, bool active, double (*s)[3][27], double (*t)[3][27],
                                             double f[3], Sync sync) {
  const int x = q % 3, y = (q / 3) % 3, z = q / 9;
  if (active)  // along z
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      t[c][0][q] = line<false, true>(B, z, s[c][0] + q - 9 * z, 9, 0.0);
      t[c][1][q] = line<false, true>(B, z, s[c][1] + q - 9 * z, 9, 0.0);
      t[c][2][q] = line<true, true>(B, z, s[c][2] + q - 9 * z, 9, 0.0);
    }
  sync();
  if (active)  // along y: s[c][0] still needs the x derivative, s[c][1] the x value
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s[c][0][q] = line<false, true>(B, y, t[c][0] + q - 3 * y, 3, 0.0);
      s[c][1][q] = line<true, true>(B, y, t[c][1] + q - 3 * y, 3, line<false, true>(B, y, t[c][2] + q - 3 * y, 3, 0.0));
    }
  sync();
  if (active)  // along x
#pragma unroll
    for (int c = 0; c < 3; ++c)
      f[c] = line<true, true>(B, x, s[c][0] + q - x, 1, line<false, true>(B, x, s[c][1] + q - x, 1, 0.0));
}

// ------------------------------------------------------------------ the same in FP32, a line per thread
// A thread that owns a whole line of three nodes (or points) of one component reads each value once for
// all three results, and the basis values are constants in the instructions, those of the middle point
// (0, 1, 0 and -1/2, 0, 1/2) left out.  Every constant keeps a second word (hi + lo): its rounding,
// the same at every element, would otherwise be half of the error of an operator product.
// acc + sum over k of p_k times the value (DER: derivative) of basis k at point I, or (TEST) of basis I at
// point k
template <bool DER, bool TEST, int I>
__device__ __forceinline__ float line_at(const float (&p)[3], float acc) {
  constexpr double c0 = DER ? (TEST ? q2_d(I, 0) : q2_d(0, I)) : (TEST ? q2_v(I, 0) : q2_v(0, I));
  constexpr double c1 = DER ? (TEST ? q2_d(I, 1) : q2_d(1, I)) : (TEST ? q2_v(I, 1) : q2_v(1, I));
  constexpr double c2 = DER ? (TEST ? q2_d(I, 2) : q2_d(2, I)) : (TEST ? q2_v(I, 2) : q2_v(2, I));
  constexpr float h0 = float(c0), h1 = float(c1), h2 = float(c2);
  constexpr float l0 = float(c0 - double(h0)), l1 = float(c1 - double(h1)), l2 = float(c2 - double(h2));
  if constexpr (l0 != 0.f) acc = fmaf(p[0], l0, acc);
  if constexpr (l1 != 0.f) acc = fmaf(p[1], l1, acc);
  if constexpr (l2 != 0.f) acc = fmaf(p[2], l2, acc);
  if constexpr (h0 != 0.f) acc = fmaf(p[0], h0, acc);
  if constexpr (h1 != 0.f) acc = fmaf(p[1], h1, acc);
  if constexpr (h2 != 0.f) acc = fmaf(p[2], h2, acc);
  return acc;
}
// out[i step] for the three i of a line
template <bool DER, bool TEST>
__device__ __forceinline__ void line_all(const float (&p)[3], float* out, int step) {
  out[0] = line_at<DER, TEST, 0>(p, 0.f);
  out[step] = line_at<DER, TEST, 1>(p, 0.f);
  out[2 * step] = line_at<DER, TEST, 2>(p, 0.f);
}
__device__ __forceinline__ void load_line(const float* p, int step, float (&v)[3]) {
  v[0] = p[0], v[1] = p[step], v[2] = p[2 * step];
}

}  // namespace gdsw
