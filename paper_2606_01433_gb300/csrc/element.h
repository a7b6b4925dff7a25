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
// a barrier over the element's threads.  In FP32 the basis values keep a second word (hi + lo): their
// rounding, the same at every element, would otherwise be half of the error of an operator product.
template <typename T>
struct Grad1D {
  T v[3][3], d[3][3];   // [basis][point]
};
template <>
struct Grad1D<float> {
  float v[3][3], d[3][3], vl[3][3], dl[3][3];
};
__device__ __forceinline__ void fill_grad1d(Grad1D<double>& B, int tid) {
  if (tid < 9) {
    B.v[tid / 3][tid % 3] = q2_v(tid / 3, tid % 3);
    B.d[tid / 3][tid % 3] = q2_d(tid / 3, tid % 3);
  }
}
inline void host_grad1d(Grad1D<float>& B) {
  for (int a = 0; a < 3; ++a)
    for (int q = 0; q < 3; ++q) {
      B.v[a][q] = float(q2_v(a, q));
      B.vl[a][q] = float(q2_v(a, q) - double(B.v[a][q]));
      B.d[a][q] = float(q2_d(a, q));
      B.dl[a][q] = float(q2_d(a, q) - double(B.d[a][q]));
    }
}
// acc + sum over k of p[k step] times the values (DER: derivatives) of basis k at point i, or (TEST) of
// basis i at point k
template <bool DER, bool TEST>
__device__ __forceinline__ double line(const Grad1D<double>& B, int i, const double* p, int step, double acc) {
  const double(*b)[3] = DER ? B.d : B.v;
  return fma(p[2 * step], TEST ? b[i][2] : b[2][i],
             fma(p[step], TEST ? b[i][1] : b[1][i], fma(p[0], TEST ? b[i][0] : b[0][i], acc)));
}
template <bool DER, bool TEST>
__device__ __forceinline__ float line(const Grad1D<float>& B, int i, const float* p, int step, float acc) {
  const float(*h)[3] = DER ? B.d : B.v;
  const float(*l)[3] = DER ? B.dl : B.vl;
  const float p0 = p[0], p1 = p[step], p2 = p[2 * step];
  acc = fmaf(p2, TEST ? l[i][2] : l[2][i], fmaf(p1, TEST ? l[i][1] : l[1][i], fmaf(p0, TEST ? l[i][0] : l[0][i], acc)));
  return fmaf(p2, TEST ? h[i][2] : h[2][i], fmaf(p1, TEST ? h[i][1] : h[1][i], fmaf(p0, TEST ? h[i][0] : h[0][i], acc)));
}

template <typename T, typename Sync>
__device__ __forceinline__ void element_gradient(const Grad1D<T>& B, int q, bool active, const T (*u)[27],
                                                 T (*s)[3][27], T (*t)[3][27], T gr[3][3], Sync sync) {
  const int x = q % 3, y = (q / 3) % 3, z = q / 9;
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // along x: values s[0], derivatives s[1]
      s[0][c][q] = line<false, false>(B, x, u[c] + q - x, 1, T(0));
      s[1][c][q] = line<true, false>(B, x, u[c] + q - x, 1, T(0));
    }
  sync();
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // along y: dx t[0], dy t[1], no derivative t[2]
      t[0][c][q] = line<false, false>(B, y, s[1][c] + q - 3 * y, 3, T(0));
      t[1][c][q] = line<true, false>(B, y, s[0][c] + q - 3 * y, 3, T(0));
      t[2][c][q] = line<false, false>(B, y, s[0][c] + q - 3 * y, 3, T(0));
    }
  sync();
  if (active)
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // along z
      gr[c][0] = line<false, false>(B, z, t[0][c] + q - 9 * z, 9, T(0));
      gr[c][1] = line<false, false>(B, z, t[1][c] + q - 9 * z, 9, T(0));
      gr[c][2] = line<true, false>(B, z, t[2][c] + q - 9 * z, 9, T(0));
    }
}

// The transposed steps: with the stress s[c][l] (weights included) given at the Gauss points, f[c] =
// sum over points and l of s[c][l] d_l phi_q for node q.  s and t are overwritten.
template <typename T, typename Sync>
__device__ __forceinline__ void element_test(const Grad1D<T>& B, int q, bool active, T (*s)[3][27], T (*t)[3][27],
                                             T f[3], Sync sync) {
  const int x = q % 3, y = (q / 3) % 3, z = q / 9;
  if (active)  // along z
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      t[c][0][q] = line<false, true>(B, z, s[c][0] + q - 9 * z, 9, T(0));
      t[c][1][q] = line<false, true>(B, z, s[c][1] + q - 9 * z, 9, T(0));
      t[c][2][q] = line<true, true>(B, z, s[c][2] + q - 9 * z, 9, T(0));
    }
  sync();
  if (active)  // along y: s[c][0] still needs the x derivative, s[c][1] the x value
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s[c][0][q] = line<false, true>(B, y, t[c][0] + q - 3 * y, 3, T(0));
      s[c][1][q] = line<true, true>(B, y, t[c][1] + q - 3 * y, 3, line<false, true>(B, y, t[c][2] + q - 3 * y, 3, T(0)));
    }
  sync();
  if (active)  // along x
#pragma unroll
    for (int c = 0; c < 3; ++c)
      f[c] = line<true, true>(B, x, s[c][0] + q - x, 1, line<false, true>(B, x, s[c][1] + q - x, 1, T(0)));
}

}  // namespace gdsw
