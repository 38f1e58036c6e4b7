// Device code of Eqs. (polarization) and (Ewald) shared by several passes:
// p for many e-field angles from one set of per-voxel sums, and a detector
// pixel from its two q_z bins.
#pragma once

#include "rsx_device.cuh"
#include "rsx_kernels.h"

namespace rsx {

constexpr double kFourPi = 12.566370614359172953850573533118;

// FP32: the SFU approximation, which is accurate (absolute error ~1e-6) only
// near [-pi, pi].  The Euler angles of Sec. 3.1 are not restricted, so x is
// first reduced to r = x - n 2 pi, n = rint(x / 2 pi), by Cody and Waite's
// method with a two-part constant: hi = float(2 pi), lo = float(2 pi - hi),
// each product subtracted in one fused multiply-add.  For |x| up to ~1e4
// the reduced angle is off by less than one ulp of pi, far below the FP32
// contrast tolerance.  FP64 keeps the library call, which reduces any range.
__device__ __forceinline__ float reduce_2pi(float x) {
  constexpr double two_pi = 6.283185307179586476925286766559;
  constexpr float hi = (float)two_pi;
  constexpr float lo = (float)(two_pi - (double)hi);
  const float n = rintf(x * (float)(1.0 / two_pi));
  return fmaf(-n, lo, fmaf(-n, hi, x));
}
__device__ __forceinline__ void sincos_r(float x, float* s, float* c) {
  __sincosf(reduce_2pi(x), s, c);
}
__device__ __forceinline__ void sincos_r(double x, double* s, double* c) { sincos(x, s, c); }

// Loads of data read once per pass (the morphology, N_t): streaming hint, so
// that they do not push the x-transformed slices out of L2 before the y pass
// reads them back.
__device__ __forceinline__ float4 ld_stream(const float4* p) { return __ldcs(p); }
__device__ __forceinline__ double4_32a ld_stream(const double4_32a* p) { return *p; }
__device__ __forceinline__ float2 ld_stream(const float2* p) { return __ldcs(p); }
__device__ __forceinline__ double2 ld_stream(const double2* p) { return __ldcs(p); }

// The angle-independent part of Eq. (polarization) at one voxel, summed
// over components j with g_j = b_j (2 a_j + b_j) (a_j = v (1 + tau'_j),
// b_j = v s dpar_j) and the director d_j:
//   p(e) = [ ((sum_j v_j^2 - 1) + sum_j v_j^2 tau'_j (2 + tau'_j)) e + T e ] / (4 pi),
//   T = sum_j g_j d_j d_j^T  (complex symmetric),
// of which e = (cos a, sin a, 0) meets only the entries xx, xy, yy, xz, yz.
// Summing T instead of T e lets one read of the morphology serve several
// e-field angles; each angle's p is then formed exactly as Eq.
// (polarization) prescribes (the same products, summed in another order).
template <typename R> struct TAcc {
  R aw;        // sum_j v_j^2
  R as[2];     // sum_j v_j^2 tau'_j (2 + tau'_j)
  R t[5][2];   // T: xx, xy, yy, xz, yz
};

template <typename R> __device__ __forceinline__ void tacc_zero(TAcc<R>& a) {
  a.aw = R(0);
  a.as[0] = a.as[1] = R(0);
#pragma unroll
  for (int q = 0; q < 5; ++q) a.t[q][0] = a.t[q][1] = R(0);
}

// A row of k_slice_means: the sums' mean over a slice in the order t, as, aw - 1
// (from N_t: PTen's, see pten_less).  Starting the sums at minus the mean takes it off without an operation (aw -
// 1 is formed after the sum, so aw starts at minus the mean of aw - 1).
constexpr int kMeanStride = 16;
template <typename R> struct MeanRow {
  R t[5][2], as[2], aw1;
};
__device__ __forceinline__ void mean_load(const float* m, MeanRow<float>& v) {
  const float4* q = reinterpret_cast<const float4*>(m);
  const float4 a = q[0], b = q[1], c = q[2];
  v.t[0][0] = a.x, v.t[0][1] = a.y, v.t[1][0] = a.z, v.t[1][1] = a.w;
  v.t[2][0] = b.x, v.t[2][1] = b.y, v.t[3][0] = b.z, v.t[3][1] = b.w;
  v.t[4][0] = c.x, v.t[4][1] = c.y, v.as[0] = c.z, v.as[1] = c.w;
  v.aw1 = m[12];
}
__device__ __forceinline__ void mean_load(const double* m, MeanRow<double>& v) {
  const double2* q = reinterpret_cast<const double2*>(m);
#pragma unroll
  for (int e = 0; e < 5; ++e) v.t[e][0] = q[e].x, v.t[e][1] = q[e].y;
  v.as[0] = q[5].x, v.as[1] = q[5].y, v.aw1 = m[12];
}
template <typename R> __device__ __forceinline__ void tacc_start(TAcc<R>& a, const R* mean) {
  MeanRow<R> v;
  mean_load(mean, v);
  a.aw = -v.aw1;
  a.as[0] = -v.as[0];
  a.as[1] = -v.as[1];
#pragma unroll
  for (int q = 0; q < 5; ++q) a.t[q][0] = -v.t[q][0], a.t[q][1] = -v.t[q][1];
}

// Adds component j with the director (dx, dy, dz).
template <typename R>
__device__ __forceinline__ void tacc_add_d(TAcc<R>& acc, R v, R s, R dx, R dy, R dz,
                                           const PolParams<R>& pp, int j) {
  const R v2 = v * v, v2s = v2 * s, v2s2 = v2s * s;
  acc.aw += v2;
  acc.as[0] += v2 * pp.q[j][0][0] + v2s * pp.q[j][1][0] + v2s2 * pp.q[j][2][0];
  acc.as[1] += v2 * pp.q[j][0][1] + v2s * pp.q[j][1][1] + v2s2 * pp.q[j][2][1];
  const R gr = v2s * pp.q[j][3][0] + v2s2 * pp.q[j][4][0];
  const R gi = v2s * pp.q[j][3][1] + v2s2 * pp.q[j][4][1];
  const R hxr = gr * dx, hxi = gi * dx, hyr = gr * dy, hyi = gi * dy;
  acc.t[0][0] += hxr * dx; acc.t[0][1] += hxi * dx;
  acc.t[1][0] += hxr * dy; acc.t[1][1] += hxi * dy;
  acc.t[2][0] += hyr * dy; acc.t[2][1] += hyi * dy;
  acc.t[3][0] += hxr * dz; acc.t[3][1] += hxi * dz;
  acc.t[4][0] += hyr * dz; acc.t[4][1] += hyi * dz;
}

template <typename R>
__device__ __forceinline__ void tacc_add(TAcc<R>& acc, R v, R s, R phi, R theta,
                                         const PolParams<R>& pp, int j) {
  R sp, cp, st, ct;
  sincos_r(phi, &sp, &cp);
  sincos_r(theta, &st, &ct);
  tacc_add_d(acc, v, s, cp * st, sp * st, ct, pp, j);
}

// The sums as the angles use them, ten reals per voxel: with
// ar = [(sum v^2 - 1) + sum v^2 tau'(2 + tau')] / (4 pi) (complex; the
// reference constant left out; the large part first, then the small optical
// one) and t = T / (4 pi), for e = (c, s, 0) = (cos a, sin a, 0) and b = T e:
//   literal (p <- U^T p):  p0 = ar + c b_x + s b_y = [ar + (txx + tyy)/2]
//                               + cos 2a (txx - tyy)/2 + sin 2a txy
//                          p1 = -s b_x + c b_y = cos 2a txy - sin 2a (txx - tyy)/2
//   lab:                   p0 = c (ar + txx) + s txy,  p1 = c txy + s (ar + tyy)
//   both:                  p2 = b_z = c txz + s tyz,
// so a and b hold the two bracketed terms of the frame in use.  (12 operations
// per voxel and angle and ten registers, where p from the twelve sums took 16
// and twelve; the z-first pass, whose polarisation warps were the later to
// finish, 53.4 -> 48.9 ms per energy at 1024 x 1024 x 128.)
template <typename R> struct PTen {
  R a[2], b[2], xy[2], xz[2], yz[2];
};
template <typename R> __device__ __forceinline__ void pten_zero(PTen<R>& p) {
#pragma unroll
  for (int i = 0; i < 2; ++i) p.a[i] = p.b[i] = p.xy[i] = p.xz[i] = p.yz[i] = R(0);
}
// From t and ar (both already divided by 4 pi).
template <typename R>
__device__ __forceinline__ void pten_of(PTen<R>& p, const R (&ar)[2], const R (&t)[5][2],
                                        bool literal) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    p.a[i] = literal ? ar[i] + R(0.5) * (t[0][i] + t[2][i]) : ar[i] + t[0][i];
    p.b[i] = literal ? R(0.5) * (t[0][i] - t[2][i]) : ar[i] + t[2][i];
    p.xy[i] = t[1][i];
    p.xz[i] = t[3][i];
    p.yz[i] = t[4][i];
  }
}
// From the sums over the components.
template <typename R>
__device__ __forceinline__ void pten_of(PTen<R>& p, TAcc<R>& acc, bool literal) {
  const R inv = R(1.0 / kFourPi);
  const R ar[2] = {((acc.aw - R(1)) + acc.as[0]) * inv, acc.as[1] * inv};
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    acc.t[q][0] *= inv;
    acc.t[q][1] *= inv;
  }
  pten_of(p, ar, acc.t, literal);
}
// Less a slice's mean of PTen (k_slice_means from N_t; t holds a, xy, b, xz, yz).
template <typename R> __device__ __forceinline__ void pten_less(PTen<R>& p, const R* mean) {
  MeanRow<R> m;
  mean_load(mean, m);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    p.a[i] -= m.t[0][i];
    p.xy[i] -= m.t[1][i];
    p.b[i] -= m.t[2][i];
    p.xz[i] -= m.t[3][i];
    p.yz[i] -= m.t[4][i];
  }
}
// p for one angle: c, s = cos a, sin a; c2, s2 = cos 2a, sin 2a.
template <typename R>
__device__ __forceinline__ void p_from_pten(const PTen<R>& p, R c, R s, R c2, R s2, bool literal,
                                            typename RT<R>::C* out) {
  if (literal) {
    out[0] = RT<R>::mk(fma(c2, p.b[0], fma(s2, p.xy[0], p.a[0])),
                       fma(c2, p.b[1], fma(s2, p.xy[1], p.a[1])));
    out[1] = RT<R>::mk(fma(c2, p.xy[0], -s2 * p.b[0]), fma(c2, p.xy[1], -s2 * p.b[1]));
  } else {
    out[0] = RT<R>::mk(fma(c, p.a[0], s * p.xy[0]), fma(c, p.a[1], s * p.xy[1]));
    out[1] = RT<R>::mk(fma(c, p.xy[0], s * p.b[0]), fma(c, p.xy[1], s * p.b[1]));
  }
  out[2] = RT<R>::mk(fma(c, p.xz[0], s * p.yz[0]), fma(c, p.xz[1], s * p.yz[1]));
}

// |(I - r r) v|^2 = sum_k |v_k - r_k (r . v)|^2 for one bin.
template <typename R>
__device__ __forceinline__ R proj_norm2(const typename RT<R>::C v[3], R rx, R ry, R rz) {
  const R sr = rx * v[0].x + ry * v[1].x + rz * v[2].x;
  const R si = rx * v[0].y + ry * v[1].y + rz * v[2].y;
  const R y0r = v[0].x - rx * sr, y0i = v[0].y - rx * si;
  const R y1r = v[1].x - ry * sr, y1i = v[1].y - ry * si;
  const R y2r = v[2].x - rz * sr, y2i = v[2].y - rz * si;
  return y0r * y0r + y0i * y0i + y1r * y1r + y1i * y1i + y2r * y2r + y2i * y2i;
}

template <typename R>
__device__ __forceinline__ R ewald_value(const Geo<R>& g, const typename RT<R>::C a0[3],
                                         const typename RT<R>::C a1[3]) {
  const R x0 = proj_norm2<R>(a0, g.rx, g.ry, g.rz);
  const R x1 = proj_norm2<R>(a1, g.rx, g.ry, g.rz);
  return g.k4 * ((R(1) - g.w) * x0 + g.w * x1);
}

}  // namespace rsx
