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

// p for e = (c, s, 0) = (cos a, sin a, 0) from the sums, already divided by
// 4 pi (ar + i ai = [(sum v^2 - 1) + sum v^2 tau'(2 + tau')] / (4 pi), the
// reference constant left out; t = T / (4 pi)), in the frame of `literal`:
// with b = T e,
//   literal (p <- U^T p):  p0 = ar + c b_x + s b_y = ar + c^2 Txx + 2cs Txy + s^2 Tyy
//                          p1 = -s b_x + c b_y    = cs (Tyy - Txx) + (c^2 - s^2) Txy
//   lab:                   p0 = c ar + b_x,  p1 = s ar + b_y,
//   both:                  p2 = b_z = c Txz + s Tyz.
template <typename R>
__device__ __forceinline__ void p_from_tacc(R ar, R ai, const R (&t)[5][2], R c, R s, bool literal,
                                            typename RT<R>::C out[3]) {
  if (literal) {
    const R c2 = c * c, s2 = s * s, cs2 = R(2) * c * s, cs = c * s, d2 = c2 - s2;
    out[0] = RT<R>::mk(fma(s2, t[2][0], fma(cs2, t[1][0], fma(c2, t[0][0], ar))),
                       fma(s2, t[2][1], fma(cs2, t[1][1], fma(c2, t[0][1], ai))));
    out[1] = RT<R>::mk(fma(d2, t[1][0], cs * (t[2][0] - t[0][0])),
                       fma(d2, t[1][1], cs * (t[2][1] - t[0][1])));
  } else {
    out[0] = RT<R>::mk(fma(c, ar + t[0][0], s * t[1][0]), fma(c, ai + t[0][1], s * t[1][1]));
    out[1] = RT<R>::mk(fma(s, ar + t[2][0], c * t[1][0]), fma(s, ai + t[2][1], c * t[1][1]));
  }
  out[2] = RT<R>::mk(fma(c, t[3][0], s * t[4][0]), fma(c, t[3][1], s * t[4][1]));
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
