// The general planes path: Algorithm 1 or 2 for any grid with nz <= 254 in
// either precision, a batch of e-field angles at a time.
//
//   k_pol_planes    per pixel column: the angle-independent sums of Eq.
//                   (polarization) once, then for each angle p, its z
//                   transform, and only the ns q_z planes the detector reads
//                   (the run kb .. kb + ns - 1 mod nz; see rsx_zfirst_plan).
//   (x-FFT, y-FFT)  the lateral transforms of those planes, in place.
//   k_plane_images  Eqs. (3Dscatter) and (Ewald): each pixel's two planes to
//                   the detector image, for every angle of the batch.
// The rotation and average follow as on the other paths.  The 3-D DFT is
// separable, so the values are the full transform's up to rounding order.
#include "rsx_device.cuh"
#include "rsx_kernels.h"
#include "rsx_pol.cuh"

namespace rsx {
namespace {

// A voxel pair's field after the fold below: sum and difference.
template <typename C> struct Folded {
  C s, d;
};

constexpr int kPlThreads = 256, kPlSlots = 2, kPlPairs = kPlThreads * kPlSlots;

// A block owns PX adjacent pixels (flat index y nx + x) by the whole stack.
// The z transform is evaluated as a sum over the bins that are kept, with the
// voxels z and nz - z folded first: with S = p(z) + p(nz - z) and
// D = p(z) - p(nz - z),
//   X(k) = sum_{z = 0}^{nz/2} cos(t) S - i sin(t) D,  t = 2 pi k z / nz
// (z = 0 and, for even nz, z = nz/2 stand alone with D = 0), which halves the
// multiplies: 2 ns fused multiply-adds per voxel and field.  At the kept
// fraction of the bins (ns / nz ~ 0.28 at 5 nm and 300 eV) that is 14 per
// voxel and field at nz = 16 and 28 at nz = 45, against ~10 to 25 for an FFT
// that would need a plan for every nz.
// A thread keeps the sums of its kPlSlots voxel pairs in registers for all
// angles.  Per step of A angles: every thread forms p of its voxels for each
// angle and stores S and D (three fields) to shared memory; then the block's
// threads take (angle, field, group of SB bins, pixel) items, a pixel's
// S and D read once per SB bins (with SB = 8, 32 fused multiply-adds per
// 16-byte shared read of S and D and 4 broadcast reads of the twiddles).
// SRC 0: morphology (dir: FP64's cached director); 1: Algorithm 2's N_t.
// twt: exp(-2 pi i j / nz), j < nz.
template <typename R, int SRC, int SB>
__global__ void __launch_bounds__(kPlThreads, sizeof(R) == 4 ? 2 : 1) k_pol_planes(
    const typename RT<R>::V4* __restrict__ M, const typename RT<R>::C* __restrict__ nt,
    const R* __restrict__ dir, long long npix, int nz, int PX, int A, int kb, int ns,
    const __grid_constant__ PolParams<R> pp, const __grid_constant__ AngleBatch<R> ang,
    typename RT<R>::C* __restrict__ out, const typename RT<R>::C* __restrict__ twz) {
  using C = typename RT<R>::C;
  using F = Folded<C>;
  constexpr int SBP = (SB + 1) & ~1;  // twiddles of a group, padded to pairs
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int t = threadIdx.x;
  const int H1 = nz / 2 + 1, G = (ns + SB - 1) / SB, NSP = G * SBP;
  F* buf = reinterpret_cast<F*>(smem_raw);        // [A][H1][3][PX]
  C* tw = reinterpret_cast<C*>(buf + (size_t)A * H1 * 3 * PX);  // [H1][NSP]
  const long long N = npix * nz;
  const long long pix0 = (long long)blockIdx.x * PX;
  const int npx = npix - pix0 < PX ? (int)(npix - pix0) : PX;
  for (int i = t; nz > 1 && i < H1 * NSP; i += kPlThreads) {  // (nz = 1 has no shared memory)
    const int z = i / NSP, r = i - z * NSP, g = r / SBP, b = g * SB + (r - g * SBP);
    tw[i] = twz[(int)(((long long)(kb + b) * z) % nz)];
  }

  // this thread's voxel pairs: the sums of Eq. (polarization), divided by 4 pi
  TAcc<R> acc[kPlSlots][2];
  int at[kPlSlots];    // shared-memory place of the pair (field 0, angle 0); -1: none
  bool two[kPlSlots];  // the pair has a second voxel, nz - z
#pragma unroll
  for (int sl = 0; sl < kPlSlots; ++sl) {
    const int q = t + sl * kPlThreads, z = q / PX, px = q - z * PX;
    at[sl] = z < H1 && px < npx ? (z * 3) * PX + px : -1;
    two[sl] = at[sl] >= 0 && z > 0 && 2 * z < nz;
    tacc_zero(acc[sl][0]);
    tacc_zero(acc[sl][1]);
    if (at[sl] < 0) continue;
    const size_t i0 = (size_t)z * npix + pix0 + px, i1 = (size_t)(nz - z) * npix + pix0 + px;
    if constexpr (SRC == 1) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h && !two[sl]) break;
        acc[sl][h].aw = R(0);
#pragma unroll
        for (int e = 0; e < 5; ++e) {
          const C v = ld_stream(nt + (size_t)e * N + (h ? i1 : i0));
          acc[sl][h].t[e][0] = v.x;
          acc[sl][h].t[e][1] = v.y;
        }
      }
    } else {
      for (int j = 0; j < pp.c; ++j) {
        const typename RT<R>::V4* Mj = M + (size_t)j * N;
        const typename RT<R>::V4 m0 = ld_stream(Mj + i0);
        typename RT<R>::V4 m1 = m0;
        if (two[sl]) m1 = ld_stream(Mj + i1);
        if (dir) {
          const R* dj = dir + (size_t)j * 3 * N;
          tacc_add_d(acc[sl][0], (R)m0.x, (R)m0.y, dj[i0], dj[N + i0], dj[2 * N + i0], pp, j);
          if (two[sl])
            tacc_add_d(acc[sl][1], (R)m1.x, (R)m1.y, dj[i1], dj[N + i1], dj[2 * N + i1], pp, j);
        } else {
          tacc_add(acc[sl][0], (R)m0.x, (R)m0.y, (R)m0.z, (R)m0.w, pp, j);
          if (two[sl]) tacc_add(acc[sl][1], (R)m1.x, (R)m1.y, (R)m1.z, (R)m1.w, pp, j);
        }
      }
      const R inv = R(1.0 / kFourPi);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        TAcc<R>& a = acc[sl][h];
        a.aw = ((a.aw - R(1)) + a.as[0]) * inv;
        a.as[1] *= inv;
#pragma unroll
        for (int e = 0; e < 5; ++e) {
          a.t[e][0] *= inv;
          a.t[e][1] *= inv;
        }
      }
    }
  }

  const bool literal = pp.literal != 0;
  const size_t fstride = (size_t)ns * npix, kstride = 3 * fstride;
  if (nz == 1) {  // no z transform: the pixel's p is its plane
    for (int k = 0; k < ang.n; ++k) {
#pragma unroll
      for (int sl = 0; sl < kPlSlots; ++sl) {
        if (at[sl] < 0) continue;
        C p[3];
        p_from_tacc(acc[sl][0].aw, acc[sl][0].as[1], acc[sl][0].t, ang.ce[k], ang.se[k], literal, p);
        C* o = out + k * kstride + pix0 + at[sl];
        o[0] = p[0];
        o[fstride] = p[1];
        o[2 * fstride] = p[2];
      }
    }
    return;
  }
  for (int a0 = 0; a0 < ang.n; a0 += A) {
    const int na = ang.n - a0 < A ? ang.n - a0 : A;
    if (a0 > 0) __syncthreads();  // the previous step's reads are done
    for (int a = 0; a < na; ++a) {
      const R ce = ang.ce[a0 + a], se = ang.se[a0 + a];
      F* ba = buf + (size_t)a * H1 * 3 * PX;
#pragma unroll
      for (int sl = 0; sl < kPlSlots; ++sl) {
        if (at[sl] < 0) continue;
        C p[3], q[3];
        p_from_tacc(acc[sl][0].aw, acc[sl][0].as[1], acc[sl][0].t, ce, se, literal, p);
        p_from_tacc(acc[sl][1].aw, acc[sl][1].as[1], acc[sl][1].t, ce, se, literal, q);
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          F v;
          v.s = two[sl] ? cadd(p[f], q[f]) : p[f];
          v.d = two[sl] ? csub(p[f], q[f]) : RT<R>::mk(R(0), R(0));
          ba[at[sl] + f * PX] = v;
        }
      }
    }
    __syncthreads();
    const int items = na * 3 * G * PX;
    for (int it = t; it < items; it += kPlThreads) {
      int r = it / PX;
      const int px = it - r * PX;
      const int g = r % G;
      r /= G;
      const int f = r % 3, a = r / 3;
      if (px >= npx) continue;
      C x[SB];
#pragma unroll
      for (int i = 0; i < SB; ++i) x[i] = RT<R>::mk(R(0), R(0));
      const F* b = buf + ((size_t)a * H1 * 3 + f) * PX + px;
      const C* w = tw + g * SBP;
      for (int z = 0; z < H1; ++z) {
        const F v = b[z * 3 * PX];
        C wv[SBP];
#pragma unroll
        for (int i = 0; i < SBP; ++i) wv[i] = w[z * NSP + i];
#pragma unroll
        for (int i = 0; i < SB; ++i) {  // (cos, -sin) = (wv.x, wv.y)
          x[i].x = fma(wv[i].x, v.s.x, fma(-wv[i].y, v.d.y, x[i].x));
          x[i].y = fma(wv[i].x, v.s.y, fma(wv[i].y, v.d.x, x[i].y));
        }
      }
      C* o = out + (size_t)(a0 + a) * kstride + (size_t)f * fstride + pix0 + px;
#pragma unroll
      for (int i = 0; i < SB; ++i)
        if (g * SB + i < ns) o[(size_t)(g * SB + i) * npix] = x[i];
    }
  }
}

// Images of the angles of a batch from their transformed planes: per pixel
// its two planes (b - kb mod nz) of the three fields, the constant left out
// of p before the transform returned at q = 0 (its x and y parts per angle),
// the projection and the interpolation; written in fftshift order.  A thread
// takes AP angles of one pixel, so the 32-byte geometry is read once for
// them; planes has kstride = 3 ns npix complex per angle.
template <typename R, int AP>
__global__ void __launch_bounds__(256) k_plane_images(const typename RT<R>::C* __restrict__ planes,
                                                      int nx, int ny, int nz, int kb, int ns,
                                                      const Geo<R>* __restrict__ geo,
                                                      const __grid_constant__ ImageDc<R> dc,
                                                      R* __restrict__ imgs) {
  using C = typename RT<R>::C;
  const long long npix = (long long)nx * ny;
  const long long pix = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (pix >= npix) return;
  const Geo<R> g = geo[pix];
  const int my = (int)(pix / nx), mx = (int)(pix - (long long)my * nx);
  int sy = my + ny / 2, sx = mx + nx / 2;
  if (sy >= ny) sy -= ny;
  if (sx >= nx) sx -= nx;
  R* dst = imgs + (size_t)sy * nx + sx;
  const int a0 = blockIdx.y * AP;
  const size_t fstride = (size_t)ns * npix, kstride = 3 * fstride;
  int s0 = g.b0 - kb, s1 = g.b1 - kb;
  if (s0 < 0) s0 += nz;
  if (s1 < 0) s1 += nz;
#pragma unroll
  for (int i = 0; i < AP; ++i) {
    const int a = a0 + i;
    if (a >= dc.n) return;
    R val = R(0);
    if (g.b0 >= 0) {
      const C* src = planes + a * kstride + pix;
      C v0[3], v1[3];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        v0[f] = src[f * fstride + (size_t)s0 * npix];
        v1[f] = src[f * fstride + (size_t)s1 * npix];
      }
      if (pix == 0) {
        if (g.b0 == 0) v0[0].x += dc.x[a], v0[1].x += dc.y[a];
        if (g.b1 == 0) v1[0].x += dc.x[a], v1[1].x += dc.y[a];
      }
      val = ewald_value<R>(g, v0, v1);
    }
    dst[(size_t)a * npix] = val;
  }
}

// Groups of at most 8 bins, as even as they come.
int bins_per_group(int ns) {
  const int G = (ns + 7) / 8, SB = (ns + G - 1) / G;
  return SB < 2 ? 2 : SB;
}

template <typename R, int SRC, int SB>
cudaError_t pol_planes_sb(const void* M, const void* nt, const void* dir, long long npix, int nz,
                          const PolParams<R>& pp, const AngleBatch<R>& ang, void* out, int kb,
                          int ns, const void* twz, cudaStream_t s) {
  using C = typename RT<R>::C;
  using F = Folded<C>;
  const int H1 = nz / 2 + 1, G = (ns + SB - 1) / SB, NSP = G * ((SB + 1) & ~1);
  // pixels of a block: all pair slots in use, whole 32-byte sectors per plane row
  constexpr int unit = 32 / (int)sizeof(C);
  const int PX = kPlPairs / H1 / unit * unit;
  if (PX < unit) return cudaErrorInvalidValue;
  // angles per step: up to 4 within ~100 KB (two FP32 blocks per SM), the
  // fewest idle threads in the last round of the items
  const size_t per = (size_t)H1 * 3 * PX * sizeof(F), twb = (size_t)H1 * NSP * sizeof(C);
  int A = 1;
  double best = 0.0;
  for (int a = 1; a <= 4 && a <= ang.n; ++a) {
    if (a > 1 && a * per + twb > 104 * 1024) break;
    const int items = a * 3 * G * PX, rounds = (items + kPlThreads - 1) / kPlThreads;
    const double eff = (double)items / (rounds * kPlThreads) + 0.02 * a;
    if (eff > best) best = eff, A = a;
  }
  const size_t smem = nz == 1 ? 0 : A * per + twb;
  auto kern = k_pol_planes<R, SRC, SB>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)((npix + PX - 1) / PX), kPlThreads, smem, s>>>(
      (const typename RT<R>::V4*)M, (const C*)nt, (const R*)dir, npix, nz, PX, A, kb, ns, pp, ang,
      (C*)out, (const C*)twz);
  return cudaGetLastError();
}

template <typename R, int SRC>
cudaError_t pol_planes_src(const void* M, const void* nt, const void* dir, long long npix, int nz,
                           const PolParams<R>& pp, const AngleBatch<R>& ang, void* out, int kb,
                           int ns, const void* twz, cudaStream_t s) {
#define RSX_PL(B) \
  case B: return pol_planes_sb<R, SRC, B>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, s);
  switch (bins_per_group(ns)) {
    RSX_PL(3) RSX_PL(4) RSX_PL(5) RSX_PL(6) RSX_PL(7) RSX_PL(8)
    default: return pol_planes_sb<R, SRC, 2>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, s);
  }
#undef RSX_PL
}
}  // namespace

bool pol_planes_fits(int precision, int nz, int ns) {
  if (nz < 1 || nz > kMaxPlanesNz || ns < 1 || ns > nz) return false;
  const size_t cs = precision == 32 ? sizeof(float2) : sizeof(double2);
  const int H1 = nz / 2 + 1, SB = bins_per_group(ns), G = (ns + SB - 1) / SB;
  return (2 * 3 * (size_t)kPlPairs + (size_t)H1 * G * ((SB + 1) & ~1)) * cs <= 220 * 1024;
}

template <typename R>
cudaError_t launch_pol_planes(const void* M, const void* nt, const void* dir, long long npix,
                              int nz, const PolParams<R>& pp, const AngleBatch<R>& ang, void* out,
                              int kb, int ns, const void* twz, cudaStream_t s) {
  if (nz < 1 || nz > kMaxPlanesNz || ns < 1 || ns > nz || kb < 0 || kb >= nz || ang.n < 1 ||
      ang.n > kMaxAngleBatch)
    return cudaErrorInvalidValue;
  return nt ? pol_planes_src<R, 1>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, s)
            : pol_planes_src<R, 0>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, s);
}

template <typename R>
cudaError_t launch_plane_images(const void* planes, int nx, int ny, int nz, int kb, int ns,
                                const Geo<R>* geo, const ImageDc<R>& dc, void* imgs,
                                cudaStream_t s) {
  using C = typename RT<R>::C;
  const long long npix = (long long)nx * ny;
  const unsigned gx = (unsigned)((npix + 255) / 256);
  // four angles per thread once one angle's pixels fill the chip
  if (npix >= (1 << 18))
    k_plane_images<R, 4><<<dim3(gx, (dc.n + 3) / 4), 256, 0, s>>>((const C*)planes, nx, ny, nz, kb,
                                                                  ns, geo, dc, (R*)imgs);
  else
    k_plane_images<R, 1><<<dim3(gx, dc.n), 256, 0, s>>>((const C*)planes, nx, ny, nz, kb, ns, geo,
                                                        dc, (R*)imgs);
  return cudaGetLastError();
}

#define RSX_INST(R)                                                                               \
  template cudaError_t launch_pol_planes<R>(const void*, const void*, const void*, long long, int, \
                                            const PolParams<R>&, const AngleBatch<R>&, void*, int, \
                                            int, const void*, cudaStream_t);                      \
  template cudaError_t launch_plane_images<R>(const void*, int, int, int, int, int,               \
                                              const Geo<R>*, const ImageDc<R>&, void*,            \
                                              cudaStream_t);
RSX_INST(float)
RSX_INST(double)
#undef RSX_INST

}  // namespace rsx
