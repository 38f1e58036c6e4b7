// The general planes path: Algorithm 1 or 2 for any grid with nz <= 255 in
// either precision, a batch of e-field angles at a time, and (z transform
// first too) the linearity path's five entries of N_t.
//
//   k_slice_means   a constant near each slice's mean, left out of p.
//   k_pol_planes, k_pol_planes_fft   per pixel column: the angle-independent
//                   sums of Eq. (polarization) once, then for each angle p, its
//                   z transform, and only the ns q_z planes the detector reads
//                   (the run kb .. kb + ns - 1 mod nz; see rsx_zfirst_plan).
//   k_x_planes, k_y_planes   the lateral transforms of those planes, in place,
//                   for tuned sizes (others: the general row and column FFTs).
//   k_plane_images  Eqs. (3Dscatter) and (Ewald): each pixel's two planes to
//                   the detector image, for every angle of the batch.
//   k_bins5_planes  the same for the linearity path's bins.
// The rotation and average follow as on the other paths.  The 3-D DFT is
// separable, so the values are the full transform's up to rounding order.
#include <cuda.h>  // CUtensorMap (the type only)
#include <string.h>

#include "rsx_device.cuh"
#include "rsx_kernels.h"
#include "rsx_pol.cuh"

namespace rsx {
namespace {

// The mean of each slice, left out of every voxel's sums before the z
// transform and returned at q = 0 (its transform lies there alone).  With the
// z transform first, the mean would ride through the lateral transforms of
// the few planes next to bin 0 and leave its rounding in every pixel of them.
// (FP32, unrotated image away from q = 0, error against 64 bits, in units of
// 1e-7, with the mean in and without, and transforming x and y first: six
// materials at 300 x 180 x 45 21, 2.0 and 5.3; with a substrate below the film
// 11, 1.3 and 1.6; one material at 45 x 512 x 16 6.4, 2.6 and 3.7.  Over 19
// shapes and 11 morphologies, relative to x and y first: 1.24 and 0.82.)
// Any constant near the mean serves, so it is that of 16 runs of 16 pixels
// (FP64, whose arithmetic is slow: 8 of 8), one pixel a thread, so that its few
// loads are all that is waited for.  Run r starts at floor((npix - len + 1)
// frac(r / golden ratio)), which no period of a lattice resonates with.
// means: [nz][kMeanStride] (MeanRow).
template <typename R> constexpr int kMeanRun = sizeof(R) == 4 ? 16 : 8;
template <typename R> constexpr int kMeanSample = kMeanRun<R> * kMeanRun<R>;
constexpr int kMeanVals = 13;

template <typename R>
__global__ void __launch_bounds__(kMeanSample<R>) k_slice_means(
    const typename RT<R>::V4* __restrict__ M, const typename RT<R>::C* __restrict__ nt,
    const R* __restrict__ dir, long long npix, int nz, const __grid_constant__ PolParams<R> pp,
    int literal, R* __restrict__ means) {
  using C = typename RT<R>::C;
  constexpr int LEN = kMeanRun<R>, NS = kMeanSample<R>, NW = NS / 32;
  const int t = threadIdx.x, z = blockIdx.x;
  const long long N = npix * nz;
  const int S = npix < NS ? (int)npix : NS;
  TAcc<R> a;
  tacc_zero(a);
  if (t < S) {
    const unsigned long long g = (unsigned)(t / LEN) * 2654435769u;  // 2^32 frac(run / golden ratio)
    const size_t v =
        (size_t)z * npix +
        (npix <= NS ? (size_t)t : (size_t)(g * (npix - LEN + 1) >> 32) + (size_t)(t % LEN));
    if (nt) {
#pragma unroll
      for (int e = 0; e < 5; ++e) {
        const C q = nt[(size_t)e * N + v];
        a.t[e][0] = q.x;
        a.t[e][1] = q.y;
      }
      PTen<R> p;
      pten_of(p, a.as, a.t, literal != 0);  // (a.as is 0)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        a.t[0][i] = p.a[i];
        a.t[2][i] = p.b[i];
      }
    } else {
#pragma unroll 4
      for (int j = 0; j < pp.c; ++j) {
        const typename RT<R>::V4 m = M[(size_t)j * N + v];
        if (dir) {
          const R* dj = dir + (size_t)j * 3 * N + v;
          tacc_add_d(a, (R)m.x, (R)m.y, dj[0], dj[N], dj[2 * N], pp, j);
        } else {
          tacc_add(a, (R)m.x, (R)m.y, (R)m.z, (R)m.w, pp, j);
        }
      }
      a.aw -= R(1);
    }
  }
  __shared__ R part[NW][kMeanVals];
#pragma unroll
  for (int q = 0; q < kMeanVals; ++q) {
    R s = q < 10 ? a.t[q >> 1][q & 1] : q < 12 ? a.as[q & 1] : a.aw;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if ((t & 31) == 0) part[t >> 5][q] = s;
  }
  __syncthreads();
  if (t < kMeanVals) {
    R m = R(0);
#pragma unroll
    for (int k = 0; k < NW; ++k) m += part[k][t];
    means[(size_t)z * kMeanStride + t] = m / (R)S;
  }
}

// What leaving the means out takes from p at q = 0: PTen's ten numbers of npix
// times their sum over z, in double.  A block of 256 threads calls
// means_total, then those that want the result means_pten (FP64 arithmetic:
// not more threads than need be).  from_nt: the rows are PTen's already.  The
// value at q = 0 is rounded once, when what was left out has been added: it
// outweighs the rest of the image.
template <typename R>
__device__ __forceinline__ void means_total(const R* __restrict__ means, int nz, long long npix,
                                            double* total) {
  const int t = threadIdx.x, q = t >> 4;
  double m = 0.0;
  if (q < kMeanVals)
    for (int k = t & 15; k < nz; k += 16) m += (double)means[(size_t)k * kMeanStride + q];
#pragma unroll
  for (int d = 8; d > 0; d >>= 1) m += __shfl_xor_sync(0xffffffffu, m, d);
  if ((t & 15) == 0 && q < kMeanVals) total[q] = m * (double)npix;
  __syncthreads();
}
__device__ __forceinline__ void means_pten(const double* total, bool literal, bool from_nt,
                                           PTen<double>& out) {
  const double sc = from_nt ? 1.0 : 1.0 / kFourPi;
  const bool half = literal && !from_nt;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double* q = total + i;
    const double ar = q[10] + (i == 0 ? total[12] : 0.0);
    out.a[i] = sc * (half ? ar + 0.5 * (q[0] + q[4]) : ar + q[0]);
    out.b[i] = sc * (half ? 0.5 * (q[0] - q[4]) : ar + q[4]);
    out.xy[i] = sc * q[2];
    out.xz[i] = sc * q[6];
    out.yz[i] = sc * q[8];
  }
}

// A field at a fold's voxels: sum and difference.
template <typename C> struct Folded {
  C s, d;
};

constexpr int kPlThreads = 256, kPlVoxels = 4;  // voxels a thread holds

// it / d for it < 2^11 and d <= 512, with magic(d): exact while it d < 2^20
__host__ __device__ constexpr unsigned magic(unsigned d) { return (1u << 20) / d + 1; }
__device__ __forceinline__ int div_by(int it, unsigned m) { return (int)(((unsigned)it * m) >> 20); }

// A block owns PX adjacent pixels (flat index y nx + x) by the whole stack.
// The z transform is evaluated as a sum over the bins that are kept, the
// voxels folded first.  Odd nz: with S = p(z) + p(nz - z), D = p(z) - p(nz - z),
//   X(k) = sum_{z <= nz/2} cos(t) S - i sin(t) D,  t = 2 pi k z / nz
// (z = 0 alone).  EVEN nz, L = nz / 2: the even bins see a(z) = p(z) +
// p(z + L) and the odd ones b(z) = p(z) - p(z + L), z < L, each folded once
// more: S = a(z) + a(L - z), D = a(z) - a(L - z), or S = b(z) - b(L - z),
// D = b(z) + b(L - z), in the same sum over z <= L/2 (z = 0 and L/2 alone).
// So a kept bin takes 2 fused multiply-adds per voxel and field for odd nz
// and 1 for even: ns of them, 7 at nz = 16 and 28 at nz = 45 (5 nm, 270 eV),
// against ~10 to 25 for an FFT that would need a plan for every nz.  Before
// the sum its z = 0 term is taken off the even bins' whole column and
// returned to bin 0 (the other bins of a constant are 0): of a column that
// hardly changes along z (a lattice of rods, less the slices' means) the sum
// as it stands would leave its rounding in every bin, where the first stages
// of an FFT cancel it.
// A thread keeps the angle-independent sums of its 4 voxels (one quad, or
// two pairs) in registers for all angles.  Per step of A angles: every thread
// forms p of its voxels for each angle and stores the folds (three fields) to
// shared memory; then the block's threads take (angle, field, group of SB
// bins of one parity, pixel) items.
// SRC 0: morphology (dir: FP64's cached director); 1: Algorithm 2's N_t.
// twt: exp(-2 pi i j / nz), j < nz.
template <typename R, int SRC, int SB, bool EVEN>
__global__ void __launch_bounds__(kPlThreads, sizeof(R) == 4 ? 2 : 1) k_pol_planes(
    const typename RT<R>::V4* __restrict__ M, const typename RT<R>::C* __restrict__ nt,
    const R* __restrict__ dir, long long npix, int nz, int PX, int A, int kb, int ns,
    const __grid_constant__ PolParams<R> pp, const __grid_constant__ AngleBatch<R> ang,
    typename RT<R>::C* __restrict__ out, const typename RT<R>::C* __restrict__ twz,
    const R* __restrict__ means) {
  using C = typename RT<R>::C;
  using F = Folded<C>;
  constexpr int SBP = (SB + 1) & ~1;  // twiddles of a group, padded to pairs
  constexpr int NP = EVEN ? 2 : 1;    // parities of the bins
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int t = threadIdx.x;
  const int L = EVEN ? nz / 2 : nz, H = L / 2 + 1;  // terms of the folded sum
  const int odd0 = kb & 1;                          // parity of plane 0's bin
  const int n0 = EVEN ? (ns + 1 - odd0) / 2 : ns;   // kept bins of parity 0
  const int G0 = (n0 + SB - 1) / SB, G = G0 + (EVEN ? (ns - n0 + SB - 1) / SB : 0);
  const int NSP = G * SBP;
  F* buf = reinterpret_cast<F*>(smem_raw);                        // [A][NP][H][3][PX]
  C* tw = reinterpret_cast<C*>(buf + (size_t)A * NP * H * 3 * PX);  // [H][NSP]
  const long long N = npix * nz;
  const long long pix0 = (long long)blockIdx.x * PX;
  const int npx = npix - pix0 < PX ? (int)(npix - pix0) : PX;
  // bin i of group g: plane first(g) + NP i
  auto first = [&](int g) {
    return !EVEN ? g * SB : g < G0 ? odd0 + 2 * g * SB : 1 - odd0 + 2 * (g - G0) * SB;
  };
  for (int i = t; nz > 1 && i < H * NSP; i += kPlThreads) {  // (nz = 1 has no shared memory)
    const int z = i / NSP, r = i - z * NSP, g = r / SBP, b = first(g) + NP * (r - g * SBP);
    tw[i] = twz[(unsigned)((kb + b) * z) % (unsigned)nz];  // ((kb + b) z < 2^16)
  }

  // this thread's voxels: the sums of Eq. (polarization), divided by 4 pi.
  // EVEN: z, z + L, L - z, nz - z of one pixel; else z, nz - z of two
  const bool literal = pp.literal != 0;
  PTen<R> ten[kPlVoxels];
  int at[2];     // shared-memory place of each fold (field 0, angle 0); -1: none
  bool two[2];   // its second half exists (z is not alone)
#pragma unroll
  for (int sl = 0; sl < 2; ++sl) {
    const int q = EVEN ? t : t + sl * kPlThreads, z = q / PX, px = q - z * PX;
    const bool in = z < H && px < npx;
    at[sl] = in ? z * 3 * PX + px : -1;
    two[sl] = in && z > 0 && 2 * z != L;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      pten_zero(ten[2 * sl + h]);
      // EVEN: slot 0 holds z and z + L, slot 1 L - z and nz - z
      const int zv = EVEN ? (sl ? L - z : z) + (h ? L : 0) : h ? nz - z : z;
      const bool have = EVEN ? (sl ? two[sl] : in) : h ? two[sl] : in;
      if (!have) continue;
      const size_t i = (size_t)(EVEN && sl && h ? nz - z : zv) * npix + pix0 + px;
      if constexpr (SRC == 1) {
        const R none[2] = {R(0), R(0)};
        R tt[5][2];
#pragma unroll
        for (int e = 0; e < 5; ++e) {
          const C v = ld_stream(nt + (size_t)e * N + i);
          tt[e][0] = v.x;
          tt[e][1] = v.y;
        }
        pten_of(ten[2 * sl + h], none, tt, literal);
        if (means) pten_less(ten[2 * sl + h], means + zv * kMeanStride);
      } else {
        TAcc<R> a;
        if (means) tacc_start(a, means + zv * kMeanStride);
        else tacc_zero(a);
        for (int j = 0; j < pp.c; ++j) {
          const typename RT<R>::V4 m = ld_stream(M + (size_t)j * N + i);
          if (dir) {
            const R* dj = dir + (size_t)j * 3 * N + i;
            tacc_add_d(a, (R)m.x, (R)m.y, dj[0], dj[N], dj[2 * N], pp, j);
          } else {
            tacc_add(a, (R)m.x, (R)m.y, (R)m.z, (R)m.w, pp, j);
          }
        }
        pten_of(ten[2 * sl + h], a, literal);
      }
    }
  }

  const size_t fstride = (size_t)ns * npix, kstride = 3 * fstride;
  if (nz == 1) {  // no z transform: the pixel's p is its plane
    for (int k = 0; k < ang.n; ++k) {
#pragma unroll
      for (int sl = 0; sl < 2; ++sl) {
        if (at[sl] < 0) continue;
        C p[3];
        p_from_pten(ten[2 * sl], ang.ce[k], ang.se[k], ang.c2[k], ang.s2[k], literal, p);
        C* o = out + k * kstride + pix0 + at[sl];
        o[0] = p[0];
        o[fstride] = p[1];
        o[2 * fstride] = p[2];
      }
    }
    return;
  }
  const unsigned mpx = magic(PX), mg = magic(G), m3 = magic(3);
  const int s_bin0 = kb == 0 ? 0 : nz - kb;  // bin 0's plane
  for (int a0 = 0; a0 < ang.n; a0 += A) {
    const int na = ang.n - a0 < A ? ang.n - a0 : A;
    if (a0 > 0) __syncthreads();  // the previous step's reads are done
    for (int a = 0; a < na; ++a) {
      const R ce = ang.ce[a0 + a], se = ang.se[a0 + a], c2 = ang.c2[a0 + a], s2 = ang.s2[a0 + a];
      F* ba = buf + (size_t)a * NP * H * 3 * PX;
      if constexpr (EVEN) {
        if (at[0] < 0) continue;
        C p[4][3];
#pragma unroll
        for (int v = 0; v < 4; ++v)
          p_from_pten(ten[v], ce, se, c2, s2, literal, p[v]);
#pragma unroll
        for (int f = 0; f < 3; ++f) {  // (a voxel that does not exist has p = 0)
          const C a1 = cadd(p[0][f], p[1][f]), b1 = csub(p[0][f], p[1][f]);
          const C a2 = cadd(p[2][f], p[3][f]), b2 = csub(p[2][f], p[3][f]);
          F v;
          v.s = cadd(a1, a2);
          v.d = csub(a1, a2);
          ba[at[0] + f * PX] = v;
          v.s = csub(b1, b2);
          v.d = cadd(b1, b2);
          ba[at[0] + (H * 3 + f) * PX] = v;
        }
      } else {
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
          if (at[sl] < 0) continue;
          C p[3], q[3];
          p_from_pten(ten[2 * sl], ce, se, c2, s2, literal, p);
          p_from_pten(ten[2 * sl + 1], ce, se, c2, s2, literal, q);
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            F v;
            v.s = cadd(p[f], q[f]);
            v.d = csub(p[f], q[f]);
            ba[at[sl] + f * PX] = v;
          }
        }
      }
    }
    __syncthreads();
    const int items = na * 3 * G * PX;
    for (int it = t; it < items; it += kPlThreads) {
      int r = div_by(it, mpx);
      const int px = it - r * PX;
      int q = div_by(r, mg);
      const int g = r - q * G, a = div_by(q, m3), f = q - 3 * a;
      if (px >= npx) continue;
      const int par = EVEN && g >= G0;
      const F* b = buf + ((size_t)(a * NP + par) * H * 3 + f) * PX + px;
      const C* w = tw + g * SBP;
      // z = 0: the even bins' base (see above), the odd bins' first term
      const C p0 = b[0].s;
      C x[SB];
#pragma unroll
      for (int i = 0; i < SB; ++i) x[i] = par ? p0 : RT<R>::mk(R(0), R(0));
      const R once = par ? R(0) : R(1), twice = par ? R(0) : R(2);
      for (int z = 1; z < H; ++z) {
        F v = b[z * 3 * PX];
        const R n = 2 * z == L ? once : twice;
        v.s.x = fma(-n, p0.x, v.s.x);
        v.s.y = fma(-n, p0.y, v.s.y);
        C wv[SBP];
#pragma unroll
        for (int i = 0; i < SBP; ++i) wv[i] = w[z * NSP + i];
#pragma unroll
        for (int i = 0; i < SB; ++i) {  // (cos, -sin) = (wv.x, wv.y)
          x[i].x = fma(wv[i].x, v.s.x, fma(-wv[i].y, v.d.y, x[i].x));
          x[i].y = fma(wv[i].x, v.s.y, fma(wv[i].y, v.d.x, x[i].y));
        }
      }
      const int s0 = first(g);
      C* o = out + (size_t)(a0 + a) * kstride + (size_t)f * fstride + (size_t)s0 * npix + pix0 + px;
#pragma unroll
      for (int i = 0; i < SB; ++i) {
        if (s0 + NP * i == s_bin0) {
          x[i].x = fma(R(L), p0.x, x[i].x);
          x[i].y = fma(R(L), p0.y, x[i].y);
        }
        if (s0 + NP * i < ns) o[(size_t)(NP * i) * npix] = x[i];
      }
    }
  }
}

// The same pass for nz = 4 Q, Q = 2, 4, 8, 16 or 32, by a decimation in
// frequency: z = n2 + Q n1, and plane s = 4 s2 + s1 holds bin kb + s:
//   X(kb + s) = sum_n2 W_Q^(n2 s2) W_nz^(n2 (kb + s1)) sum_n1 x[n2 + Q n1] W_4^(n1 (kb + s1)).
// A block owns PX = 256 / Q pixels; thread (n2, pixel) holds the
// angle-independent sums of its four voxels n1 in registers for all angles.
// Per step of A angles it forms their p, does the 4-point transform over n1
// and the twiddles (its own four, in registers) and stores u[s1][n2] of the
// three fields to shared memory (thread order: contiguous); then the threads
// take (angle, field, s1, pixel) items: a Q-point transform over n2 in
// registers, whose first outputs s2 go straight to their planes (Q = 32: only
// the kept ones are evaluated).  119 instructions per voxel and angle at
// nz = 16 and 74 % issue (1024 x 1024 x 16, c = 3, 18 angles: 1.22 ms), where the
// folded sums above took 160 at 64 % (1.88 ms).  Two energies of 91 angles there:
// the pass 19.0 ms, 12.2 so; Algorithm 2 at 1024 x 1024 x 32, 37 angles: 16.5 and
// 12.3 (FP32, nz <= 32: three blocks per SM).
// NF = 3: the fields of p of every angle.  NF = 5: the linearity path's five
// entries of N_t (xx, xy, yy, xz, yz, the constant left out), once.
template <typename R, int Q> struct PlFft {
  static constexpr int PX = kPlThreads / Q;
  // u's stride between s1: padded where a half-warp spans two of them
  static constexpr int KS = kPlThreads + (PX * (int)sizeof(typename RT<R>::C) < 128 ? PX : 0);
  // angles per step: the items (12 PX per angle) fill the block
  static constexpr int A = sizeof(R) == 8 ? (Q >= 8 ? 2 : 1) : Q >= 16 ? 4 : Q == 8 ? 2 : 1;
};

template <typename R, int SRC, int Q, int NF>
__global__ void __launch_bounds__(kPlThreads, sizeof(R) == 8 ? 1 : Q <= 8 && NF == 3 ? 3 : 2) k_pol_planes_fft(
    const typename RT<R>::V4* __restrict__ M, const typename RT<R>::C* __restrict__ nt,
    const R* __restrict__ dir, long long npix, int kb, int ns,
    const __grid_constant__ PolParams<R> pp, const __grid_constant__ AngleBatch<R> ang,
    typename RT<R>::C* __restrict__ out, const typename RT<R>::C* __restrict__ twz,
    const R* __restrict__ means) {
  using C = typename RT<R>::C;
  using P = PlFft<R, Q>;
  constexpr int NZ = 4 * Q, PX = P::PX, KS = P::KS, A = NF == 3 ? P::A : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // N_t: the rows of the slices' means a warp needs (4 n1, NR n2), fetched by
  // the warp itself, so that no warp waits for another's loads
  constexpr int NR = PX >= 32 ? 1 : 32 / PX, kRow = kMeanStride * (int)sizeof(R);
  constexpr int NM = SRC == 1 ? kPlThreads / 32 * 4 * NR * kRow : 0;
  unsigned char* const mean_s = smem_raw + (threadIdx.x >> 5) * 4 * NR * kRow;
  C* buf = reinterpret_cast<C*>(smem_raw + NM);  // [A][NF][4][KS]
  const int t = threadIdx.x, px = t % PX, n2 = t / PX;
  if constexpr (SRC == 1) {
    constexpr int CH = 10 * (int)sizeof(R) / 16 + (sizeof(R) == 4);  // 16-byte pieces in use
    const int first = (t & ~31) / PX;                                // the warp's lowest n2
    for (int i = t & 31; i < 4 * NR * CH; i += 32) {
      const int r = i / CH, c = i % CH, z = first + r % NR + Q * (r / NR);
      cp_async_pair(reinterpret_cast<float2*>(mean_s + r * kRow + c * 16),
                    reinterpret_cast<const float2*>(
                        reinterpret_cast<const unsigned char*>(means) + z * kRow + c * 16));
    }
  }
  const long long N = npix * NZ;
  const long long pix0 = (long long)blockIdx.x * PX;
  const int npx = npix - pix0 < PX ? (int)(npix - pix0) : PX;
  // NF = 5: the lab frame's terms are N_t's entries themselves
  const bool literal = NF == 3 && pp.literal != 0;
  PTen<R> ten[4];
  C w[4];
#pragma unroll
  for (int n1 = 0; n1 < 4; ++n1) {
    w[n1] = twz[(n2 * (kb + n1)) % NZ];
    pten_zero(ten[n1]);
  }
  if (px < npx) {
    const size_t i = (size_t)n2 * npix + pix0 + px, step = (size_t)Q * npix;
    if constexpr (SRC == 1) {
      const R none[2] = {R(0), R(0)};
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) {
        R tt[5][2];
#pragma unroll
        for (int e = 0; e < 5; ++e) {
          const C v = ld_stream(nt + (size_t)e * N + i + n1 * step);
          tt[e][0] = v.x;
          tt[e][1] = v.y;
        }
        pten_of(ten[n1], none, tt, literal);
      }
    } else {
      TAcc<R> acc[4];
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) tacc_start(acc[n1], means + (n2 + Q * n1) * kMeanStride);
      for (int j = 0; j < pp.c; ++j) {
        const typename RT<R>::V4* Mj = M + (size_t)j * N + i;
        typename RT<R>::V4 m[4];
#pragma unroll
        for (int n1 = 0; n1 < 4; ++n1) m[n1] = ld_stream(Mj + n1 * step);
        const R* dj = dir + (size_t)j * 3 * N + i;
#pragma unroll
        for (int n1 = 0; n1 < 4; ++n1) {
          if (dir)
            tacc_add_d(acc[n1], (R)m[n1].x, (R)m[n1].y, dj[n1 * step], dj[N + n1 * step],
                       dj[2 * N + n1 * step], pp, j);
          else
            tacc_add(acc[n1], (R)m[n1].x, (R)m[n1].y, (R)m[n1].z, (R)m[n1].w, pp, j);
        }
      }
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) pten_of(ten[n1], acc[n1], literal);
    }
  }
  if constexpr (SRC == 1) {
    // (the means come while N_t does, and are taken off when both are here)
    cp_async_wait_all();
    __syncwarp();
    if (px < npx) {
      const int j = n2 - (t & ~31) / PX;
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1)
        pten_less(ten[n1], reinterpret_cast<const R*>(mean_s + (n1 * NR + j) * kRow));
    }
  }
  const size_t fstride = (size_t)ns * npix;
  const int rot = kb & 3;  // s1 = 0 takes output kb mod 4 of the 4-point transform
  const int nang = NF == 3 ? ang.n : 1;
  for (int a0 = 0; a0 < nang; a0 += A) {
    const int na = nang - a0 < A ? nang - a0 : A;
    if (a0 > 0) __syncthreads();  // the previous step's reads are done
    for (int a = 0; a < na; ++a) {
      C p[4][NF];
      if constexpr (NF == 3) {
        const R ce = ang.ce[a0 + a], se = ang.se[a0 + a], c2 = ang.c2[a0 + a], s2 = ang.s2[a0 + a];
#pragma unroll
        for (int n1 = 0; n1 < 4; ++n1) p_from_pten(ten[n1], ce, se, c2, s2, literal, p[n1]);
      } else {
#pragma unroll
        for (int n1 = 0; n1 < 4; ++n1) {
          const PTen<R>& q = ten[n1];
          p[n1][0] = RT<R>::mk(q.a[0], q.a[1]);
          p[n1][1] = RT<R>::mk(q.xy[0], q.xy[1]);
          p[n1][2] = RT<R>::mk(q.b[0], q.b[1]);
          p[n1][NF - 2] = RT<R>::mk(q.xz[0], q.xz[1]);
          p[n1][NF - 1] = RT<R>::mk(q.yz[0], q.yz[1]);
        }
      }
      C* b = buf + a * NF * 4 * KS + t;
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        dft4(p[0][f], p[1][f], p[2][f], p[3][f]);
        // output k1 goes to s1 = (k1 - kb) mod 4 (uniform)
#pragma unroll
        for (int s1 = 0; s1 < 4; ++s1) {
          const C v = rot == 0   ? p[s1][f]
                      : rot == 1 ? p[(s1 + 1) & 3][f]
                      : rot == 2 ? p[(s1 + 2) & 3][f]
                                 : p[(s1 + 3) & 3][f];
          b[(f * 4 + s1) * KS] = cmul(v, w[s1]);
        }
      }
    }
    __syncthreads();
    const int items = na * 4 * NF * PX;
    for (int it = t; it < items; it += kPlThreads) {
      const int q = it % PX, r = it / PX, s1 = r & 3, af = r >> 2;  // af = NF a + f
      if (q >= npx) continue;
      const C* b = buf + r * KS + q;
      C v[Q];
#pragma unroll
      for (int n = 0; n < Q; ++n) v[n] = b[n * PX];
      C* o = out + (size_t)(NF * a0 + af) * fstride + (size_t)s1 * npix + pix0 + q;
      const int mine = (ns - s1 + 3) >> 2;  // kept s2 of this s1
      if constexpr (Q == 32) {
        if (ns <= 64) {
          dft32_first(v, (ns + 3) >> 2, [&](int s2, C x) {
            if (s2 < mine) o[(size_t)(4 * s2) * npix] = x;
          });
        } else {
          dft32(v);
#pragma unroll
          for (int s2 = 0; s2 < 32; ++s2)
            if (s2 < mine) o[(size_t)(4 * s2) * npix] = v[s2];
        }
      } else {
        dft_reg<Q>(v);
#pragma unroll
        for (int s2 = 0; s2 < Q; ++s2)
          if (s2 < mine) o[(size_t)(4 * s2) * npix] = v[out_pos<Q>(s2)];
      }
    }
  }
}

// Images of the angles of a batch from their transformed planes: per pixel
// its two planes (b - kb mod nz) of the three fields, what was left out of p
// before the transform returned at q = 0 (the constant's x and y parts per
// angle, and the slices' means, null: none), the projection and the
// interpolation; written in fftshift order.  A thread takes AP angles of one
// pixel, so the 32-byte geometry is read once for them; q = 0 has a block of its own, and with AP = 4 the registers are held to
// what the other blocks need (2048 x 2048 film, 182 angles: 5.05 ms; 5.37 with
// q = 0's 40 registers, 6.4 with its code behind the loop).
// planes has kstride = 3 ns npix complex per angle.
template <typename R, int AP>
__global__ void __launch_bounds__(256, sizeof(R) == 8 ? 4 : AP == 4 ? 8 : 5) k_plane_images(const typename RT<R>::C* __restrict__ planes,
                                                      int nx, int ny, int nz, int kb, int ns,
                                                      const Geo<R>* __restrict__ geo,
                                                      const __grid_constant__ ImageDc<R> dc,
                                                      const R* __restrict__ means, int literal,
                                                      int from_nt, R* __restrict__ imgs) {
  using C = typename RT<R>::C;
  const long long npix = (long long)nx * ny;
  const size_t fstride = (size_t)ns * npix, kstride = 3 * fstride;
  if (blockIdx.x == 0) {  // q = 0, an angle per thread: with what was left out
    if (blockIdx.y > 0) return;
    const int a = threadIdx.x;
    // (the loads first: they and the means' arrive together)
    const Geo<R> g = geo[0];
    const int s0 = g.b0 < kb ? g.b0 - kb + nz : g.b0 - kb, s1 = g.b1 < kb ? g.b1 - kb + nz : g.b1 - kb;
    C v0[3], v1[3];
    if (a < dc.n) {
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const C* src = planes + a * kstride + f * fstride;
        v0[f] = src[(size_t)s0 * npix];
        v1[f] = src[(size_t)s1 * npix];
      }
    }
    __shared__ double sum[kMeanVals];
    if (means) means_total<R>(means, nz, npix, sum);
    if (a >= dc.n) return;
    PTen<double> total;
    pten_zero(total);
    if (means) means_pten(sum, literal != 0, from_nt != 0, total);
    double2 d[3];
    p_from_pten<double>(total, dc.ce[a], dc.se[a], dc.c2[a], dc.s2[a], literal != 0, d);
    d[0].x += dc.x[a];
    d[1].x += dc.y[a];
    auto plus = [](C v, double2 w) { return RT<R>::mk((R)(v.x + w.x), (R)(v.y + w.y)); };
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if (g.b0 == 0) v0[f] = plus(v0[f], d[f]);
      if (g.b1 == 0) v1[f] = plus(v1[f], d[f]);
    }
    imgs[(size_t)a * npix + (size_t)(ny / 2) * nx + nx / 2] = ewald_value<R>(g, v0, v1);
    return;
  }
  const long long pix = (long long)(blockIdx.x - 1) * blockDim.x + threadIdx.x;
  if (pix == 0 || pix >= npix) return;
  const Geo<R> g = geo[pix];
  const int my = (int)(pix / nx), mx = (int)(pix - (long long)my * nx);
  int sy = my + ny / 2, sx = mx + nx / 2;
  if (sy >= ny) sy -= ny;
  if (sx >= nx) sx -= nx;
  R* dst = imgs + (size_t)sy * nx + sx;
  const int a0 = blockIdx.y * AP;
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
      val = ewald_value<R>(g, v0, v1);
    }
    dst[(size_t)a * npix] = val;
  }
}

// --------------------------------------------------- y pass of the planes
// In-place y-FFT of the kept planes (FP32, ny = 512, 1024 or 2048, nx a
// multiple of 16) that stores only what the image reads: a pixel's value in a
// plane is kept when that plane is one of the pixel's two bins.
//
// The planes a column meets: the bins of its pixels run from the one at the
// largest |q_y| up to the one at q_y = 0, so a 16-column group needs one run
// of planes (YRuns, bounds from the host).  Summed over the groups that is
// ~52 % of the planes (1024 x 1024 x 128 at 5 nm and 270 eV); the rest is
// never read here.
//
// A step is one (angle, field, 16-column group, plane): TPG = ny / 512 tiles
// of 8192 elements (a group's 128-byte lines are read by one block, tile
// after tile).  The steps are cut into one contiguous range per persistent
// block of two 256-thread groups; thread group g takes the block's tiles
// i = g, g + 2, ...  Three tile buffers rotate: while two tiles are
// transformed the next is in flight.  A tile arrives by tensor copies; each
// thread holds 32 of its elements in registers, transforms them, and the
// tile is transposed through the buffer it came in (three 256-thread barriers
// a tile; one shared write and two reads per element, where the
// split-halves form this replaces took three and four).
//   ny = 1024 = 32 x 32: 8 columns; thread (n1, col) does the 32-point DFT over n2
//       (n = n1 + 32 n2), W1024^(n1 k2), then thread (k2, col) the one over
//       n1: rows k2 + 32 k1.
//   ny = 2048: 4 columns; threads 0-127 the even outputs, 128-255 the odd
//       ones (a radix-2 decimation in frequency as the tile is read:
//       a = x[n] + x[n + 1024], b = (x[n] - x[n + 1024]) W2048^n), each a
//       1024-point transform as above: rows 2 (k2 + 32 k1) + odd.
//   ny = 512 = 16 x 32: 16 columns; thread (n1, col) does the 32-point DFT
//       over n2 (n = n1 + 16 n2), W512^(n1 k2), then two 16-point DFTs, k2
//       and k2 + 16: rows k2 + 32 k1.
// A thread's pixels' plane indices are packed as bytes in registers, loaded
// when the column group changes.  Waits are bounded; on a timeout the block
// sets *err and its abort flag, both groups leave their loops, and thread 0
// waits (bounded) for the copies in flight.
template <int NY> struct YTile {
  static constexpr int TX = 8192 / NY, TPG = 16 / TX;
  static constexpr int BUF = NY == 512 ? 8192 : 8448;  // elements: the tile, or its padded transpose
  static constexpr int NTW = NY == 2048 ? 1024 + 1024 : NY;
  static constexpr int NQ = NY == 2048 ? 2 : 1;  // tiles of a step one thread group sees
};
constexpr int kYBufs = 3;

// v[n] *= tw[n * stride] for n = 1..31
template <int STRIDE>
__device__ __forceinline__ void tw_rows(float2* v, const float2* tw) {
#pragma unroll
  for (int n = 1; n < 32; ++n) v[n] = cmul(v[n], tw[n * STRIDE]);
}

template <int NY>
__global__ void __launch_bounds__(512, 1) k_y_planes(
    const __grid_constant__ CUtensorMap tmap, const __grid_constant__ YRuns runs, int nx, int nz,
    int kb, int ns, int L, int T, const unsigned short* __restrict__ b0idx,
    const float2* __restrict__ tw_g, const float2* __restrict__ twy_g, float2* __restrict__ p,
    int* __restrict__ err, unsigned poll) {
  using C = float2;
  using Y = YTile<NY>;
  constexpr int TX = Y::TX, TPG = Y::TPG, BUF = Y::BUF, NQ = Y::NQ;
  constexpr unsigned kPoll = 1u << 22;
  extern __shared__ __align__(128) unsigned char smem_a128[];
  C* bufs = reinterpret_cast<C*>(smem_a128);  // [kYBufs][BUF]
  C* tw = bufs + kYBufs * BUF;                 // [NTW]
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(tw + Y::NTW);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar + kYBufs);
  volatile int* issued = abort_flag + 1;  // [kYBufs] loads issued into each buffer
  const int t = threadIdx.x & 255, g = threadIdx.x >> 8;
  const int s0 = (int)blockIdx.x * L;
  const int s1 = s0 + L < T ? s0 + L : T;
  if (s0 >= s1) return;
  const int ntile = (s1 - s0) * TPG;
  const int S = runs.start[runs.n];
  const size_t npix = (size_t)NY * nx;

  // step -> (angle and field af, column group cg, plane z); next() advances
  struct Step {
    int af, cg, z;
  };
  auto locate = [&](int st) {
    Step q;
    q.af = st / S;
    const int r = st - q.af * S;
    int lo = 0, hi = runs.n - 1;  // the last group with start <= r that has steps
    while (lo < hi) {
      const int m = (lo + hi + 1) >> 1;
      if (runs.start[m] <= r) lo = m;
      else hi = m - 1;
    }
    q.cg = lo;
    q.z = runs.first[lo] + (r - runs.start[lo]);
    return q;
  };
  auto next = [&](Step& q) {
    if (q.z - runs.first[q.cg] + 1 < runs.start[q.cg + 1] - runs.start[q.cg]) {
      ++q.z;
      return;
    }
    do {
      if (++q.cg == runs.n) q.cg = 0, ++q.af;
    } while (runs.start[q.cg + 1] == runs.start[q.cg]);
    q.z = runs.first[q.cg];
  };
  auto issue = [&](const Step& q, int i) {  // tile i of the block (one thread)
    const int b = i % kYBufs, x = q.cg * 32 + (i % TPG) * (2 * TX);
    mbar_expect_tx(&bar[b], 8192 * sizeof(C));
#pragma unroll
    for (int k = 0; k < NY / 256; ++k)
      tma_load_3d(bufs + b * BUF + k * 256 * TX, &tmap, x, k * 256, q.af * ns + q.z, &bar[b]);
    __threadfence_block();  // the count follows the barrier's arrival
    issued[b] = issued[b] + 1;
  };

  if (threadIdx.x == 0) {
    for (int b = 0; b < kYBufs; ++b) {
      mbar_init(&bar[b], 1);
      issued[b] = 0;
    }
    *abort_flag = 0;
    fence_proxy_async();
  }
  // W1024^(n1 k2) as [32][32] (1024 and 2048 rows; then W2048^n, n < 1024), or W512^j
  for (int i = threadIdx.x; i < (NY == 512 ? 512 : 1024); i += 512) tw[i] = tw_g[i];
  if constexpr (NY == 2048)
    for (int i = threadIdx.x; i < 1024; i += 512) tw[1024 + i] = twy_g[i];
  __syncthreads();
  if (threadIdx.x == 0) {
    Step q = locate(s0);
    for (int i = 0; i < kYBufs && i < ntile; ++i) {
      issue(q, i);
      if ((i + 1) % TPG == 0 && i + 1 < ntile) next(q);
    }
  }

  // this thread's place: c its column; stage 1 line n1, stage 2 line k2
  const int c = t & (TX - 1), hi = t / TX;
  const int odd = NY == 2048 ? hi >> 5 : 0;    // warp-uniform
  const int ln = NY == 2048 ? hi & 31 : hi;    // n1 in stage 1, k2 in stage 2
  Step q = locate(s0), ahead = q;  // this group's tile; the tile kYBufs later (thread t = 0)
  int qi = 0, ai = 0;              // their step numbers, relative to s0
  int last_af = -1, last_cg = -1;
  uint4 sb[NQ][2];  // plane indices of this thread's 32 pixels, as bytes
  for (int i = g; i < ntile; i += 2) {
    while (qi < i / TPG) next(q), ++qi;
    const int b = i % kYBufs, x0 = q.cg * 16 + (i % TPG) * TX;
    if (q.cg != last_cg || q.af != last_af) {
      last_cg = q.cg;
      last_af = q.af;
#pragma unroll
      for (int h = 0; h < NQ; ++h) {
        // 2048 rows: the group's tiles are quarters g (h = 0) and g + 2
        const int col = NY == 2048 ? q.cg * 16 + (g + 2 * h) * TX + c : x0 + c;
        unsigned w[8];
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          const int row = NY == 512 ? (k & 15) * 32 + ln + (k >> 4) * 16
                          : NY == 2048 ? 2 * (ln + 32 * k) + odd
                                       : ln + 32 * k;
          int d = (int)b0idx[(size_t)row * nx + col] - kb;
          if (d < 0) d += nz;
          w[k >> 2] = (k & 3) ? w[k >> 2] | (unsigned)d << (8 * (k & 3)) : (unsigned)d;
        }
        sb[h][0] = make_uint4(w[0], w[1], w[2], w[3]);
        sb[h][1] = make_uint4(w[4], w[5], w[6], w[7]);
      }
    }
    // The other thread group issues this tile once it has read tile
    // i - kYBufs from the same buffer; until then the barrier may still be in
    // that tile's phase, where this tile's parity would read as complete.
    bool ok = false;
    for (unsigned n = 0; n < poll; ++n) {
      if (issued[b] > i / kYBufs &&
          (ok = mbar_try_wait(&bar[b], (unsigned)((i / kYBufs) & 1))))
        break;
      if (*abort_flag) break;
    }
    C* const in = bufs + b * BUF;
    C v[32];
    if (ok) {
      if constexpr (NY == 2048) {
#pragma unroll
        for (int n2 = 0; n2 < 32; ++n2) {
          const int n = ln + 32 * n2;
          const C x1 = in[n * TX + c], x2 = in[(n + 1024) * TX + c];
          v[n2] = odd ? cmul(csub(x1, x2), tw[1024 + n]) : cadd(x1, x2);
        }
      } else {
#pragma unroll
        for (int n2 = 0; n2 < 32; ++n2) v[n2] = in[(ln + (NY / 32) * n2) * TX + c];
      }
    }
    if (named_bar_or(1 + g, 256, !ok)) {  // the tile has been read (or not all of it came)
      if (t == 0) {
        atomicOr(err, 1);
        *abort_flag = 1;
      }
      break;
    }
    dft32(v);
    if constexpr (NY == 512) {
#pragma unroll
      for (int k2 = 1; k2 < 32; ++k2) v[k2] = cmul(v[k2], tw[ln * k2]);
#pragma unroll
      for (int k2 = 0; k2 < 32; ++k2) in[k2 * 256 + t] = v[k2];  // t = n1 16 + c
    } else {
      tw_rows<32>(v, tw + ln);
      C* tr = in + (NY == 2048 ? odd * 32 * 33 * TX : 0) + ln * TX + c;
#pragma unroll
      for (int k2 = 0; k2 < 32; ++k2) tr[k2 * 33 * TX] = v[k2];
    }
    named_bar_sync(1 + g, 256);
    if constexpr (NY == 512) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int n1 = 0; n1 < 16; ++n1) v[16 * h + n1] = in[(ln + 16 * h) * 256 + n1 * 16 + c];
    } else {
      const C* tr = in + (NY == 2048 ? odd * 32 * 33 * TX : 0) + ln * 33 * TX + c;
#pragma unroll
      for (int n1 = 0; n1 < 32; ++n1) v[n1] = tr[n1 * TX];
    }
    named_bar_sync(1 + g, 256);  // the buffer is free
    if (t == 0 && i + kYBufs < ntile) {
      while (ai < (i + kYBufs) / TPG) next(ahead), ++ai;
      fence_proxy_async();
      issue(ahead, i + kYBufs);
    }
    if constexpr (NY == 512) {
      dft_reg<16>(v);
      dft_reg<16>(v + 16);
    } else {
      dft32(v);
    }
    C* o = p + ((size_t)q.af * ns + q.z) * npix + x0 + c;
    const uint4 sa = NQ == 2 && (i % TPG) >= 2 ? sb[NQ - 1][0] : sb[0][0];
    const uint4 sc = NQ == 2 && (i % TPG) >= 2 ? sb[NQ - 1][1] : sb[0][1];
    const unsigned w[8] = {sa.x, sa.y, sa.z, sa.w, sc.x, sc.y, sc.z, sc.w};
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const int d = q.z - (int)((w[k >> 2] >> (8 * (k & 3))) & 0xffu);
      if ((unsigned)d <= 1u) {
        const int row = NY == 512 ? (k & 15) * 32 + ln + (k >> 4) * 16
                        : NY == 2048 ? 2 * (ln + 32 * k) + odd
                                     : ln + 32 * k;
        o[(size_t)row * nx] = NY == 512 ? v[(k & 16) + out_pos<16>(k & 15)] : v[k];
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag)
    for (int b = 0; b < kYBufs; ++b)
      if (issued[b] > 0) mbar_wait_bounded(&bar[b], (unsigned)((issued[b] - 1) & 1), kPoll);
}

// --------------------------------------------------- x pass of the planes
// x-FFT of the planes' rows in place (FP32, nx = NX = 512, 1024 or 2048), one
// warp per row, storing only the column groups (NX / 32 columns each) that
// the y pass reads from the row's plane (mask.m[plane], a bit per group;
// ~53 % of them at 1024 x 1024 x 128, 5 nm, 270 eV).  HBM-bound: a row comes to
// shared memory by asynchronous 16-byte copies (no registers held), and a
// persistent warp issues the next row's as soon as its transform has read
// the buffer for the last time, so that they overlap the second half of the
// transform and the stores.
//   NX = 1024: four-step 32 x 32 in registers with one padded transpose; 512:
//   16 x 32, the 32-point half split over lane pairs; 2048: a radix-2
//   decimation in frequency as the row is read, then two 1024-point
//   transforms, kept in registers (64 complex a lane) so that the even and
//   odd outputs leave as one 16-byte store; 12 warps, one block per SM, share
//   one twiddle table (two blocks of 4 warps, one row each: 55.7 ms per energy at
//   2048 x 2048 x 64, 91 angles, 4.5 TB/s; 36.0 ms, 7.0 TB/s so).
// tw_g: W512^j; W1024^(n1 k2) as [32][32]; for 2048 that, then W2048^n, n < 1024.
template <int NX> struct XRow {
  static constexpr int FS = NX == 2048 ? 2 * 1056 : (NX / 32) * 33;
  static constexpr int NTW = NX;
  static constexpr int W = NX == 2048 ? 12 : 8, BPS = NX == 2048 ? 1 : 2;  // warps, blocks per SM
};

// The first half of a 1024-point transform up to and including the
// transpose: v[n2] in, the second stage's inputs out.
__device__ __forceinline__ void fft1024_half(float2* v, float2* F, const float2* tw4, int lane) {
  dft32(v);
  tw_rows<32>(v, tw4 + lane);
  __syncwarp();
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) F[k2 * 33 + lane] = v[k2];
  __syncwarp();
#pragma unroll
  for (int n1 = 0; n1 < 32; ++n1) v[n1] = F[lane * 33 + n1];
}

template <int NX>
__global__ void __launch_bounds__(32 * XRow<NX>::W, XRow<NX>::BPS) k_x_planes(
    float2* __restrict__ data, long long nrows, int ny, int ns, const __grid_constant__ XMask mask,
    const float2* __restrict__ tw_g) {
  using C = float2;
  constexpr int FS = XRow<NX>::FS, NTW = XRow<NX>::NTW, W = XRow<NX>::W;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* F = tw + NTW + (threadIdx.x >> 5) * FS;
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * W;
  long long row = (long long)blockIdx.x * W + (threadIdx.x >> 5);
  // this warp's next row with columns to keep, from row on; its mask in m
  unsigned m = 0;
  auto seek = [&] {
    for (; row < nrows; row += stride)
      if ((m = mask.m[(int)((row / ny) % ns)])) return;
    m = 0;
  };
  auto fetch = [&] {
    const C* r = data + (size_t)row * NX;
#pragma unroll
    for (int j = 0; j < NX / 64; ++j) {
      const int n = 2 * (lane + 32 * j);
      cp_async_pair(F + (NX == 2048 && n >= 1024 ? n + 32 : n), r + n);
    }
  };
  seek();
  if (m) fetch();
  for (int i = threadIdx.x; i < NTW; i += 32 * W) tw[i] = tw_g[i];
  __syncthreads();
  while (m) {
    cp_async_wait_all();
    __syncwarp();
    const unsigned mr = m;  // this row's, and its place
    C* const r = data + (size_t)row * NX;
    C v[32];
    if constexpr (NX == 1024) {
#pragma unroll
      for (int n2 = 0; n2 < 32; ++n2) v[n2] = F[lane + 32 * n2];
      fft1024_half(v, F, tw, lane);
      __syncwarp();
      row += stride;
      seek();
      if (m) fetch();
      dft32(v);
#pragma unroll
      for (int k1 = 0; k1 < 32; ++k1)
        if (mr >> k1 & 1u) r[lane + 32 * k1] = v[k1];
    } else if constexpr (NX == 2048) {
      C u[32];
#pragma unroll
      for (int n2 = 0; n2 < 32; ++n2) {
        const int n = lane + 32 * n2;
        const C a = F[n], b = F[1056 + n];
        v[n2] = cadd(a, b);
        u[n2] = cmul(csub(a, b), tw[1024 + n]);
      }
      fft1024_half(v, F, tw, lane);
      fft1024_half(u, F + 1056, tw, lane);
      __syncwarp();
      row += stride;
      seek();
      if (m) fetch();
      dft32(v);
      dft32(u);
#pragma unroll
      for (int k1 = 0; k1 < 32; ++k1)
        if (mr >> k1 & 1u)
          reinterpret_cast<float4*>(r)[lane + 32 * k1] =
              make_float4(v[k1].x, v[k1].y, u[k1].x, u[k1].y);
    } else {
#pragma unroll
      for (int n2 = 0; n2 < 16; ++n2) v[n2] = F[lane + 32 * n2];
      dft_reg<16>(v);
      C u[16];
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) u[k2] = cmul(v[out_pos<16>(k2)], tw[lane * k2]);
      __syncwarp();
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) F[k2 * 33 + lane] = u[k2];
      __syncwarp();
      const int k2 = lane & 15, h = lane >> 4;
#pragma unroll
      for (int n = 0; n < 16; ++n) v[n] = F[k2 * 33 + 2 * n + h];
      __syncwarp();
      row += stride;
      seek();
      if (m) fetch();
      dft32_pair(v, u, h);
      const unsigned mh = mr >> (16 * h);
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (mh >> k & 1u) r[k2 + 256 * h + 16 * k] = u[k];
    }
  }
}

// The pass's shape for a stack: terms of the folded sum, bins of the larger
// parity, groups of at most 8 bins of one parity, as even as they come.
struct PlShape {
  int np, H, SB, G;
};
PlShape pl_shape(int nz, int kb, int ns) {
  PlShape p;
  const bool even = nz % 2 == 0;
  p.np = even ? 2 : 1;
  p.H = (even ? nz / 2 : nz) / 2 + 1;
  const int n0 = even ? (ns + 1 - (kb & 1)) / 2 : ns, n1 = ns - n0, most = n0 > n1 ? n0 : n1;
  const int g = (most + 7) / 8;
  p.SB = (most + g - 1) / g;
  if (p.SB < 2) p.SB = 2;
  p.G = (n0 + p.SB - 1) / p.SB + (even ? (n1 + p.SB - 1) / p.SB : 0);
  return p;
}

// Its launch for nang angles: pixels of a block (its threads' folds in use,
// whole 32-byte sectors per plane row), angles per step (up to 4 within ~100
// KB, two FP32 blocks per SM, with the fewest idle threads in the last round
// of the items), rounds of the items, shared memory.
struct PlLaunch {
  int PX, A, rounds;
  size_t smem;
};
PlLaunch pl_launch(const PlShape& sh, bool even, size_t cs, int nang) {
  PlLaunch l;
  const int unit = 32 / (int)cs;
  l.PX = (even ? kPlThreads : 2 * kPlThreads) / sh.H / unit * unit;
  const size_t per = (size_t)sh.np * sh.H * 3 * l.PX * 2 * cs,
               twb = (size_t)sh.H * sh.G * ((sh.SB + 1) & ~1) * cs;
  l.A = 1;
  double best = 0.0;
  for (int a = 1; a <= 4 && a <= nang; ++a) {
    const int items = a * 3 * sh.G * l.PX, rounds = (items + kPlThreads - 1) / kPlThreads;
    if (a > 1 && (a * per + twb > 104 * 1024 || items >= 2048)) break;
    const double eff = (double)items / (rounds * kPlThreads) + 0.02 * a;
    if (eff > best) best = eff, l.A = a;
  }
  l.rounds = (l.A * 3 * sh.G * l.PX + kPlThreads - 1) / kPlThreads;
  l.smem = l.A * per + twb;
  return l;
}

template <typename R, int SRC, int SB, bool EVEN>
cudaError_t pol_planes_sb(const void* M, const void* nt, const void* dir, long long npix, int nz,
                          const PolParams<R>& pp, const AngleBatch<R>& ang, void* out, int kb,
                          int ns, const void* twz, const void* means, cudaStream_t s) {
  using C = typename RT<R>::C;
  const PlShape sh = pl_shape(nz, kb, ns);
  const PlLaunch l = pl_launch(sh, EVEN, sizeof(C), ang.n);
  if (l.PX < 1 || 3 * sh.G * l.PX >= 2048 || l.A * 3 * sh.G >= 2048)
    return cudaErrorInvalidValue;  // (div_by's range)
  const size_t smem = nz == 1 ? 0 : l.smem;
  auto kern = k_pol_planes<R, SRC, SB, EVEN>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)((npix + l.PX - 1) / l.PX), kPlThreads, smem, s>>>(
      (const typename RT<R>::V4*)M, (const C*)nt, (const R*)dir, npix, nz, l.PX, l.A, kb, ns, pp,
      ang, (C*)out, (const C*)twz, (const R*)means);
  return cudaGetLastError();
}

// The linearity path's bins ([5][2][npix]) from the transformed planes of
// N_t's entries: per pixel its two planes of each; returned at q = 0 (by block
// 0): the constant to xx and yy, and the slices' means (a, xy, b, xz, yz of the
// lab frame's PTen are xx, xy, yy, xz, yz).
template <typename R>
__global__ void __launch_bounds__(256) k_bins5_planes(const typename RT<R>::C* __restrict__ planes,
                                                      long long npix, int nz, int kb, int ns,
                                                      const Geo<R>* __restrict__ geo, double dc,
                                                      const R* __restrict__ means, int from_nt,
                                                      typename RT<R>::C* __restrict__ bins) {
  using C = typename RT<R>::C;
  const long long pix =
      blockIdx.x == 0 ? 0 : (long long)(blockIdx.x - 1) * blockDim.x + threadIdx.x;
  if (pix >= npix || (blockIdx.x > 0 && pix == 0)) return;
  const Geo<R> g = geo[pix];
  if (blockIdx.x == 0) {
    __shared__ double sum[kMeanVals];
    means_total<R>(means, nz, npix, sum);
    if (threadIdx.x > 0) return;
    PTen<double> m;
    means_pten(sum, false, from_nt != 0, m);
    const double2 d[5] = {{m.a[0] + dc, m.a[1]}, {m.xy[0], m.xy[1]}, {m.b[0] + dc, m.b[1]},
                          {m.xz[0], m.xz[1]}, {m.yz[0], m.yz[1]}};
    for (int b = 0; b < 2; ++b) {
      const int bin = b ? g.b1 : g.b0, s = bin < kb ? bin - kb + nz : bin - kb;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        C v = planes[((size_t)q * ns + s) * npix];
        if (bin == 0) v = RT<R>::mk((R)(v.x + d[q].x), (R)(v.y + d[q].y));
        bins[(size_t)(2 * q + b) * npix] = v;
      }
    }
    return;
  }
  if (g.b0 < 0) return;  // off the sphere: the bins are not read
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int bin = b ? g.b1 : g.b0;
    const int s = bin < kb ? bin - kb + nz : bin - kb;
#pragma unroll
    for (int q = 0; q < 5; ++q)
      bins[(size_t)(2 * q + b) * npix + pix] = planes[((size_t)q * ns + s) * npix + pix];
  }
}

template <typename R, int SRC, int Q, int NF = 3>
cudaError_t pol_planes_fft(const void* M, const void* nt, const void* dir, long long npix,
                           const PolParams<R>& pp, const AngleBatch<R>& ang, void* out, int kb,
                           int ns, const void* twz, const void* means, cudaStream_t s) {
  using C = typename RT<R>::C;
  using P = PlFft<R, Q>;
  constexpr int NR = P::PX >= 32 ? 1 : 32 / P::PX;  // (as in the kernel)
  const size_t smem = (SRC == 1 ? (size_t)kPlThreads / 32 * 4 * NR * kMeanStride * sizeof(R) : 0) +
                      (size_t)(NF == 3 ? P::A : 1) * 4 * NF * P::KS * sizeof(C);
  auto kern = k_pol_planes_fft<R, SRC, Q, NF>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)((npix + P::PX - 1) / P::PX), kPlThreads, smem, s>>>(
      (const typename RT<R>::V4*)M, (const C*)nt, (const R*)dir, npix, kb, ns, pp, ang, (C*)out,
      (const C*)twz, (const R*)means);
  return cudaGetLastError();
}

template <typename R, int SRC, bool EVEN>
cudaError_t pol_planes_src(const void* M, const void* nt, const void* dir, long long npix, int nz,
                           const PolParams<R>& pp, const AngleBatch<R>& ang, void* out, int kb,
                           int ns, const void* twz, const void* means, cudaStream_t s) {
  if (nz > 1 && !means) return cudaErrorInvalidValue;
  if constexpr (EVEN) {
    // FP64 at nz = 128 would not fit its registers (64 of data, 96 of sums)
    switch (nz) {
      case 8: return pol_planes_fft<R, SRC, 2>(M, nt, dir, npix, pp, ang, out, kb, ns, twz, means, s);
      case 16: return pol_planes_fft<R, SRC, 4>(M, nt, dir, npix, pp, ang, out, kb, ns, twz, means, s);
      case 32: return pol_planes_fft<R, SRC, 8>(M, nt, dir, npix, pp, ang, out, kb, ns, twz, means, s);
      case 64: return pol_planes_fft<R, SRC, 16>(M, nt, dir, npix, pp, ang, out, kb, ns, twz, means, s);
      case 128:
        if constexpr (sizeof(R) == 4)
          return pol_planes_fft<R, SRC, 32>(M, nt, dir, npix, pp, ang, out, kb, ns, twz, means, s);
        break;
      default: break;
    }
  }
#define RSX_PL(B) \
  case B: return pol_planes_sb<R, SRC, B, EVEN>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, means, s);
  switch (pl_shape(nz, kb, ns).SB) {
    RSX_PL(2) RSX_PL(3) RSX_PL(4) RSX_PL(5) RSX_PL(6) RSX_PL(7) RSX_PL(8)
    default: return cudaErrorInvalidValue;
  }
#undef RSX_PL
}
}  // namespace

bool lin_planes_fits(int precision, int nz) {
  return nz == 8 || nz == 16 || nz == 32 || nz == 64 || (nz == 128 && precision == 32);
}

template <typename R>
cudaError_t launch_lin_planes(const void* M, const void* nt, long long npix, int nz,
                              const PolParams<R>& pp, void* out, int kb, int ns, const void* twz,
                              const void* means, cudaStream_t s) {
  if (!means || !lin_planes_fits(8 * (int)sizeof(R), nz) || ns < 1 || ns > nz || kb < 0 || kb >= nz)
    return cudaErrorInvalidValue;
  AngleBatch<R> none;
  memset(&none, 0, sizeof(none));
#define RSX_LIN(Q)                                                                                \
  return nt ? pol_planes_fft<R, 1, Q, 5>(M, nt, nullptr, npix, pp, none, out, kb, ns, twz, means, s) \
            : pol_planes_fft<R, 0, Q, 5>(M, nt, nullptr, npix, pp, none, out, kb, ns, twz, means, s);
  switch (nz) {
    case 8: RSX_LIN(2)
    case 16: RSX_LIN(4)
    case 32: RSX_LIN(8)
    case 64: RSX_LIN(16)
    default: break;
  }
  if constexpr (sizeof(R) == 4) { RSX_LIN(32) }
#undef RSX_LIN
  return cudaErrorInvalidValue;
}

template <typename R>
cudaError_t launch_bins5_planes(const void* planes, int nx, int ny, int nz, int kb, int ns,
                                const Geo<R>* geo, double dc, const void* means, bool from_nt,
                                void* bins, cudaStream_t s) {
  using C = typename RT<R>::C;
  const long long npix = (long long)nx * ny;
  if (!means) return cudaErrorInvalidValue;
  k_bins5_planes<R><<<(unsigned)((npix + 255) / 256) + 1, 256, 0, s>>>(
      (const C*)planes, npix, nz, kb, ns, geo, dc, (const R*)means, from_nt ? 1 : 0, (C*)bins);
  return cudaGetLastError();
}

PlanesWork pol_planes_work(int precision, int nz, int kb, int ns, int nang) {
  PlanesWork w;
  memset(&w, 0, sizeof(w));
  w.fft = nz == 1 || lin_planes_fits(precision, nz);
  if (w.fft) return w;
  const PlShape sh = pl_shape(nz, kb, ns);
  const PlLaunch l =
      pl_launch(sh, nz % 2 == 0, precision == 32 ? sizeof(float2) : sizeof(double2), nang);
  if (l.PX < 1) return w;
  const double vox = (double)l.PX * nz;
  w.slots = kPlThreads * kPlVoxels / vox;
  w.sums = (double)l.rounds * kPlThreads * sh.H * sh.SB / (l.A * vox);
  w.lone = l.smem > 112 * 1024;
  w.px = l.PX;
  return w;
}

bool pol_planes_fits(int precision, int nz, int kb, int ns) {
  if (nz < 1 || nz > kMaxPlanesNz || ns < 1 || ns > nz) return false;
  const size_t cs = precision == 32 ? sizeof(float2) : sizeof(double2);
  const PlShape sh = pl_shape(nz, kb, ns);
  return (4 * 3 * (size_t)kPlThreads + (size_t)sh.H * sh.G * ((sh.SB + 1) & ~1)) * cs <= 220 * 1024;
}

template <typename R>
cudaError_t launch_pol_planes(const void* M, const void* nt, const void* dir, long long npix,
                              int nz, const PolParams<R>& pp, const AngleBatch<R>& ang, void* out,
                              int kb, int ns, const void* twz, const void* means, cudaStream_t s) {
  if (nz < 1 || nz > kMaxPlanesNz || ns < 1 || ns > nz || kb < 0 || kb >= nz || ang.n < 1 ||
      ang.n > kMaxAngleBatch)
    return cudaErrorInvalidValue;
  if (nz % 2)
    return nt ? pol_planes_src<R, 1, false>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, means, s)
              : pol_planes_src<R, 0, false>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, means, s);
  return nt ? pol_planes_src<R, 1, true>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, means, s)
            : pol_planes_src<R, 0, true>(M, nt, dir, npix, nz, pp, ang, out, kb, ns, twz, means, s);
}

template <typename R>
cudaError_t launch_plane_images(const void* planes, int nx, int ny, int nz, int kb, int ns,
                                const Geo<R>* geo, const ImageDc<R>& dc, const void* means,
                                bool from_nt, bool literal, void* imgs, cudaStream_t s) {
  using C = typename RT<R>::C;
  const long long npix = (long long)nx * ny;
  const unsigned gx = (unsigned)((npix + 255) / 256) + 1;  // block 0: q = 0
  // four angles per thread once one angle's pixels fill the chip
  const bool big = npix >= (1 << 18);
  auto kern = big ? k_plane_images<R, 4> : k_plane_images<R, 1>;
  kern<<<dim3(gx, big ? (dc.n + 3) / 4 : dc.n), 256, 0, s>>>(
      (const C*)planes, nx, ny, nz, kb, ns, geo, dc, (const R*)means, literal ? 1 : 0,
      from_nt ? 1 : 0, (R*)imgs);
  return cudaGetLastError();
}

size_t slice_means_bytes(int precision, int nz) {
  return (size_t)nz * kMeanStride * (precision / 8);
}

template <typename R>
cudaError_t launch_slice_means(const void* M, const void* nt, const void* dir, long long npix,
                               int nz, const PolParams<R>& pp, bool literal, void* means,
                               cudaStream_t s) {
  if (!means || nz < 1 || npix < 1) return cudaErrorInvalidValue;
  k_slice_means<R><<<nz, kMeanSample<R>, 0, s>>>((const typename RT<R>::V4*)M,
                                                 (const typename RT<R>::C*)nt, (const R*)dir, npix,
                                                 nz, pp, literal ? 1 : 0, (R*)means);
  return cudaGetLastError();
}

bool y_planes_ok(int nx, int ny) {
  return (ny == 512 || ny == 1024 || ny == 2048) && nx >= 16 && nx <= 4096 && nx % 16 == 0;
}

template <int NY>
static cudaError_t y_planes_impl(const void* tmap, void* p, int nx, int nz, int kb, int ns,
                                 long long nfields, const YRuns& runs,
                                 const unsigned short* b0idx, const void* tw, const void* twy,
                                 int* err, int n_sm, unsigned poll, cudaStream_t s) {
  using Y = YTile<NY>;
  const long long T = nfields * runs.start[runs.n];
  if (T <= 0) return cudaSuccess;
  if (n_sm <= 0 || T > (1 << 30) || (NY == 2048 && !twy) || !tw || !b0idx)
    return cudaErrorInvalidValue;
  const long long L = (T + n_sm - 1) / n_sm;
  const size_t smem = (size_t)(kYBufs * Y::BUF + Y::NTW) * sizeof(float2) + kYBufs * 8 +
                      (1 + kYBufs) * sizeof(int);
  auto kern = k_y_planes<NY>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)((T + L - 1) / L), 512, smem, s>>>(
      *(const CUtensorMap*)tmap, runs, nx, nz, kb, ns, (int)L, (int)T, b0idx, (const float2*)tw,
      (const float2*)twy, (float2*)p, err, poll);
  return cudaGetLastError();
}

cudaError_t launch_y_planes(const void* tmap, void* p, int nx, int ny, int nz, int kb, int ns,
                            long long nfields, const YRuns& runs, const unsigned short* b0idx,
                            const void* tw, const void* twy, int* err, int n_sm, unsigned poll,
                            cudaStream_t s) {
  if (!y_planes_ok(nx, ny) || ns < 1 || (ns >= nz && nz > 1) || nz > kMaxPlanesNz || kb < 0 ||
      kb >= nz ||
      runs.n != nx / 16)
    return cudaErrorInvalidValue;
  for (int i = 0; i < runs.n; ++i)
    if (runs.start[i + 1] < runs.start[i] ||
        runs.first[i] + (runs.start[i + 1] - runs.start[i]) > ns)
      return cudaErrorInvalidValue;
  if (ny == 512)
    return y_planes_impl<512>(tmap, p, nx, nz, kb, ns, nfields, runs, b0idx, tw, twy, err, n_sm,
                              poll, s);
  if (ny == 1024)
    return y_planes_impl<1024>(tmap, p, nx, nz, kb, ns, nfields, runs, b0idx, tw, twy, err, n_sm,
                               poll, s);
  return y_planes_impl<2048>(tmap, p, nx, nz, kb, ns, nfields, runs, b0idx, tw, twy, err, n_sm,
                             poll, s);
}

template <int NX>
static cudaError_t x_planes_impl(void* data, long long nrows, int ny, int ns, const XMask& mask,
                                 const void* tw, int n_sm, cudaStream_t s) {
  using X = XRow<NX>;
  const size_t smem = ((size_t)X::NTW + (size_t)X::W * X::FS) * sizeof(float2);
  auto kern = k_x_planes<NX>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long want = (nrows + X::W - 1) / X::W, most = (long long)n_sm * X::BPS;
  kern<<<(unsigned)(want < most ? want : most), 32 * X::W, smem, s>>>(
      (float2*)data, nrows, ny, ns, mask, (const float2*)tw);
  return cudaGetLastError();
}

cudaError_t launch_x_planes(void* data, int nx, int ny, int ns, long long nfields,
                            const XMask& mask, const void* tw, int n_sm, cudaStream_t s) {
  const long long nrows = nfields * ns * ny;
  if (nrows <= 0) return cudaSuccess;
  // 16-byte row copies
  if (!tw || ((uintptr_t)data & 15) || ns < 1 || ns > kMaxPlanesNz || n_sm <= 0)
    return cudaErrorInvalidValue;
  if (nx == 1024) return x_planes_impl<1024>(data, nrows, ny, ns, mask, tw, n_sm, s);
  if (nx == 2048) return x_planes_impl<2048>(data, nrows, ny, ns, mask, tw, n_sm, s);
  if (nx == 512) return x_planes_impl<512>(data, nrows, ny, ns, mask, tw, n_sm, s);
  return cudaErrorInvalidValue;
}

#define RSX_INST(R)                                                                               \
  template cudaError_t launch_pol_planes<R>(const void*, const void*, const void*, long long, int, \
                                            const PolParams<R>&, const AngleBatch<R>&, void*, int, \
                                            int, const void*, const void*, cudaStream_t);         \
  template cudaError_t launch_lin_planes<R>(const void*, const void*, long long, int,             \
                                            const PolParams<R>&, void*, int, int, const void*,    \
                                            const void*, cudaStream_t);                           \
  template cudaError_t launch_bins5_planes<R>(const void*, int, int, int, int, int,               \
                                              const Geo<R>*, double, const void*, bool, void*,    \
                                              cudaStream_t);                                      \
  template cudaError_t launch_plane_images<R>(const void*, int, int, int, int, int,               \
                                              const Geo<R>*, const ImageDc<R>&, const void*, bool, \
                                              bool, void*, cudaStream_t);                               \
  template cudaError_t launch_slice_means<R>(const void*, const void*, const void*, long long,    \
                                             int, const PolParams<R>&, bool, void*, cudaStream_t);
RSX_INST(float)
RSX_INST(double)
#undef RSX_INST

}  // namespace rsx
