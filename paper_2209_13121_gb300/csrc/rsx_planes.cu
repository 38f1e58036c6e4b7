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
#include <cuda.h>  // CUtensorMap (the type only)

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
// multiplies: 2 ns fused multiply-adds per voxel and field.  p(0) is taken off
// the whole column first and nz p(0) returned to bin 0 (the other bins of a
// constant are 0): summed as it stands, a column's mean would leave its
// rounding in every bin, where the first stages of an FFT cancel it (one
// material, 45 x 40 x 40, unrotated image against 64 bits away from q = 0:
// 3.9e-6 with it, 2.1e-6 without; transforming every slice first 1.4e-6).  At the kept
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
      const C p0 = b[0].s;  // taken off the column: its bin 0 gets nz p0 back
      for (int z = 1; z < H1; ++z) {
        F v = b[z * 3 * PX];
        const R n = 2 * z == nz ? R(1) : R(2);
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
      C* o = out + (size_t)(a0 + a) * kstride + (size_t)f * fstride + pix0 + px;
      const int zero = (kb == 0 ? 0 : nz - kb) - g * SB;  // the group's place of bin 0
#pragma unroll
      for (int i = 0; i < SB; ++i) {
        if (i == zero) {
          x[i].x = fma(R(nz), p0.x, x[i].x);
          x[i].y = fma(R(nz), p0.y, x[i].y);
        }
        if (g * SB + i < ns) o[(size_t)(g * SB + i) * npix] = x[i];
      }
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
// ~53 % of them at 1024 x 1024 x 128, 5 nm, 270 eV).  HBM-bound: the row goes to
// shared memory by asynchronous 16-byte copies (a lane keeps all NX / 64 of
// its copies in flight, no registers held), issued before the twiddle
// table's loads so that the two overlap.
//   NX = 1024: four-step 32 x 32 in registers with one padded transpose; 512:
//   16 x 32, the 32-point half split over lane pairs; 2048: a radix-2
//   decimation in frequency as the row is read, then two 1024-point
//   transforms, kept in registers (64 complex a lane) so that the even and
//   odd outputs leave as one 16-byte store.
// tw_g: W512^j; W1024^(n1 k2) as [32][32]; for 2048 that, then W2048^n, n < 1024.
template <int NX> struct XRow {
  static constexpr int FS = NX == 2048 ? 2 * 1056 : (NX / 32) * 33;
  static constexpr int NTW = NX;
  static constexpr int W = NX == 2048 ? 4 : 8;  // warps per block, two blocks per SM
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
__global__ void __launch_bounds__(32 * XRow<NX>::W, 2) k_x_planes(
    float2* __restrict__ data, long long nrows, int ny, int ns, const __grid_constant__ XMask mask,
    const float2* __restrict__ tw_g) {
  using C = float2;
  constexpr int FS = XRow<NX>::FS, NTW = XRow<NX>::NTW, W = XRow<NX>::W;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* F = tw + NTW + (threadIdx.x >> 5) * FS;
  const int lane = threadIdx.x & 31;
  const long long row = (long long)blockIdx.x * W + (threadIdx.x >> 5);
  const unsigned m = row < nrows ? mask.m[(int)((row / ny) % ns)] : 0u;
  C* r = data + (size_t)row * NX;
  if (m) {
#pragma unroll
    for (int j = 0; j < NX / 64; ++j) {
      const int n = 2 * (lane + 32 * j);
      cp_async_pair(F + (NX == 2048 && n >= 1024 ? n + 32 : n), r + n);
    }
  }
  for (int i = threadIdx.x; i < NTW; i += 32 * W) tw[i] = tw_g[i];
  __syncthreads();
  if (!m) return;
  cp_async_wait_all();
  __syncwarp();
  C v[32];
  if constexpr (NX == 1024) {
#pragma unroll
    for (int n2 = 0; n2 < 32; ++n2) v[n2] = F[lane + 32 * n2];
    fft1024_half(v, F, tw, lane);
    dft32(v);
#pragma unroll
    for (int k1 = 0; k1 < 32; ++k1)
      if (m >> k1 & 1u) r[lane + 32 * k1] = v[k1];
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
    dft32(v);
    dft32(u);
#pragma unroll
    for (int k1 = 0; k1 < 32; ++k1)
      if (m >> k1 & 1u)
        reinterpret_cast<float4*>(r)[lane + 32 * k1] = make_float4(v[k1].x, v[k1].y, u[k1].x, u[k1].y);
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
    dft32_pair(v, u, h);
    const unsigned mh = m >> (16 * h);
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (mh >> k & 1u) r[k2 + 256 * h + 16 * k] = u[k];
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
  if (!y_planes_ok(nx, ny) || ns < 1 || ns >= nz || nz > kMaxPlanesNz || kb < 0 || kb >= nz ||
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
                                 const void* tw, cudaStream_t s) {
  using X = XRow<NX>;
  const size_t smem = ((size_t)X::NTW + (size_t)X::W * X::FS) * sizeof(float2);
  auto kern = k_x_planes<NX>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)((nrows + X::W - 1) / X::W), 32 * X::W, smem, s>>>(
      (float2*)data, nrows, ny, ns, mask, (const float2*)tw);
  return cudaGetLastError();
}

cudaError_t launch_x_planes(void* data, int nx, int ny, int ns, long long nfields,
                            const XMask& mask, const void* tw, cudaStream_t s) {
  const long long nrows = nfields * ns * ny;
  if (nrows <= 0) return cudaSuccess;
  // 16-byte row copies
  if (!tw || ((uintptr_t)data & 15) || ns < 1 || ns > kMaxPlanesNz) return cudaErrorInvalidValue;
  if (nx == 1024) return x_planes_impl<1024>(data, nrows, ny, ns, mask, tw, s);
  if (nx == 2048) return x_planes_impl<2048>(data, nrows, ny, ns, mask, tw, s);
  if (nx == 512) return x_planes_impl<512>(data, nrows, ny, ns, mask, tw, s);
  return cudaErrorInvalidValue;
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
