// cg_healpix.cuh -- device-side HEALPix RING geometry shared by the sample
// index (k_healpix.cu) and the degridder's target index (k_degrid.cu):
// ring geometry, the closed-form pixel intervals of a disc on a ring (the
// per-ring treatment of the paper's Sect. 3.3), the RING index of a sample
// from its double-float sine with exact FP64 fallback, and binary search.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "cg_common.cuh"
#include "cg_internal.h"
#include "cg_trig.cuh"

namespace cg {
namespace {

// The disc queries propose candidates; the support cut decides every pair
// exactly afterwards, so an interval only has to contain the pixels that a
// disc meets.  They run in FP32 (GB300 executes 1.6 FP64 operations per clock
// and SM; the same queries in FP64 took 4.4 ms per pass over the 24,576 tiles
// of an nside-256 HEALPix target grid): every angle below is good to ~5e-7
// rad, and the discs are widened by kQueryMargin, which covers those errors
// and widens the intervals by at most 4 % of a pixel of nside 8192.
constexpr float kQueryMargin = 4e-6f;
constexpr float kPiF = 3.14159265f;

// A disc on the sphere: colatitude, longitude (radians), radius (< 0: none)
// and the constants of its half-widths: sin(tc), and the colatitude where the
// disc is widest (cos ts = cos tc / cos R; -1 if the disc holds a pole).
struct Disc {
  float tc, pc, R, st, ts;
};

__host__ __device__ __forceinline__ Disc make_disc_f(float x, float y, float z, float R) {
  Disc d;
  const float rho = sqrtf(x * x + y * y);
  // colatitude from the nearer pole: accurate next to it, unlike acos(z)
  const float tn = atan2f(rho, fabsf(z));
  d.tc = z < 0.f ? kPiF - tn : tn;
  d.pc = atan2f(y, x);
  d.R = R + kQueryMargin;
  d.st = sinf(tn);
  // sin^2(ts / 2) = sin((tc + R) / 2) sin((tc - R) / 2) / cos R
  d.ts = -1.f;
  if (d.R < 1.5f && tn > d.R) {
    const float q = sinf(0.5f * (tn + d.R)) * sinf(0.5f * (tn - d.R)) / cosf(d.R);
    const float ts = 2.f * asinf(fminf(1.f, sqrtf(q)));
    d.ts = z < 0.f ? kPiF - ts : ts;
  }
  return d;
}

// Half-width in longitude of the disc at its widest within the colatitude
// band [ta, tb]: -1 if it misses the band, >= 4 if it may cover every
// longitude there.  With u = t - tc, the haversine form
//   sin^2(dphi / 2) = sin((R + u) / 2) sin((R - u) / 2) / (sin t sin tc)
// has no cancellation; the half-width grows towards ts and falls beyond it,
// so the band's colatitude nearest to ts is the widest.
__host__ __device__ __forceinline__ float disc_halfwidth(const Disc& d, float ta, float tb) {
  if (tb < d.tc - d.R || ta > d.tc + d.R) return -1.f;
  if (ta <= 0.f && d.tc <= d.R) return 4.f;
  if (tb >= kPiF && d.tc + d.R >= kPiF) return 4.f;
  if (d.R >= 1.5f || !(d.st > 0.f)) return 4.f;
  const float lo = fmaxf(fmaxf(ta, d.tc - d.R), 0.f);
  const float hi = fminf(fminf(tb, d.tc + d.R), kPiF);
  // a disc that holds a pole is widest at the end of the band nearest to it
  float t = d.ts;
  if (t < 0.f) t = (d.tc < 1.5707964f) ? lo : hi;
  t = fminf(fmaxf(t, lo), hi);
  const float u = t - d.tc;
  const float num = fmaxf(sinf(0.5f * (d.R + u)), 0.f) * fmaxf(sinf(0.5f * (d.R - u)), 0.f);
  const float den = sinf(t) * d.st;
  if (!(num < den)) return 4.f;
  return 2.f * asinf(sqrtf(num / den));
}

// Colatitude of ring i = 0 .. 4 ns: sin(theta / 2) = k / (ns sqrt 6) on the
// caps' rings (z = 1 - k^2 / (3 ns^2)), acos(z) in the belt.
__host__ __device__ __forceinline__ float ring_colat(int ns, int i) {
  if (i <= 0) return 0.f;
  if (i >= 4 * ns) return kPiF;
  const float inv = 1.f / (float)ns;
  if (i < ns) return 2.f * asinf((float)i * inv * 0.40824829f);
  if (i > 3 * ns) return kPiF - 2.f * asinf((float)(4 * ns - i) * inv * 0.40824829f);
  return acosf((float)(2 * ns - i) * inv * (2.f / 3.f));
}

// Continuous ring number of colatitude t (the inverse of ring_colat).
__host__ __device__ __forceinline__ float ring_coord(int ns, float t) {
  const float z = cosf(t);
  if (fabsf(z) <= 2.f / 3.f) return (float)ns * (2.f - 1.5f * z);
  if (z > 0.f) return (float)ns * 2.4494897f * sinf(0.5f * t);
  return (float)ns * (4.f - 2.4494897f * sinf(0.5f * (kPiF - t)));
}

// The rings that a colatitude span [tlo, thi] meets, two on each side for the
// pixels' extent and the rounding of the inverse.
__host__ __device__ __forceinline__ void ring_span(int ns, float tlo, float thi, int& ilo, int& ihi) {
  ilo = (int)floorf(ring_coord(ns, fmaxf(0.f, tlo))) - 2;
  ihi = (int)ceilf(ring_coord(ns, fminf(kPiF, thi))) + 2;
  ilo = ilo < 1 ? 1 : ilo;
  ihi = ihi > 4 * ns - 1 ? 4 * ns - 1 : ihi;
}

struct RingGeo {
  int count, first;
  float phase, dphi;
};
__host__ __device__ __forceinline__ RingGeo ring_geo(int ns, int i) {
  RingGeo r;
  r.phase = 0.5f;
  if (i < ns) {
    r.count = 4 * i;
    r.first = 2 * i * (i - 1);
  } else if (i <= 3 * ns) {
    r.count = 4 * ns;
    r.first = 2 * ns * (ns - 1) + (i - ns) * 4 * ns;
    r.phase = (((i - ns) & 1) == 0) ? 0.5f : 0.f;
  } else {
    const int k = 4 * ns - i;
    r.count = 4 * k;
    r.first = 12 * ns * ns - 2 * k * (k + 1);
  }
  r.dphi = 2.f * kPiF / (float)r.count;
  return r;
}

// Pixels of ring i whose centres lie in the longitude interval [lo, hi] (full:
// all): up to 2 ranges into out.
__host__ __device__ __forceinline__ int ring_pixels(const RingGeo& g, int i, float lo, float hi, bool full,
                                                    Range* out) {
  int jlo = 0, jhi = g.count - 1;
  if (!full) {
    // interval ends in pixels: good to ~1e-2 of a pixel at nside 8192, and
    // the half pixel in the discs' half-widths reaches to the pixel centres
    jlo = (int)ceilf(lo / g.dphi - g.phase - 0.02f);
    jhi = (int)floorf(hi / g.dphi - g.phase + 0.02f);
    if (jhi < jlo) return 0;
    if (jhi - jlo + 1 >= g.count) full = true;
  }
  if (full) {
    out[0] = Range{g.first, g.first + g.count - 1, i, 0};
    return 1;
  }
  int a = jlo % g.count, b = jhi % g.count;
  if (a < 0) a += g.count;
  if (b < 0) b += g.count;
  if (a <= b) {
    out[0] = Range{g.first + a, g.first + b, i, 0};
    return 1;
  }
  out[0] = Range{g.first, g.first + b, i, 0};
  out[1] = Range{g.first + a, g.first + g.count - 1, i, 0};
  return 2;
}

// Pixel ranges of ring i met by the union of nd discs (the hull of their
// pixel intervals on the ring, a superset); writes up to 2 into out.
__host__ __device__ inline int ring_ranges(int ns, int i, const Disc* discs, int nd, Range* out) {
  const RingGeo g = ring_geo(ns, i);
  const float ta = ring_colat(ns, i - 1), tb = ring_colat(ns, i + 1);
  bool any = false, full = false;
  float lo = 0.f, hi = 0.f;   // hull of [pc - W, pc + W], unwrapped near the first disc
  for (int q = 0; q < nd && !full; ++q) {
    if (discs[q].R < 0.f) continue;   // empty group
    const float hw = disc_halfwidth(discs[q], ta, tb);
    if (hw < 0.f) continue;
    const float W = hw + 0.5f * g.dphi + 2e-6f;
    if (W >= kPiF) { full = true; break; }
    float c = discs[q].pc;
    if (any) {  // move c to within pi of the hull's centre
      const float ref = 0.5f * (lo + hi);
      if (c - ref > kPiF) c -= 2.f * kPiF;
      if (ref - c > kPiF) c += 2.f * kPiF;
      lo = fminf(lo, c - W);
      hi = fmaxf(hi, c + W);
      if (hi - lo >= 2.f * kPiF) full = true;
    } else {
      lo = c - W;
      hi = c + W;
      any = true;
    }
  }
  if (!any && !full) return 0;
  return ring_pixels(g, i, lo, hi, full, out);
}

__device__ __forceinline__ bool valid_coord(double lon, double lat) {
  return isfinite(lon) && isfinite(lat) && lat >= -90.0 && lat <= 90.0;
}

// HEALPix RING index from an approximate z = sin(lat) (|error| ~1e-14):
// the same decisions as ang2pix_ring_f64, each checked for a margin that the
// FP64 evaluation's own rounding cannot cross; *ok = false when a value lies
// within that margin of a decision boundary (then the exact FP64 routine
// decides).  For nside <= 16384 a truncated quantity is at most 4 nside =
// 65536 and FP64 and this evaluation differ by < 1e-9 there; the margin is
// 1e-6.
__device__ __forceinline__ int64_t ang2pix_ring_fast(int64_t ns, double lon_deg, double z,
                                                     bool* ok) {
  constexpr double M = 1e-6;
  const double za = fabs(z);
  const double phi = lon_fold_deg(lon_deg);
  const double tt = phi * (1.0 / 90.0);
  const double dns = (double)ns;
  bool good = fabs(za - 2.0 / 3.0) > 1e-9;
  int64_t pix;
  if (za <= 2.0 / 3.0) {
    const double u = dns * (0.5 + tt);
    const double v = dns * (z * 0.75);
    const double A = u - v, B = u + v;
    const double fa = A - floor(A), fb = B - floor(B);
    good = good && fa > M && fa < 1.0 - M && fb > M && fb < 1.0 - M;
    const int64_t asc = (int64_t)A;
    const int64_t dsc = (int64_t)B;
    const int64_t k = ns + 1 + asc - dsc;
    const int64_t odd = k & 1;
    int64_t j = (asc + dsc - ns + (1 - odd) + 1) / 2;
    j %= 4 * ns;
    if (j < 0) j += 4 * ns;
    pix = 2 * ns * (ns - 1) + (k - 1) * 4 * ns + j;
  } else {
    const double ft = tt - floor(tt);
    // near a pole sqrt(1 - za) magnifies the error of z (<= 1e-13): with
    // 1 - za > 1e-5 the error of x stays below 0.5e-13 nside sqrt(3) /
    // sqrt(1e-5) < 5e-7 for nside <= 16384, inside the margin; nearer the
    // pole FP64 decides
    good = good && ft > 1e-12 && ft < 1.0 - 1e-12 && 1.0 - za > 1e-5;
    const double x = dns * sqrt(3.0 * (1.0 - za));
    const double P = ft * x, Q = (1.0 - ft) * x;
    const double fp = P - floor(P), fq = Q - floor(Q);
    good = good && fp > M && fp < 1.0 - M && fq > M && fq < 1.0 - M;
    const int64_t a = (int64_t)P;
    const int64_t b = (int64_t)Q;
    const int64_t k = a + b + 1;
    const double J = tt * (double)k;
    const double fj = J - floor(J);
    good = good && fj > M && fj < 1.0 - M;
    int64_t j = (int64_t)J;
    j %= 4 * k;
    if (j < 0) j += 4 * k;
    pix = (z > 0.0) ? 2 * k * (k - 1) + j : 12 * ns * ns - 2 * k * (k + 1) + j;
  }
  *ok = good;
  return pix;
}

// floor of a double-float and its fractional part (as FP32).
__device__ __forceinline__ float df_floor(df32 a, float& frac) {
  float f = floorf(a.hi);
  if (f == a.hi && a.lo < 0.f) f -= 1.f;   // a sits just below the integer a.hi
  frac = (a.hi - f) + a.lo;                 // a.hi - f is exact
  return f;
}

// ang2pix_ring_fast in double-float arithmetic (no FP64 operations):
// longitude lon (degrees, double-float, folded here), z = sin lat as a
// double-float (|error| ~1e-14).  *ok = false near the cap/belt boundary
// (| |z| - 2/3 | <= 1e-6), within 1e-5 of a pole's z, at a quadrant boundary
// of the caps, or when a truncated quantity lies within the 1e-6 margin of an
// integer: df32 evaluates the truncated quantities (at most 4 nside = 65536)
// to ~1e-8 absolute, so the decisions outside the margin are those of the
// FP64 definition.
__device__ __forceinline__ int64_t ang2pix_ring_df(int64_t ns, df32 lon, df32 z, bool* ok) {
  constexpr float M = 1e-6f;
  constexpr float kZb = (float)(2.0 / 3.0);
  const float za = fabsf(z.hi);
  const bool belt = za < kZb - 1e-6f;
  if (!(belt || (za > kZb + 1e-6f && za < 1.f - 1e-5f)) || ns > 16384) {
    *ok = false;
    return 0;
  }
  // phi in [0, 360): fold by whole turns (exact in FP32 for |lon| < 2^24)
  if (lon.hi < 0.f || lon.hi >= 360.f) {
    const float k = floorf(lon.hi * (1.f / 360.f));
    lon = df_add(lon, df32{-360.f * k, 0.f});
    if (lon.hi < 0.f) lon = df_add(lon, df32{360.f, 0.f});
    if (lon.hi >= 360.f) lon = df_add(lon, df32{-360.f, 0.f});
  }
  constexpr double kInv90 = 1.0 / 90.0;
  const df32 tt = df_mul(lon, df32{(float)kInv90, (float)(kInv90 - (double)(float)kInv90)});
  const float dns = (float)ns;                           // exact: ns <= 16384
  if (belt) {
    // diamonds between ascending and descending edge lines
    const df32 u = df_mul(df_add(tt, df32{0.5f, 0.f}), df32{dns, 0.f});
    const df32 v = df_mul(z, df32{0.75f * dns, 0.f});
    const df32 A = df_add(u, df_neg(v)), B = df_add(u, v);
    float fa, fb;
    const float Af = df_floor(A, fa), Bf = df_floor(B, fb);
    *ok = fa > M && fa < 1.f - M && fb > M && fb < 1.f - M;
    const int64_t asc = (int64_t)Af;
    const int64_t dsc = (int64_t)Bf;
    int64_t k = ns + 1 + asc - dsc;
    k = k < 1 ? 1 : (k > 2 * ns + 1 ? 2 * ns + 1 : k);
    const int64_t odd = k & 1;
    int64_t j = (asc + dsc - ns + (1 - odd) + 1) / 2;
    j %= 4 * ns;
    if (j < 0) j += 4 * ns;
    return 2 * ns * (ns - 1) + (k - 1) * 4 * ns + j;
  }
  // polar caps: ring counted from the pole = sum of the two edge indices + 1,
  // the edge indices from the fraction ft of the quadrant and
  // x = nside sqrt(3 (1 - |z|))
  float ftf;
  const float tf = df_floor(tt, ftf);
  const df32 ft = df_add(tt, df32{-tf, 0.f});             // tt - floor(tt), as a double-float
  const df32 omft = df_add(df32{1.f, 0.f}, df_neg(ft));
  const df32 zabs = z.hi < 0.f ? df_neg(z) : z;
  const df32 w = df_mul(df32{3.f, 0.f}, df_add(df32{1.f, 0.f}, df_neg(zabs)));
  // square root: FP32 estimate and one Newton step on the double-float residual
  const float s0 = sqrtf(w.hi);
  const df32 res = df_add(w, df_neg(df_two_prod(s0, s0)));
  const df32 sq = df_fast_two_sum(s0, res.hi * (0.5f / s0));
  const df32 x = df_mul(sq, df32{dns, 0.f});
  const df32 P = df_mul(ft, x), Q = df_mul(omft, x);
  float fp, fq;
  const float Pf = df_floor(P, fp), Qf = df_floor(Q, fq);
  bool good = ft.hi > 1e-12f && omft.hi > 1e-12f;
  good = good && fp > M && fp < 1.f - M && fq > M && fq < 1.f - M;
  const int64_t k = (int64_t)Pf + (int64_t)Qf + 1;
  const df32 J = df_mul(tt, df32{(float)k, 0.f});           // k <= nside: exact in FP32
  float fj;
  const float Jf = df_floor(J, fj);
  *ok = good && fj > M && fj < 1.f - M;
  int64_t j = (int64_t)Jf;
  j %= 4 * k;
  if (j < 0) j += 4 * k;
  return (z.hi > 0.f) ? 2 * k * (k - 1) + j : 12 * ns * ns - 2 * k * (k + 1) + j;
}

// RING index of a valid sample with z from the double-float sine; exact
// FP64 fallback near decision boundaries.
__device__ __forceinline__ int64_t ang2pix_ring_dual(int64_t ns, double lon, double lat,
                                                     df32 sb) {
  if (ns > 16384) return ang2pix_ring_f64(ns, lon, lat);
  bool ok;
  const int64_t p = ang2pix_ring_fast(ns, lon, (double)sb.hi + (double)sb.lo, &ok);
  return ok ? p : ang2pix_ring_f64(ns, lon, lat);
}

__device__ __forceinline__ int32_t lower_bound_u32(const uint32_t* __restrict__ a, int32_t lo,
                                                   int32_t hi, uint32_t v) {
  while (lo < hi) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    if (a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Ring number (1 .. 4 ns - 1) of RING pixel p; integer arithmetic with an FP32
// square-root estimate corrected exactly (nside <= 8192).
__device__ __forceinline__ int ring_of_pix(int ns, int p) {
  const int npix = 12 * ns * ns, ncap = 2 * ns * (ns - 1);
  if (p >= ncap && p < npix - ncap) return ns + (p - ncap) / (4 * ns);
  const int q = p < ncap ? p : npix - 1 - p;
  int k = (int)(0.5f * (1.f + sqrtf(1.f + 2.f * (float)q)));
  while (k > 1 && 2 * k * (k - 1) > q) --k;
  while (2 * (k + 1) * k <= q) ++k;
  return p < ncap ? k : 4 * ns - k;
}

// First pixel of ring i = 0 .. 4 ns (ring 0 is empty, ring 4 ns past the end).
__device__ __forceinline__ int64_t ring_first(int64_t ns, int64_t i) {
  if (i < ns) return i < 1 ? 0 : 2 * i * (i - 1);
  if (i <= 3 * ns) return 2 * ns * (ns - 1) + (i - ns) * 4 * ns;
  const int64_t k = 4 * ns - i;
  return 12 * ns * ns - 2 * k * (k + 1);
}

}  // namespace
}  // namespace cg
