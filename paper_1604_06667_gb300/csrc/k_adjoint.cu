// k_adjoint.cu -- the adjoint (degridding) and the normalised interpolation for
// circular kernels: every sample gathers the targets within the support,
//   xhat[n][c] = omega_n sum_p w_pn (y[p][c] / W_p)   or   sum_p w_pn y[p][c] / sum_p w_pn,
// so that no two threads write the same output.  Every warp works alone:
//
//   samples  8 or 16 per warp, consecutive in the sorted order of the last add with
//            every other ring reversed (so that the run turns round at the end
//            of a ring instead of jumping across the field): a short strip;
//   query    lane = ring: the pixel interval of the strip's disc widened by r
//            (FP32, cg_healpix.cuh) and its targets in the sorted target index
//            (two binary searches);
//   weights  lanes over the targets of those intervals, loaded one batch of 32
//            ahead; samples in packed f32x2 pairs; pair vectors are differences
//            of double-float unit vectors, as in the general kernel;
//   sums     up to 8 channels: in the lanes, added up by a transposing
//            butterfly; more: lanes over channels, the weights through the
//            warp's shared memory, rows straight from L2.
//
// The map's rows come in the index's order, times 1 / W (k_adjoint_rows).
// Bound by instruction issue (57 % of the slots with one channel, 47 % with 64)
// and by the latency of the searches.  Measured on GB300 against one warp per 32
// samples with the targets one after another (k_degrid.cu, which stays for the
// elliptical kernel and for maps with non-finite or out-of-range values): 1e6
// samples, one channel 3.6 -> 0.7 ms; 2e5 samples, 64 channels 3.8 -> 0.41 ms; 16
// channels 1.9 -> 0.36 ms.  A form with
// tiles of 64 samples, targets staged for 8 warps and listed by each, took
// 0.75 ms for the first and 1.9 ms for the second: a third of the staged
// targets was in reach of a warp.
#include <algorithm>

#include "cg_common.cuh"
#include "cg_cut.cuh"
#include "cg_healpix.cuh"
#include "cg_internal.h"
#include "cg_pair.cuh"

namespace cg {
namespace {

constexpr int kNTh = 256;
constexpr int kNWarps = kNTh / 32;
constexpr uint32_t kAll = 0xffffffffu;

template <int NG>
struct AdjWarp {
  alignas(16) float2 pair[NG / 2][6];        // per pair of samples: hi x, y, z, lo x, y, z
  float4 s_hi[NG], s_lo[NG];           // (w of s_hi: omega); dead ones at (4, 4, 4)
  uint32_t s_idx[NG];                   // output row (0xffffffff: none)
  int lo[64];                            // target intervals of a batch of rings
  int pre[65];                           // targets before each
};

__device__ __forceinline__ float4 lds4(const void* q) {
  const uint32_t p = (uint32_t)__cvta_generic_to_shared(q);
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(p));
  return v;
}

// Samples 0 .. n - 1 of the warp whose pair with the target lies in the guard band
// and outside the support after all (cut decided from the coordinates).
__device__ __noinline__ uint32_t adjoint_band(int n, const float4* s_hi, const float4* s_lo,
                                              const uint32_t* s_idx, float4 th, float4 tl,
                                              double2 tll, const double2* sll, float c2_in,
                                              float c2_out, float c2r_hi, float c2r_lo,
                                              float c2r_tol, double r_rad) {
  uint32_t kill = 0;
  for (int t = 0; t < n; ++t) {
    const float dx = df_diff(s_hi[t].x, s_lo[t].x, th.x, tl.x);
    const float dy = df_diff(s_hi[t].y, s_lo[t].y, th.y, tl.y);
    const float dz = df_diff(s_hi[t].z, s_lo[t].z, th.z, tl.z);
    const float c2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    if (c2 >= c2_in && c2 <= c2_out && s_idx[t] != 0xffffffffu &&
        !pair_inside(tll, sll[s_idx[t]], c2r_hi, c2r_lo, c2r_tol, r_rad))
      kill |= 1u << t;
  }
  return kill;
}

// The warp's samples into its shared memory, and its discs: one around the
// strip, or (`sparse`: samples spread over many supports, as on a ring that the
// field's edge barely cuts, or across a gap of the coverage) one per sample, to
// be gathered one after another.
struct Strip {
  bool sparse, live;
  float gx, gy, gz, R;                   // the strip's disc
};

template <int NG>
__device__ __forceinline__ Strip load_strip(const AdjointArgs& a, AdjWarp<NG>& S, int64_t p0) {
  const int lane = threadIdx.x & 31;
  float4 h = make_float4(4.f, 4.f, 4.f, 0.f), l = make_float4(0.f, 0.f, 0.f, 0.f);
  if (lane < NG) {
    const int64_t p = p0 + lane;
    uint32_t idx = kAll;
    if (p < a.n) {
      int64_t s = p;
      const uint32_t key = a.skey[p];
      if (key < (uint32_t)(12 * a.ns * a.ns)) {
        const int ring = ring_of_pix(a.ns, (int)key);
        if (ring & 1) s = (int64_t)a.ring_off[ring] + a.ring_off[ring + 1] - 1 - p;
        h = a.s_hi[s];
        l = a.s_lo[s];
      }
      idx = a.sval[s];
    }
    S.s_hi[lane] = h;
    S.s_lo[lane] = l;
    S.s_idx[lane] = idx;
    float2* q = S.pair[lane >> 1];
    float* f = reinterpret_cast<float*>(q) + (lane & 1);
    f[0] = h.x;
    f[2] = h.y;
    f[4] = h.z;
    f[6] = l.x;
    f[8] = l.y;
    f[10] = l.z;
  }
  __syncwarp();
  const float4 p = S.s_hi[lane & (NG - 1)];     // copies of the strip
  const bool on = p.x < 3.f;
  float sx = on ? p.x : 0.f, sy = on ? p.y : 0.f, sz = on ? p.z : 0.f;
#pragma unroll
  for (int o = NG / 2; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(kAll, sx, o);
    sy += __shfl_xor_sync(kAll, sy, o);
    sz += __shfl_xor_sync(kAll, sz, o);
  }
  Strip t;
  t.live = __any_sync(kAll, on);
  const float nrm = sqrtf(sx * sx + sy * sy + sz * sz);
  const bool ok = nrm > 1e-3f;           // else: all over the sphere, sparse
  t.gx = ok ? sx / nrm : 0.f;
  t.gy = ok ? sy / nrm : 0.f;
  t.gz = ok ? sz / nrm : 1.f;
  const float ex = p.x - t.gx, ey = p.y - t.gy, ez = p.z - t.gz;
  float rad2 = on ? ex * ex + ey * ey + ez * ez : 0.f;
#pragma unroll
  for (int o = NG / 2; o > 0; o >>= 1) rad2 = fmaxf(rad2, __shfl_xor_sync(kAll, rad2, o));
  const float rad = sqrtf(rad2);
  t.sparse = rad > 3.f * sqrtf(a.kc.c2_out);
  t.R = 2.f * asinf(fminf(1.f, 0.5f * rad)) * (1.f + 1e-5f) + 1e-6f + (float)a.kd.r_rad;
  return t;
}

// Target intervals of rings rb .. rb + 31 (of those up to ihi) of a disc into
// the warp's shared memory; their number of targets.
template <int NG>
__device__ __forceinline__ int query_rings(const AdjointArgs& a, AdjWarp<NG>& S, const Disc& d, int rb,
                                           int ihi) {
  const int lane = threadIdx.x & 31;
  const int ring = rb + lane;
  int lo[2] = {0, 0}, len[2] = {0, 0};
  if (ring <= ihi) {
    const int32_t ta = a.t_ring_off[ring], tb = a.t_ring_off[ring + 1];
    Range rr[2];
    const int nr = tb > ta ? ring_ranges(a.ns, ring, &d, 1, rr) : 0;
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (q < nr) {
        lo[q] = lower_bound_u32(a.t_key, ta, tb, (uint32_t)rr[q].pix_lo);
        len[q] = lower_bound_u32(a.t_key, lo[q], tb, (uint32_t)rr[q].pix_hi + 1u) - lo[q];
      }
  }
  int incl = len[0] + len[1];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kAll, incl, o);
    if (lane >= o) incl += y;
  }
  const int before = incl - len[0] - len[1];
  __syncwarp();
  S.lo[2 * lane] = lo[0];
  S.lo[2 * lane + 1] = lo[1];
  S.pre[2 * lane] = before;
  S.pre[2 * lane + 1] = before + len[0];
  __syncwarp();
  return __shfl_sync(kAll, incl, 31);
}

// Place of target v of the intervals in the sorted index.
template <int NG>
__device__ __forceinline__ int locate(const AdjWarp<NG>& S, int v) {
  int lo = 0, hi = 63;                   // last interval with pre <= v
#pragma unroll
  for (int b = 0; b < 6; ++b) {
    const int mid = (lo + hi + 1) >> 1;
    if (S.pre[mid] <= v) lo = mid; else hi = mid - 1;
  }
  return S.lo[lo] + (v - S.pre[lo]);
}

// Weights of this lane's target (h, l; place t in the index) against the
// warp's samples (only sample `part` if it is not negative).
template <int FORM, int NG>
__device__ __forceinline__ void pair_weights(const AdjointArgs& a, const AdjWarp<NG>& S, float4 h, float4 l,
                                             int t, int part, float2 (&w)[NG / 2]) {
  const WeightConst& kc = a.kc;
  float near = INFINITY;
#pragma unroll
  for (int j = 0; j < NG / 2; ++j) {
    const float4 u0 = lds4(&S.pair[j][0]), u1 = lds4(&S.pair[j][2]), u2 = lds4(&S.pair[j][4]);
    const float2 dx = __fadd2_rn(__fadd2_rn(make_float2(u0.x, u0.y), f2(-h.x)),
                                 __fadd2_rn(make_float2(u1.z, u1.w), f2(-l.x)));
    const float2 dy = __fadd2_rn(__fadd2_rn(make_float2(u0.z, u0.w), f2(-h.y)),
                                 __fadd2_rn(make_float2(u2.x, u2.y), f2(-l.y)));
    const float2 dz = __fadd2_rn(__fadd2_rn(make_float2(u1.x, u1.y), f2(-h.z)),
                                 __fadd2_rn(make_float2(u2.z, u2.w), f2(-l.z)));
    const float2 c2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    const float2 v = weight2<FORM>(kc, a.kd, c2, dx, dy, dz, Axes2{});
    const bool i0 = c2.x <= kc.c2_out, i1 = c2.y <= kc.c2_out;
    w[j] = make_float2(i0 ? v.x : 0.f, i1 ? v.y : 0.f);
    near = band_near(kc, c2, near);
  }
  uint32_t kill = part >= 0 ? ~(1u << part) : 0u;
  if (near <= kc.hw)
    kill |= adjoint_band(NG, S.s_hi, S.s_lo, S.s_idx, h, l, a.tll[a.t_slot[t]], a.sll, a.kd.c2_in, a.kd.c2_out,
                         a.kd.c2r_hi, a.kd.c2r_lo, a.kd.c2r_tol, a.kd.r_rad);
  if (kill) {
#pragma unroll
    for (int j = 0; j < NG / 2; ++j) {
      if (kill & (1u << (2 * j))) w[j].x = 0.f;
      if (kill & (2u << (2 * j))) w[j].y = 0.f;
    }
  }
}

// Every batch of up to 32 targets near the warp's samples: use(v, part) with
// v < total the lane's target of the batch's intervals.  The intervals are
// computed once per call, in batches of 32 rings.
template <int NG, class F>
__device__ __forceinline__ void for_targets(const AdjointArgs& a, AdjWarp<NG>& S, const Strip& strip, F use) {
  if (!strip.live) return;
#pragma unroll 1
  for (int part = 0; part < (strip.sparse ? NG : 1); ++part) {
    Disc d;
    if (strip.sparse) {
      const float4 h = S.s_hi[part];
      if (!(h.x < 3.f)) continue;
      d = make_disc_f(h.x, h.y, h.z, (float)a.kd.r_rad + 1e-6f);
    } else {
      d = make_disc_f(strip.gx, strip.gy, strip.gz, strip.R);
    }
    int ilo, ihi;
    ring_span(a.ns, d.tc - d.R, d.tc + d.R, ilo, ihi);
#pragma unroll 1
    for (int rb = ilo; rb <= ihi; rb += 32) {
      const int total = query_rings(a, S, d, rb, ihi);
      if (total > 0) use(total, strip.sparse ? part : -1);
    }
  }
}

// Up to 8 channels, in the lanes; 16 samples per warp for one or two channels
// (the query is shared by more of them: 1.13 -> 1.09 ms per map-making iteration
// of 1e6 samples), 8 where the sums take the registers.
template <int CN, int NG, int FORM, bool INTERP>
__global__ void __launch_bounds__(kNTh, CN <= 2 ? 3 : 2) k_adjoint(const __grid_constant__ AdjointArgs a) {
  __shared__ AdjWarp<NG> SW[kNWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t p0 = ((int64_t)blockIdx.x * kNWarps + warp) * NG;
  if (p0 >= a.n) return;
  AdjWarp<NG>& S = SW[warp];
  const int c_base = blockIdx.y * CN;
  const Strip strip = load_strip(a, S, p0);

  float2 acc[CN][NG / 2], vs[NG / 2];
#pragma unroll
  for (int j = 0; j < NG / 2; ++j) {
    vs[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < CN; ++c) acc[c][j] = make_float2(0.f, 0.f);
  }
  for_targets(a, S, strip, [&](int total, int part) {
    struct Tgt {
      float4 h, l;
      float d[CN];
      int t;
    };
    auto fetch = [&](int v) {
      Tgt g;                             // padding lies far from every sample
      g.h = make_float4(-4.f, -4.f, -4.f, 0.f);
      g.l = make_float4(0.f, 0.f, 0.f, 0.f);
      g.t = 0;
#pragma unroll
      for (int k = 0; k < CN; ++k) g.d[k] = 0.f;
      if (v < total) {
        g.t = locate(S, v);
        g.h = a.t_hi[g.t];
        g.l = a.t_lo[g.t];
        const float* src = a.rows + (size_t)g.t * a.cpad + c_base;
        if constexpr (CN == 1) {
          g.d[0] = src[0];
        } else if constexpr (CN == 2) {
          const float2 q = *reinterpret_cast<const float2*>(src);
          g.d[0] = q.x; g.d[1] = q.y;
        } else {
#pragma unroll
          for (int k = 0; k < CN; k += 4) {
            const float4 q = *reinterpret_cast<const float4*>(src + k);
            g.d[k] = q.x; g.d[k + 1] = q.y; g.d[k + 2] = q.z; g.d[k + 3] = q.w;
          }
        }
      }
      return g;
    };
    Tgt nx = fetch(lane);
#pragma unroll 1
    for (int b = 0; b < total; b += 32) {
      const Tgt g = nx;
      if (b + 32 < total) nx = fetch(b + 32 + lane);
      float2 w[NG / 2];
      pair_weights<FORM, NG>(a, S, g.h, g.l, g.t, part, w);
#pragma unroll
      for (int j = 0; j < NG / 2; ++j) {
        if (INTERP) vs[j] = __fadd2_rn(vs[j], w[j]);
#pragma unroll
        for (int k = 0; k < CN; ++k) acc[k][j] = __ffma2_rn(w[j], f2(g.d[k]), acc[k][j]);
      }
    }
  });

  // ---- the lanes' sums: value e = t CN + c of the warp's NG CN sums; every
  // step halves the values a lane holds, keeping the half of its lane bit ----
  float v[NG * CN];
#pragma unroll
  for (int t = 0; t < NG; ++t)
#pragma unroll
    for (int c = 0; c < CN; ++c) v[t * CN + c] = (t & 1) ? acc[c][t >> 1].y : acc[c][t >> 1].x;
  int e0 = 0;
#pragma unroll
  for (int o = 16, half = NG * CN / 2; o > 0; o >>= 1, half >>= 1) {
    if (half >= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < (half >= 1 ? half : 1); ++i) {
        const float keep = up ? v[i + half] : v[i], send = up ? v[i] : v[i + half];
        v[i] = keep + __shfl_xor_sync(kAll, send, o);
      }
      e0 += up ? half : 0;
    } else {
      v[0] += __shfl_xor_sync(kAll, v[0], o);
    }
  }
  float vsum = 0.f;                      // lane t < NG: sample t's sum of weights
  if (INTERP) {
#pragma unroll
    for (int t = 0; t < NG; ++t) {
      float x = (t & 1) ? vs[t >> 1].y : vs[t >> 1].x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kAll, x, o);
      if (lane == t) vsum = x;
    }
    if (a.vsum && blockIdx.y == 0 && lane < NG && S.s_idx[lane] != kAll) a.vsum[S.s_idx[lane]] = vsum;
  }
  constexpr int kVals = NG * CN >= 32 ? NG * CN / 32 : 1;    // values per lane
  const bool writes = NG * CN >= 32 || (lane & (32 / (NG * CN) - 1)) == 0;
#pragma unroll
  for (int i = 0; i < kVals; ++i) {
    const int e = e0 + i, t = e / CN, c = c_base + e % CN;
    const float W = __shfl_sync(kAll, vsum, t);
    const uint32_t idx = S.s_idx[t];
    if (!writes || idx == kAll || c >= a.C) continue;
    float x;
    if (INTERP) x = W > 0.f ? v[i] / W : __int_as_float(0x7fc00000);
    else x = S.s_hi[t].x < 3.f ? v[i] * S.s_hi[t].w : 0.f;
    a.out[(size_t)idx * a.C + c] = x;
  }
}

// More channels: lanes over 32 CL channels (a slab per grid.y); the weights of
// a batch go through the warp's shared memory, its targets with a weight are
// visited one by one, four rows in flight.
constexpr int kNG = 8;                   // samples per warp of the wide form
template <int CL, int FORM, bool INTERP>
__global__ void __launch_bounds__(kNTh, 2) k_adjoint_wide(const __grid_constant__ AdjointArgs a) {
  __shared__ AdjWarp<kNG> SW[kNWarps];
  __shared__ __align__(16) float sw[kNWarps][32][kNG];         // weights of listed targets
  __shared__ int st[kNWarps][32];                              // their places in the index
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t p0 = ((int64_t)blockIdx.x * kNWarps + warp) * kNG;
  if (p0 >= a.n) return;
  AdjWarp<kNG>& S = SW[warp];
  const int c_lane = blockIdx.y * 32 * CL + CL * lane;         // this lane's first channel
  const bool mine = c_lane < a.cpad;                           // (rows are padded to cpad)
  const Strip strip = load_strip(a, S, p0);

  float2 acc[kNG][CL / 2], vs[4];
#pragma unroll
  for (int t = 0; t < kNG; ++t)
#pragma unroll
    for (int c = 0; c < CL / 2; ++c) acc[t][c] = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < 4; ++j) vs[j] = make_float2(0.f, 0.f);
  for_targets(a, S, strip, [&](int total, int part) {
    struct Tgt {
      float4 h, l;
      int t;
    };
    auto fetch = [&](int v) {
      Tgt g{make_float4(-4.f, -4.f, -4.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f), 0};
      if (v < total) {
        g.t = locate(S, v);
        g.h = a.t_hi[g.t];
        g.l = a.t_lo[g.t];
      }
      return g;
    };
    Tgt nx = fetch(lane);
#pragma unroll 1
    for (int b = 0; b < total; b += 32) {
      const Tgt g = nx;
      if (b + 32 < total) nx = fetch(b + 32 + lane);
      float2 w[4];
      pair_weights<FORM, kNG>(a, S, g.h, g.l, g.t, part, w);
      bool any = false;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        any |= w[j].x != 0.f || w[j].y != 0.f;
        if (INTERP) vs[j] = __fadd2_rn(vs[j], w[j]);
      }
      const uint32_t m = __ballot_sync(kAll, any);
      if (any) {
        const int q = __popc(m & ((1u << lane) - 1u));
        st[warp][q] = g.t;
        *reinterpret_cast<float4*>(&sw[warp][q][0]) = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
        *reinterpret_cast<float4*>(&sw[warp][q][4]) = make_float4(w[2].x, w[2].y, w[3].x, w[3].y);
      }
      __syncwarp();
      const int cnt = __popc(m);
#pragma unroll 4
      for (int k = 0; k < cnt; ++k) {
        const float* src = a.rows + (size_t)st[warp][k] * a.cpad + c_lane;
        float2 d[CL / 2];
        if constexpr (CL == 2) {
          d[0] = mine ? *reinterpret_cast<const float2*>(src) : make_float2(0.f, 0.f);
        } else {
          const float4 q = mine ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
          d[0] = make_float2(q.x, q.y);
          d[1] = make_float2(q.z, q.w);
        }
        const float4 w0 = *reinterpret_cast<const float4*>(&sw[warp][k][0]);
        const float4 w1 = *reinterpret_cast<const float4*>(&sw[warp][k][4]);
        const float wt[kNG] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
        for (int t = 0; t < kNG; ++t)
#pragma unroll
          for (int c = 0; c < CL / 2; ++c) acc[t][c] = __ffma2_rn(f2(wt[t]), d[c], acc[t][c]);
      }
      __syncwarp();
    }
  });

#pragma unroll
  for (int t = 0; t < kNG; ++t) {
    float W = 0.f;
    if (INTERP) {
      W = (t & 1) ? vs[t >> 1].y : vs[t >> 1].x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) W += __shfl_xor_sync(kAll, W, o);
    }
    const uint32_t idx = S.s_idx[t];
    if (idx == kAll) continue;
    if (INTERP && a.vsum && blockIdx.y == 0 && lane == 0) a.vsum[idx] = W;
    const float om = S.s_hi[t].w;
    const bool live = S.s_hi[t].x < 3.f;
#pragma unroll
    for (int c = 0; c < CL; ++c) {
      if (c_lane + c >= a.C) continue;
      const float v = (c & 1) ? acc[t][c >> 1].y : acc[t][c >> 1].x;
      float x;
      if (INTERP) x = W > 0.f ? v / W : __int_as_float(0x7fc00000);
      else x = live ? v * om : 0.f;
      a.out[(size_t)idx * a.C + c_lane + c] = x;
    }
  }
}

// Whether v = x / W of a target leaves the range in which sums over v and then the
// sample's weight give what sums over w omega / W x give: too large, as for a
// small W (0 x inf would reach other samples of the strip), or small because of
// a large W, so that products with w fall below the normal numbers.  (An ordinary
// W leaves small map values alone, such as the tails of a model's sources.)
__device__ __forceinline__ bool out_of_range(float v, float x, float iw) {
  return !(fabsf(v) <= 0x1p100f) || (iw < 0x1p-20f && x != 0.f && fabsf(v) < 0x1p-100f);
}

// Rows of the map in the order of the sorted target index, times 1 / W_p (0
// where W_p <= 0 or not finite) or as they are (interpolation), padded to cpad
// channels.  Non-finite or out-of-range values become 0 and set *dirty: the
// general kernel then computes the result again.
__global__ void __launch_bounds__(256) k_adjoint_rows(const float* __restrict__ y, int C, int cpad,
                                                      const uint32_t* __restrict__ t_slot,
                                                      const uint32_t* __restrict__ perm,
                                                      const float* __restrict__ wmap,
                                                      const float2* __restrict__ acc_w, int interp,
                                                      int64_t n, float* __restrict__ rows,
                                                      uint32_t* __restrict__ dirty) {
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= n * cpad) return;
  const int64_t t = e / cpad;
  const int c = (int)(e - t * cpad);
  const uint32_t slot = t_slot[t], u = perm[slot];
  float v = 0.f;
  if (u != 0xffffffffu && c < C) {
    const float iw = target_factor(slot, u, wmap, acc_w, interp);
    if (iw != 0.f) {
      const float x = y[(size_t)u * C + c];
      v = iw * x;
      if (interp ? !isfinite(x) : out_of_range(v, x, iw)) {
        v = 0.f;
        *dirty = 1u;
      }
    }
  }
  rows[e] = v;
}

// The largest channel count whose sums stay in the lanes (16 channels: two
// passes in the lanes 1.46 ms per training step, lanes over channels 1.29).
constexpr int kLaneC = 8;

template <class K>
cudaError_t go(const AdjointArgs& a, int ng, int channels, K k, cudaStream_t s) {
  const dim3 grid((unsigned)((a.n + ng * kNWarps - 1) / (ng * kNWarps)),
                  (unsigned)((a.C + channels - 1) / channels));
  k<<<grid, kNTh, 0, s>>>(a);
  return cudaGetLastError();
}

template <int CN, int NG>
cudaError_t launch_adjoint(const AdjointArgs& a, cudaStream_t s) {
  const bool any = weight_form(a.kd) == kWAny;
  if (a.interp)
    return any ? go(a, NG, CN, k_adjoint<CN, NG, kWAny, true>, s) : go(a, NG, CN, k_adjoint<CN, NG, kWGauss1, true>, s);
  return any ? go(a, NG, CN, k_adjoint<CN, NG, kWAny, false>, s) : go(a, NG, CN, k_adjoint<CN, NG, kWGauss1, false>, s);
}

template <int CL>
cudaError_t launch_adjoint_wide(const AdjointArgs& a, cudaStream_t s) {
  const bool any = weight_form(a.kd) == kWAny;
  if (a.interp)
    return any ? go(a, kNG, 32 * CL, k_adjoint_wide<CL, kWAny, true>, s)
               : go(a, kNG, 32 * CL, k_adjoint_wide<CL, kWGauss1, true>, s);
  return any ? go(a, kNG, 32 * CL, k_adjoint_wide<CL, kWAny, false>, s)
             : go(a, kNG, 32 * CL, k_adjoint_wide<CL, kWGauss1, false>, s);
}

}  // namespace

int adjoint_cpad(int C) {
  return C <= 1 ? 1 : (C <= 2 ? 2 : (C <= 4 ? 4 : (C <= kLaneC ? (C + 7) / 8 * 8 : (C + 3) / 4 * 4)));
}

cudaError_t grid_adjoint(AdjointArgs a, const float* y, const float* wmap, const float2* acc_w,
                         int64_t n_targets, cudaStream_t s) {
  a.kc = weight_const(a.kd);
  k_adjoint_rows<<<ceil_div(n_targets * a.cpad, 256), 256, 0, s>>>(
      y, a.C, a.cpad, a.t_slot, a.perm, wmap, acc_w, a.interp, n_targets, a.rows, a.dirty);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (a.C > 64) return launch_adjoint_wide<4>(a, s);
  if (a.C > kLaneC) return launch_adjoint_wide<2>(a, s);
  switch (a.cpad) {
    case 1: return launch_adjoint<1, 16>(a, s);
    case 2: return launch_adjoint<2, 16>(a, s);
    case 4: return launch_adjoint<4, 8>(a, s);
    default: return launch_adjoint<8, 8>(a, s);
  }
}

}  // namespace cg
