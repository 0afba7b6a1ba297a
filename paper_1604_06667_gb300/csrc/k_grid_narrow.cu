// k_grid_narrow.cu -- tile gridder for at most 8 channels (paper Eq. 1-2).
//
// With few channels the weights are the work: every candidate costs ~13
// instructions per target and the channel sums almost nothing.  So the lanes
// of a warp run over candidates and each lane keeps the sums of the warp's
// targets in registers; no weight ever goes through shared memory.
//
//   CTA      one tile of 64 targets (and one share of its candidates); 8
//            warps of 8 targets each, a compact k-d leaf;
//   stage    256 candidates per step (double-buffered, loaded one step ahead
//            into registers): tile-relative vector and weight, and the
//            channel values, which k_rows_sorted has put in sorted order so
//            that they load coalesced;
//   cull     each warp tests the step's candidates against the disc of its
//            8 targets widened by r and lists those in reach, so that the
//            weights run on full warps: a 64-target tile meets 8 % (Example
//            1) to 35 % of its candidates per target, the 8-target leaf
//            three times as many of those it lists;
//   weights  8 targets as 4 packed f32x2 pairs per lane: chord, kernel value,
//            cut (guard band decided from the coordinates), weight sums
//            (Kahan) and channel sums;
//   end      the lanes' sums meet by shuffles that halve the targets a lane holds
//            at every step (compensated for W).
// Maps of few samples per tile run k_grid_sparse, below.
//
// Bound by the barrier per step and by issue slots (1e7 samples onto 8,100
// targets: 48 % of the issue slots used, the barrier the largest stall, ALU pipe
// 32 %).  Measured on GB300 against the register-blocked form it replaced (one
// target per thread, weights through shared memory, every candidate of the tile
// evaluated): 1e8 samples onto 8,100 targets 36.6 -> 8.0 ms, 1e6 samples onto
// 512 x 512 targets 0.95 -> 0.32 ms, 1.2e7 samples on the sphere onto 786,432
// targets 4.48 -> 1.29 ms; the sums of 32 lanes are
// also ten times more accurate than one long one.  The bounds of 3 CTAs per
// SM (2 above two channels, where the sums take the registers) measured best:
// 17.91 ms per call of 1e8 samples against 18.44 (2) and 18.02 (4).  One
// distance from the centre of the guard band per packed pair, instead of two
// comparisons of each lane, and packed Kahan sums: 17.91 -> 17.25 ms, 2e4
// samples onto 100 x 100 targets 95 -> 92.8 us.
#include <cuda_bf16.h>

#include <algorithm>

#include "cg_common.cuh"
#include "cg_cut.cuh"
#include "cg_internal.h"
#include "cg_pair.cuh"

namespace cg {
namespace {

constexpr int kNTh = 256;              // threads per CTA, candidates per step
constexpr int kNWarps = kNTh / 32;
constexpr int kNG = kTile / kNWarps;   // targets per warp
constexpr int kNRanges = 256;          // sample ranges held in shared memory
static_assert(kNG == 8, "eight targets per warp, four packed pairs");

template <int CN>
struct NarrowSmem {
  float4 rec[2][kNTh];                 // tile-relative vector, sample weight
  alignas(16) float dat[2][kNTh * CN]; // channel values
  uint32_t idx[2][kNTh];               // row of the caller's arrays
  float4 tv[kTile];                    // tile-relative target vectors
  // per pair of targets, packed: x, y, z and (elliptical) axis directions
  alignas(16) float2 pair[kNWarps][4][10];
  uint16_t list[kNWarps][kNTh];        // candidates of the step in reach of the warp
  int2 rg[kNRanges];
  int rg_pre[kNRanges + 1];            // candidates before each range of the batch
};

struct NarrowArgs {
  GridArgs g;
  const int32_t* range_c;              // the tile's candidates before each range
  const float* rows;                   // [n][CN] channel values in sorted order (null: CN = 1
                                       // and the values came with the index, in s_lo.w)
  bool sparse;                         // few candidates per tile (k_grid_sparse)
  WeightConst kc;
};

// Targets 0 .. 7 of the warp whose pair with the candidate lies in the guard
// band and outside the support after all (cut decided from the coordinates).
__device__ __noinline__ uint32_t narrow_band(const float4* tv, float4 cand, const double2* tll,
                                             double2 sll, float c2_in, float c2_out,
                                             float c2r_hi, float c2r_lo, float c2r_tol,
                                             double r_rad) {
  uint32_t kill = 0;
  for (int t = 0; t < kNG; ++t) {
    const float dx = tv[t].x - cand.x, dy = tv[t].y - cand.y, dz = tv[t].z - cand.z;
    const float c2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    if (c2 >= c2_in && c2 <= c2_out && !pair_inside(tll[t], sll, c2r_hi, c2r_lo, c2r_tol, r_rad))
      kill |= 1u << t;
  }
  return kill;
}

// Shared-memory loads that stay where they are written.
__device__ __forceinline__ float4 lds4(uint32_t p) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(p));
  return v;
}
__device__ __forceinline__ float2 lds2(uint32_t p) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(p));
  return v;
}

// A candidate's channel values: row s of rows (null: one channel, in the record).
template <int CN>
__device__ __forceinline__ void load_row(const float* rows, int64_t s, float in_rec, float (&d)[CN]) {
  const float* row = rows + (size_t)s * CN;
  if constexpr (CN == 1) {
    d[0] = rows ? row[0] : in_rec;
  } else if constexpr (CN == 2) {
    const float2 q = *reinterpret_cast<const float2*>(row);
    d[0] = q.x; d[1] = q.y;
  } else {
#pragma unroll
    for (int k = 0; k < CN; k += 4) {
      const float4 q = *reinterpret_cast<const float4*>(row + k);
      d[k] = q.x; d[k + 1] = q.y; d[k + 2] = q.z; d[k + 3] = q.w;
    }
  }
}

// A group's targets 2 lane, 2 lane + 1 (lane < 4) as a packed pair: vectors and, for
// the elliptical kernel, axis directions.
template <int FORM>
__device__ __forceinline__ void load_pair(const GridArgs& a, float2* A, int64_t sa) {
  const float4 p = a.tgt_a[sa], q = a.tgt_a[sa + 1];
  A[0] = make_float2(p.x, q.x);
  A[1] = make_float2(p.y, q.y);
  A[2] = make_float2(p.z, q.z);
  if (FORM != kWGauss1 && FORM != kWGauss1Ds && a.kd.type == CG_GAUSS2D) {
    const float4 f1a = a.tgt_f1[sa], f1b = a.tgt_f1[sa + 1];
    const float4 f2a = a.tgt_f2[sa], f2b = a.tgt_f2[sa + 1];
    A[4] = make_float2(f1a.x, f1b.x);
    A[5] = make_float2(f1a.y, f1b.y);
    A[6] = make_float2(f1a.z, f1b.z);
    A[7] = make_float2(f2a.x, f2b.x);
    A[8] = make_float2(f2a.y, f2b.y);
    A[9] = make_float2(f2a.z, f2b.z);
  }
}

// Disc of a group of 8 targets (p: target lane & 7; empty slots sit at (4, 4, 4)),
// widened by the support: centre and squared reach (chords; -1: no target).
__device__ __forceinline__ float4 group_reach(float4 p, float c2_out) {
  const bool on = p.x < 3.f;
  float sx = on ? p.x : 0.f, sy = on ? p.y : 0.f, sz = on ? p.z : 0.f, sn = on ? 1.f : 0.f;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
    sz += __shfl_xor_sync(0xffffffffu, sz, o);
    sn += __shfl_xor_sync(0xffffffffu, sn, o);
  }
  const float inv = sn > 0.f ? 1.f / sn : 0.f;
  const float gx = sx * inv, gy = sy * inv, gz = sz * inv;
  const float ex = p.x - gx, ey = p.y - gy, ez = p.z - gz;
  float rad2 = on ? ex * ex + ey * ey + ez * ez : 0.f;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) rad2 = fmaxf(rad2, __shfl_xor_sync(0xffffffffu, rad2, o));
  const float reach = sqrtf(rad2) + sqrtf(c2_out);
  return make_float4(gx, gy, gz, sn > 0.f ? reach * reach * 1.0001f + 1e-12f : -1.f);
}

// A lane's sums over its candidates: 8 targets as 4 packed pairs.
template <int CN>
struct LaneSums {
  float2 acc[CN][4], ws[4], wc[4];
  unsigned npair;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      ws[j] = wc[j] = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < CN; ++c) acc[c][j] = make_float2(0.f, 0.f);
    }
    npair = 0;
  }
};

// The warp's list of the first 32 B candidates in reach of its group; their number.
template <int B>
__device__ __forceinline__ int list_near(const float4* rec, float4 g, uint16_t* list) {
  const int lane = threadIdx.x & 31;
  int cnt = 0;
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const float4 p = rec[32 * b + lane];
    const float ex = p.x - g.x, ey = p.y - g.y, ez = p.z - g.z;
    const bool in = fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= g.w;
    const uint32_t m = __ballot_sync(0xffffffffu, in);
    if (in) list[cnt + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(32 * b + lane);
    cnt += __popc(m);
  }
  __syncwarp();
  return cnt;
}

// Weights and sums of cnt listed candidates, 32 at a time; pair_s: the group's
// packed pairs, tv and slot0: its targets.
template <int CN, int FORM>
__device__ __forceinline__ void add_listed(const NarrowArgs& na, LaneSums<CN>& L, const uint16_t* list, int cnt,
                                           const float4* rec, const float* dat, const uint32_t* idx,
                                           uint32_t pair_s, const float4* tv, int64_t slot0) {
  const GridArgs& a = na.g;
  const WeightConst& kc = na.kc;
  const int lane = threadIdx.x & 31;
  for (int b = 0; b < cnt; b += 32) {
    float4 p = make_float4(-4.f, -4.f, -4.f, 0.f);
    int ci = 0;
    float d[CN];
#pragma unroll
    for (int k = 0; k < CN; ++k) d[k] = 0.f;
    if (b + lane < cnt) {
      ci = list[b + lane];
      p = rec[ci];
#pragma unroll
      for (int k = 0; k < CN; ++k) d[k] = dat[ci * CN + k];
    }
    const float2 nx = f2(-p.x), ny = f2(-p.y), nz = f2(-p.z), om = f2(p.w);
    float2 w[4];
    float near = INFINITY;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // read for every batch: held in registers they would be spilled
      const uint32_t q6 = pair_s + j * (uint32_t)(10 * sizeof(float2));
      const float4 xy = lds4(q6);
      const float2 dx = __fadd2_rn(make_float2(xy.x, xy.y), nx);
      const float2 dy = __fadd2_rn(make_float2(xy.z, xy.w), ny);
      const float2 dz = __fadd2_rn(lds2(q6 + 16), nz);
      const float2 c2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
      Axes2 A{};
      if (FORM != kWGauss1 && FORM != kWGauss1Ds) {
        const float4 u0 = lds4(q6 + 32), u1 = lds4(q6 + 48), u2 = lds4(q6 + 64);
        A.ax = make_float2(u0.x, u0.y); A.ay = make_float2(u0.z, u0.w);
        A.az = make_float2(u1.x, u1.y); A.bx = make_float2(u1.z, u1.w);
        A.by = make_float2(u2.x, u2.y); A.bz = make_float2(u2.z, u2.w);
      }
      const float2 v = __fmul2_rn(weight2<FORM>(kc, a.kd, c2, dx, dy, dz, A), om);
      const bool i0 = c2.x <= kc.c2_out, i1 = c2.y <= kc.c2_out;
      // outside the support: -0.0 adds nothing to any finite sum
      w[j] = make_float2(i0 ? v.x : -0.f, i1 ? v.y : -0.f);
      L.npair += (i0 ? 1u : 0u) + (i1 ? 1u : 0u);
      near = band_near(kc, c2, near);
    }
    if (near <= kc.hw) {
      const uint32_t kill = narrow_band(tv, p, a.tgt_ll + slot0, a.sll[idx[ci]],
                                        a.kd.c2_in, a.kd.c2_out, a.kd.c2r_hi, a.kd.c2r_lo,
                                        a.kd.c2r_tol, a.kd.r_rad);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (kill & (1u << (2 * j))) { w[j].x = -0.f; --L.npair; }
        if (kill & (2u << (2 * j))) { w[j].y = -0.f; --L.npair; }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      kahan2(L.ws[j], L.wc[j], w[j]);
#pragma unroll
      for (int k = 0; k < CN; ++k) L.acc[k][j] = __ffma2_rn(w[j], f2(d[k]), L.acc[k][j]);
    }
  }
}

// Sum over the lanes of 8 targets' values: every step halves the targets a lane
// holds, keeping those of its lane bit; lanes 4 t .. 4 t + 3 end with target t.
__device__ __forceinline__ float lanes_sum(const float2 (&v)[4]) {
  const int lane = threadIdx.x & 31;
  float x[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) x[t] = (t & 1) ? v[t >> 1].y : v[t >> 1].x;
#pragma unroll
  for (int o = 16, half = 4; half > 0; o >>= 1, half >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float keep = up ? x[i + half] : x[i], send = up ? x[i] : x[i + half];
      x[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  x[0] += __shfl_xor_sync(0xffffffffu, x[0], 2);
  return x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
}
// The same for compensated sums.
__device__ __forceinline__ float2 lanes_comp(const float2 (&s)[4], const float2 (&c)[4]) {
  const int lane = threadIdx.x & 31;
  float x[8], y[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    x[t] = (t & 1) ? s[t >> 1].y : s[t >> 1].x;
    y[t] = (t & 1) ? c[t >> 1].y : c[t >> 1].x;
  }
#pragma unroll
  for (int o = 16, half = 4; half > 0; o >>= 1, half >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float xs = up ? x[i] : x[i + half], ys = up ? y[i] : y[i + half];
      const float xr = __shfl_xor_sync(0xffffffffu, xs, o), yr = __shfl_xor_sync(0xffffffffu, ys, o);
      x[i] = up ? x[i + half] : x[i];
      y[i] = up ? y[i + half] : y[i];
      comp_add(x[i], y[i], xr, yr);
    }
  }
#pragma unroll
  for (int o = 2; o > 0; o >>= 1)
    comp_add(x[0], y[0], __shfl_xor_sync(0xffffffffu, x[0], o), __shfl_xor_sync(0xffffffffu, y[0], o));
  return make_float2(x[0], y[0]);
}

// A target's sums into the one-shot map, the accumulators or a share's partial
// sums.
template <int CN>
__device__ __forceinline__ void write_target(const GridArgs& a, int64_t slot, float wsum, float wcor,
                                             const float (&num)[CN], int split) {
  const uint32_t u = a.tgt_perm[slot];
  if (u == 0xffffffffu) return;
  // A non-finite channel value of a candidate outside the support reaches the
  // target through 0 x NaN: such rows are computed again by the fix-up pass
  // with only the pairs inside the support.
  float chk = 0.f;
#pragma unroll
  for (int k = 0; k < CN; ++k) chk += num[k];
  const bool bad = !isfinite(chk);
  if (bad) {
    atomicOr(&a.nf_bits[slot >> 5], 1u << (slot & 31));
    atomicOr(a.nf_any, 1u);
  }
  if (a.out) {
    const float W = wsum + wcor;
    if (a.out_w) a.out_w[u] = W;
    if (!bad) {
#pragma unroll
      for (int k = 0; k < CN; ++k)
        if (k < a.C) a.out[(size_t)u * a.C + k] = (W > 0.f) ? num[k] / W : __int_as_float(0x7fc00000);
    }
    if (!a.keep) return;
  }
  const bool splits = a.n_split > 1;
  if (!bad) {
    float* dst = splits ? a.part_num + ((size_t)split * a.n_slots + slot) * a.C
                        : a.acc_num + (size_t)slot * a.C;
    const bool add = a.accumulate && !splits;
#pragma unroll
    for (int k = 0; k < CN; ++k)
      if (k < a.C) dst[k] = add ? dst[k] + num[k] : num[k];
  }
  if (splits) {
    a.part_w[(size_t)split * a.n_slots + slot] = make_float2(wsum, wcor);
    return;
  }
  float2 old = a.accumulate ? a.acc_w[slot] : make_float2(0.f, 0.f);
  comp_add(old.x, old.y, wsum, wcor);
  a.acc_w[slot] = old;
}

// Adds up the lanes' sums and writes the group's targets.
template <int CN>
__device__ __forceinline__ void write_group(const NarrowArgs& na, LaneSums<CN>& L, int64_t slot0, int split) {
  const GridArgs& a = na.g;
  const int lane = threadIdx.x & 31;
  const float2 w = lanes_comp(L.ws, L.wc);
  const float wsum = w.x, wcor = w.y;
  float num[CN];
#pragma unroll
  for (int k = 0; k < CN; ++k) num[k] = lanes_sum(L.acc[k]);
  unsigned npair = __reduce_add_sync(0xffffffffu, L.npair);
  if (lane == 0 && npair && a.pairs) atomicAdd(a.pairs, (unsigned long long)npair);
  if (lane & 3) return;
  const int64_t slot = slot0 + (lane >> 2);
  write_target<CN>(a, slot, wsum, wcor, num, split);
}

template <int CN, int FORM>
__global__ void __launch_bounds__(kNTh, CN <= 2 ? 3 : 2)
    k_grid_narrow(const __grid_constant__ NarrowArgs na) {
  __shared__ NarrowSmem<CN> S;
  const GridArgs& a = na.g;
  if (a.hold && hold_gives_up(a.hold, a.hold_cycles, a.err)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tile = blockIdx.x;
  const int split = blockIdx.z;
  const int64_t slot0 = tile * kTile + warp * kNG;   // the warp's first target
  const float4 chi = a.tile_chi[tile], clo = a.tile_clo[tile];
  const uint32_t pair_s = (uint32_t)__cvta_generic_to_shared(&S.pair[warp][0][0]);
  // ---- the warp's targets: packed pairs in shared memory (read by all lanes
  // at once); centre and reach of the group (empty slots sit at (4, 4, 4)) ----
  if (tid < kTile) S.tv[tid] = a.tgt_a[tile * kTile + tid];
  if (lane < 4) load_pair<FORM>(a, S.pair[warp][lane], slot0 + 2 * lane);
  const float4 near = group_reach(a.tgt_a[slot0 + (lane & 7)], a.kd.c2_out);   // four copies of the group
  LaneSums<CN> L;
  L.clear();

  const int64_t r0 = a.range_off[tile], r1 = a.range_off[tile + 1];
  int c_lo = 0, c_hi = 0x7fffffff;
  if (a.n_split > 1) {
    const int total = a.tile_cand[tile];
    const int per = ((total + a.n_split - 1) / a.n_split + kNTh - 1) / kNTh * kNTh;
    c_lo = split * per;
    c_hi = min(total, c_lo + per);
  }

  int cbase = 0;
  for (int64_t rb = r0; rb < r1 && cbase < c_hi; rb += kNRanges) {
    const int nr = (int)((r1 - rb) < kNRanges ? (r1 - rb) : kNRanges);
    __syncthreads();   // the previous batch's steps are done with rg / rg_pre
    if (tid < nr) {
      const int2 r = a.range_s[rb + tid];
      const int pre = na.range_c[rb + tid] - cbase;
      S.rg[tid] = r;
      S.rg_pre[tid] = pre;
      if (tid == nr - 1) S.rg_pre[nr] = pre + (r.y - r.x);
    }
    __syncthreads();
    const int total = S.rg_pre[nr];
    const int v_lo = max(0, min(total, c_lo - cbase));
    const int v_hi = max(0, min(total, c_hi - cbase));
    cbase += total;
    const int n_steps = (v_hi - v_lo + kNTh - 1) / kNTh;
    if (n_steps <= 0) continue;

    struct Cand {
      float4 h, l;
      uint32_t idx;
      float d[CN];
    };
    auto fetch = [&](int v0) {
      // padding lies far from every target and from the empty slots
      Cand c;
      c.h = make_float4(-4.f, -4.f, -4.f, 0.f);
      c.l = make_float4(0.f, 0.f, 0.f, 0.f);
      c.idx = 0xffffffffu;
#pragma unroll
      for (int k = 0; k < CN; ++k) c.d[k] = 0.f;
      const int v = v0 + tid;
      if (v < v_hi) {
        int lo = 0, hi = nr - 1;   // last range with rg_pre <= v
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (S.rg_pre[mid] <= v) lo = mid; else hi = mid - 1;
        }
        const int64_t s = S.rg[lo].x + (v - S.rg_pre[lo]);
        c.h = a.s_hi[s];
        c.l = a.s_lo[s];
        c.idx = a.perm[s];
        load_row<CN>(na.rows, s, c.l.w, c.d);
      }
      return c;
    };
    auto put = [&](const Cand& c, int st) {
      S.rec[st][tid] = make_float4(df_diff(c.h.x, c.l.x, chi.x, clo.x), df_diff(c.h.y, c.l.y, chi.y, clo.y),
                                   df_diff(c.h.z, c.l.z, chi.z, clo.z), c.h.w);
      S.idx[st][tid] = c.idx;
      // a sample of weight zero does not take part, whatever its values
#pragma unroll
      for (int k = 0; k < CN; ++k) S.dat[st][tid * CN + k] = c.h.w != 0.f ? c.d[k] : 0.f;
    };

    Cand pre = fetch(v_lo);
    put(pre, 0);
    if (n_steps > 1) pre = fetch(v_lo + kNTh);
    __syncthreads();
    for (int q = 0; q < n_steps; ++q) {
      const int st = q & 1;
      if (q + 1 < n_steps) {
        put(pre, st ^ 1);
        if (q + 2 < n_steps) pre = fetch(v_lo + (q + 2) * kNTh);
      }
      // (a step's loads and ballots at once; a nearly empty last one apart)
      const int cnt = v_hi - v_lo - q * kNTh > kNTh / 4 ? list_near<kNTh / 32>(S.rec[st], near, S.list[warp])
                                                        : list_near<kNTh / 128>(S.rec[st], near, S.list[warp]);
      add_listed<CN, FORM>(na, L, S.list[warp], cnt, S.rec[st], S.dat[st], S.idx[st], pair_s, S.tv + warp * kNG, slot0);
      __syncthreads();   // the stage may be rewritten; the next one is visible
    }
  }

  write_group(na, L, slot0, split);
}

// The same for tiles of few candidates.  A tile is some five dependent loads and
// little work, so what counts is how many run at a time: two warps per tile
// (twelve tiles per SM against three).  Up to 64 candidates, lanes over targets:
// no list, no sums over lanes.  More: four groups per warp, one after the other
// on candidates that are staged once (above 128: again for every group).
// Measured on GB300 per call, one channel, gauss1d, onto 2048 x 1024 targets of
// the whole sky: 1e5 samples 559 -> 187 us (register-blocked form 280), 3e5 594 ->
// 244 (413); 1e6 x 7 1290 -> 928 (927); 8,000 x 3 onto 500 x 500 129 -> 72 (72).
constexpr int kSpTh = 64, kSpStep = 128, kSpRanges = 128;
constexpr int kSpDirect = 64;   // tiles of so few candidates: a lane per target
template <int CN>
struct SparseSmem {
  float4 rec[kSpStep];
  alignas(16) float dat[kSpStep * CN];
  uint32_t idx[kSpStep];
  float4 tv[kTile];
  alignas(16) float2 pair[kTile / kNG][4][10];
  uint16_t list[kSpTh / 32][kSpStep];
  int2 rg[kSpRanges];
  int rg_c[kSpRanges];
};

template <int CN, int FORM>
__global__ void __launch_bounds__(kSpTh, CN <= 2 ? 12 : 8) k_grid_sparse(const __grid_constant__ NarrowArgs na) {
  __shared__ SparseSmem<CN> S;
  const GridArgs& a = na.g;
  if (a.hold && hold_gives_up(a.hold, a.hold_cycles, a.err)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tile = blockIdx.x;
  const float4 chi = a.tile_chi[tile], clo = a.tile_clo[tile];
  const int total = a.tile_cand[tile];
  const int64_t r0 = a.range_off[tile];
  const int nr = (int)(a.range_off[tile + 1] - r0);
  const bool rg_in = nr <= kSpRanges;   // more are searched in global memory
  if (rg_in)
    for (int r = tid; r < nr; r += kSpTh) {
      S.rg[r] = a.range_s[r0 + r];
      S.rg_c[r] = na.range_c[r0 + r];
    }
  S.tv[tid] = a.tgt_a[tile * kTile + tid];
  if (lane < 16) {
    const int p = 16 * warp + lane;   // pair of the tile
    load_pair<FORM>(a, S.pair[p >> 2][p & 3], tile * kTile + 2 * p);
  }
  __syncthreads();

  auto stage = [&](int v0) {
    for (int i = tid; i < kSpStep; i += kSpTh) {
      const int v = v0 + i;
      // padding lies far from every target and from the empty slots
      float4 rec = make_float4(-4.f, -4.f, -4.f, 0.f);
      float d[CN];
#pragma unroll
      for (int k = 0; k < CN; ++k) d[k] = 0.f;
      if (v < total) {
        int lo = 0, hi = nr - 1;   // last range with so many candidates before it
        int64_t s;
        if (rg_in) {
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (S.rg_c[mid] <= v) lo = mid; else hi = mid - 1;
          }
          s = S.rg[lo].x + (v - S.rg_c[lo]);
        } else {
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (na.range_c[r0 + mid] <= v) lo = mid; else hi = mid - 1;
          }
          s = a.range_s[r0 + lo].x + (v - na.range_c[r0 + lo]);
        }
        const float4 h = a.s_hi[s], l = a.s_lo[s];
        rec = make_float4(df_diff(h.x, l.x, chi.x, clo.x), df_diff(h.y, l.y, chi.y, clo.y),
                          df_diff(h.z, l.z, chi.z, clo.z), h.w);
        S.idx[i] = a.perm[s];
        load_row<CN>(na.rows, s, l.w, d);
      }
      S.rec[i] = rec;
      // a sample of weight zero does not take part, whatever its values
#pragma unroll
      for (int k = 0; k < CN; ++k) S.dat[i * CN + k] = rec.w != 0.f ? d[k] : 0.f;
    }
  };

  if (total <= kSpDirect) {
    // ---- lanes over targets: no list, and no sum over lanes ----
    stage(0);
    __syncthreads();
    const int64_t slot = tile * kTile + tid;
    const float4 at = S.tv[tid];
    Axes2 A{};
    if (FORM != kWGauss1 && FORM != kWGauss1Ds && a.kd.type == CG_GAUSS2D) {
      const float4 u = a.tgt_f1[slot], v = a.tgt_f2[slot];
      A.ax = f2(u.x); A.ay = f2(u.y); A.az = f2(u.z);
      A.bx = f2(v.x); A.by = f2(v.y); A.bz = f2(v.z);
    }
    const WeightConst& kc = na.kc;
    // four chains of additions: candidates 4 k, 4 k + 1, ... apart (short chains
    // keep the digits that sums over lanes keep in the other forms)
    float2 ws[2], wc[2], acc[2][CN];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      ws[h] = wc[h] = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < CN; ++c) acc[h][c] = make_float2(0.f, 0.f);
    }
    unsigned npair = 0;
#pragma unroll 1
    for (int k0 = 0; k0 < total; k0 += 4) {   // (padding follows the last one)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = k0 + 2 * h;
        const float4 p = S.rec[k], q = S.rec[k + 1];
        const float2 dx = __fadd2_rn(f2(at.x), make_float2(-p.x, -q.x));
        const float2 dy = __fadd2_rn(f2(at.y), make_float2(-p.y, -q.y));
        const float2 dz = __fadd2_rn(f2(at.z), make_float2(-p.z, -q.z));
        const float2 c2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        const float2 v = __fmul2_rn(weight2<FORM>(kc, a.kd, c2, dx, dy, dz, A), make_float2(p.w, q.w));
        bool i0 = c2.x <= kc.c2_out, i1 = c2.y <= kc.c2_out;
        if (band_near(kc, c2, INFINITY) <= kc.hw) {
          // guard band: the cut is decided from the coordinates
          const double2 tll = a.tgt_ll[slot];
          if (i0 && c2.x >= a.kd.c2_in)
            i0 = pair_inside(tll, a.sll[S.idx[k]], a.kd.c2r_hi, a.kd.c2r_lo, a.kd.c2r_tol, a.kd.r_rad);
          if (i1 && c2.y >= a.kd.c2_in)
            i1 = pair_inside(tll, a.sll[S.idx[k + 1]], a.kd.c2r_hi, a.kd.c2r_lo, a.kd.c2r_tol, a.kd.r_rad);
        }
        npair += (i0 ? 1u : 0u) + (i1 ? 1u : 0u);
        const float2 w = make_float2(i0 ? v.x : -0.f, i1 ? v.y : -0.f);
        kahan2(ws[h], wc[h], w);
#pragma unroll
        for (int c = 0; c < CN; ++c)
          acc[h][c] = __ffma2_rn(w, make_float2(S.dat[k * CN + c], S.dat[(k + 1) * CN + c]), acc[h][c]);
      }
    }
    float num[CN];
#pragma unroll
    for (int c = 0; c < CN; ++c) num[c] = (acc[0][c].x + acc[0][c].y) + (acc[1][c].x + acc[1][c].y);
    comp_add(ws[0].x, wc[0].x, ws[0].y, wc[0].y);
    comp_add(ws[1].x, wc[1].x, ws[1].y, wc[1].y);
    comp_add(ws[0].x, wc[0].x, ws[1].x, wc[1].x);
    npair = __reduce_add_sync(0xffffffffu, npair);
    if (lane == 0 && npair && a.pairs) atomicAdd(a.pairs, (unsigned long long)npair);
    write_target<CN>(a, slot, ws[0].x, wc[0].x, num, 0);
    return;
  }

  const int n_steps = (total + kSpStep - 1) / kSpStep;
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    const int group = 4 * warp + q;
    const int64_t slot0 = tile * kTile + group * kNG;
    const float4 near = group_reach(S.tv[group * kNG + (lane & 7)], a.kd.c2_out);
    const uint32_t pair_s = (uint32_t)__cvta_generic_to_shared(&S.pair[group][0][0]);
    LaneSums<CN> L;
    L.clear();
    for (int step = 0; step < n_steps; ++step) {
      if (q == 0 || n_steps > 1) {
        __syncthreads();   // everyone is done with what was staged before
        stage(step * kSpStep);
        __syncthreads();
      }
      const int cnt = list_near<kSpStep / 32>(S.rec, near, S.list[warp]);
      add_listed<CN, FORM>(na, L, S.list[warp], cnt, S.rec, S.dat, S.idx, pair_s, S.tv + group * kNG, slot0);
      __syncwarp();        // the warp's list is rewritten
    }
    write_group(na, L, slot0, 0);
  }
}

// Channel rows in sorted order, padded to CN channels (BF16 values as FP32).
template <typename DT, int CN>
__global__ void __launch_bounds__(256) k_rows_sorted(const DT* __restrict__ data,
                                                     const uint32_t* __restrict__ perm, int64_t n,
                                                     int C, float* __restrict__ rows) {
  const int64_t s = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (s >= n) return;
  const DT* src = data + (size_t)perm[s] * C;
  float v[CN];
#pragma unroll
  for (int k = 0; k < CN; ++k) v[k] = k < C ? (float)src[k] : 0.f;
  float* dst = rows + (size_t)s * CN;
  if constexpr (CN == 1) {
    dst[0] = v[0];
  } else if constexpr (CN == 2) {
    *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int k = 0; k < CN; k += 4)
      *reinterpret_cast<float4*>(dst + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
  }
}

template <int CN>
cudaError_t launch_narrow(const NarrowArgs& na, int64_t n_tiles, int64_t n, int dtype, float* rows,
                          cudaStream_t s) {
  if (!rows) {
  } else if (dtype == CG_BF16)
    k_rows_sorted<__nv_bfloat16, CN><<<ceil_div(n, 256), 256, 0, s>>>(
        static_cast<const __nv_bfloat16*>(na.g.data), na.g.perm, n, na.g.C, rows);
  else
    k_rows_sorted<float, CN><<<ceil_div(n, 256), 256, 0, s>>>(
        static_cast<const float*>(na.g.data), na.g.perm, n, na.g.C, rows);
  const dim3 grid((unsigned)n_tiles, 1, (unsigned)na.g.n_split);
  auto go = [&](auto dense, auto sparse) {
    if (na.sparse) sparse<<<(unsigned)n_tiles, kSpTh, 0, s>>>(na);
    else dense<<<grid, kNTh, 0, s>>>(na);
  };
  switch (weight_form(na.g.kd)) {
    case kWGauss1: go(k_grid_narrow<CN, kWGauss1>, k_grid_sparse<CN, kWGauss1>); break;
    case kWGauss2: go(k_grid_narrow<CN, kWGauss2>, k_grid_sparse<CN, kWGauss2>); break;
    case kWGauss1Ds: go(k_grid_narrow<CN, kWGauss1Ds>, k_grid_sparse<CN, kWGauss1Ds>); break;
    default: go(k_grid_narrow<CN, kWAny>, k_grid_sparse<CN, kWAny>); break;
  }
  return cudaGetLastError();
}

}  // namespace

int narrow_width(int C) { return C <= 1 ? 1 : (C <= 2 ? 2 : (C <= 4 ? 4 : 8)); }

// Candidate shares per tile: enough CTAs for ~16 rounds of the resident ones
// (456 at three per SM) where the targets form few tiles, but at least ~4
// steps of candidates each (a tile sees about twice the samples it holds).
int narrow_splits(int64_t n_tiles, int64_t n, int n_sms) {
  const int64_t want = ((int64_t)n_sms * 3 * 16 + n_tiles - 1) / n_tiles;
  const int64_t most = 2 * n / n_tiles / (4 * kNTh);
  return (int)std::max<int64_t>(1, std::min<int64_t>(64, std::min(want, most)));
}

// Where k_grid_sparse is the faster form: few samples per tile (a tile sees two to
// four times those), and the more tiles the more, because the dense form's CTAs
// are few per SM.  Measured on GB300, sparse / dense, one channel: 32,768 tiles 12
// samples each 0.58, 25 0.84, 32 0.99, 40 1.08; 2048 tiles 8 0.84, 18 0.95, 25
// 1.05; seven channels: 32,768 tiles 28 0.80, 36 0.91, 48 0.98; 3633 tiles 20 0.86,
// 28 0.97, 36 1.04.  Around one tile per SM a tile's own latency counts, which is
// shorter with eight warps (156 tiles, 13 samples each: 1.12).
bool sparse_tiles(int64_t n_tiles, int64_t n, int C, int n_sms) {
  if (2 * n_tiles < 3 * n_sms) return false;
  const int most = n_tiles < 20 * n_sms ? 16 : (n_tiles < 60 * n_sms ? 26 : (C <= 2 ? 30 : 44));
  return n < most * n_tiles;
}

cudaError_t grid_narrow(const GridArgs& a, const Tiling& t, int64_t n, int dtype, float* rows, int n_sms,
                        cudaStream_t s) {
  NarrowArgs na;
  na.g = a;
  na.range_c = t.range_c;
  na.rows = rows;
  na.sparse = a.n_split == 1 && sparse_tiles(t.n_tiles, n, a.C, n_sms);
  na.kc = weight_const(a.kd);
  switch (narrow_width(a.C)) {
    case 1: return launch_narrow<1>(na, t.n_tiles, n, dtype, rows, s);
    case 2: return launch_narrow<2>(na, t.n_tiles, n, dtype, rows, s);
    case 4: return launch_narrow<4>(na, t.n_tiles, n, dtype, rows, s);
    default: return launch_narrow<8>(na, t.n_tiles, n, dtype, rows, s);
  }
}

}  // namespace cg
