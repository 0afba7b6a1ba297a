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
//   end      the lanes' sums are added up by shuffles (compensated for W).
//
// Bound by issue slots and by the barrier per step (58 % of the issue slots
// used, ALU pipe 46 %).  Measured on GB300 against the register-blocked form
// it replaced (one target per thread, weights through shared memory, every
// candidate of the tile evaluated): 1e8 samples onto 8,100 targets 36.6 ->
// 8.3 ms, 1e6 samples onto 512 x 512 targets 0.95 -> 0.33 ms, 1.2e7 samples on
// the sphere onto 786,432 targets 4.48 -> 1.37 ms; the sums of 32 lanes are
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
  const WeightConst& kc = na.kc;

  const uint32_t pair_s = (uint32_t)__cvta_generic_to_shared(&S.pair[warp][0][0]);
  // ---- the warp's targets: packed pairs in shared memory (read by all lanes
  // at once); centre and reach of the group (empty slots sit at (4, 4, 4)) ----
  if (tid < kTile) S.tv[tid] = a.tgt_a[tile * kTile + tid];
  if (lane < 4) {
    float2* A = S.pair[warp][lane];
    const int64_t sa = slot0 + 2 * lane;
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
  float gx, gy, gz, reach2;
  {
    const float4 p = a.tgt_a[slot0 + (lane & 7)];   // four copies of the group
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
    gx = sx * inv;
    gy = sy * inv;
    gz = sz * inv;
    const float ex = p.x - gx, ey = p.y - gy, ez = p.z - gz;
    float rad2 = on ? ex * ex + ey * ey + ez * ez : 0.f;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) rad2 = fmaxf(rad2, __shfl_xor_sync(0xffffffffu, rad2, o));
    const float reach = sqrtf(rad2) + sqrtf(a.kd.c2_out);
    reach2 = sn > 0.f ? reach * reach * 1.0001f + 1e-12f : -1.f;
  }

  float2 acc[CN][4], ws[4], wc[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    ws[j] = wc[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < CN; ++c) acc[c][j] = make_float2(0.f, 0.f);
  }
  unsigned npair = 0;

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
        const float* row = na.rows + (size_t)s * CN;
        if constexpr (CN == 1) {
          c.d[0] = na.rows ? row[0] : c.l.w;
        } else if constexpr (CN == 2) {
          const float2 q = *reinterpret_cast<const float2*>(row);
          c.d[0] = q.x; c.d[1] = q.y;
        } else {
#pragma unroll
          for (int k = 0; k < CN; k += 4) {
            const float4 q = *reinterpret_cast<const float4*>(row + k);
            c.d[k] = q.x; c.d[k + 1] = q.y; c.d[k + 2] = q.z; c.d[k + 3] = q.w;
          }
        }
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
      // ---- list the candidates in reach of the warp's targets ----
      int cnt = 0;
#pragma unroll
      for (int b = 0; b < kNTh / 32; ++b) {
        const float4 p = S.rec[st][32 * b + lane];
        const float ex = p.x - gx, ey = p.y - gy, ez = p.z - gz;
        const bool in = fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= reach2;
        const uint32_t m = __ballot_sync(0xffffffffu, in);
        if (in) S.list[warp][cnt + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(32 * b + lane);
        cnt += __popc(m);
      }
      __syncwarp();
      // ---- weights and sums, 32 listed candidates at a time ----
      for (int b = 0; b < cnt; b += 32) {
        float4 p = make_float4(-4.f, -4.f, -4.f, 0.f);
        int ci = 0;
        float d[CN];
#pragma unroll
        for (int k = 0; k < CN; ++k) d[k] = 0.f;
        if (b + lane < cnt) {
          ci = S.list[warp][b + lane];
          p = S.rec[st][ci];
#pragma unroll
          for (int k = 0; k < CN; ++k) d[k] = S.dat[st][ci * CN + k];
        }
        const float2 nx = f2(-p.x), ny = f2(-p.y), nz = f2(-p.z), om = f2(p.w);
        float2 w[4];
        float near = INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // read for every batch: held in registers they would be spilled
          const uint32_t q6 = pair_s + j * (uint32_t)sizeof(S.pair[0][0]);
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
          npair += (i0 ? 1u : 0u) + (i1 ? 1u : 0u);
          near = band_near(kc, c2, near);
        }
        if (near <= kc.hw) {
          const uint32_t kill = narrow_band(S.tv + warp * kNG, p, a.tgt_ll + slot0, a.sll[S.idx[st][ci]],
                                            a.kd.c2_in, a.kd.c2_out, a.kd.c2r_hi, a.kd.c2r_lo,
                                            a.kd.c2r_tol, a.kd.r_rad);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (kill & (1u << (2 * j))) { w[j].x = -0.f; --npair; }
            if (kill & (2u << (2 * j))) { w[j].y = -0.f; --npair; }
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          kahan2(ws[j], wc[j], w[j]);
#pragma unroll
          for (int k = 0; k < CN; ++k) acc[k][j] = __ffma2_rn(w[j], f2(d[k]), acc[k][j]);
        }
      }
      __syncthreads();   // the stage may be rewritten; the next one is visible
    }
  }

  // ---- the lanes' sums ----
  float wsum = 0.f, wcor = 0.f, num[CN];
#pragma unroll
  for (int k = 0; k < CN; ++k) num[k] = 0.f;
#pragma unroll
  for (int t = 0; t < kNG; ++t) {
    float s = (t & 1) ? ws[t >> 1].y : ws[t >> 1].x;
    float c = (t & 1) ? wc[t >> 1].y : wc[t >> 1].x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
      comp_add(s, c, s2, c2);
    }
    if (lane == t) { wsum = s; wcor = c; }
#pragma unroll
    for (int k = 0; k < CN; ++k) {
      float v = (t & 1) ? acc[k][t >> 1].y : acc[k][t >> 1].x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == t) num[k] = v;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) npair += __shfl_xor_sync(0xffffffffu, npair, o);
  if (lane == 0 && npair && a.pairs) atomicAdd(a.pairs, (unsigned long long)npair);
  if (lane >= kNG) return;
  const int64_t slot = slot0 + lane;
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
  switch (weight_form(na.g.kd)) {
    case kWGauss1: k_grid_narrow<CN, kWGauss1><<<grid, kNTh, 0, s>>>(na); break;
    case kWGauss2: k_grid_narrow<CN, kWGauss2><<<grid, kNTh, 0, s>>>(na); break;
    case kWGauss1Ds: k_grid_narrow<CN, kWGauss1Ds><<<grid, kNTh, 0, s>>>(na); break;
    default: k_grid_narrow<CN, kWAny><<<grid, kNTh, 0, s>>>(na); break;
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

cudaError_t grid_narrow(const GridArgs& a, const Tiling& t, int64_t n, int dtype, float* rows,
                        cudaStream_t s) {
  NarrowArgs na;
  na.g = a;
  na.range_c = t.range_c;
  na.rows = rows;
  na.kc = weight_const(a.kd);
  switch (narrow_width(a.C)) {
    case 1: return launch_narrow<1>(na, t.n_tiles, n, dtype, rows, s);
    case 2: return launch_narrow<2>(na, t.n_tiles, n, dtype, rows, s);
    case 4: return launch_narrow<4>(na, t.n_tiles, n, dtype, rows, s);
    default: return launch_narrow<8>(na, t.n_tiles, n, dtype, rows, s);
  }
}

}  // namespace cg
