// k_healpix.cu -- the HEALPix lookup of the paper (Sect. 2.2, 3.3, 3.4) on
// the GPU, reorganised around target tiles instead of per-sample discs:
//
//   samples:  RING index of every sample (Sect. 2.2 step 3a), a stable sort by
//             index (replacing the hash tables of Sect. 3.4), per-ring offsets
//             into the sorted order, and the sorted samples' unit vectors;
//   tiles:    one disc query per tile of targets (Sect. 2.2 step 3b, done once
//             per tile rather than once per sample), radius = tile radius +
//             support, as closed-form pixel intervals per ring (the per-ring
//             treatment of Sect. 3.3);
//   ranges:   each pixel interval becomes a contiguous range of sorted samples
//             by two binary searches inside its ring.
#include "cg_common.cuh"
#include "cg_internal.h"
#include "cg_trig.cuh"
#include "cg_healpix.cuh"

namespace cg {
namespace {

// One warp per tile; mode 0 counts ranges, mode 1 writes them.  The tile's
// candidates are the samples within r of any of its 4-target groups' discs
// (radius group radius + r): per ring, the hull of those discs' pixel
// intervals, which follows the outline of the tile widened by r (one disc of
// radius tile radius + r around the centre would hold ~1.4x as many samples
// for a square tile).  Bound by the arithmetic of 32 lanes (rings) x 32 discs,
// in FP32 (cg_healpix.cuh).
constexpr int kQueryWarps = 8;
constexpr int kMaxDiscs = 32;

__global__ void __launch_bounds__(32 * kQueryWarps) k_tile_query(
    const float4* __restrict__ grp, int n_grp,
    int64_t n_tiles, int ns, float r_rad, int64_t* __restrict__ counts,
    const int64_t* __restrict__ offs, Range* __restrict__ out, int mode) {
  __shared__ Disc sdisc[kQueryWarps][kMaxDiscs];
  const int64_t tile = (int64_t)blockIdx.x * kQueryWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  if (tile >= n_tiles) return;
  Disc* discs = sdisc[wq];
  const int nd = n_grp;
  if (lane < nd) {
    const float4 gc = grp[tile * nd + lane];
    Disc d = make_disc_f(gc.x, gc.y, gc.z, gc.w + r_rad);
    if (gc.w < 0.f) d.R = -1.f;   // empty group
    discs[lane] = d;
  }
  __syncwarp();
  // colatitude span of all discs
  float tlo = kPiF, thi = 0.f;
  for (int q = 0; q < nd; ++q) {
    if (discs[q].R < 0.f) continue;
    tlo = fminf(tlo, discs[q].tc - discs[q].R);
    thi = fmaxf(thi, discs[q].tc + discs[q].R);
  }
  if (thi < tlo) {  // no member at all
    if (mode == 0 && lane == 0) counts[tile] = 0;
    return;
  }
  int ilo, ihi;
  ring_span(ns, tlo, thi, ilo, ihi);
  int64_t pos = (mode == 1) ? offs[tile] : 0;
  int64_t total = 0;
  for (int base = ilo; base <= ihi; base += 32) {
    const int i = base + lane;
    Range rr[2];
    const int n = (i <= ihi) ? ring_ranges(ns, i, discs, nd, rr) : 0;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int sum = __shfl_sync(0xffffffffu, incl, 31);
    if (mode == 1) {
      for (int q = 0; q < n; ++q) {
        rr[q].pad = (int32_t)tile;
        out[pos + incl - n + q] = rr[q];
      }
      pos += sum;
    }
    total += sum;
  }
  if (mode == 0 && lane == 0) counts[tile] = total;
}


// off[i] = sum of counts[0 .. i), i = 0 .. n: one CTA, a run of consecutive
// counts per thread and step (n is the number of tiles, at most ~1e5 in use).
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 8;
__global__ void __launch_bounds__(kScanThreads) k_count_scan(const int64_t* __restrict__ counts,
                                                             int64_t n, int64_t* __restrict__ off) {
  __shared__ int64_t wsum[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int64_t carry = 0;
  for (int64_t base = 0; base < n; base += kScanThreads * kScanPer) {
    int64_t v[kScanPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      const int64_t i = base + (int64_t)tid * kScanPer + k;
      v[k] = i < n ? counts[i] : 0;
      sum += v[k];
    }
    int64_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int64_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < 32; ++w) {
      if (w < warp) before += wsum[w];
      all += wsum[w];
    }
    int64_t x = carry + before + incl - sum;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      const int64_t i = base + (int64_t)tid * kScanPer + k;
      if (i < n) off[i] = x;
      x += v[k];
    }
    carry += all;
    __syncthreads();   // wsum is rewritten by the next step
  }
  if (tid == 0) off[n] = carry;
}

// RING index of a valid direction and the double-float sine / cosine of its
// latitude and longitude.  Ordinary angles (|lon| < 2048 deg) take an FP64-free
// path: the inputs are split into double-float pairs with integer operations,
// the trigonometry and the index arithmetic run in double-float, and only a
// decision within the margin of a pixel boundary, the cap/belt boundary, the
// immediate neighbourhood of a pole and the caps' quadrant boundaries go to
// the FP64 routines.
__device__ __forceinline__ int64_t key_and_sincos(int64_t ns, double lo, double la, df32& sb,
                                                  df32& cb, df32& sl, df32& cl) {
  const bool fast = df_split_ok(lo) && df_split_ok(la) &&
                    (__double_as_longlong(lo) & 0x7ff0000000000000ll) < (1034ll << 52);
  bool ok = false;
  int64_t kpix = 0;
  if (fast) {
    const df32 lon_d = df_split(lo), lat_d = df_split(la);
    df_sincos_deg_df(lat_d, sb, cb);
    df_sincos_deg_df(lon_d, sl, cl);
    kpix = ang2pix_ring_df(ns, lon_d, sb, &ok);
  } else {
    df_sincos_deg(la, sb, cb);
    df_sincos_deg(lo, sl, cl);
  }
  return ok ? kpix : ang2pix_ring_dual(ns, lo, la, sb);
}

__global__ void k_ang2pix_export(int64_t ns, const double* __restrict__ lon,
                                 const double* __restrict__ lat, int64_t n,
                                 int64_t* __restrict__ pix) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double lo = lon[i], la = lat[i];
  if (!valid_coord(lo, la)) {
    pix[i] = -1;
    return;
  }
  df32 sb, cb, sl, cl;
  pix[i] = key_and_sincos(ns, lo, la, sb, cb, sl, cl);
}

// Unit vectors (double-float) of n directions, as FP64 [n][3].
__global__ void k_unit_vectors(const double* __restrict__ lon, const double* __restrict__ lat,
                               int64_t n, double* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  df32 sb, cb, sl, cl;
  df_sincos_deg(lat[i], sb, cb);
  df_sincos_deg(lon[i], sl, cl);
  const df32 x = df_mul(cb, cl), y = df_mul(cb, sl);
  out[3 * i + 0] = (double)x.hi + (double)x.lo;
  out[3 * i + 1] = (double)y.hi + (double)y.lo;
  out[3 * i + 2] = (double)sb.hi + (double)sb.lo;
}

// Per sample (input order): RING key (invalid samples get npix and sort to
// the end), identity value for the sort, and the unit vector as (hi, lo)
// FP32 pairs with w = sample weight, one 32-byte record u[2 i], u[2 i + 1].
// A single channel's value takes the record's last word: the gather into
// sorted order moves it in the sector that it reads anyway (a gather of its
// own took 1.58 ms for 1e8 samples).
__global__ void k_sample_keys(int64_t ns, const double* __restrict__ lon,
                              const double* __restrict__ lat,
                              const float* __restrict__ weights, int64_t n,
                              const void* __restrict__ values, int bf16,
                              uint32_t* __restrict__ key, uint32_t* __restrict__ val,
                              float4* __restrict__ u, double2* __restrict__ sll, unsigned* err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double lo = lon[i], la = lat[i];
  val[i] = (uint32_t)i;
  sll[i] = make_double2(lo, la);
  if (!valid_coord(lo, la)) {
    key[i] = (uint32_t)(12 * ns * ns);
    u[2 * i] = make_float4(4.f, 4.f, 4.f, 0.f);
    u[2 * i + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
    set_error(err, ERR_BAD_SAMPLE);
    return;
  }
  df32 sb, cb, sl, cl;
  key[i] = (uint32_t)key_and_sincos(ns, lo, la, sb, cb, sl, cl);
  const df32 x = df_mul(cb, cl), y = df_mul(cb, sl);
  float w = 1.f;
  if (weights) {
    w = weights[i];
    if (!(w >= 0.f) || !isfinite(w)) {
      set_error(err, ERR_BAD_SAMPLE);
      w = 0.f;
    }
  }
  float v = 0.f;
  if (values)
    v = bf16 ? __uint_as_float((uint32_t)static_cast<const uint16_t*>(values)[i] << 16)
             : static_cast<const float*>(values)[i];
  u[2 * i] = make_float4(x.hi, y.hi, sb.hi, w);
  u[2 * i + 1] = make_float4(x.lo, y.lo, sb.lo, v);
}


// Sorted order: gather the unit vectors (CTAs 0 .. nb - 1, one thread per
// sample), and ring_off[i] = first sorted position with ring >= i, i = 0 ..
// 4 ns (the CTAs after them, one thread per ring: a binary search for the
// ring's first pixel).  Latency-bound: when the thread at a gap of the
// coverage filled the entries of all the rings in the gap one by one, a small
// field (thousands of empty rings before its first sample) paid for a serial
// chain of thousands of stores: 2e4 samples at nside 4096 took 29.7 us, 1e6
// samples 47 us; the searches run side by side with the gather.
__global__ void __launch_bounds__(256) k_sample_gather(
    int64_t ns, int64_t nb, const uint32_t* __restrict__ skey, const uint32_t* __restrict__ sval,
    const float4* __restrict__ u_hi, const float4* __restrict__ u_lo, int stride, int64_t n,
    float4* __restrict__ s_hi, float4* __restrict__ s_lo, int32_t* __restrict__ ring_off) {
  if (blockIdx.x >= nb) {
    const int64_t i = (int64_t)(blockIdx.x - nb) * 256 + threadIdx.x;
    if (i <= 4 * ns) ring_off[i] = lower_bound_u32(skey, 0, (int32_t)n, (uint32_t)ring_first(ns, i));
    return;
  }
  const int64_t s = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (s >= n) return;
  const int64_t idx = (int64_t)sval[s] * stride;
  s_hi[s] = u_hi[idx];
  s_lo[s] = u_lo[idx];
}


// One warp per tile: the sorted-sample interval [lo, hi) of each of the
// tile's pixel ranges (binary search inside the range's ring), the number of
// the tile's candidates before each range (cum), and the tile's total.
__global__ void k_tile_ranges(const Range* __restrict__ ranges,
                              const int64_t* __restrict__ range_off, int64_t n_tiles,
                              const int32_t* __restrict__ ring_off,
                              const uint32_t* __restrict__ skey, int2* __restrict__ out,
                              int32_t* __restrict__ cum, int32_t* __restrict__ tile_cand) {
  const int64_t tile = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (tile >= n_tiles) return;
  const int64_t r0 = range_off[tile], r1 = range_off[tile + 1];
  int32_t running = 0;
  for (int64_t b = r0; b < r1; b += 32) {
    const int64_t r = b + lane;
    int32_t lo = 0, hi = 0;
    if (r < r1) {
      const Range q = ranges[r];
      const int32_t a = ring_off[q.ring], e = ring_off[q.ring + 1];
      lo = a;
      hi = a;
      if (e > a) {
        lo = lower_bound_u32(skey, a, e, (uint32_t)q.pix_lo);
        hi = lower_bound_u32(skey, lo, e, (uint32_t)q.pix_hi + 1u);
      }
    }
    const int32_t cnt = hi - lo;
    int32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (r < r1) {
      out[r] = make_int2(lo, hi);
      cum[r] = running + incl - cnt;
    }
    running += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) tile_cand[tile] = running;
}

__global__ void k_export(const uint32_t* __restrict__ skey, const uint32_t* __restrict__ sval,
                         int64_t n, int64_t* __restrict__ pix, int64_t* __restrict__ perm) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  pix[s] = skey[s];
  perm[s] = sval[s];
}

__global__ void k_export_ring(const int32_t* __restrict__ ro, int64_t m, int64_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) out[i] = ro[i];
}

}  // namespace

// ---------------------------------------------------------------------------
// Fused batches: the sample index of all jobs at once.
// ---------------------------------------------------------------------------
namespace {

// Largest j with off[j] <= x (off[0] = 0, x < off[n]).
__device__ __forceinline__ int batch_job(const int64_t* __restrict__ off, int n, int64_t x) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// k_sample_keys for every job: composite key (job key base + RING key at the
// job's nside), the sample's index within its job, its unit vector record
// and FP64 lon/lat at its batch position.  CTA b serves 256 samples of the
// job whose CTA range (blk: prefix of the jobs' CTA counts) holds b.
__global__ void __launch_bounds__(256) k_batch_keys(const BatchIndexJob* __restrict__ jobs,
                                                    const int64_t* __restrict__ blk, int n_jobs,
                                                    uint64_t* __restrict__ key,
                                                    uint32_t* __restrict__ val,
                                                    float4* __restrict__ u,
                                                    double2* __restrict__ sll, unsigned* err) {
  __shared__ int s_job;
  if (threadIdx.x == 0) s_job = batch_job(blk, n_jobs, blockIdx.x);
  __syncthreads();
  const int j = s_job;
  const BatchIndexJob& J = jobs[j];
  const int64_t li = (int64_t)(blockIdx.x - blk[j]) * 256 + threadIdx.x;
  if (li >= J.n) return;
  const int64_t i = J.off + li;
  const int64_t ns = J.nside;
  const double lo = J.lon[li], la = J.lat[li];
  val[i] = (uint32_t)li;
  sll[i] = make_double2(lo, la);
  if (!valid_coord(lo, la)) {
    key[i] = J.key_base + (uint64_t)(12 * ns * ns);
    u[2 * i] = make_float4(4.f, 4.f, 4.f, 0.f);
    u[2 * i + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
    set_error(err, ERR_BAD_SAMPLE);
    return;
  }
  df32 sb, cb, sl, cl;
  key[i] = J.key_base + (uint64_t)key_and_sincos(ns, lo, la, sb, cb, sl, cl);
  const df32 x = df_mul(cb, cl), y = df_mul(cb, sl);
  float w = 1.f;
  if (J.weights) {
    w = J.weights[li];
    if (!(w >= 0.f) || !isfinite(w)) {
      set_error(err, ERR_BAD_SAMPLE);
      w = 0.f;
    }
  }
  u[2 * i] = make_float4(x.hi, y.hi, sb.hi, w);
  u[2 * i + 1] = make_float4(x.lo, y.lo, sb.lo, 0.f);
}

// First of the sorted composite keys [lo, hi) that is at least v.
__device__ __forceinline__ int64_t lower_bound_u64(const uint64_t* __restrict__ a, int64_t lo,
                                                   int64_t hi, uint64_t v) {
  while (lo < hi) {
    const int64_t mid = lo + ((hi - lo) >> 1);
    if (a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// k_sample_gather for every job: a job's CTAs (blk: prefix of the jobs' CTA
// counts) serve its ceil(n / 256) blocks of samples and then its 4 nside + 1
// ring offsets, which are relative to the job's segment, so that each job
// sees its own index as if it ran alone.
__global__ void __launch_bounds__(256) k_batch_gather(const BatchIndexJob* __restrict__ jobs,
                                                      const int64_t* __restrict__ blk, int n_jobs,
                                                      const uint64_t* __restrict__ skey64,
                                                      const uint32_t* __restrict__ sval,
                                                      const float4* __restrict__ u,
                                                      float4* __restrict__ s_hi,
                                                      float4* __restrict__ s_lo,
                                                      uint32_t* __restrict__ skey,
                                                      int32_t* __restrict__ ring_off) {
  __shared__ int s_job;
  if (threadIdx.x == 0) s_job = batch_job(blk, n_jobs, blockIdx.x);
  __syncthreads();
  const int j = s_job;
  const BatchIndexJob& J = jobs[j];
  const int64_t b = (int64_t)blockIdx.x - blk[j];
  const int64_t nb = (J.n + 255) / 256;
  if (b >= nb) {
    const int64_t i = (b - nb) * 256 + threadIdx.x;
    if (i <= 4 * J.nside)
      ring_off[J.ring_base + i] =
          (int32_t)(lower_bound_u64(skey64, J.off, J.off + J.n,
                                    J.key_base + (uint64_t)ring_first(J.nside, i)) -
                    J.off);
    return;
  }
  const int64_t s = b * 256 + threadIdx.x;
  if (s >= J.n) return;
  const int64_t gs = J.off + s;
  const int64_t rec = 2 * (J.off + (int64_t)sval[gs]);
  s_hi[gs] = u[rec];
  s_lo[gs] = u[rec + 1];
  skey[gs] = (uint32_t)(skey64[gs] - J.key_base);
}

// k_tile_ranges for the tiles of every job (one warp per tile).
__global__ void k_batch_ranges(const BatchIndexJob* __restrict__ jobs,
                               const int64_t* __restrict__ tile_off, int n_jobs, int64_t n_tiles,
                               const int32_t* __restrict__ ring_off_all,
                               const uint32_t* __restrict__ skey_all) {
  const int64_t gt = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (gt >= n_tiles) return;
  const int j = batch_job(tile_off, n_jobs, gt);
  const BatchIndexJob& J = jobs[j];
  const int64_t tile = gt - tile_off[j];
  const int32_t* ring_off = ring_off_all + J.ring_base;
  const uint32_t* skey = skey_all + J.off;
  const int64_t r0 = J.range_off[tile], r1 = J.range_off[tile + 1];
  int32_t running = 0;
  for (int64_t b = r0; b < r1; b += 32) {
    const int64_t r = b + lane;
    int32_t lo = 0, hi = 0;
    if (r < r1) {
      const Range q = J.ranges[r];
      const int32_t a = ring_off[q.ring], e = ring_off[q.ring + 1];
      lo = a;
      hi = a;
      if (e > a) {
        lo = lower_bound_u32(skey, a, e, (uint32_t)q.pix_lo);
        hi = lower_bound_u32(skey, lo, e, (uint32_t)q.pix_hi + 1u);
      }
    }
    const int32_t cnt = hi - lo;
    int32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (r < r1) {
      J.range_s[r] = make_int2(lo, hi);
      J.range_c[r] = running + incl - cnt;
    }
    running += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) J.tile_cand[tile] = running;
}

}  // namespace

cudaError_t batch_index_alloc(BatchIndex& bi, cudaStream_t s) {
  const size_t n = (size_t)bi.N;
  cudaError_t e;
  if ((e = dalloc(&bi.key, n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&bi.val, n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&bi.u_rec, 2 * n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&bi.sll, n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&bi.s_hi, n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&bi.s_lo, n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&bi.skey, n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&bi.ring_off, (size_t)bi.n_ring, s)) != cudaSuccess) return e;
  return cudaSuccess;
}

void batch_index_free(BatchIndex& bi, cudaStream_t s) {
  dfree(bi.jobs, s);
  dfree(bi.key_blk, s);
  dfree(bi.gth_blk, s);
  dfree(bi.tile_off, s);
  dfree(bi.key, s);
  dfree(bi.val, s);
  dfree(bi.u_rec, s);
  dfree(bi.sll, s);
  dfree(bi.s_hi, s);
  dfree(bi.s_lo, s);
  dfree(bi.skey, s);
  dfree(bi.ring_off, s);
  if (bi.sw.keys_alt) cudaFreeAsync(bi.sw.keys_alt, s);
  bi.sw.keys_alt = nullptr;
  dfree(bi.sw.vals_alt, s);
  dfree(bi.sw.hist, s);
  dfree(bi.sw.totals, s);
  dfree(bi.sw.status, s);
  dfree(bi.sw.os_meta, s);
  bi.sw = SortWork();
  bi.sorted_key = nullptr;
  bi.sorted_val = nullptr;
}

cudaError_t batch_index_run(BatchIndex& bi, unsigned* err, cudaStream_t s, int64_t* launches) {
  if (bi.N <= 0) return cudaSuccess;
  k_batch_keys<<<(unsigned)bi.n_key_blk, 256, 0, s>>>(bi.jobs, bi.key_blk, bi.n_jobs, bi.key,
                                                      bi.val, bi.u_rec, bi.sll, err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = radix_sort_u64(bi.key, bi.val, bi.N, bi.key_bits, bi.sw, s, &bi.sorted_key, &bi.sorted_val);
  if (e != cudaSuccess) return e;
  k_batch_gather<<<(unsigned)bi.n_gth_blk, 256, 0, s>>>(
      bi.jobs, bi.gth_blk, bi.n_jobs, bi.sorted_key, bi.sorted_val, bi.u_rec, bi.s_hi,
      bi.s_lo, bi.skey, bi.ring_off);
  if (bi.n_tiles > 0) {
    const int warps = 8;
    k_batch_ranges<<<ceil_div(bi.n_tiles, warps), 32 * warps, 0, s>>>(
        bi.jobs, bi.tile_off, bi.n_jobs, bi.n_tiles, bi.ring_off, bi.skey);
  }
  if (launches) *launches += 3 + 3 * ((bi.key_bits + 7) / 8);
  return cudaGetLastError();
}

int key_bits_for(int64_t ns) {
  const uint64_t maxkey = (uint64_t)(12 * ns * ns);  // sentinel for invalid samples
  int b = 0;
  while (b < 32 && (maxkey >> b) != 0) ++b;
  return b;
}

cudaError_t ang2pix_export(int nside, const double* lon, const double* lat, int64_t n,
                           int64_t* pix, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_ang2pix_export<<<ceil_div(n, 256), 256, 0, s>>>(nside, lon, lat, n, pix);
  return cudaGetLastError();
}

cudaError_t unit_vectors(const double* lon, const double* lat, int64_t n, double* out,
                         cudaStream_t s) {
  if (n > 0) k_unit_vectors<<<ceil_div(n, 256), 256, 0, s>>>(lon, lat, n, out);
  return cudaGetLastError();
}

void tiling_free(Tiling& t, cudaStream_t s) {
  dfree(t.chi, s);
  dfree(t.clo, s);
  dfree(t.a, s);
  dfree(t.tile_cand, s);
  dfree(t.order, s);
  t.cap_order = 0;
  dfree(t.grp, s);
  dfree(t.subf, s);
  dfree(t.range_off, s);
  dfree(t.ranges, s);
  dfree(t.range_s, s);
  dfree(t.range_c, s);
  t.n_ranges = 0;
}

// Both tilings' candidate ranges: count, exclusive scan, write.  The host
// waits once, for the two totals that size the range arrays.
cudaError_t tiles_query(cg_grid* g) {
  cudaStream_t s = g->stream;
  const float r = (float)(g->support_deg * kDeg2Rad);
  Tiling* ts[2] = {&g->t64, &g->t128};
  int64_t* counts[2] = {nullptr, nullptr};
  int64_t total[2] = {0, 0};
  cudaError_t e = cudaSuccess;
  for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
    Tiling& t = *ts[q];
    dfree(t.range_off, s);
    dfree(t.ranges, s);
    dfree(t.range_s, s);
    dfree(t.range_c, s);
    t.n_ranges = 0;
    e = dalloc(&counts[q], (size_t)t.n_tiles, s);
    if (e == cudaSuccess) e = dalloc(&t.range_off, (size_t)t.n_tiles + 1, s);
    if (e != cudaSuccess) break;
    k_tile_query<<<ceil_div(t.n_tiles, kQueryWarps), 32 * kQueryWarps, 0, s>>>(
        t.grp, t.T / 4, t.n_tiles, g->nside, r, counts[q], nullptr, nullptr, 0);
    k_count_scan<<<1, kScanThreads, 0, s>>>(counts[q], t.n_tiles, t.range_off);
    g->n_launches += 2;
    e = cudaMemcpyAsync(&total[q], t.range_off + t.n_tiles, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
    Tiling& t = *ts[q];
    t.n_ranges = total[q];
    if ((e = dalloc(&t.ranges, (size_t)t.n_ranges, s)) != cudaSuccess) break;
    if ((e = dalloc(&t.range_s, (size_t)t.n_ranges, s)) != cudaSuccess) break;
    if ((e = dalloc(&t.range_c, (size_t)t.n_ranges, s)) != cudaSuccess) break;
    k_tile_query<<<ceil_div(t.n_tiles, kQueryWarps), 32 * kQueryWarps, 0, s>>>(
        t.grp, t.T / 4, t.n_tiles, g->nside, r, nullptr, t.range_off, t.ranges, 1);
    g->n_launches += 1;
    e = cudaGetLastError();
  }
  for (int q = 0; q < 2; ++q) dfree(counts[q], s);
  if (e != cudaSuccess) return e;
  dfree(g->ring_off, s);
  return dalloc(&g->ring_off, (size_t)(4 * g->nside + 1), s);
}

static cudaError_t ensure_samples(cg_grid* g, int64_t n) {
  if (g->cap_n >= (size_t)n) return cudaSuccess;
  cudaStream_t s = g->stream;
  dfree(g->key, s);
  dfree(g->val, s);
  dfree(g->s_hi, s);
  dfree(g->s_lo, s);
  dfree(g->u_rec, s);
  dfree(g->s_ll, s);
  g->cap_n = 0;
  cudaError_t e;
  if ((e = dalloc(&g->key, (size_t)n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->val, (size_t)n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->s_hi, (size_t)n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->s_lo, (size_t)n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->u_rec, 2 * (size_t)n, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->s_ll, (size_t)n, s)) != cudaSuccess) return e;
  g->cap_n = (size_t)n;
  return cudaSuccess;
}

cudaError_t samples_keys(cg_grid* g, const double* lon, const double* lat, const float* weights,
                         int64_t n, const void* values, int dtype) {
  cudaError_t e = ensure_samples(g, n);
  if (e != cudaSuccess) return e;
  k_sample_keys<<<ceil_div(n, 256), 256, 0, g->stream>>>(g->nside, lon, lat, weights, n, values,
                                                         dtype == CG_BF16, g->key, g->val, g->u_rec, g->s_ll,
                                                         g->d_err);
  g->n_launches += 1;
  return cudaGetLastError();
}

cudaError_t samples_sort(cg_grid* g, int64_t n) {
  const int bits = key_bits_for(g->nside);
  g->n_launches += radix_sort_u32_launches(n, bits);
  g->sw.err = g->d_err;
  return radix_sort_u32(g->key, g->val, n, bits, g->sw, g->stream, &g->sorted_key,
                        &g->sorted_val);
}

cudaError_t sorted_gather(int64_t ns, const uint32_t* skey, const uint32_t* sval,
                          const float4* u_hi, const float4* u_lo, int stride, int64_t n,
                          float4* s_hi, float4* s_lo, int32_t* ring_off, cudaStream_t s) {
  const int64_t nb = ceil_div(n, 256);
  k_sample_gather<<<(unsigned)(nb + ceil_div(4 * ns + 1, 256)), 256, 0, s>>>(
      ns, nb, skey, sval, u_hi, u_lo, stride, n, s_hi, s_lo, ring_off);
  return cudaGetLastError();
}

cudaError_t samples_prepare(cg_grid* g, int64_t n) {
  cudaStream_t s = g->stream;
  const int64_t ns = g->nside;
  cudaError_t e = sorted_gather(ns, g->sorted_key, g->sorted_val, g->u_rec, g->u_rec + 1, 2, n, g->s_hi,
                                g->s_lo, g->ring_off, s);
  if (e != cudaSuccess) return e;
  g->n_launches += 1;
  g->last_n = n;
  return cudaGetLastError();
}

cudaError_t tiles_ranges(cg_grid* g, Tiling& t) {
  if (t.n_tiles > 0) {
    const int warps = 8;
    k_tile_ranges<<<ceil_div(t.n_tiles, warps), 32 * warps, 0, g->stream>>>(
        t.ranges, t.range_off, t.n_tiles, g->ring_off, g->sorted_key, t.range_s, t.range_c,
        t.tile_cand);
    g->n_launches += 1;
  }
  return cudaGetLastError();
}

cudaError_t export_index(cg_grid* g, int64_t* sorted_pix, int64_t* perm, int64_t* ring_off,
                         int64_t n) {
  cudaStream_t s = g->stream;
  if (n > 0) k_export<<<ceil_div(n, 256), 256, 0, s>>>(g->sorted_key, g->sorted_val, n,
                                                      sorted_pix, perm);
  if (ring_off) {
    const int64_t m = 4 * (int64_t)g->nside + 1;
    k_export_ring<<<ceil_div(m, 256), 256, 0, s>>>(g->ring_off, m, ring_off);
  }
  return cudaGetLastError();
}

}  // namespace cg
