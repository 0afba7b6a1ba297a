// k_targets.cu -- target geometry and tiling (set-up, once per handle).
//
// The paper grids onto the pixel centres of a WCS map or onto a list of sight
// lines (Sect. 3.5, WcsGrid / SlGrid).  Here targets are always a list of
// directions.  To give each CTA a compact group of targets (its "tile"), the
// targets are split by a k-d tree over their unit vectors: every node is
// sorted along the wider of its axes and cut at a multiple of the leaf size, so
// all leaves hold exactly that many targets (except the last) and each leaf is a
// compact box.  The axes are east, north and outward at one of the node's
// targets: along x, y and z the cuts of a field away from those axes are oblique
// and its leaves lozenges, which reach further.  1e6 samples x 256 channels onto
// 512 x 512 targets at latitude 30: 6.19 -> 5.85 million candidates, in BF16
// 1.072 -> 0.984 ms per call, in FP32 4.10 -> 3.78; 2.5e5 x 128 1.35 -> 1.26 ms.  The tree is cut to 128-target leaves, then each leaf into
// 64 + 64, 32 + 32 and on down to groups of 4, so a 128-tile is two 64-tiles,
// four 32-target quarters and thirty-two 4-target groups, all compact
// (consecutive slots).  A position's node at any level follows from its index
// alone (the cuts depend on counts only).
//
// A new set of targets is part of every new map, so the build is a path of its
// own: levels of nodes above 4096 targets run over the whole array (bounding
// boxes, 16-bit coordinates within the node's box, one radix sort of the
// 32-bit (node, coordinate) keys per level), all levels below in shared
// memory, one CTA per node.  786,432 sight lines: 18 levels of 64-bit
// three-kernel sort passes with per-target atomics and FP64 geometry took
// 18 ms of kernels.
// Each tile stores
//   - its centre e_c (near the targets' mean) and, for every member,
//     u_t - e_c in FP32 (accurate relative to its size; u_t as a double-float);
//   - the local east / north unit vectors (for the elliptical kernel);
//   - the member's longitude / latitude in FP64 (guard-band recomputation);
//   - the discs of its 4-target groups and (128-tiles) 32-target quarters.
#include <algorithm>

#include "cg_common.cuh"
#include "cg_internal.h"
#include "cg_trig.cuh"

namespace cg {
namespace {

__host__ __device__ __forceinline__ uint32_t orderable_bits(uint32_t b) {
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ uint32_t orderable(float f) { return orderable_bits(__float_as_uint(f)); }
__device__ __forceinline__ float from_orderable(uint32_t u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

__device__ __forceinline__ bool valid_coord(double lon, double lat) {
  return isfinite(lon) && isfinite(lat) && lat >= -90.0 && lat <= 90.0;
}

// Double-float sine and cosine of a longitude or latitude in degrees (FP64
// operations only for angles beyond the split's range).
__device__ __forceinline__ void sincos_deg(double a, df32& s, df32& c) {
  if (df_split_ok(a) && fabs(a) < 2048.0) {
    df_sincos_deg_df(df_split(a), s, c);
  } else {
    double sd, cd;
    sincos(a * kDeg2Rad, &sd, &cd);
    split_f64(sd, s.hi, s.lo);
    split_f64(cd, c.hi, c.lo);
  }
}

__global__ void __launch_bounds__(256) k_target_init(const double* __restrict__ lon,
                                                     const double* __restrict__ lat, int64_t P,
                                                     float4* __restrict__ u_hi,
                                                     float4* __restrict__ u_lo,
                                                     uint32_t* __restrict__ ord, unsigned* err) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= P) return;
  const double lo = lon[i], la = lat[i];
  float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
  if (valid_coord(lo, la)) {
    df32 sb, cb, sl, cl;
    sincos_deg(la, sb, cb);
    sincos_deg(lo, sl, cl);
    const df32 x = df_mul(cb, cl), y = df_mul(cb, sl);
    h = make_float4(x.hi, y.hi, sb.hi, 0.f);
    l = make_float4(x.lo, y.lo, sb.lo, 0.f);
  } else {
    set_error(err, ERR_BAD_TARGET);
  }
  u_hi[i] = h;
  u_lo[i] = l;
  ord[i] = (uint32_t)i;
}

// ---- k-d tree ----
constexpr int kNodeCap = 4096;     // targets of a node finished in shared memory
constexpr int kNodeThreads = 1024;

struct Node {
  uint32_t id, start, cnt;         // id: path from the root (0 left, 1 right)
};

// The part of node q that holds position s after its cut at a multiple of leaf.
__device__ __forceinline__ void descend(Node& q, uint32_t s, uint32_t leaf) {
  q.id *= 2u;
  if (q.cnt <= leaf) return;
  const uint32_t left = leaf * (((q.cnt + leaf - 1) / leaf) / 2);
  if (s - q.start >= left) {
    q.id += 1u;
    q.start += left;
    q.cnt -= left;
  } else {
    q.cnt = left;
  }
}

__device__ __forceinline__ Node node_at(uint32_t s, uint32_t P, int level) {
  Node q{0u, 0u, P};
  for (int l = 0; l < level; ++l) descend(q, s, (uint32_t)kTile2);
  return q;
}

// Axes of a node: east, north and outward at the target in its middle (in the
// order reached so far) where its targets agree on them, else x, y and z.  They
// agree where the node spans at most 20 degrees and the meridians turn by less
// than 15 degrees across it; parts of one node cut along directions that differ
// more become triangles (whole sky, 4096 x 2048 targets, 32 channels: 11.1 ms
// with the rule, 16.6 with local axes at all levels).
struct Frame {
  float3 c, e, n, r;
};

__device__ __forceinline__ Frame world_frame() {
  return {make_float3(0.f, 0.f, 0.f), make_float3(1.f, 0.f, 0.f), make_float3(0.f, 1.f, 0.f),
          make_float3(0.f, 0.f, 1.f)};
}

// The local axes at a target; reach receives the largest extent of a node along
// x, y or z for which they are used.
__device__ __forceinline__ Frame local_frame(const float4 c, float& reach) {
  const float h2 = c.x * c.x + c.y * c.y;
  if (!(h2 > 1e-6f)) {
    reach = -1.f;
    return world_frame();
  }
  const float i = rsqrtf(h2);
  reach = fminf(0.35f, 0.26f * h2 * i / fmaxf(fabsf(c.z), 1e-6f));
  return {make_float3(c.x, c.y, c.z), make_float3(-c.y * i, c.x * i, 0.f),
          make_float3(-c.z * c.x * i, -c.z * c.y * i, h2 * i), make_float3(c.x, c.y, c.z)};
}

__device__ __forceinline__ float3 in_frame(const Frame& f, const float4 v) {
  const float x = v.x - f.c.x, y = v.y - f.c.y, z = v.z - f.c.z;
  return make_float3(x * f.e.x + y * f.e.y + z * f.e.z, x * f.n.x + y * f.n.y + z * f.n.z,
                     x * f.r.x + y * f.r.y + z * f.r.z);
}

// Extent of a box (order-preserving minima, complements of maxima).
__device__ __forceinline__ float3 box_extent(const uint32_t* b) {
  return make_float3(from_orderable(~b[3]) - from_orderable(b[0]),
                     from_orderable(~b[4]) - from_orderable(b[1]),
                     from_orderable(~b[5]) - from_orderable(b[2]));
}

// Bounding boxes of the nodes of a level along x, y, z and along their local
// axes: box[12 n] = the minima, then the complements of the maxima
// (order-preserving integers, so one fill of ones and one atomic minimum serve
// both), and the same again.  A warp covers 256 positions and reduces before its
// atomics (nodes start at multiples of 128): with one atomic per target and side
// the first levels serialised on a few addresses (13 ms for 786,432 targets).
__global__ void __launch_bounds__(256) k_kd_box(const float4* __restrict__ pos,
                                                const uint32_t* __restrict__ ord, uint32_t P,
                                                int level, uint32_t* __restrict__ box) {
  const int lane = threadIdx.x & 31;
  const uint32_t s0 = (blockIdx.x * 8u + (threadIdx.x >> 5)) * 256u;
  uint32_t b[12], cur = 0xffffffffu;
  Frame f{};
#pragma unroll
  for (int k = 0; k < 12; ++k) b[k] = 0xffffffffu;
  auto flush = [&]() {
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const uint32_t m = __reduce_min_sync(0xffffffffu, b[k]);
      if (lane == 0) atomicMin(&box[12 * cur + k], m);
      b[k] = 0xffffffffu;
    }
  };
  for (int r = 0; r < 8; ++r) {
    const uint32_t sw = s0 + 32u * r;   // uniform over the warp
    if (sw >= P) break;
    const Node q = node_at(sw, P, level);
    if (q.id != cur) {
      if (cur != 0xffffffffu) flush();
      cur = q.id;
      float reach;
      f = local_frame(pos[ord[q.start + q.cnt / 2]], reach);
    }
    const uint32_t s = sw + lane;
    if (s < P) {
      const float4 w = pos[ord[s]];
      const float3 v = in_frame(f, w);
      const float c[6] = {w.x, w.y, w.z, v.x, v.y, v.z};
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const uint32_t x = orderable(c[k]);
        const int at = k < 3 ? k : k + 3;
        b[at] = min(b[at], x);
        b[at + 3] = min(b[at + 3], ~x);
      }
    }
  }
  if (cur != 0xffffffffu) flush();
}

// Sort key: (node, coordinate within the node's box along its widest axis).
// ord may be val: every position is rewritten with what it holds.
__global__ void __launch_bounds__(256) k_kd_keys(const float4* __restrict__ pos,
                                                 const uint32_t* ord, uint32_t P, int level,
                                                 const uint32_t* __restrict__ box,
                                                 uint32_t* __restrict__ key, uint32_t* val) {
  const uint32_t s = blockIdx.x * 256u + threadIdx.x;
  if (s >= P) return;
  const Node nd = node_at(s, P, level);
  const uint32_t* b = box + 12 * (size_t)nd.id;
  float reach;
  Frame f = local_frame(pos[ord[nd.start + nd.cnt / 2]], reach);
  float3 ext = box_extent(b);
  if (fmaxf(ext.x, fmaxf(ext.y, ext.z)) <= reach) {
    b += 6;
    ext = box_extent(b);
  } else {
    f = world_frame();
  }
  const uint32_t o = ord[s];
  const float3 v = in_frame(f, pos[o]);
  const int ax = (ext.x >= ext.y && ext.x >= ext.z) ? 0 : (ext.y >= ext.z ? 1 : 2);
  const float c = (ax == 0 ? v.x : (ax == 1 ? v.y : v.z)) - from_orderable(b[ax]);
  const float ex = ax == 0 ? ext.x : (ax == 1 ? ext.y : ext.z);
  key[s] = kd_key(nd.id, level, ex > 0.f ? c / ex : 0.f);
  val[s] = o;
}

struct NodeSmem {
  uint64_t key[kNodeCap];          // (segment, coordinate, place in the node)
  float pos[3][kNodeCap];
  uint32_t box[128][6];            // segments of at least 32 targets
};

// All levels below `level` of node blockIdx.x, down to groups of 4: per level
// the segments' boxes, then a sort along each segment's widest axis.  Bound by
// the barriers of the bitonic sorts; segments of at most 128 targets start at
// multiples of their power-of-two size, so only their own steps run.
__global__ void __launch_bounds__(kNodeThreads) k_kd_node(const float4* __restrict__ pos,
                                                          const uint32_t* __restrict__ ord,
                                                          uint32_t P, int level, int levels2,
                                                          uint32_t* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char raw[];
  NodeSmem& S = *reinterpret_cast<NodeSmem*>(raw);
  const int tid = threadIdx.x, lane = tid & 31;
  // the node: descend along the bits of its id
  Node nd{0u, 0u, P};
  for (int l = 0; l < level; ++l) {
    const uint32_t leaf = (uint32_t)kTile2;
    const uint32_t left = nd.cnt > leaf ? leaf * (((nd.cnt + leaf - 1) / leaf) / 2) : nd.cnt;
    if ((blockIdx.x >> (level - 1 - l)) & 1u) {
      nd.start += left;
      nd.cnt -= left;
    } else {
      nd.cnt = left;
    }
  }
  const uint32_t n = nd.cnt;
  uint32_t np = 128;
  while (np < n) np <<= 1;
  constexpr int kPer = kNodeCap / kNodeThreads;
  Node seg[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const uint32_t i = tid + k * kNodeThreads;
    seg[k] = Node{0u, 0u, n};
    if (i < np) S.key[i] = i < n ? (uint64_t)i : ~0ull;
  }
  // the node's axes
  if (tid < 6) S.box[0][tid] = 0xffffffffu;
  __syncthreads();
  float4 w[kPer];
  {
    uint32_t b[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) b[d] = 0xffffffffu;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t i = tid + k * kNodeThreads;
      if (i >= n) continue;
      w[k] = pos[ord[nd.start + i]];
      const float c[3] = {w[k].x, w[k].y, w[k].z};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        b[d] = min(b[d], orderable(c[d]));
        b[d + 3] = min(b[d + 3], ~orderable(c[d]));
      }
    }
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const uint32_t m = __reduce_min_sync(0xffffffffu, b[d]);
      if (lane == 0 && m != 0xffffffffu) atomicMin(&S.box[0][d], m);
    }
  }
  __syncthreads();
  if (n > 0u) {
    float reach;
    Frame f = local_frame(pos[ord[nd.start + n / 2]], reach);
    const float3 ext = box_extent(S.box[0]);
    if (!(fmaxf(ext.x, fmaxf(ext.y, ext.z)) <= reach)) f = world_frame();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t i = tid + k * kNodeThreads;
      if (i >= n) continue;
      const float3 v = in_frame(f, w[k]);
      S.pos[0][i] = v.x;
      S.pos[1][i] = v.y;
      S.pos[2][i] = v.z;
    }
  }
  __syncthreads();
  for (int l = level; l < levels2 + 5; ++l) {
    // size of the level's segments: multiples of 128 down to tiles, then halves
    const uint32_t cap = l <= levels2 ? 128u : (128u >> (l - levels2));
    const bool small = l >= levels2;     // segments of at most cap targets, aligned to cap
    if (cap >= 32u) {
      for (int i = tid; i < 128 * 6; i += kNodeThreads) S.box[i / 6][i % 6] = 0xffffffffu;
      __syncthreads();
    }
    uint32_t lo[kPer][3], hc[kPer][3];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t i = tid + k * kNodeThreads;
#pragma unroll
      for (int d = 0; d < 3; ++d) lo[k][d] = hc[k][d] = 0xffffffffu;
      if (i < n) {
        const uint32_t e = (uint32_t)S.key[i] & 0xfffu;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const uint32_t x = orderable(S.pos[d][e]);
          lo[k][d] = x;
          hc[k][d] = ~x;
        }
      }
      const int width = cap < 32u ? (int)cap : 32;
      for (int o = width >> 1; o > 0; o >>= 1) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          lo[k][d] = min(lo[k][d], __shfl_xor_sync(0xffffffffu, lo[k][d], o));
          hc[k][d] = min(hc[k][d], __shfl_xor_sync(0xffffffffu, hc[k][d], o));
        }
      }
      if (cap >= 32u && lane == 0 && i < n) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          atomicMin(&S.box[seg[k].id][d], lo[k][d]);
          atomicMin(&S.box[seg[k].id][3 + d], hc[k][d]);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t i = tid + k * kNodeThreads;
      if (i >= n) continue;
      if (cap >= 32u) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          lo[k][d] = S.box[seg[k].id][d];
          hc[k][d] = S.box[seg[k].id][3 + d];
        }
      }
      const float ex = from_orderable(~hc[k][0]) - from_orderable(lo[k][0]);
      const float ey = from_orderable(~hc[k][1]) - from_orderable(lo[k][1]);
      const float ez = from_orderable(~hc[k][2]) - from_orderable(lo[k][2]);
      const int ax = (ex >= ey && ex >= ez) ? 0 : (ey >= ez ? 1 : 2);
      const uint32_t e = (uint32_t)S.key[i] & 0xfffu;
      S.key[i] = ((uint64_t)seg[k].id << 44) | ((uint64_t)orderable(S.pos[ax][e]) << 12) | e;
    }
    __syncthreads();
    const uint32_t top = small ? cap : np;
    for (uint32_t kk = 2; kk <= top; kk <<= 1) {
      for (uint32_t jj = kk >> 1; jj > 0; jj >>= 1) {
        for (uint32_t t = tid; t < np / 2; t += kNodeThreads) {
          const uint32_t i = 2u * t - (t & (jj - 1u)), m = i + jj;
          const bool up = kk == top || (i & kk) == 0u;
          const uint64_t x = S.key[i], y = S.key[m];
          if ((x > y) == up) {
            S.key[i] = y;
            S.key[m] = x;
          }
        }
        __syncthreads();
      }
    }
    const uint32_t leaf = l < levels2 ? (uint32_t)kTile2 : ((uint32_t)kTile >> (l - levels2));
#pragma unroll
    for (int k = 0; k < kPer; ++k) descend(seg[k], tid + k * kNodeThreads, leaf);
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const uint32_t i = tid + k * kNodeThreads;
    if (i < n) out[nd.start + i] = ord[nd.start + ((uint32_t)S.key[i] & 0xfffu)];
  }
}

// One CTA of T threads per tile: centre and tile-relative vectors, the discs
// of its groups.  The T = kTile2 build also writes the per-slot data shared by
// both tilings and the quarters' discs.  FP32 throughout: the unit vectors are
// double-float, and the centre may be any point near the targets.
template <int T>
__global__ void __launch_bounds__(T) k_tile_build(
    const double* __restrict__ lon, const double* __restrict__ lat, int64_t P,
    const uint32_t* __restrict__ order, const float4* __restrict__ u_hi,
    const float4* __restrict__ u_lo, float4* __restrict__ tile_chi,
    float4* __restrict__ tile_clo, float4* __restrict__ tgt_a, uint32_t* __restrict__ tgt_perm,
    float4* __restrict__ tgt_e, float4* __restrict__ tgt_n, double2* __restrict__ tgt_ll,
    float4* __restrict__ subf, float4* __restrict__ grp) {
  __shared__ float red[3][T / 32];
  const int64_t tile = blockIdx.x;
  const int j = threadIdx.x, lane = j & 31;
  const int64_t s = tile * T + j;
  const bool valid = s < P;
  float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
  uint32_t u = 0xffffffffu;
  if (valid) {
    u = order[s];
    h = u_hi[u];
    l = u_lo[u];
  }
  auto warp_sum = [](float v, int width) {
    for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  auto warp_max = [](float v, int width) {
    for (int o = width >> 1; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
  };
  {
    const float sx = warp_sum(h.x, 32), sy = warp_sum(h.y, 32), sz = warp_sum(h.z, 32);
    if (lane == 0) {
      red[0][j >> 5] = sx;
      red[1][j >> 5] = sy;
      red[2][j >> 5] = sz;
    }
  }
  __syncthreads();
  float cx = 0.f, cy = 0.f, cz = 0.f;
#pragma unroll
  for (int w = 0; w < T / 32; ++w) {
    cx += red[0][w];
    cy += red[1][w];
    cz += red[2][w];
  }
  const float nrm = sqrtf(cx * cx + cy * cy + cz * cz);
  if (nrm > 1e-3f) {
    cx /= nrm;
    cy /= nrm;
    cz /= nrm;
  } else {  // targets all over the sphere: the first member
    const float4 f = u_hi[order[tile * T]];
    cx = f.x;
    cy = f.y;
    cz = f.z;
  }
  const float dx = df_diff(h.x, l.x, cx, 0.f), dy = df_diff(h.y, l.y, cy, 0.f),
              dz = df_diff(h.z, l.z, cz, 0.f);
  // an empty slot sits far outside every support radius
  tgt_a[s] = valid ? make_float4(dx, dy, dz, 0.f) : make_float4(4.f, 4.f, 4.f, 0.f);
  if (tgt_perm) {
    tgt_perm[s] = u;
    const double lo = valid ? lon[u] : 0.0, la = valid ? lat[u] : 0.0;
    if (valid && valid_coord(lo, la)) {
      df32 sb, cb, sl, cl;
      sincos_deg(la, sb, cb);
      sincos_deg(lo, sl, cl);
      tgt_e[s] = make_float4(-sl.hi, cl.hi, 0.f, 0.f);
      tgt_n[s] = make_float4(-sb.hi * cl.hi, -sb.hi * sl.hi, cb.hi, 0.f);
      tgt_ll[s] = make_double2(lo, la);
    } else {
      tgt_e[s] = make_float4(0.f, 0.f, 0.f, 0.f);
      tgt_n[s] = make_float4(0.f, 0.f, 0.f, 0.f);
      tgt_ll[s] = make_double2(0.0, 0.0);
    }
  }
  if (subf) {
    // 32-target quarters: mean and largest distance, relative to the tile
    // centre (an empty quarter: the tile centre, radius 0)
    const float m = warp_sum(valid ? 1.f : 0.f, 32);
    const float inv = m > 0.f ? 1.f / m : 0.f;
    const float qx = warp_sum(valid ? dx : 0.f, 32) * inv, qy = warp_sum(valid ? dy : 0.f, 32) * inv,
                qz = warp_sum(valid ? dz : 0.f, 32) * inv;
    const float ex = dx - qx, ey = dy - qy, ez = dz - qz;
    const float r = warp_max(valid ? sqrtf(ex * ex + ey * ey + ez * ez) : 0.f, 32);
    if (lane == 0) subf[tile * (T / 32) + (j >> 5)] = make_float4(qx, qy, qz, r * (1.f + 1e-6f) + 1e-12f);
  }
  // 4-target groups (lanes 4 g .. 4 g + 3): the direction of their mean and
  // their largest angle from it, widened by the rounding; empty: radius -1
  const float m = warp_sum(valid ? 1.f : 0.f, 4);
  float gx = warp_sum(h.x, 4), gy = warp_sum(h.y, 4), gz = warp_sum(h.z, 4);
  const float gn = sqrtf(gx * gx + gy * gy + gz * gz);
  if (gn > 1e-3f) {
    gx /= gn;
    gy /= gn;
    gz /= gn;
  } else {  // degenerate spread: the tile centre (the radius still covers)
    gx = cx;
    gy = cy;
    gz = cz;
  }
  const float ex = h.x - gx, ey = h.y - gy, ez = h.z - gz;
  const float ch = warp_max(valid ? sqrtf(ex * ex + ey * ey + ez * ez) : 0.f, 4);
  if ((j & 3) == 0)
    grp[tile * (T / 4) + (j >> 2)] = make_float4(
        gx, gy, gz, m > 0.f ? 2.f * asinf(fminf(1.f, 0.5f * ch)) * (1.f + 1e-5f) + 1e-6f : -1.f);
  if (j == 0) {
    tile_chi[tile] = make_float4(cx, cy, cz, 0.f);
    tile_clo[tile] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

__global__ void k_set_axes(const float4* __restrict__ e, const float4* __restrict__ n,
                           float4* __restrict__ f1, float4* __restrict__ f2, int64_t slots,
                           float cpa, float spa) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= slots) return;
  const float4 E = e[i], N = n[i];
  // major axis at position angle PA from north through east
  f1[i] = make_float4(N.x * cpa + E.x * spa, N.y * cpa + E.y * spa, N.z * cpa + E.z * spa, 0.f);
  f2[i] = make_float4(E.x * cpa - N.x * spa, E.y * cpa - N.y * spa, E.z * cpa - N.z * spa, 0.f);
}

}  // namespace

static cudaError_t tiling_alloc(Tiling& t, int T, int64_t P, cudaStream_t s) {
  t.T = T;
  t.n_tiles = (P + T - 1) / T;
  cudaError_t e;
  if ((e = dalloc(&t.chi, (size_t)t.n_tiles, s)) != cudaSuccess) return e;
  if ((e = dalloc(&t.clo, (size_t)t.n_tiles, s)) != cudaSuccess) return e;
  if ((e = dalloc(&t.a, (size_t)(t.n_tiles * T), s)) != cudaSuccess) return e;
  if ((e = dalloc(&t.tile_cand, (size_t)t.n_tiles, s)) != cudaSuccess) return e;
  if ((e = dalloc(&t.grp, (size_t)(t.n_tiles * (T / 4)), s)) != cudaSuccess) return e;
  if (T == kTile2) {
    if ((e = dalloc(&t.subf, (size_t)(t.n_tiles * 4), s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t targets_build(cg_grid* g, const double* lon, const double* lat) {
  cudaStream_t s = g->stream;
  const int64_t P = g->P;
  cudaError_t e;
  if ((e = tiling_alloc(g->t64, kTile, P, s)) != cudaSuccess) return e;
  if ((e = tiling_alloc(g->t128, kTile2, P, s)) != cudaSuccess) return e;
  g->n_slots = g->t128.n_tiles * kTile2;
  const int64_t slots = g->n_slots;
  if ((e = dalloc(&g->tgt_perm, slots, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->tgt_e, slots, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->tgt_n, slots, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->tgt_f1, slots, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->tgt_f2, slots, s)) != cudaSuccess) return e;
  if ((e = dalloc(&g->tgt_ll, slots, s)) != cudaSuccess) return e;

  // levels to 128-target leaves; the first `top` of them over the whole array,
  // until a node has at most kNodeCap targets
  int levels2 = 0;
  const int top = kd_top_levels(g->t128.n_tiles, kTile2, kNodeCap);
  while (((int64_t)1 << levels2) < g->t128.n_tiles) ++levels2;
  float4 *u_hi = nullptr, *u_lo = nullptr;
  uint32_t *ord = nullptr, *key = nullptr, *val = nullptr, *box = nullptr;
  SortWork w;
  w.err = g->d_err;
  e = dalloc(&u_hi, (size_t)P, s);
  if (e == cudaSuccess) e = dalloc(&u_lo, (size_t)P, s);
  if (e == cudaSuccess) e = dalloc(&ord, (size_t)P, s);
  if (e == cudaSuccess) e = dalloc(&val, (size_t)P, s);
  if (e == cudaSuccess && top > 0) e = dalloc(&key, (size_t)P, s);
  if (e == cudaSuccess && top > 0) e = dalloc(&box, (size_t)12 << (top - 1), s);
  const unsigned nb = ceil_div(P, 256);
  if (e == cudaSuccess) {
    k_target_init<<<nb, 256, 0, s>>>(lon, lat, P, u_hi, u_lo, ord, g->d_err);
    g->n_launches += 1;
  }
  uint32_t* cur = ord;   // the targets in the order reached so far
  for (int l = 0; l < top && e == cudaSuccess; ++l) {
    e = cudaMemsetAsync(box, 0xff, sizeof(uint32_t) * ((size_t)12 << l), s);
    if (e != cudaSuccess) break;
    k_kd_box<<<ceil_div(P, 2048), 256, 0, s>>>(u_hi, cur, (uint32_t)P, l, box);
    k_kd_keys<<<nb, 256, 0, s>>>(u_hi, cur, (uint32_t)P, l, box, key, val);
    uint32_t* sk = nullptr;
    const int bits = kd_coord_bits(l) + l;
    e = radix_sort_u32(key, val, P, bits, w, s, &sk, &cur);
    g->n_launches += 2 + radix_sort_u32_launches(P, bits);
  }
  if (e == cudaSuccess) {
    // (`ord` is free unless nothing has been sorted: then val takes the result)
    uint32_t* fin = cur == ord ? val : ord;
    e = cudaFuncSetAttribute(k_kd_node, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(NodeSmem));
    if (e == cudaSuccess) {
      k_kd_node<<<1u << top, kNodeThreads, sizeof(NodeSmem), s>>>(u_hi, cur, (uint32_t)P, top,
                                                                  levels2, fin);
      k_tile_build<kTile2><<<(unsigned)g->t128.n_tiles, kTile2, 0, s>>>(
          lon, lat, P, fin, u_hi, u_lo, g->t128.chi, g->t128.clo, g->t128.a, g->tgt_perm,
          g->tgt_e, g->tgt_n, g->tgt_ll, g->t128.subf, g->t128.grp);
      k_tile_build<kTile><<<(unsigned)g->t64.n_tiles, kTile, 0, s>>>(
          lon, lat, P, fin, u_hi, u_lo, g->t64.chi, g->t64.clo, g->t64.a, nullptr, nullptr,
          nullptr, nullptr, nullptr, g->t64.grp);
      g->n_launches += 3;
      e = cudaGetLastError();
    }
  }
  if (w.keys_alt) cudaFreeAsync(w.keys_alt, s);
  dfree(w.vals_alt, s);
  dfree(w.hist, s);
  dfree(w.totals, s);
  dfree(w.status, s);
  dfree(w.os_meta, s);
  dfree(u_hi, s);
  dfree(u_lo, s);
  dfree(ord, s);
  dfree(val, s);
  dfree(key, s);
  dfree(box, s);
  return e;
}

cudaError_t targets_set_axes(cg_grid* g, double pa_deg) {
  const int64_t slots = g->n_slots;
  const double pa = pa_deg * kDeg2Rad;
  k_set_axes<<<ceil_div(slots, 256), 256, 0, g->stream>>>(g->tgt_e, g->tgt_n, g->tgt_f1,
                                                          g->tgt_f2, slots, (float)cos(pa),
                                                          (float)sin(pa));
  return cudaGetLastError();
}

}  // namespace cg
