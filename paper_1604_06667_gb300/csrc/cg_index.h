// cg_index.h -- index arithmetic of the kernels that a host compiler can check
// as well (plain C++; under nvcc the functions serve both sides).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define CG_HD __host__ __device__ __forceinline__
#else
#define CG_HD inline
#endif

namespace cg {

constexpr uint32_t kEmptySlot = 0xffffffffu;   // tgt_perm of a slot without a target

// Shares that a tile of `total` candidates is worked on in, of at most n_split
// (the wide FP32 form; shares of fewer than eight stages cost more than they
// give).
CG_HD int wide_shares(int total, int n_split) {
  const int s = total / 256;
  return s < 1 ? 1 : (s < n_split ? s : n_split);
}

// Chunks of kc candidates between two folds of the wide form's sums: a tile's
// `total` candidates in up to n_fold parts, of at least two chunks each (one part:
// never).
CG_HD int wide_fold_chunks(int total, int n_fold, int kc) {
  const int chunks = total / kc + (total % kc ? 1 : 0);
  const int parts = chunks / 2 < n_fold ? chunks / 2 : n_fold;
  return parts < 2 ? 1 << 30 : (chunks + parts - 1) / parts;
}

// Partial sums of a slot: the shares of its tile, 0 for an empty slot.  Slots
// come in whole 128-target tiles, candidate counts in 64-target tiles that hold
// at least one target, so an empty slot's tile may lie past the last count: it
// is not looked up.  tile_cand null: every tile has n_split shares.
template <class Perm, class Cand>
CG_HD int slot_shares(Perm perm, Cand tile_cand, int64_t slot, int tile, int n_split) {
  if (perm[slot] == kEmptySlot) return 0;
  return tile_cand ? wide_shares(tile_cand[slot / tile], n_split) : n_split;
}

// Targets' k-d tree: levels of nodes that are sorted over the whole array, until
// a node of the `n_tiles` tiles of `tile` targets holds at most `cap` targets.
CG_HD int kd_top_levels(int64_t n_tiles, int tile, int cap) {
  int top = 0;
  while (((n_tiles + ((int64_t)1 << top) - 1) >> top) * tile > cap) ++top;
  return top;
}

// Such a level's 32-bit sort key: the node's number (`level` bits) above the
// coordinate, which gives way from level 17 on (more than 2^29 targets).
CG_HD int kd_coord_bits(int level) { return level > 16 ? 32 - level : 16; }
CG_HD uint32_t kd_key(uint32_t node, int level, float t) {   // t: 0 .. 1 across the node
  const int bits = kd_coord_bits(level);
  const uint32_t most = (1u << bits) - 1u, q = (uint32_t)(t * (float)most);
  return (node << bits) | (q < most ? q : most);
}

}  // namespace cg
