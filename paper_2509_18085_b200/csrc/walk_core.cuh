// Step 5 of Algorithm 1 for one sequence.  The walk starts at the true block
// (node 0) and moves to the first node (ascending index) that lists the current
// one as a parent and whose state equals the current node's next state; it stops
// when there is none, or at a node with nothing left to unmask.
//
// A few nodes' children are found by a table (below), the others as follows.
// Whether node m follows node p depends on p and m alone, not on the path, so
// the links are found for all (parent, child) entries at once -- one warp per
// child, lane k owning block positions k and k + 32 -- and the walk itself is a
// chase through at most N-1 links.  The graph arrays may live in shared or
// global memory; `link` is N ints of shared memory.
#pragma once
#include "common.cuh"

namespace spiffy {

constexpr int kNoLink = 0x7fffffff;
constexpr int kTableNodes = 64;  // graphs up to here have their children in a table: what lists a node as a parent, a bit each

// A state, positions `lane` and `lane` + 32 (zeros beyond L): its still-masked positions, and a number that
// equal states share (multipliers: the golden ratio's, and the two of MurmurHash3's 32-bit finaliser, which is in the
// public domain; states of equal numbers are compared token by token, so that nothing rests on them).
__device__ __forceinline__ uint64_t masked_of(const int32_t (&state)[2], int L, int mask_id, int lane) {
  uint64_t masked = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h)
    masked |= (uint64_t)__ballot_sync(0xffffffffu, lane + 32 * h < L && state[h] == mask_id) << (32 * h);
  return masked;
}
__device__ __forceinline__ uint32_t hash_of(const int32_t (&state)[2], int lane) {
  const uint32_t a = ((uint32_t)state[0] + 0x9e3779b9u * (uint32_t)lane) * 0x85ebca6bu;
  const uint32_t b = ((uint32_t)state[1] + 0x9e3779b9u * (uint32_t)(lane + 32)) * 0xc2b2ae35u;
  return __reduce_xor_sync(0xffffffffu, (a ^ (a >> 15)) + (b ^ (b >> 13)));
}

// One warp enters node m's parents into the table (all zero beforehand).  False on a lane that met a malformed
// offset or entry, which is ignored.
__device__ __forceinline__ bool enter_parents(uint32_t (*kids)[2], const int32_t* off, const int32_t* idx, int parent_cap,
                                              int m, int lane) {
  const int e0 = off[m], e1 = off[m + 1];
  if (e0 < 0 || e1 < e0 || e1 > parent_cap) return false;
  bool good = true;
  for (int e = e0 + lane; e < e1; e += 32) {
    const int q = idx[e];
    if (q < 0 || q >= m) good = false;
    else atomicOr(&kids[q][m >> 5], 1u << (m & 31));
  }
  return good;
}

// The first of the nodes in `kids` (a bit each) whose state is `next`, kNoLink if there is none; by one warp.
__device__ __forceinline__ int child_of(const uint32_t (&kids)[2], const uint32_t* hashes, const int32_t* states,
                                        const int32_t (&next)[2], int N, int L, int lane) {
  const uint32_t hash = hash_of(next, lane);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int m0 = 32 * h;
    if (m0 >= N) break;
    unsigned like = __ballot_sync(0xffffffffu, m0 + lane < N && hashes[min(m0 + lane, N - 1)] == hash) & kids[h];
    for (; like; like &= like - 1) {
      const int m = m0 + __ffs(like) - 1;
      const int32_t* sm = states + m * L;
      if (__all_sync(0xffffffffu, (lane >= L || sm[lane] == next[0]) && (lane + 32 >= L || sm[lane + 32] == next[1])))
        return m;
    }
  }
  return kNoLink;
}

__device__ __forceinline__ int32_t walk_next_token(const int32_t* state, const int32_t* top,
                                                   uint64_t bits, int node, int L, int l) {
  return ((bits >> l) & 1ull) ? top[node * L + l] : state[node * L + l];
}

// Called by `n_warps` warps together (warp index `warp`); `link` must hold
// kNoLink everywhere beforehand and is complete after the next block-wide sync.
// Returns true on every lane of a warp that met a malformed offset or entry
// (such entries are ignored).
__device__ __forceinline__ bool walk_link_children(int N, int L, int parent_cap,
                                                   const int32_t* state, const int32_t* top,
                                                   const int32_t* off, const int32_t* idx,
                                                   const uint64_t* ubits, int* link, int warp,
                                                   int n_warps, int lane) {
  const unsigned full = 0xffffffffu;
  const int l0 = lane, l1 = lane + 32;
  bool bad = false;
  for (int m = 1 + warp; m < N; m += n_warps) {
    const int e0 = off[m], e1 = off[m + 1];
    if (e0 < 0 || e1 < e0 || e1 > parent_cap) {  // malformed offsets
      bad = true;
      continue;
    }
    const int32_t s0 = l0 < L ? state[m * L + l0] : 0;
    const int32_t s1 = l1 < L ? state[m * L + l1] : 0;
    for (int e = e0; e < e1; ++e) {
      const int p = idx[e];
      if (p < 0 || p >= m) {  // ignored entry
        bad = true;
        continue;
      }
      const uint64_t bits = ubits[p];
      if (bits == 0) continue;  // a node with nothing to unmask ends the walk
      bool eq = true;
      if (l0 < L) eq &= s0 == walk_next_token(state, top, bits, p, L, l0);
      if (l1 < L) eq &= s1 == walk_next_token(state, top, bits, p, L, l1);
      if (__all_sync(full, eq) && lane == 0) atomicMin(link + p, m);
    }
  }
  return __any_sync(full, bad);
}

// Called by one warp after the links are complete (a block-wide sync after walk_link_children): the
// node the walk ends on, the hops to it in `hops`, and the path, hops + 1 entries, in `pth`.
__device__ __forceinline__ int walk_follow(int N, const int* link, int32_t* pth, int lane, int& hops) {
  int cur = 0;
  hops = 0;
  if (lane == 0) {
    // `link` may be the path array itself: a link is read before the slot at or
    // below its node is reused for the path (hop h is stored at index h <= node)
    int m = link[0];
    pth[0] = 0;
    while (hops < N - 1 && m != kNoLink) {
      cur = m;  // accepted: its distribution replaces the target's
      m = link[cur];
      pth[++hops] = cur;
    }
  }
  hops = __shfl_sync(0xffffffffu, hops, 0);
  return __shfl_sync(0xffffffffu, cur, 0);
}

// ... and what it says about the node `cur` it ends on.
__device__ __forceinline__ void walk_end(int cur, int hops, int L, const int32_t* state, const int32_t* top,
                                         const uint64_t* ubits, int32_t* next_block, int32_t* accepted_node,
                                         int32_t* n_accepted, int lane) {
  if (lane == 0) {
    *accepted_node = cur;
    *n_accepted = hops;
  }
  const uint64_t bits = ubits[cur];
  if (lane < L) next_block[lane] = walk_next_token(state, top, bits, cur, L, lane);
  if (lane + 32 < L) next_block[lane + 32] = walk_next_token(state, top, bits, cur, L, lane + 32);
}

__device__ __forceinline__ void walk_chase(int N, int L, const int32_t* state, const int32_t* top,
                                           const uint64_t* ubits, const int* link, int32_t* pth,
                                           int32_t* next_block, int32_t* accepted_node,
                                           int32_t* n_accepted, int lane) {
  int hops;
  const int cur = walk_follow(N, link, pth, lane, hops);
  for (int i = hops + 1 + lane; i < N; i += 32) pth[i] = -1;
  walk_end(cur, hops, L, state, top, ubits, next_block, accepted_node, n_accepted, lane);
}

}  // namespace spiffy
