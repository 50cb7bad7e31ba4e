// Pieces of the population search (Sec. 4.3) that the one-launch round and the dense operators share: draws of the
// counter-based stream and the repair's decision for a node.
#pragma once

#include <algorithm>
#include <cmath>

#include "common.cuh"

static __device__ __noinline__ u32x4 draw_one(uint32_t k0, uint32_t k1, uint32_t idx, uint32_t cand, uint32_t gen, uint32_t slot) {
  const u32x4 c = {idx, cand, gen, slot};
  return philox4x32_10(c, k0, k1);
}

// Two calls that differ only in their slot (the last counter word), side by side: of the first call word
// x, of the second all.  What does not see the slot is worked out once - the first round, the first product
// of the second, the second product of the third - and of the first call's last two rounds only what its
// word x needs.
static __device__ __noinline__ void draw_two(uint32_t k0, uint32_t k1, uint32_t idx, uint32_t cand, uint32_t gen, uint32_t slot_a,
                                      uint32_t slot_b, uint32_t &a_x, u32x4 &b) {
  constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#define HI(m, v) __umulhi((m), (v))
#define LO(m, v) ((m) * (v))
  u32x4 ca, cb, na, nb;
  {
    const uint32_t x = HI(M1, gen) ^ cand ^ k0, y = LO(M1, gen), w = LO(M0, idx), h0 = HI(M0, idx);
    const uint32_t za = h0 ^ slot_a ^ k1, zb = h0 ^ slot_b ^ k1;
    k0 += W0; k1 += W1;
    ca.x = HI(M1, za) ^ y ^ k0; ca.y = LO(M1, za);
    cb.x = HI(M1, zb) ^ y ^ k0; cb.y = LO(M1, zb);
    ca.z = HI(M0, x) ^ w ^ k1; ca.w = LO(M0, x);
    k0 += W0; k1 += W1;
    const uint32_t h1 = HI(M1, ca.z), l1 = LO(M1, ca.z);
    na.x = h1 ^ ca.y ^ k0; na.y = l1; na.z = HI(M0, ca.x) ^ ca.w ^ k1; na.w = LO(M0, ca.x);
    nb.x = h1 ^ cb.y ^ k0; nb.y = l1; nb.z = HI(M0, cb.x) ^ ca.w ^ k1; nb.w = LO(M0, cb.x);
    ca = na; cb = nb;
    k0 += W0; k1 += W1;
  }
#pragma unroll
  for (int r = 3; r < 8; ++r) {
    na.x = HI(M1, ca.z) ^ ca.y ^ k0; na.y = LO(M1, ca.z); na.z = HI(M0, ca.x) ^ ca.w ^ k1; na.w = LO(M0, ca.x);
    nb.x = HI(M1, cb.z) ^ cb.y ^ k0; nb.y = LO(M1, cb.z); nb.z = HI(M0, cb.x) ^ cb.w ^ k1; nb.w = LO(M0, cb.x);
    ca = na; cb = nb;
    k0 += W0; k1 += W1;
  }
  // ninth round: of the first call y and z
  na.y = LO(M1, ca.z); na.z = HI(M0, ca.x) ^ ca.w ^ k1;
  nb.x = HI(M1, cb.z) ^ cb.y ^ k0; nb.y = LO(M1, cb.z); nb.z = HI(M0, cb.x) ^ cb.w ^ k1; nb.w = LO(M0, cb.x);
  k0 += W0; k1 += W1;
  a_x = HI(M1, na.z) ^ na.y ^ k0;
  b.x = HI(M1, nb.z) ^ nb.y ^ k0; b.y = LO(M1, nb.z); b.z = HI(M0, nb.x) ^ nb.w ^ k1; b.w = LO(M0, nb.x);
#undef HI
#undef LO
}

// What the repair decides for the occupant in this lane of a group of 16 (`have`: there is one; v: its GPUs on the
// node, 0 without; distributed: its row spans two nodes or more): the GPUs it keeps there.  rot_i, rot_c: the
// row's place in the node's two rotated job orders (below 65536; GPUs below 2048).  Called by whole warps, two nodes at a time (shuffles under the full mask; a group
// without a node has no occupants).
__device__ __forceinline__ int decide(int v, bool distributed, bool have, int most, bool intf, int tot, int cap_n, int rot_i, int rot_c) {
  const bool dist = have && intf && distributed;
  int removed = 0;
  if (__any_sync(0xffffffffu, intf)) {   // of the distributed ones only the first in rotated order stays
    int first = dist ? (rot_i << 11) | v : 0x7fffffff, all = dist ? v : 0;
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
      first = min(first, __shfl_xor_sync(0xffffffffu, first, off));
      all += __shfl_xor_sync(0xffffffffu, all, off);
    }
    if (intf) removed = all - (first & 0x7FF);
    if (dist && (first >> 11) != rot_i) v = 0;
  }
  const int excess = tot - removed - cap_n;
  int ahead = 0;                         // GPUs of the occupants that come first in rotated order
  if (__any_sync(0xffffffffu, excess > 0)) {
    const int mine = have ? (rot_c << 11) | v : 0x7fffffff;
#pragma unroll 1
    for (int k = 0; k < most; k += 4) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int other = __shfl_sync(0xffffffffu, mine, k + q, 16);
        if ((other >> 11) < rot_c && other != 0x7fffffff) ahead += other & 0x7FF;
      }
    }
  }
  if (have && excess > 0) v -= min(v, max(excess - ahead, 0));
  return v;
}

// What the repair decides for a node with more occupants than decide() takes, by a warp, from their list (bit 31 of an
// entry: distributed): of the distributed ones the first in rotated order stays; of the GPUs then left, the last that
// the node has room for stay, in the other rotated order.
struct CrowdPlaces {
  int first;                             // place of the distributed occupant that stays, -1: all do
  int upto, stay;                        // all before the place `upto` leave; of the occupant there `stay` GPUs stay
  __device__ __forceinline__ int keeps(uint32_t e, int gpus, int place_i, int place_c) const {
    if (first >= 0 && (e >> 31) && place_i != first) return 0;
    return place_c < upto ? 0 : place_c == upto ? min(gpus, stay) : gpus;
  }
};

// `upto` is found bit by bit, a pass over the list each, so the work grows with the list and not with its square.
// list(k): its k-th entry; gpus(e), rot_i(e), rot_c(e): an entry's GPUs (below 2048) and its places (below 65536, J of them).
template <class List, class Gpus, class RotI, class RotC>
__device__ __forceinline__ CrowdPlaces crowd_places(List list, int count, int J, int tot, bool intf, int cap_n, int lane, Gpus gpus,
                                                    RotI rot_i, RotC rot_c) {
  CrowdPlaces at = {-1, -1, 0};
  const bool one = count <= 32;          // an entry a lane, looked at once
  const uint32_t e0 = lane < count ? list(lane) : 0u;
  const int g0 = lane < count ? gpus(e0) : 0;
  if (intf) {
    int first = 0x7fffffff, all = 0;
#pragma unroll 1
    for (int k = lane; k < count; k += 32) {
      const uint32_t e = one ? e0 : list(k);
      if (!(e >> 31)) continue;
      first = min(first, (rot_i(e) << 11) | gpus(e));
      all += gpus(e);
    }
    first = __reduce_min_sync(0xffffffffu, first);
    tot -= __reduce_add_sync(0xffffffffu, all) - (first & 0x7FF);
    at.first = first >> 11;
  }
  if (tot <= cap_n) return at;
  const int v0 = at.keeps(e0, g0, rot_i(e0), 0), place0 = rot_c(e0);
  auto from = [&](int place) {           // GPUs from there on
    int sum = place0 >= place ? v0 : 0;
    if (!one)
#pragma unroll 1
      for (int k = lane + 32; k < count; k += 32) {
        const uint32_t e = list(k);
        if (rot_c(e) >= place) sum += at.keeps(e, gpus(e), rot_i(e), 0);
      }
    return __reduce_add_sync(0xffffffffu, sum);
  };
  int upto = 0;
#pragma unroll 1
  for (int bit = 1 << (31 - __clz(J)); bit; bit >>= 1)
    if (from(upto | bit) > cap_n) upto |= bit;
  const int stay = cap_n - from(upto + 1);
  at.upto = upto;
  at.stay = stay;
  return at;
}

// How many occupants a node's list should hold, in steps of 16 (what decide() takes) up to `most`: jobs of two GPUs on a
// full node, what a step brings on average (two of three perturbed rows take a node), and four standard deviations.
inline int listed_occupants(const sched_ctx *ctx, uint32_t thr, int most) {
  const double full = std::min(ctx->cap_max, 2 * ctx->cfg.num_jobs) / 2.0;
  const double mean = ctx->cfg.num_jobs * (thr / 4294967296.0) * (2.0 / 3.0) / ctx->cfg.num_nodes;
  const double want = std::min(full + mean + 4.0 * std::sqrt(full / 2.0 + mean), 1e6);
  return std::max(16, std::min(((int)want + 15) & ~15, most & ~15));
}
