// Radix sort of up to half a million keys inside one cooperative launch: device
// functions shared by the engine's sort (sort.cu) and the allocation-free
// deduplication (noalloc.cu).
//
// Up to that size a pass of the general radix sort is five launches of a few
// microseconds each, whose work fits a few microseconds together: 100,003 keys of
// 64 bits took 205 us in 40 launches.  Here a block keeps a tile of eight keys a
// thread in registers through a pass, the tiles' digit counts go through global
// memory, and grid barriers separate counting from scattering and one pass from
// the next.  A pass whose keys all share the digit is seen in the counts and
// skipped, with no second barrier.  One tile needs no barrier and no global traffic
// between passes: the reordered tile is read back from shared memory.  A block adds
// up the counts of all tiles itself, so the grid stays at 64 tiles; the fewer
// threads a tile has, the shorter its ranking and warp sums, so tiles are as small
// as 64 of them allow.
#pragma once
#include <type_traits>

#include "common.cuh"

struct NoPay {};

constexpr int kFItems = 8;    // keys per thread
constexpr int kFTiles = 64;   // blocks of a launch at most
constexpr u32 kFSpin = 1u << 26;  // barrier polls before a block gives up
// fused scratch, in u32 words: a head (barrier arrivals, give-up flag, blocks that
// left, padding), zero when a launch of several blocks starts, and the tiles' digit
// counts, two passes' worth (a block may still add up one pass's when another counts
// the next)
constexpr u32 kFHead = 16;
LOB_HD constexpr u64 fused_count_words(u64 tiles) { return 2 * 256 * tiles; }
LOB_HD u64 fused_scratch_words(u64 tiles) { return kFHead + fused_count_words(tiles); }

// Lanes of this warp holding the same RB-bit digit (and a valid key): the
// intersection over the digit's bits of the ballot of lanes agreeing on that bit.
template <int RB>
LOB_DEV u32 same_digit_lanes(u32 d, bool valid) {
  u32 m = __ballot_sync(0xFFFFFFFFu, valid);
#pragma unroll
  for (int b = 0; b < RB; b++) {
    const bool bit = (d >> b) & 1u;
    const u32 v = __ballot_sync(0xFFFFFFFFu, bit);
    m &= bit ? v : ~v;
  }
  return m;
}

// every block of the launch, or false when one of them gave up waiting
LOB_DEV bool fused_barrier(u32* bar, u32& gen) {
  __shared__ u32 ok;
  __syncthreads();
  if (gridDim.x == 1) return true;
  if (threadIdx.x == 0) {
    volatile u32* b = bar;
    __threadfence();
    gen++;
    atomicAdd(bar, 1u);
    const u32 want = gen * gridDim.x;
    u32 n = 0;
    while (b[0] < want && !b[1] && n < kFSpin) n++;
    if (b[0] < want) b[1] = 1;
    __threadfence();
    ok = b[1] == 0;
  }
  __syncthreads();
  return ok != 0;
}

template <class K, class P, int NT>
struct FusedSmem {
  static constexpr int kTile = NT * kFItems, kWarps = NT / 32;
  K keys[kTile];
  P pay[std::is_same<P, NoPay>::value ? 1 : kTile];
  u32 wh[kWarps][256];  // per warp: digit counts, then the warp's first rank of the digit
  u32 dstart[256], gbase[256];
  u32 sm[kWarps + 1];
  u32 all_same;
};

// A tile of the keys being sorted: thread t's keys are at offsets wofs + r * 32 + lane.
template <class K, class P, int NT>
struct FusedTile {
  static constexpr bool kPay = !std::is_same<P, NoPay>::value;
  K k[kFItems];
  P p[kFItems];
  K *src_k, *dst_k;  // the order so far (global), and the other buffer
  P *src_p, *dst_p;
  u64 tbase;
  int tile_n, wofs;

  LOB_DEV bool valid(int r) const { return wofs + r * 32 + (int)(threadIdx.x & 31) < tile_n; }
  LOB_DEV u64 at(int r) const { return tbase + wofs + r * 32 + (threadIdx.x & 31); }
  LOB_DEV void place(u64 n) {
    tbase = (u64)blockIdx.x * (NT * kFItems);
    tile_n = (int)min((u64)(NT * kFItems), n - tbase);
    wofs = (int)(threadIdx.x >> 5) * 32 * kFItems;
  }
  // stores came from other blocks: read past L1
  LOB_DEV void reload() {
#pragma unroll
    for (int r = 0; r < kFItems; r++)
      if (valid(r)) {
        k[r] = __ldcg(src_k + at(r));
        if constexpr (kPay) p[r] = __ldcg(src_p + at(r));
      }
  }
};

// Sorts by the low `bits` bits; afterwards every block's tile is in registers, and
// (unless the launch has one tile) in src_k / src_p.  False when a barrier gave up.
template <class K, class P, int NT>
LOB_DEV bool fused_passes(FusedTile<K, P, NT>& T, FusedSmem<K, P, NT>& S, u64 n, int bits, u32* head, u32* counts,
                          u32& gen) {
  constexpr bool kPay = FusedTile<K, P, NT>::kPay;
  constexpr int kWarps = NT / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u32 lt_mask = (1u << lane) - 1u;
  const u32 tiles = gridDim.x;
  int pass = 0;
  for (int shift = 0; shift < bits; shift += 8, pass++) {
    for (int i = threadIdx.x; i < kWarps * 256; i += NT) (&S.wh[0][0])[i] = 0;
    if (threadIdx.x == 0) S.all_same = 0;
    __syncthreads();
    u32 rank[kFItems];
#pragma unroll
    for (int r = 0; r < kFItems; r++) {
      const bool v = T.valid(r);
      const u32 d = v ? (u32)((T.k[r] >> shift) & (K)255) : 0u;
      const u32 peers = same_digit_lanes<8>(d, v);
      u32 base = 0;
      if (v) base = S.wh[warp][d];
      rank[r] = base + __popc(peers & lt_mask);
      __syncwarp();
      if (v && (__ffs(peers) - 1) == lane) S.wh[warp][d] = base + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    u32 mine = 0;  // this tile's keys of digit threadIdx.x
    if (threadIdx.x < 256) {
#pragma unroll
      for (int w = 0; w < kWarps; w++) {
        const u32 c = S.wh[w][threadIdx.x];
        S.wh[w][threadIdx.x] = mine;
        mine += c;
      }
    }
    u32 before = 0, total = mine;  // of the tiles before this one, of all tiles
    if (tiles > 1) {
      u32* cnt = counts + (u64)(pass & 1) * 256 * tiles;
      if (threadIdx.x < 256) cnt[blockIdx.x * 256 + threadIdx.x] = mine;
      if (!fused_barrier(head, gen)) return false;
      if (threadIdx.x < 256) {
        total = 0;
#pragma unroll 16
        for (u32 b = 0; b < tiles; b++) {
          const u32 c = __ldcg(cnt + b * 256 + threadIdx.x);
          if (b < blockIdx.x) before += c;
          total += c;
        }
      }
    }
    if (threadIdx.x < 256 && (u64)total == n) S.all_same = 1;
    // both digit scans at once: this tile's counts and the whole input's
    u64 sum;
    __shared__ u64 sm64[kWarps + 1];
    const u64 ex = block_exclusive_sum<u64>(threadIdx.x < 256 ? ((u64)total << 32) | mine : 0ull, sm64, &sum);
    if (threadIdx.x < 256) {
      S.dstart[threadIdx.x] = (u32)ex;
      S.gbase[threadIdx.x] = (u32)(ex >> 32) + before;
    }
    __syncthreads();
    if (S.all_same) {  // every key has this digit: the order stands
      __syncthreads();
      continue;
    }
#pragma unroll
    for (int r = 0; r < kFItems; r++) {
      if (T.valid(r)) {
        const u32 d = (u32)((T.k[r] >> shift) & (K)255);
        const u32 lp = S.dstart[d] + S.wh[warp][d] + rank[r];
        S.keys[lp] = T.k[r];
        if constexpr (kPay) S.pay[lp] = T.p[r];
      }
    }
    __syncthreads();
    if (tiles == 1) {
#pragma unroll
      for (int r = 0; r < kFItems; r++)
        if (T.valid(r)) {
          T.k[r] = S.keys[T.wofs + r * 32 + lane];
          if constexpr (kPay) T.p[r] = S.pay[T.wofs + r * 32 + lane];
        }
      __syncthreads();
      continue;
    }
    for (int i = threadIdx.x; i < T.tile_n; i += NT) {
      const K key = S.keys[i];
      const u32 d = (u32)((key >> shift) & (K)255);
      const u64 pos = (u64)S.gbase[d] + (u32)(i - (int)S.dstart[d]);
      T.dst_k[pos] = key;
      if constexpr (kPay) T.dst_p[pos] = S.pay[i];
    }
    { K* t = T.src_k; T.src_k = T.dst_k; T.dst_k = t; }
    { P* t = T.src_p; T.src_p = T.dst_p; T.dst_p = t; }
    if (!fused_barrier(head, gen)) return false;
    T.reload();
  }
  return true;
}
