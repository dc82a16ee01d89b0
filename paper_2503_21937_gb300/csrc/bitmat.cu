// Bit-matrix fixpoint of chain programs (unit semiring).
//
// A chain program is one whose derived relations are binary and whose rules
// link their body atoms into a path from one head variable to the other --
//   path(x,z) :- path(x,y), edge(y,z).
//   sg(x,y)   :- parent(a,x), sg(a,b), parent(b,y).
//   pt(r,o)   :- store(p,q), pt(p,r), pt(q,o).
// Each rule is then a product of boolean matrices, an atom read against its
// column order being the transpose.  A derived relation is kept as a bit matrix
// over the values that occur in the program's relations (renumbered in order, so
// that row-major bit order is the relation's key order) and an input relation as
// compressed rows.  Rows of a bit matrix are combined 128 bits a lane, so one
// instruction derives up to 4,096 candidates of a warp; the general path spends
// an atomic (or a sort of 8 bytes) on each.  Algorithm 1 is unchanged: an
// iteration evaluates every semi-naive arm on the facts the previous one left
// (recent set D, full set F), and D' = N & ~F, F |= D' ends it.
//
// What bounds it: reading the operand rows, out of L2 (the matrices of the
// benchmark's closure are 50 MB each), then the read-out of the result.
//
// Products are evaluated from the right: U = M_m, U = M_i U for i = m-1 .. 1.
//   gather   M_i x bits: row r = OR of the rows of U listed in row r of M_i
//   scatter  M_i x compressed rows: row r is built in shared memory, one
//            shared atomic OR per derivation
// The derived relations are stored transposed when that turns scatters into
// gathers (bit_eligible's rule): a left-recursive closure reads as E' P'.
//
// Measured (GB300, fixpoint only, general path before -> bit matrices): closure
// of the 20,000-node / 100,000-edge power-law graph 11.9 -> 1.5 ms; same
// generation on a 50,000-node tree 22.6 -> 6.1 ms; points-to on 400,000
// statements (8.7e9 derivations of 1.8e6 facts, 36-bit keys: sorted before)
// 418 -> 2.4 ms; closure of 1,000 nodes / 3,000 edges 0.99 -> 0.27 ms.
#include "bitmat.h"

#include <algorithm>
#include <cstring>
#include <numeric>

#include "engine.h"
#include "scan.cuh"

namespace {

constexpr int kMaxChain = 4;       // body atoms of a chain rule
constexpr int kMaxBitRels = 16;    // relations the state block holds sizes of
constexpr u32 kHeavyRow = 512;     // compressed rows longer than this are gathered by a whole block
constexpr u64 kMatrixBytes = 1ull << 30;  // largest bit matrix (92,000 values)
constexpr u64 kRunBytes = 8ull << 30;     // all matrices of a run: two to six a derived relation, two temporaries
constexpr u64 kMaxValue = 1ull << 28;     // largest id the renumbering's presence bitmap covers

// state block: done flag (1 fixpoint, 2 max_iters), iterations run, new facts
// of all iterations, derivations, words read (profiling), then per relation
// |F|, |D| and this iteration's new facts
enum : int { B_DONE = 0, B_ITER, B_NEW, B_CAND, B_WORDS, B_REL = 8 };
LOB_HD int rel_slot(int r, int f) { return B_REL + 3 * r + f; }
constexpr int kStateSlots = B_REL + 3 * kMaxBitRels;
// ... and, not read back, three list lengths for each of an iteration's products
constexpr int kMaxLists = 32;
constexpr int kAllSlots = kStateSlots + 3 * kMaxLists;
// (the loop in one launch uses the first of those as its barrier words)
constexpr int kReadSlots = kStateSlots + 1;

// set bits a warp of a scatter lists before it sets their columns (at least the
// 1,024 of one batch of words)
constexpr int kBitList = 1024;
// k_bit_gather_wide: chunks of a task, and the most entries of a row it takes (the
// rows of 512 entries that the other form takes would keep one warp for four
// chunks: closure of the power-law graph 0.86 -> 1.48 ms)
constexpr int kWide = 4;
constexpr u32 kWideRow = 8;

enum IndexKind { I_IDENT = 0, I_CSR = 1, I_BITS = 2 };

// A bit matrix.  Row r is empty, whatever its words hold, when cnt[r] (bag[r]
// when bag is set) is 0.  bag[r]: the derivations row r stands for, duplicates
// included (a stored relation's is its facts, cnt).
// What a run's iterations write, read by a launch that spans several of them
// (kLoop): past L1, which keeps lines of earlier iterations.
template <bool kLoop, class T> LOB_DEV T ldm(const T* p) {
  if constexpr (kLoop) return __ldcg(p);
  else return *p;
}
struct BMat {
  const u32* bits;
  const u32* cnt;
  const u64* bag;
  template <bool kLoop> LOB_DEV u64 weight(u32 r) const { return bag ? ldm<kLoop>(bag + r) : (u64)ldm<kLoop>(cnt + r); }
};
struct BCsr {
  const u32* ptr;
  const u32* col;
  const u32* heavy;    // rows longer than kHeavyRow
  const u32* n_heavy;
};

struct BOp {
  u32 rows, words;     // rows, words per row (a multiple of 4)
  BCsr ic;             // index matrix M_i
  BMat ib;
  BCsr mc;             // operand U
  BMat mb;
  const u32* filled;   // scatter by bits: the operand rows that are not empty, as bits
  const u32* need;     // rows of the result that a later product reads (null: all)
  // listed form: only the result rows some index entry gives anything to, as
  // k_bit_active found them (long compressed rows apart); null: every row
  u32* list;
  u32* hlist;
  u32* slist;          // (or null) rows of few entries, for k_bit_gather_wide
  u64* n_list;         // rows listed in list, hlist, slist
  // result: a temporary (out, obag) ...
  u32* out;
  u64* obag;
  // ... or the head's accumulator N (flagged rows hold something) ...
  u32* acc;
  u32* aflag;
  int diag;            // 0: all, 1: x != z, 2: x == z
  // ... or, as the iteration's last product into it, straight D' and F
  int commit;
  u32* full;
  u32* next;
  u32* ncnt;
  u32* fcnt;
  u64* n_new;
  u64* state;
  int n_skip;          // the arm is skipped when one of these relations has no old facts
  int skip[kMaxChain];
};

template <bool kLoop>
LOB_DEV bool op_idle(const BOp& P) {
  if (ldm<kLoop>(P.state + B_DONE)) return true;
  for (int i = 0; i < P.n_skip; i++)
    if (ldm<kLoop>(P.state + rel_slot(P.skip[i], 0)) == ldm<kLoop>(P.state + rel_slot(P.skip[i], 1))) return true;
  return false;
}

LOB_DEV void or4(uint4& a, const uint4& b) {
  a.x |= b.x; a.y |= b.y; a.z |= b.z; a.w |= b.w;
}
LOB_DEV bool any4(const uint4& a) { return (a.x | a.y | a.z | a.w) != 0u; }
LOB_DEV u32 popc4(const uint4& a) { return __popc(a.x) + __popc(a.y) + __popc(a.z) + __popc(a.w); }

// the rule's filter on the words [w, w + 4) of row r
LOB_DEV void diag4(uint4& a, int diag, u32 r, u32 w) {
  if (!diag) return;
  u32 m[4] = {0, 0, 0, 0};
  if ((r >> 5) >= w && (r >> 5) < w + 4) m[(r >> 5) - w] = 1u << (r & 31u);
  if (diag == 1) {
    a.x &= ~m[0]; a.y &= ~m[1]; a.z &= ~m[2]; a.w &= ~m[3];
  } else {
    a.x &= m[0]; a.y &= m[1]; a.z &= m[2]; a.w &= m[3];
  }
}

// The words [w, w + 4) of result row r go where the product's result goes;
// returns the new facts among them (commit).
template <bool kLoop>
LOB_DEV u32 put4(const BOp& P, u32 r, u32 w, uint4 a) {
  const u64 at = ((u64)r * P.words + w) / 4;
  if (P.out) {
    reinterpret_cast<uint4*>(P.out)[at] = a;
    return 0;
  }
  diag4(a, P.diag, r, w);
  if (!P.commit) {
    if (any4(a)) {
      uint4* N = reinterpret_cast<uint4*>(P.acc) + at;
      or4(a, ldm<kLoop>(N));
      *N = a;
      P.aflag[r] = 1;
    }
    return 0;
  }
  if (P.aflag && ldm<kLoop>(P.aflag + r)) {
    uint4* N = reinterpret_cast<uint4*>(P.acc) + at;
    or4(a, ldm<kLoop>(N));
    *N = make_uint4(0, 0, 0, 0);
  }
  uint4* F = reinterpret_cast<uint4*>(P.full) + at;
  if (!any4(a)) {  // nothing derived here: F stays unread
    reinterpret_cast<uint4*>(P.next)[at] = a;
    return 0;
  }
  uint4 f = ldm<kLoop>(F);
  a.x &= ~f.x; a.y &= ~f.y; a.z &= ~f.z; a.w &= ~f.w;
  reinterpret_cast<uint4*>(P.next)[at] = a;
  if (any4(a)) {
    or4(f, a);
    *F = f;
  }
  return popc4(a);
}

LOB_DEV void count_new(const BOp& P, u32 r, u32 fresh) {
  if (!fresh) return;
  atomicAdd(P.ncnt + r, fresh);
  atomicAdd(P.fcnt + r, fresh);
}

// derivations, words read and new facts of a block's threads, one atomic each
LOB_DEV void block_totals(const BOp& P, u64 cand, u64 words, u64 fresh) {
  __shared__ u64 tot[3];
  if (threadIdx.x < 3) tot[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    cand += __shfl_xor_sync(0xFFFFFFFFu, cand, o);
    words += __shfl_xor_sync(0xFFFFFFFFu, words, o);
    fresh += __shfl_xor_sync(0xFFFFFFFFu, fresh, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (cand) atomicAdd(reinterpret_cast<unsigned long long*>(&tot[0]), cand);
    if (words) atomicAdd(reinterpret_cast<unsigned long long*>(&tot[1]), words);
    if (fresh) atomicAdd(reinterpret_cast<unsigned long long*>(&tot[2]), fresh);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long* s = reinterpret_cast<unsigned long long*>(P.state);
    if (tot[0] && !P.out) atomicAdd(s + B_CAND, tot[0]);
    if (tot[1]) atomicAdd(s + B_WORDS, tot[1]);
    if (tot[2]) atomicAdd(reinterpret_cast<unsigned long long*>(P.n_new), tot[2]);
  }
}

// ---------------------------------------------------------------------------
// gather: row r of the result = OR of the operand rows listed in row r of the
// index matrix.
// A task is 128 words of a result row.  Compressed index rows: a warp a task
// (an average row of the benchmark's graph lists five operand rows), and a
// block a task for rows of more than kHeavyRow entries, whose hub of 5,000
// would otherwise keep one warp busy long after the rest have finished.  Bit
// index rows: a block a task, its warps sharing the words of the index row.
// Rows narrower than 128 words leave lanes over: lanes are split into groups of
// the row's width, each taking other operand rows, and ORed together at the end.
// Entries whose operand row is empty are dropped first (a ballot), so an
// iteration with few recent rows reads few words.
// ---------------------------------------------------------------------------
constexpr int kGatherWarps = 8;
constexpr int kListCap = 64;

struct Lanes {  // how the 32 lanes split over a task's words
  int group;    // lanes per operand row (a power of two)
  int sub, n_sub;
  u32 w;        // this lane's first word of the row
  bool in;
};
LOB_DEV Lanes split_lanes(u32 words, u32 chunk) {
  const int lane = threadIdx.x & 31;
  const u32 left = words - chunk * 128;
  int g = 32;
  while (g > 1 && (u32)(g / 2) * 4 >= left) g >>= 1;
  Lanes L;
  L.group = g;
  L.sub = lane / g;
  L.n_sub = 32 / g;
  L.w = chunk * 128 + (u32)(lane % g) * 4;
  L.in = L.w < words;
  return L;
}

// acc |= the words of the n operand rows listed in shared memory
template <bool kLoop>
LOB_DEV void gather_list(const BMat& M, u32 words, const Lanes& L, const u32* list, int n, uint4& acc) {
  if (!L.in) return;
  const uint4* base = reinterpret_cast<const uint4*>(M.bits + L.w);
  const u64 stride = words / 4;
  int k = L.sub;
  for (; k + 3 * L.n_sub < n; k += 4 * L.n_sub) {  // four rows in flight
    const uint4 a = ldm<kLoop>(base + list[k] * stride), b = ldm<kLoop>(base + list[k + L.n_sub] * stride);
    const uint4 c = ldm<kLoop>(base + list[k + 2 * L.n_sub] * stride), d = ldm<kLoop>(base + list[k + 3 * L.n_sub] * stride);
    or4(acc, a); or4(acc, b); or4(acc, c); or4(acc, d);
  }
  for (; k < n; k += L.n_sub) or4(acc, ldm<kLoop>(base + list[k] * stride));
}

LOB_DEV void or_groups(const Lanes& L, uint4& a) {
  for (int o = L.group; o < 32; o <<= 1) {
    a.x |= __shfl_xor_sync(0xFFFFFFFFu, a.x, o);
    a.y |= __shfl_xor_sync(0xFFFFFFFFu, a.y, o);
    a.z |= __shfl_xor_sync(0xFFFFFFFFu, a.z, o);
    a.w |= __shfl_xor_sync(0xFFFFFFFFu, a.w, o);
  }
}

// add one warp's batch of up to 32 candidate operand rows (idx, valid) to its
// list, reading them once the list holds 32 or more; n entries are pending
template <bool kLoop>
LOB_DEV void push_batch(const BMat& M, u32 words, const Lanes& L, u32* list, int& n, u32 idx, bool valid, bool count,
                        u64& bag, u64& read, uint4& acc, bool& any) {
  const u64 wgt = valid ? M.weight<kLoop>(idx) : 0ull;
  const bool act = wgt != 0;
  if (count) bag += wgt;
  const u32 m = __ballot_sync(0xFFFFFFFFu, act);
  if (!m) return;
  any = true;
  const int lane = threadIdx.x & 31;
  if (act) list[n + __popc(m & ((1u << lane) - 1u))] = idx;
  n += __popc(m);
  __syncwarp();
  if (n >= kListCap - 32) {
    gather_list<kLoop>(M, words, L, list, n, acc);
    if (lane == 0) read += (u64)n * (u64)min(128u, words);
    n = 0;
    __syncwarp();
  }
}
template <bool kLoop>
LOB_DEV void flush_list(const BMat& M, u32 words, const Lanes& L, u32* list, int& n, u64& read, uint4& acc) {
  if (n) {
    gather_list<kLoop>(M, words, L, list, n, acc);
    if ((threadIdx.x & 31) == 0) read += (u64)n * (u64)min(128u, words);
  }
  n = 0;
  __syncwarp();
}

// store a task's combined words; row r of a temporary always gets its weight
template <bool kLoop>
LOB_DEV u32 finish_task(const BOp& P, const Lanes& L, u32 r, bool count, const uint4& acc, bool any, u64 bag) {
  if (P.out && count && (threadIdx.x & 31) == 0) P.obag[r] = any ? bag : 0ull;
  const bool flagged = P.commit && P.aflag && ldm<kLoop>(P.aflag + r);
  if (!any && !flagged) return 0;
  u32 fresh = 0;
  if (L.in && L.sub == 0) fresh = put4<kLoop>(P, r, L.w, acc);
  if (P.commit) {
#pragma unroll
    for (int o = 16; o; o >>= 1) fresh += __shfl_xor_sync(0xFFFFFFFFu, fresh, o);
    if ((threadIdx.x & 31) == 0) {
      count_new(P, r, fresh);
      return fresh;
    }
  }
  return 0;
}

LOB_DEV u64 warp_total(u64 v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// The result rows a product has work for, a lane a row: rows with a non-empty
// operand row (compressed index; their derivations are summed on the way) or a
// non-empty index row (bits), and rows whose accumulator waits for the commit.
// Large matrices only: there most rows have nothing to do in most iterations
// (a level of same generation is a twelfth of the tree), and visiting all rows
// x chunks of a 50,000-value matrix takes 100 us where the list takes 5.
template <int IK>
__global__ void __launch_bounds__(256) k_bit_active(const __grid_constant__ BOp P, int operand_bits) {
  if (op_idle<false>(P)) return;
  const int lane = threadIdx.x & 31;
  const u64 nwarps = (u64)gridDim.x * 8;
  u64 cand = 0;
  for (u64 r0 = ((u64)blockIdx.x * 8 + (threadIdx.x >> 5)) * 32; r0 < P.rows; r0 += nwarps * 32) {
    const u32 r = (u32)r0 + lane;
    const bool in = r < P.rows;
    bool live = in && (!P.need || P.need[r]);
    u64 bag = 0;
    u32 len = 0;
    if constexpr (IK == I_BITS) {
      live = live && P.ib.weight<false>(r) != 0;
    } else {
      u32 j0 = 0;
      if constexpr (IK == I_CSR) {
        if (live) {
          j0 = P.ic.ptr[r];
          len = P.ic.ptr[r + 1] - j0;
        }
      } else {
        len = live ? 1 : 0;
      }
      if (operand_bits) {
        if (len <= 32)
          // eight entries' loads in flight (one at a time: 33 us a list of 20,000 rows, so 24)
          for (u32 j = 0; j < len; j += 8) {
            u32 x[8];
#pragma unroll
            for (int q = 0; q < 8; q++)
              if (j + q < len) x[q] = IK == I_CSR ? P.ic.col[j0 + j + q] : r;
#pragma unroll
            for (int q = 0; q < 8; q++)
              if (j + q < len) bag += P.mb.weight<false>(x[q]);
          }
        for (u32 m = __ballot_sync(0xFFFFFFFFu, len > 32); m; m &= m - 1) {
          const int src = __ffs(m) - 1;
          const u32 a = __shfl_sync(0xFFFFFFFFu, j0, src), n = __shfl_sync(0xFFFFFFFFu, len, src);
          u64 b = 0;
          for (u32 j = lane; j < n; j += 32) b += P.mb.weight<false>(P.ic.col[a + j]);
          b = warp_total(b);
          if (lane == src) bag = b;
        }
        live = bag != 0;
      } else {
        live = len != 0 && (IK == I_CSR || P.mc.ptr[r + 1] != P.mc.ptr[r]);
      }
    }
    if (in && P.out && !live) P.obag[r] = 0;
    if (in && P.out && live && operand_bits && IK != I_BITS) P.obag[r] = bag;
    cand += bag;
    live = live || (in && P.commit && P.aflag && P.aflag[r]);
    const bool heavy = live && IK == I_CSR && operand_bits && len > kHeavyRow;
    const bool brief = live && P.slist && len <= kWideRow;
    const int which = heavy ? 1 : brief ? 2 : 0;
    const u32 below = (1u << lane) - 1u;
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const u32 m = __ballot_sync(0xFFFFFFFFu, live && which == q);
      if (!m) continue;
      u32 at = 0;
      if (lane == 0) at = (u32)atomicAdd(reinterpret_cast<unsigned long long*>(P.n_list) + q, (unsigned long long)__popc(m));
      at = __shfl_sync(0xFFFFFFFFu, at, 0);
      u32* to = q == 0 ? P.list : q == 1 ? P.hlist : P.slist;
      if (live && which == q) to[at + __popc(m & below)] = r;
    }
  }
  block_totals(P, cand, 0, 0);
}

template <int IK, bool kLoop>
LOB_DEV void gather_rows(const BOp& P) {
  __shared__ u32 lists[kGatherWarps][kListCap];
  __shared__ uint4 part[kGatherWarps][32];
  __shared__ u64 pbag[kGatherWarps];
  __shared__ u32 pany[kGatherWarps];
  if (op_idle<kLoop>(P)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 chunks = (P.words + 127) / 128;
  u32* list = lists[warp];
  u64 cand = 0, read = 0, fresh = 0;
  // k_bit_active has summed the derivations of listed compressed rows
  const bool count_all = !P.list || IK == I_BITS;
  if constexpr (IK != I_BITS) {
    const u64 tasks = (P.list ? P.n_list[0] : (u64)P.rows) * chunks;
    const u64 nwarps = (u64)gridDim.x * kGatherWarps;
    for (u64 t = (u64)blockIdx.x * kGatherWarps + warp; t < tasks; t += nwarps) {
      const u32 q = (u32)(t / chunks), chunk = (u32)(t % chunks);
      const u32 r = P.list ? P.list[q] : q;
      const bool count = count_all && chunk == 0;
      const Lanes L = split_lanes(P.words, chunk);
      uint4 acc = make_uint4(0, 0, 0, 0);
      u64 bag = 0;
      int n = 0;
      bool any = false;
      if (!P.need || P.need[r]) {
        if constexpr (IK == I_IDENT) {
          push_batch<kLoop>(P.mb, P.words, L, list, n, r, lane == 0, count, bag, read, acc, any);
        } else {
          const u32 j0 = P.ic.ptr[r], j1 = P.ic.ptr[r + 1];
          if (j1 - j0 > kHeavyRow && !P.list) continue;  // below, by whole blocks
          for (u32 j = j0; j < j1; j += 32) {
            const bool v = j + lane < j1;
            push_batch<kLoop>(P.mb, P.words, L, list, n, v ? P.ic.col[j + lane] : 0u, v, count, bag, read, acc, any);
          }
        }
        flush_list<kLoop>(P.mb, P.words, L, list, n, read, acc);
        or_groups(L, acc);
      }
      bag = warp_total(bag);
      if (lane == 0) cand += bag;
      fresh += finish_task<kLoop>(P, L, r, count, acc, any, bag);
    }
  }
  if constexpr (IK != I_IDENT) {
    const u32* rows = IK == I_CSR ? (P.list ? P.hlist : P.ic.heavy) : P.list;
    const u64 nr = IK == I_CSR ? (P.list ? P.n_list[1] : (u64)*P.ic.n_heavy) : (P.list ? P.n_list[0] : (u64)P.rows);
    const u64 tasks = nr * chunks;
    for (u64 t = blockIdx.x; t < tasks; t += gridDim.x) {
      const u32 q = (u32)(t / chunks), chunk = (u32)(t % chunks);
      const u32 r = rows ? rows[q] : q;
      const bool count = count_all && chunk == 0;
      const Lanes L = split_lanes(P.words, chunk);
      uint4 acc = make_uint4(0, 0, 0, 0);
      u64 bag = 0;
      int n = 0;
      bool any = false;
      bool live = !P.need || P.need[r];
      if constexpr (IK == I_BITS) live = live && P.ib.weight<kLoop>(r) != 0;
      if (!live) {  // the same for the whole block
        if (warp == 0) fresh += finish_task<kLoop>(P, L, r, count, acc, false, 0);
        continue;
      }
      if constexpr (IK == I_CSR) {
        const u32 j0 = P.ic.ptr[r], j1 = P.ic.ptr[r + 1];
        for (u32 j = j0 + warp * 32; j < j1; j += 256) {
          const bool v = j + lane < j1;
          push_batch<kLoop>(P.mb, P.words, L, list, n, v ? P.ic.col[j + lane] : 0u, v, count, bag, read, acc, any);
        }
      } else {
        const u32* row = P.ib.bits + (u64)r * P.words;
        for (u32 w0 = warp * 32; w0 < P.words; w0 += 256) {
          const u32 mine = w0 + lane < P.words ? ldm<kLoop>(row + w0 + lane) : 0u;
          for (u32 m = __ballot_sync(0xFFFFFFFFu, mine != 0u); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const u32 word = __shfl_sync(0xFFFFFFFFu, mine, src);
            push_batch<kLoop>(P.mb, P.words, L, list, n, (w0 + src) * 32 + lane, (word >> lane) & 1u, count, bag, read, acc, any);
          }
        }
      }
      flush_list<kLoop>(P.mb, P.words, L, list, n, read, acc);
      or_groups(L, acc);
      bag = warp_total(bag);
      part[warp][lane] = acc;
      if (lane == 0) {
        pbag[warp] = bag;
        pany[warp] = any;
      }
      __syncthreads();
      if (warp == 0) {
        for (int v = 1; v < kGatherWarps; v++) {
          or4(acc, part[v][lane]);
          bag += pbag[v];
          any = any || pany[v];
        }
        if (lane == 0) cand += bag;
        fresh += finish_task<kLoop>(P, L, r, count, acc, any, bag);
      }
      __syncthreads();  // part is rewritten by the next task
    }
  }
  block_totals(P, cand, read, fresh);
}
template <int IK>
__global__ void __launch_bounds__(256) k_bit_gather(const __grid_constant__ BOp P) { gather_rows<IK, false>(P); }

// The same for the rows of few entries of wide matrices (compressed index, listed
// apart): a warp takes four chunks of a row, so that what it waits for on the way to
// the first word -- list, offsets, column, weight, one after another -- is paid
// once, and the words of two operand rows and of F come eight and four loads at a
// time.  Same generation on the 50,000-node tree, whose rows list one operand row:
// the gathers of a run 3.2 -> 2.2 ms.
__global__ void __launch_bounds__(256) k_bit_gather_wide(const __grid_constant__ BOp P) {
  if (op_idle<false>(P)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 groups = (P.words + kWide * 128 - 1) / (kWide * 128);
  const u64 stride = P.words / 4;
  u64 read = 0, fresh_all = 0;
  const u64 tasks = P.n_list[2] * groups, nwarps = (u64)gridDim.x * kGatherWarps;
  for (u64 t = (u64)blockIdx.x * kGatherWarps + warp; t < tasks; t += nwarps) {
    const u32 r = P.slist[t / groups], w0 = (u32)(t % groups) * (kWide * 128) + lane * 4;
    const u32 j0 = P.ic.ptr[r], j1 = P.ic.ptr[r + 1];
    const uint4* base = reinterpret_cast<const uint4*>(P.mb.bits + w0);
    uint4 acc[kWide];
#pragma unroll
    for (int c = 0; c < kWide; c++) acc[c] = make_uint4(0, 0, 0, 0);
    for (u32 j = j0; j < j1; j += 32) {
      const u32 idx = j + lane < j1 ? P.ic.col[j + lane] : 0u;
      u32 m = __ballot_sync(0xFFFFFFFFu, j + lane < j1 && P.mb.weight<false>(idx) != 0);
      if (lane == 0) read += (u64)__popc(m) * min(P.words - (w0 & ~127u), (u32)kWide * 128);
      while (m) {
        const u32 a = __shfl_sync(0xFFFFFFFFu, idx, __ffs(m) - 1);
        m &= m - 1;
        const u32 b = m ? __shfl_sync(0xFFFFFFFFu, idx, __ffs(m) - 1) : a;
        m &= m - 1;
        uint4 x[kWide], y[kWide];
#pragma unroll
        for (int c = 0; c < kWide; c++)
          if (w0 + c * 128 < P.words) {
            x[c] = base[a * stride + c * 32];
            y[c] = base[b * stride + c * 32];
          }
#pragma unroll
        for (int c = 0; c < kWide; c++)
          if (w0 + c * 128 < P.words) {
            or4(acc[c], x[c]);
            or4(acc[c], y[c]);
          }
      }
    }
    u32 fresh = 0;
    if (P.commit && !(P.aflag && P.aflag[r])) {
      uint4* F = reinterpret_cast<uint4*>(P.full + (u64)r * P.words + w0);
      uint4* D = reinterpret_cast<uint4*>(P.next + (u64)r * P.words + w0);
      uint4 f[kWide];
#pragma unroll
      for (int c = 0; c < kWide; c++) {
        diag4(acc[c], P.diag, r, w0 + c * 128);
        if (w0 + c * 128 < P.words && any4(acc[c])) f[c] = F[c * 32];
      }
#pragma unroll
      for (int c = 0; c < kWide; c++) {
        if (w0 + c * 128 >= P.words) continue;
        uint4 a = acc[c];
        if (any4(a)) {
          a.x &= ~f[c].x; a.y &= ~f[c].y; a.z &= ~f[c].z; a.w &= ~f[c].w;
          if (any4(a)) {
            or4(f[c], a);
            F[c * 32] = f[c];
            fresh += popc4(a);
          }
        }
        D[c * 32] = a;
      }
    } else {
#pragma unroll
      for (int c = 0; c < kWide; c++)
        if (w0 + c * 128 < P.words) fresh += put4<false>(P, r, w0 + c * 128, acc[c]);
    }
    if (P.commit) {
#pragma unroll
      for (int o = 16; o; o >>= 1) fresh += __shfl_xor_sync(0xFFFFFFFFu, fresh, o);
      if (lane == 0) {
        count_new(P, r, fresh);
        fresh_all += fresh;
      }
    }
  }
  block_totals(P, 0, read, fresh_all);
}

// ---------------------------------------------------------------------------
// scatter: row r of the result = the union of the compressed operand rows
// listed in row r of the index matrix (identity: operand row r itself), built
// in shared memory by one block.  Bounded by the shared atomics, one per
// derivation, where the global ones of the general path go to L2; rows of up
// to 92,000 values take 11.5 KB, so 8 blocks an SM stay resident.
// ---------------------------------------------------------------------------
// The columns of n operand rows, named by a warp's list (`base` added to each
// entry), are set in `row`; four of them per lane and step, so that their loads
// overlap.
template <class T>
LOB_DEV void set_list(const BCsr& M, u32* row, const T* list, u32 n, u32 base, u64& bag) {
  constexpr int kAt = 4;
  const int lane = threadIdx.x & 31;
  for (u32 i0 = 0; i0 < n; i0 += 32 * kAt) {
    u32 j[kAt], e[kAt], c[kAt];
#pragma unroll
    for (int q = 0; q < kAt; q++) {
      const u32 i = i0 + q * 32 + lane;
      const u32 y = i < n ? base + list[i] : 0u;
      j[q] = i < n ? M.ptr[y] : 0u;
      e[q] = i < n ? M.ptr[y + 1] : 0u;
    }
#pragma unroll
    for (int q = 0; q < kAt; q++) {
      c[q] = j[q] < e[q] ? M.col[j[q]] : 0u;
      bag += e[q] - j[q];
    }
#pragma unroll
    for (int q = 0; q < kAt; q++) {
      if (j[q] < e[q]) atomicOr(row + (c[q] >> 5), 1u << (c[q] & 31u));
      const bool big = e[q] - j[q] > 16;
      if (!big)
        for (u32 k = j[q] + 1; k < e[q]; k++) {
          const u32 x = M.col[k];
          atomicOr(row + (x >> 5), 1u << (x & 31u));
        }
      for (u32 m = __ballot_sync(0xFFFFFFFFu, big); m; m &= m - 1) {  // long rows: the whole warp
        const int src = __ffs(m) - 1;
        const u32 a = __shfl_sync(0xFFFFFFFFu, j[q], src), b = __shfl_sync(0xFFFFFFFFu, e[q], src);
        for (u32 k = a + lane; k < b; k += 32) {
          const u32 x = M.col[k];
          atomicOr(row + (x >> 5), 1u << (x & 31u));
        }
      }
    }
  }
}

template <int IK, bool kLoop>
LOB_DEV void scatter_rows(const BOp& P) {
  extern __shared__ __align__(16) u32 row[];
  __shared__ u64 sm[256 / 32 + 1];
  if (op_idle<kLoop>(P)) return;
  u64 cand = 0, read = 0, fresh_all = 0;
  const u32 n_rows = P.list ? (u32)P.n_list[0] : P.rows;
  for (u32 q = blockIdx.x; q < n_rows; q += gridDim.x) {
    const u32 r = P.list ? P.list[q] : q;
    bool live = !P.need || P.need[r];
    u32 j0 = 0, j1 = 0;
    if constexpr (IK == I_BITS) {
      live = live && P.ib.weight<kLoop>(r) != 0;
    } else {
      const BCsr& C = IK == I_CSR ? P.ic : P.mc;
      j0 = C.ptr[r];
      j1 = C.ptr[r + 1];
      live = live && j1 > j0;
    }
    const bool flagged = P.commit && P.aflag && ldm<kLoop>(P.aflag + r);
    if (!live && !flagged) {
      if (P.out && threadIdx.x == 0) P.obag[r] = 0;
      continue;
    }
    for (u32 w = threadIdx.x; w < P.words; w += 256) row[w] = 0;
    __syncthreads();
    u64 bag = 0;
    if (live) {
      if constexpr (IK == I_IDENT) {
        for (u32 j = j0 + threadIdx.x; j < j1; j += 256) {
          const u32 c = P.mc.col[j];
          atomicOr(row + (c >> 5), 1u << (c & 31u));
          bag++;
        }
      } else if constexpr (IK == I_CSR) {
        const u32 per = (j1 - j0 + 7) / 8, a = j0 + (threadIdx.x >> 5) * per;
        if (a < j1) set_list(P.mc, row, P.ic.col + a, min(per, j1 - a), 0, bag);
      } else {
        // A warp lists the bits of its share of the row -- those whose operand row
        // holds something -- and then sets their columns, evenly over its lanes.  (A
        // lane walking its own word's bits waits for two loads per bit, and for the
        // lane with the most bits: 4.8 ms on the 50,000-node tree, 4.2 without the
        // empty operand rows.)
        __shared__ uint16_t lists[8][kBitList];
        uint16_t* list = lists[threadIdx.x >> 5];
        const int lane = threadIdx.x & 31;
        const u32* src = P.ib.bits + (u64)r * P.words;
        const u32 share = (P.words + 7) / 8, first = (threadIdx.x >> 5) * share, end = min(P.words, first + share);
        u32 n = 0;
        for (u32 w0 = first; w0 < end; w0 += 32) {
          const u32 w = w0 + lane;
          u32 m = w < end ? ldm<kLoop>(src + w) & P.filled[w] : 0u;
          const u32 inc = warp_inclusive_sum((u32)__popc(m));
          const u32 tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
          if (n + tot > (u32)kBitList) {
            __syncwarp();
            set_list(P.mc, row, list, n, first * 32, bag);
            __syncwarp();
            n = 0;
          }
          u32 at = n + inc - __popc(m);
          for (; m; m &= m - 1) list[at++] = (uint16_t)((w - first) * 32 + (u32)__ffs(m) - 1);
          n += tot;
        }
        __syncwarp();
        set_list(P.mc, row, list, n, first * 32, bag);
        read += threadIdx.x == 0 ? P.words : 0;
      }
    }
    u64 tot;
    block_exclusive_sum<u64>(bag, sm, &tot);  // also the barrier before the row is read
    if (threadIdx.x == 0) cand += tot;
    if (P.out && threadIdx.x == 0) P.obag[r] = tot;
    u32 fresh = 0;
    if (!P.out || tot)
      for (u32 w = threadIdx.x * 4; w < P.words; w += 1024) fresh += put4<kLoop>(P, r, w, *reinterpret_cast<const uint4*>(row + w));
    if (P.commit) {
#pragma unroll
      for (int o = 16; o; o >>= 1) fresh += __shfl_xor_sync(0xFFFFFFFFu, fresh, o);
      if ((threadIdx.x & 31) == 0) {
        count_new(P, r, fresh);
        fresh_all += fresh;
      }
    }
    __syncthreads();  // the row is cleared for the next one
  }
  block_totals(P, cand, read, fresh_all);
}
template <int IK>
__global__ void __launch_bounds__(256) k_bit_scatter(const __grid_constant__ BOp P) { scatter_rows<IK, false>(P); }

// D' = N & ~F, F |= D' of the rows some product added to; N is cleared
template <bool kLoop>
LOB_DEV void commit_rows(const BOp& P) {
  if (ldm<kLoop>(P.state + B_DONE)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 chunks = (P.words + 127) / 128;
  const u64 tasks = (u64)P.rows * chunks, nwarps = (u64)gridDim.x * kGatherWarps;
  u64 fresh_all = 0, read = 0;
  for (u64 t = (u64)blockIdx.x * kGatherWarps + warp; t < tasks; t += nwarps) {
    const u32 r = (u32)(t / chunks);
    if (!ldm<kLoop>(P.aflag + r)) continue;
    const u32 w = (u32)(t % chunks) * 128 + lane * 4;
    u32 fresh = w < P.words ? put4<kLoop>(P, r, w, make_uint4(0, 0, 0, 0)) : 0u;
#pragma unroll
    for (int o = 16; o; o >>= 1) fresh += __shfl_xor_sync(0xFFFFFFFFu, fresh, o);
    if (lane == 0) {
      read += 3ull * min(128u, P.words);
      count_new(P, r, fresh);
      fresh_all += fresh;
    }
  }
  block_totals(P, 0, read, fresh_all);
}
__global__ void __launch_bounds__(256) k_bit_commit(const __grid_constant__ BOp P) { commit_rows<false>(P); }

struct BEnd {
  u32 rows;
  int n_rel;
  int rel[kMaxBitRels];
  u32* old_cnt[kMaxBitRels];   // row counts of the recent set this iteration read: the next one writes there
  u32* aflag[kMaxBitRels];
  u32* tcnt[kMaxBitRels];      // row counts of its transposed copy (or null)
  u32 max_iters;
  u64* state;
};
// End of an iteration: sizes, the stop decision, cleared row counts and flags.
// Only block 0 writes the state; a block that sees the new done flag skips
// clearing what no later iteration reads.
template <bool kLoop>
LOB_DEV void end_iteration(const BEnd& E) {
  u64* s = E.state;
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (int i = 0; i < E.n_rel; i++)
    for (u64 q = (u64)blockIdx.x * blockDim.x + threadIdx.x; q < E.rows; q += stride) {
      E.old_cnt[i][q] = 0;
      if (E.aflag[i]) E.aflag[i][q] = 0;
      if (E.tcnt[i]) E.tcnt[i][q] = 0;
    }
  if (blockIdx.x || threadIdx.x) return;
  u64 total = 0;
  for (int i = 0; i < E.n_rel; i++) {
    const int r = E.rel[i];
    const u64 n = ldm<kLoop>(s + rel_slot(r, 2));
    s[rel_slot(r, 0)] = ldm<kLoop>(s + rel_slot(r, 0)) + n;
    s[rel_slot(r, 1)] = n;
    s[rel_slot(r, 2)] = 0;
    total += n;
  }
  if constexpr (!kLoop)
    for (int i = 0; i < 3 * kMaxLists; i++) s[kStateSlots + i] = 0;
  s[B_NEW] = ldm<kLoop>(s + B_NEW) + total;
  const u64 it = ldm<kLoop>(s + B_ITER) + 1;
  s[B_ITER] = it;
  if (!total) s[B_DONE] = 1;
  else if (it >= E.max_iters) s[B_DONE] = 2;
}
__global__ void __launch_bounds__(256) k_bit_end(const __grid_constant__ BEnd E) {
  if (E.state[B_DONE]) return;
  end_iteration<false>(E);
}

// ---------------------------------------------------------------------------
// transpose: 256 x 256 bits a block.  Each warp takes 32 rows, turns eight
// 32 x 32 squares by ballots, and the block stores 32-byte pieces of 256 result
// rows.  With `full`, the same bits are ORed into a second matrix (F' follows D').
// ---------------------------------------------------------------------------
struct BTrans {
  BMat src;
  u32 rows, words;
  u32 *dst, *dcnt, *full, *fcnt;
  const u64* state;
};
template <bool kLoop>
LOB_DEV void transpose_rows(const BTrans& X) {
  const BMat& src = X.src;
  const u32 rows = X.rows, words = X.words;
  u32 *dst = X.dst, *dcnt = X.dcnt, *full = X.full, *fcnt = X.fcnt;
  const u64* state = X.state;
  __shared__ u32 tile[256][9];  // result row within the block, its 8 words (+1: no bank conflicts)
  if (state && ldm<kLoop>(state + B_DONE)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 bw = (words + 7) / 8;
  const u64 tiles = (u64)((rows + 255) / 256) * bw;
  for (u64 t = blockIdx.x; t < tiles; t += gridDim.x) {
    const u32 r0 = (u32)(t / bw) * 256, w0 = (u32)(t % bw) * 8;
    const u32 r = r0 + warp * 32 + lane;
    const bool live = r < rows && src.weight<kLoop>(r) != 0;
    u32 x[8];
#pragma unroll
    for (int j = 0; j < 8; j += 4) {
      uint4 v = make_uint4(0, 0, 0, 0);
      if (live && w0 + j < words) v = ldm<kLoop>(reinterpret_cast<const uint4*>(src.bits + (u64)r * words + w0 + j));
      x[j] = v.x; x[j + 1] = v.y; x[j + 2] = v.z; x[j + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < 8; j++) {
      u32 mine = 0;
      if (__any_sync(0xFFFFFFFFu, x[j] != 0u)) {
#pragma unroll
        for (int b = 0; b < 32; b++) {
          const u32 v = __ballot_sync(0xFFFFFFFFu, (x[j] >> b) & 1u);
          if (lane == b) mine = v;
        }
      }
      tile[j * 32 + lane][warp] = mine;
    }
    __syncthreads();
    const u32 orow = w0 * 32 + threadIdx.x, ow = r0 / 32;
    if (orow < rows) {
      u32 c = 0;
      u32 y[8];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        y[j] = tile[threadIdx.x][j];
        c += __popc(y[j]);
      }
#pragma unroll
      for (int j = 0; j < 8; j += 4)
        if (ow + j < words) {
          const u64 at = ((u64)orow * words + ow + j) / 4;
          uint4 v = make_uint4(y[j], y[j + 1], y[j + 2], y[j + 3]);
          reinterpret_cast<uint4*>(dst)[at] = v;
          if (full && any4(v)) {
            uint4* f = reinterpret_cast<uint4*>(full) + at;
            or4(v, ldm<kLoop>(f));
            *f = v;
          }
        }
      if (c && dcnt) atomicAdd(dcnt + orow, c);
      if (c && fcnt) atomicAdd(fcnt + orow, c);
    }
    __syncthreads();
  }
}
__global__ void __launch_bounds__(256) k_bit_transpose(const __grid_constant__ BTrans X) { transpose_rows<false>(X); }

// ---------------------------------------------------------------------------
// The whole run in one cooperative launch, for matrices of at most kLoopTasks
// tasks (rows x 128-word chunks).  A closure over 1,000 nodes takes 15 iterations of two
// kernels that do a microsecond's work each, plus the iterations queued past the
// fixpoint: the steps of an iteration, described in global memory, run one after
// another with a grid barrier between them, and the loop ends where the state says
// so.  One block per eight tasks of a step, up to four per SM.
// Measured (GB300, whole passes): closure of 67 nodes 554 -> 425 us, of 1,000
// nodes 609 -> 491 us; points-to over 2,681 values, whose products fill the GPU by
// themselves, 2.96 -> 3.33 ms, so the line lies at 2,048 tasks.
// ---------------------------------------------------------------------------
enum StepKind { K_GATHER, K_SCATTER, K_COMMIT, K_TRANSPOSE };
struct BStep {
  int kind, ik;
  BOp P;
  BTrans X;
};
struct BLoop {
  const BStep* steps;
  int first[4];   // steps of: the first iteration, those on recent buffer 1, on buffer 0
  BEnd end[2];    // by recent buffer
  const BStep* after;  // transposes that follow an iteration's end, by the buffer it wrote
  int after_first[3];
  u64* state;
  u32* bar;       // arrivals, give-up flag
};
constexpr u64 kLoopTasks = 2048;
constexpr u32 kLoopSpin = 1u << 26;  // barrier polls before a block gives up

LOB_DEV bool loop_barrier(u32* bar, u32& gen) {
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
    while ((int)(b[0] - want) < 0 && !b[1] && n < kLoopSpin) n++;
    if ((int)(b[0] - want) < 0) b[1] = 1;
    __threadfence();
    ok = b[1] == 0;
  }
  __syncthreads();
  return ok != 0;
}

LOB_DEV void run_step(const BStep& S) {
  if (S.kind == K_GATHER) {
    if (S.ik == I_IDENT) gather_rows<I_IDENT, true>(S.P);
    else if (S.ik == I_CSR) gather_rows<I_CSR, true>(S.P);
    else gather_rows<I_BITS, true>(S.P);
  } else if (S.kind == K_SCATTER) {
    if (S.ik == I_IDENT) scatter_rows<I_IDENT, true>(S.P);
    else if (S.ik == I_CSR) scatter_rows<I_CSR, true>(S.P);
    else scatter_rows<I_BITS, true>(S.P);
  } else if (S.kind == K_COMMIT) {
    commit_rows<true>(S.P);
  } else {
    transpose_rows<true>(S.X);
  }
}

__global__ void __launch_bounds__(256, 4) k_bit_loop(const __grid_constant__ BLoop L) {
  __shared__ BStep step;
  u32 gen = 0;
  for (u32 it = 1;; it++) {
    const int cur = (it - 1) & 1, list = it == 1 ? 0 : (cur ? 1 : 2);
    for (int i = L.first[list]; i < L.first[list + 1]; i++) {
      for (u32 q = threadIdx.x; q < sizeof(BStep) / 4; q += blockDim.x)
        reinterpret_cast<u32*>(&step)[q] = reinterpret_cast<const u32*>(L.steps + i)[q];
      __syncthreads();
      run_step(step);
      if (!loop_barrier(L.bar, gen)) return;
    }
    end_iteration<true>(L.end[cur]);
    if (!loop_barrier(L.bar, gen)) return;
    if (ldm<true>(L.state + B_DONE)) return;
    for (int i = L.after_first[cur ^ 1]; i < L.after_first[(cur ^ 1) + 1]; i++) {
      for (u32 q = threadIdx.x; q < sizeof(BStep) / 4; q += blockDim.x)
        reinterpret_cast<u32*>(&step)[q] = reinterpret_cast<const u32*>(L.after + i)[q];
      __syncthreads();
      run_step(step);
      if (!loop_barrier(L.bar, gen)) return;
    }
  }
}

// ---------------------------------------------------------------------------
// renumbering: the values that occur get consecutive codes in value order
// ---------------------------------------------------------------------------
struct KeyCols {
  const void* keys;
  int key64;
  u64 n;
  int shift[2], width[2];
};
struct Codes {       // code of value v: pref[v / 32] + bits of pres[v / 32] below v (null pref: v itself)
  const u32* pres;
  const u32* pref;
  LOB_DEV u32 operator()(u32 v) const {
    return pref ? pref[v >> 5] + __popc(pres[v >> 5] & ((1u << (v & 31u)) - 1u)) : v;
  }
};

__global__ void k_mark_values(KeyCols K, u32* __restrict__ pres) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < K.n; i += stride) {
    const u64 k = load_key(K.keys, K.key64, i);
    touch_bit(pres, field_of(k, K.shift[0], K.width[0]));
    touch_bit(pres, field_of(k, K.shift[1], K.width[1]));
  }
}
__global__ void k_word_bits(const u32* __restrict__ pres, u64 nw, u32* __restrict__ out) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += stride) out[i] = __popc(pres[i]);
}
__global__ void k_code_values(const u32* __restrict__ pres, const u32* __restrict__ pref, u64 nw, u32* __restrict__ dict) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += stride) {
    u32 at = pref[i];
    for (u32 m = pres[i]; m; m &= m - 1) dict[at++] = (u32)i * 32 + (u32)__ffs(m) - 1;
  }
}

// compressed rows of an input relation: row lengths (and which values occur as
// columns), then, after a scan, the columns; a row's columns are in no
// particular order (a product does not depend on it)
__global__ void k_csr_count(KeyCols K, Codes code, int inv, u32* __restrict__ len, u32* __restrict__ colflag) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < K.n; i += stride) {
    const u64 k = load_key(K.keys, K.key64, i);
    atomicAdd(len + code((u32)field_of(k, K.shift[inv], K.width[inv])), 1u);
    colflag[code((u32)field_of(k, K.shift[inv ^ 1], K.width[inv ^ 1]))] = 1u;
  }
}
__global__ void k_csr_fill(KeyCols K, Codes code, int inv, const u32* __restrict__ ptr, u32* __restrict__ used,
                           u32* __restrict__ col, u32* __restrict__ heavy, u32* __restrict__ n_heavy) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < K.n; i += stride) {
    const u64 k = load_key(K.keys, K.key64, i);
    const u32 r = code((u32)field_of(k, K.shift[inv], K.width[inv]));
    const u32 q = atomicAdd(used + r, 1u);
    col[ptr[r] + q] = code((u32)field_of(k, K.shift[inv ^ 1], K.width[inv ^ 1]));
    if (q == kHeavyRow) heavy[atomicAdd(n_heavy, 1u)] = r;  // one entry of a longer row gets here
  }
}
// bit r of the result: row r holds something; a warp a word
__global__ void __launch_bounds__(256) k_filled_rows(const u32* __restrict__ ptr, u32 rows, u32 words, u32* __restrict__ out) {
  const u32 lane = threadIdx.x & 31;
  for (u32 w = blockIdx.x * 8 + (threadIdx.x >> 5); w < words; w += gridDim.x * 8) {
    const u32 r = w * 32 + lane;
    const u32 x = __ballot_sync(0xFFFFFFFFu, r < rows && ptr[r] != ptr[r + 1]);
    if (lane == 0) out[w] = x;
  }
}
// facts loaded into a derived relation: F and D start with them
__global__ void k_set_facts(KeyCols K, Codes code, int inv, u32 words, u32* full, u32* recent, u32* cnt, u32* fcnt) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < K.n; i += stride) {
    const u64 k = load_key(K.keys, K.key64, i);
    const u32 r = code((u32)field_of(k, K.shift[inv], K.width[inv]));
    const u32 c = code((u32)field_of(k, K.shift[inv ^ 1], K.width[inv ^ 1]));
    atomicOr(full + (u64)r * words + (c >> 5), 1u << (c & 31u));
    atomicOr(recent + (u64)r * words + (c >> 5), 1u << (c & 31u));
    atomicAdd(cnt + r, 1u);  // keys are distinct
    atomicAdd(fcnt + r, 1u);
  }
}

// bits per row of a matrix (every row's words are valid): a warp a row
__global__ void __launch_bounds__(256) k_row_counts(const u32* __restrict__ bits, u32 rows, u32 words,
                                                    u32* __restrict__ cnt) {
  const int lane = threadIdx.x & 31;
  const u64 nwarps = (u64)gridDim.x * 8;
  for (u64 r = (u64)blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += nwarps) {
    const uint4* a = reinterpret_cast<const uint4*>(bits + r * words);
    u32 c = 0;
    for (u32 w = lane; w < words / 4; w += 32) c += popc4(a[w]);
#pragma unroll
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
    if (lane == 0) cnt[r] = c;
  }
}

// A warp stores n consecutive words: up to the next 16-byte boundary one by one,
// then four a lane (value / four: the word, the four words, from an offset on).
template <class F, class G>
LOB_DEV void store_run(u32* __restrict__ p, u32 n, int lane, F&& value, G&& four) {
  const u32 head = min(n, (u32)(0 - (reinterpret_cast<uintptr_t>(p) >> 2)) & 3u);
  const u32 quads = (n - head) / 4;
  for (u32 q = lane; q < quads; q += 32) {
    const u32 s = head + 4 * q;
    *reinterpret_cast<uint4*>(p + s) = four(s);
  }
  const u32 rest = n - 4 * quads;  // at most six
  if ((u32)lane < rest) {
    const u32 s = (u32)lane < head ? (u32)lane : 4 * quads + (u32)lane;
    p[s] = value(s);
  }
}

// Read-out: a warp walks a row 32 words at a time; a scan of the words' bit
// counts places each lane's columns in the warp's shared-memory stage (16 bits each,
// counted from the batch's first), and the warp stores them to consecutive
// addresses, 16 bytes a lane; the columns that are the same for the whole row are
// stored in one run before.  Bound by the chain of a batch (scan, stage, store):
// 7.5e8 pairs in 3.0 ms, 2.0 TB/s; with every column a batch at a time 3.4.
__global__ void __launch_bounds__(256) k_bit_read(const u32* __restrict__ bits, u32 rows, u32 words,
                                                  const u64* __restrict__ off, const u32* __restrict__ dict,
                                                  u32* __restrict__ c0, u32* __restrict__ c1, float* __restrict__ tags,
                                                  u32* __restrict__ samples) {
  __shared__ __align__(16) uint16_t stages[8][1024 + 8];  // columns from the batch's first on
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint16_t* stage = stages[warp];
  const u64 nwarps = (u64)gridDim.x * 8;
  for (u64 r = (u64)blockIdx.x * 8 + warp; r < rows; r += nwarps) {
    u64 base = off[r];
    if (off[r + 1] == base) continue;
    const u32 x = dict ? dict[r] : (u32)r;
    const u32* row = bits + r * words;
    u32 nextw = lane < words ? row[lane] : 0u;
    // what is the same for the whole row in one run
    const u32 n_row = (u32)(off[r + 1] - base), one = __float_as_uint(1.0f);
    store_run(c0 + base, n_row, lane, [&](u32) { return x; }, [&](u32) { return make_uint4(x, x, x, x); });
    if (tags)
      store_run(reinterpret_cast<u32*>(tags) + base, n_row, lane, [&](u32) { return one; },
                [&](u32) { return make_uint4(one, one, one, one); });
    if (samples)
      store_run(samples + base, n_row, lane, [&](u32) { return 0u; }, [&](u32) { return make_uint4(0, 0, 0, 0); });
    for (u32 w0 = 0; w0 < words; w0 += 32) {
      const u32 m0 = nextw;
      nextw = w0 + 32 + lane < words ? row[w0 + 32 + lane] : 0u;
      const u32 c = __popc(m0);
      const u32 inc = warp_inclusive_sum(c);
      const u32 tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
      if (!tot) continue;
      // staged at the offset the destination has within 16 bytes
      const u32 skew = (u32)(reinterpret_cast<uintptr_t>(c1 + base) >> 2) & 3u;
      u32 pos = inc - c + skew;
      for (u32 m = m0; m; m &= m - 1) stage[pos++] = (uint16_t)(lane * 32 + __ffs(m) - 1);
      __syncwarp();
      const u32 k0 = w0 * 32;
      store_run(c1 + base, tot, lane, [&](u32 s) { return dict ? dict[k0 + stage[s + skew]] : k0 + stage[s + skew]; },
                [&](u32 s) {
                  const ushort4 z = *reinterpret_cast<const ushort4*>(stage + s + skew);
                  const uint4 y = make_uint4(k0 + z.x, k0 + z.y, k0 + z.z, k0 + z.w);
                  return dict ? make_uint4(dict[y.x], dict[y.y], dict[y.z], dict[y.w]) : y;
                });
      __syncwarp();
      base += tot;
    }
  }
}

// ---------------------------------------------------------------------------
// Does a run fill its matrices?  They cost n^2 / 8 bytes each to clear, scan and
// read out whatever they hold, so on many values with few facts the general path,
// whose cost goes with the facts, is the faster one.  For a program of one linear
// recursive rule, head = L head R with L and R products of input relations, and base
// rules of sum B, iteration k + 1 makes at most sum(L^k B R^k) derivations, in rows
// where L^k 1 is not zero: both are counted for kWalkSteps iterations by vectors of n
// floats -- (L^T)^k 1, R^k 1, L^k 1, each a pass over the facts.  Operations that
// depend on each other follow in launches of their own, about 3 us each.
// ---------------------------------------------------------------------------
constexpr int kWalkSteps = 16, kWalkOps = 8;
struct WalkOp {      // y[column] += x[row] (or the other way, back) over a link's facts;
  KeyCols K;         // with sum: *sum += x[row] z[column]
  int inv, back;
  const float *x, *z;
  float* y;
  double* sum;
};
struct WalkOps {
  WalkOp op[kWalkOps];
  Codes code;
};
__global__ void __launch_bounds__(256) k_bit_walks(const __grid_constant__ WalkOps W) {
  const WalkOp& P = W.op[blockIdx.y];
  const u64 stride = (u64)gridDim.x * blockDim.x;
  const u64 n = (P.K.n + 31) & ~31ull;  // whole warps
  double sum = 0.0;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const bool in = i < P.K.n;
    const u64 k = load_key(P.K.keys, P.K.key64, in ? i : P.K.n - 1);
    const u32 r = W.code((u32)field_of(k, P.K.shift[P.inv], P.K.width[P.inv]));
    const u32 c = W.code((u32)field_of(k, P.K.shift[P.inv ^ 1], P.K.width[P.inv ^ 1]));
    float v = in ? P.x[P.back ? c : r] : 0.0f;
    if (P.sum) {
      const float z = P.z[c];
      if (v != 0.0f && z != 0.0f) sum += (double)v * (double)z;  // (no infinity times 0)
      continue;
    }
    const u32 to = P.back ? r : c;
    int same;
    __match_all_sync(0xFFFFFFFFu, to, &same);
    if (same) {  // a hub's facts: one atomic a warp
#pragma unroll
      for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if (threadIdx.x & 31) v = 0.0f;
    }
    if (v != 0.0f) atomicAdd(P.y + to, v);
  }
  if (!P.sum) return;
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
  if ((threadIdx.x & 31) == 0 && sum != 0.0) atomicAdd(P.sum, sum);
}

struct WalkRows {
  const float* x[kWalkSteps + 1];
};
__global__ void __launch_bounds__(256) k_bit_walk_rows(const __grid_constant__ WalkRows W, u32 n, double* out) {
  const u32 stride = gridDim.x * blockDim.x;
  u32 c = 0;
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) c += W.x[blockIdx.y][i] != 0.0f;
  c = __reduce_add_sync(0xFFFFFFFFu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out + blockIdx.y, (double)c);
}

// ---------------------------------------------------------------------------
// planning
// ---------------------------------------------------------------------------
struct Link {
  u32 rel;
  int inv;   // 1: read from its second column to its first
  int atom;  // body position
};
struct Chain {
  u32 head;
  std::vector<Link> links;  // from head column 0 to head column 1
  int diag = 0;
  std::vector<int> order;   // links by body position: order[a] = link of body atom a
};

bool find_chain(const lob_engine& e, const RuleAst& R, Chain& C) {
  if (R.computes() || R.head.args.size() != 2 || R.body.empty() || R.body.size() > (size_t)kMaxChain) return false;
  const Term &hx = R.head.args[0], &hz = R.head.args[1];
  if (!hx.var || !hz.var || hx.v == hz.v) return false;
  std::vector<int> uses(R.var_names.size(), 0);
  for (const AtomAst& a : R.body) {
    if (a.args.size() != 2 || !a.args[0].var || !a.args[1].var || a.args[0].v == a.args[1].v) return false;
    uses[a.args[0].v]++;
    uses[a.args[1].v]++;
  }
  for (size_t v = 0; v < uses.size(); v++)
    if (uses[v] != ((u32)v == hx.v || (u32)v == hz.v ? 1 : 2)) return false;
  for (const FilterAst& F : R.filters) {  // only x != z or x == z, once
    if (F.prog || !F.a.var || !F.b.var || C.diag) return false;
    if (!((F.a.v == hx.v && F.b.v == hz.v) || (F.a.v == hz.v && F.b.v == hx.v))) return false;
    C.diag = F.eq ? 2 : 1;
  }
  C.head = R.head.rel;
  C.order.assign(R.body.size(), -1);
  u32 at = hx.v;
  for (size_t n = 0; n < R.body.size(); n++) {
    bool found = false;
    for (size_t i = 0; i < R.body.size() && !found; i++) {
      if (C.order[i] >= 0) continue;
      const u32 a = R.body[i].args[0].v, b = R.body[i].args[1].v;
      if (a != at && b != at) continue;
      C.order[i] = (int)C.links.size();
      C.links.push_back({R.body[i].rel, b == at, (int)i});
      at = b == at ? a : b;
      found = true;
    }
    if (!found) return false;
  }
  return at == hz.v;
}

bool chains_of(const lob_engine& e, std::vector<Chain>& out) {
  for (const RuleAst& R : e.rules) {
    Chain C;
    if (!find_chain(e, R, C)) return false;
    out.push_back(std::move(C));
  }
  return !out.empty();
}

// Store the derived relations transposed?  Costs of an iteration's products:
// one per scatter, one per derived relation read both ways (its transposed
// copy is kept too), half for the final transpose.
bool store_transposed(const lob_engine& e, const std::vector<Chain>& chains) {
  double cost[2] = {0, 0.5};
  for (int t = 0; t < 2; t++) {
    std::vector<char> both(e.rels.size(), 0);
    for (const Chain& C : chains) {
      bool recursive = false;
      for (const Link& l : C.links) recursive = recursive || e.rels[l.rel].idb;
      if (!recursive) continue;
      const Link& last = t ? C.links.front() : C.links.back();
      if (C.links.size() > 1 && !e.rels[last.rel].idb) cost[t] += 1;
      for (const Link& l : C.links)
        if (e.rels[l.rel].idb && l.inv != 0) both[l.rel] = 1;
    }
    for (char b : both) cost[t] += b;
  }
  return cost[1] < cost[0];
}

unsigned warp_grid(u64 tasks) {
  const u64 b = (tasks + kGatherWarps - 1) / kGatherWarps;
  return (unsigned)std::max<u64>(1, std::min<u64>(b, 152ull * 8));
}
unsigned block_grid(u64 tasks) { return (unsigned)std::max<u64>(1, std::min<u64>(tasks, 152ull * 8)); }
unsigned elem_grid(u64 n) { return (unsigned)std::max<u64>(1, std::min<u64>((n + 255) / 256, 152ull * 16)); }

KeyCols key_cols(const RelSt& r) {
  const ViewSt& V = r.views[0];
  KeyCols K{};
  K.keys = V.keys.p;
  K.key64 = V.lay.key64;
  K.n = V.n;
  for (int j = 0; j < 2; j++) {
    K.shift[j] = V.lay.shift[j];
    K.width[j] = V.lay.width[j];
  }
  return K;
}

}  // namespace

bool bit_eligible(const lob_engine& e) {
  // Options that ask for one of the general path's strategies get that path.
  if (!e.opt_bit_matrix || e.semiring != SR_UNIT || e.swidth) return false;
  if (!e.opt_packed_join || e.opt_warp_join != 1 || e.opt_bitmap_delta != 1 || e.opt_emit_filter != 1 ||
      !e.opt_cross_join || e.opt_join_index || e.opt_sort_algo || e.opt_max_cand < (1ull << 30))
    return false;
  if (e.rels.size() > (size_t)kMaxBitRels) return false;
  for (const RelSt& r : e.rels)
    if (r.idb && r.arity != 2) return false;
  std::vector<Chain> chains;
  if (!chains_of(e, chains)) return false;
  for (const Chain& C : chains)
    for (const Link& l : C.links)
      for (int c = 0; c < 2; c++)
        if (e.rels[l.rel].width[c] > 28) return false;
  return true;
}

namespace {

struct Run {
  lob_engine& e;
  BitRun& B;
  std::vector<Chain> chains;
  bool linear = true;      // every rule reads at most one derived atom
  u64 heavy_slots = 0;
  int n_temp = 0;
  std::vector<char> accumulates;  // per relation: some iteration has more than one product into it

  explicit Run(lob_engine& en) : e(en), B(*en.bit) {}

  void launch_check(const char* what) {
    e.after_launch(what);
    e.launches++;
  }

  // codes of the program's values; false when a matrix would be too large
  bool domain() {
    int width = 1;
    std::vector<char> used(e.rels.size(), 0);
    for (auto& C : chains) {
      used[C.head] = 1;
      for (auto& l : C.links) used[l.rel] = 1;
    }
    for (size_t r = 0; r < e.rels.size(); r++)
      if (used[r])
        for (int c = 0; c < 2; c++) width = std::max(width, e.rels[r].width[c]);
    // widths are bitlen(max + 1): all values are below 2^width
    u64 D = 1ull << width;
    if (D > kMaxValue) return false;
    B.mapped = false;
    if (D > 4096) {
      const u64 nw = D / 32;
      e.ensure(B.pres, nw * 4);
      e.ensure(B.pref, nw * 4);
      e.check(cudaMemsetAsync(B.pres.p, 0, nw * 4, e.stream), "values");
      for (size_t r = 0; r < e.rels.size(); r++)
        if (used[r] && e.rels[r].views[0].n) {
          const KeyCols K = key_cols(e.rels[r]);
          k_mark_values<<<elem_grid(K.n), 256, 0, e.stream>>>(K, B.pres.as<u32>());
          launch_check("values");
        }
      k_word_bits<<<elem_grid(nw), 256, 0, e.stream>>>(B.pres.as<u32>(), nw, B.pref.as<u32>());
      launch_check("values");
      e.ensure(e.scratch, scan_scratch_elems(nw) * 4 + 64);
      e.check(cudaMemsetAsync(e.counts.as<u64>() + 1, 0, sizeof(u64), e.stream), "values");
      exclusive_scan<u32, u32>(B.pref.as<u32>(), B.pref.as<u32>(), nw, reinterpret_cast<u32*>(e.counts.as<u64>() + 1),
                               e.scratch.as<u32>(), e.stream);
      e.after_launch("values");
      e.launches += scan_launches(nw);
      D = std::max<u64>(1, e.read_u64(e.counts.as<u64>() + 1) & 0xFFFFFFFFull);
      u64 top = 0;
      for (size_t r = 0; r < e.rels.size(); r++)
        if (used[r])
          for (int c = 0; c < 2; c++) top = std::max<u64>(top, e.rels[r].maxv[c]);
      B.mapped = D != top + 1;  // else every value up to the largest occurs: it is its own code
    }
    B.rows = (u32)D;
    B.words = (u32)((D + 127) / 128 * 4);
    if ((u64)B.rows * B.words * 4 > kMatrixBytes) return false;
    // A matrix per derived relation for F, D and D', one for N where an iteration has
    // several products, transposed copies where it is read both ways; the temporaries.
    u64 matrices = n_temp;
    for (size_t r = 0; r < e.rels.size(); r++)
      if (e.rels[r].idb) matrices += 3 + accumulates[r] + (B.rel[r].need_t ? (linear ? 1 : 2) : 0);
    if (matrices * mat_bytes() > kRunBytes || !fills()) return false;
    if (B.mapped) {
      const u64 nw = (1ull << width) / 32;
      e.ensure(B.dict, (u64)B.rows * 4);
      k_code_values<<<elem_grid(nw), 256, 0, e.stream>>>(B.pres.as<u32>(), B.pref.as<u32>(), nw, B.dict.as<u32>());
      launch_check("values");
    }
    return true;
  }

  Codes codes() const {
    Codes c{};
    if (B.mapped) {
      c.pres = B.pres.as<u32>();
      c.pref = B.pref.as<u32>();
    }
    return c;
  }

  // Up to kSureRows values (a matrix is as large as L2 then) the matrices are taken as
  // they are; up to kSureRows2 when a rule joins derived relations (an index row is
  // scanned once for every 128 words of the result).  Beyond, a program whose
  // derivations can be counted (k_bit_walks) runs on matrices when they exceed a 256th
  // of the pairs or still grow, or when the time estimated for them is the lower one;
  // any other one starts on the general path, which gives up in favour of the matrices
  // when an iteration is about to derive a 32nd of the pairs (bit_watch).
  // Measured (GB300, whole passes in ms, general path / bit matrices).  Left-recursive
  // closure: a random tree of 20,000 nodes 1.6 / 1.1, 35,000 1.9 / 2.2, 90,000 2.7 / 9.1;
  // disjoint edges 0.42 / 0.49, 0.59 / 0.71, 0.38 / 2.4; 0.9 random edges a node 35,000 6.2
  // / 2.6, 90,000 7.3 / 4.5; 60,000 of them on 50,000 nodes (2.5e8 facts) 72 / 11.
  // Right-recursive: trees 35,000 1.9 / 1.1, 90,000 2.6 / 2.0; chains of 40 35,000 4.9 /
  // 3.6, 50,000 5.0 / 5.9, 90,000 7.0 / 14.  Same generation: trees of 200 nodes 35,000 2.0
  // / 1.9, 50,000 2.2 / 2.8, 90,000 3.0 / 6.5; one tree of 50,000 (9.1e8 facts) 29 / 9.7.
  // p.p closure: trees 12,000 1.6 / 1.2, 20,000 1.7 / 2.1, 90,000 3.4 / 55; chains 10,000
  // 2.1 / 2.1, 14,000 2.1 / 3.7, 90,000 4.2 / 275; 24,000 random edges on 20,000 nodes
  // 641 / 22.  The general path with the walks before it takes 0.1 ms more than alone.
  static constexpr u32 kSureRows = 32768, kSureRows2 = 12288;
  bool fills() {
    if (e.bit_force || B.rows <= (linear ? kSureRows : kSureRows2)) return true;
    e.bit_watch = B.rows;
    const Chain* rec = nullptr;
    size_t bases = 0;
    for (const Chain& C : chains) {
      const bool derived = std::any_of(C.links.begin(), C.links.end(), [&](const Link& l) { return e.rels[l.rel].idb; });
      if (C.head != chains[0].head || (derived && rec)) return false;
      if (derived) rec = &C;
      else bases++;
    }
    if (!linear || bases > 4) return false;
    return many_walks(rec);
  }
  bool many_walks(const Chain* rec) {
    const u32 head = chains[0].head;
    const int steps = rec ? kWalkSteps : 0;
    std::vector<std::vector<Link>> base;
    for (const Chain& C : chains)
      if (&C != rec) base.push_back(C.links);
    if (e.rels[head].views[0].n) base.push_back({Link{head, 0, 0}});
    std::vector<Link> left, right;
    for (bool past = false; rec && left.size() + right.size() + 1 < rec->links.size();) {
      const Link& l = rec->links[left.size() + right.size() + past];
      if (l.rel == head) past = true;
      else (past ? right : left).push_back(l);
    }
    size_t inner = 0;
    for (auto& b : base) inner += b.size() - 1;
    const std::vector<Link>& row_links = B.transposed ? right : left;  // of the matrices as stored
    const u64 n = (B.rows + 31) & ~31u;
    const u64 vectors = 1 + steps * (left.size() + right.size() + row_links.size()) + (steps + 1) * inner;
    const u64 pad = 128;  // floats: the derivations and live rows of each step
    e.ensure(e.scratch, (pad + vectors * n) * 4);
    e.check(cudaMemsetAsync(e.scratch.p, 0, (pad + vectors * n) * 4, e.stream), "walks");
    double* sums = e.scratch.as<double>();
    float* next = e.scratch.as<float>() + pad;
    struct Vec { const float* p; int at; };  // a vector, and the launch before which it is complete
    std::vector<std::vector<WalkOp>> launches;
    const auto put = [&](int at, WalkOp op) {
      if ((int)launches.size() <= at) launches.resize(at + 1);
      launches[at].push_back(op);
    };
    const auto apply = [&](const Link& l, Vec v, int back) {
      WalkOp op{key_cols(e.rels[l.rel]), l.inv, back, v.p, nullptr, next, nullptr};
      if (op.K.n) put(v.at, op);
      next += n;
      return Vec{op.y, v.at + 1};
    };
    const Vec ones{next, 0};
    fill_f32(next, B.rows, 1.0f, e.stream);
    next += n;
    Vec a = ones, b = ones, live = ones;
    WalkRows rows{};
    std::vector<double> s(2 * (kWalkSteps + 1));
    size_t done = 0;
    int ran = 0, live_done = 0;
    const double many = (double)B.rows * B.rows / 256.0;
    for (int k = 0; k <= steps; k++) {
      if (k) {
        for (const Link& l : left) a = apply(l, a, 0);
        for (size_t i = right.size(); i--;) b = apply(right[i], b, 1);
        if (B.transposed)
          for (const Link& l : right) live = apply(l, live, 0);
        else
          for (size_t i = left.size(); i--;) live = apply(left[i], live, 1);
      }
      rows.x[k] = live.p;
      for (auto& links : base) {
        Vec c = a;
        for (size_t i = 0; i + 1 < links.size(); i++) c = apply(links[i], c, 0);
        WalkOp op{key_cols(e.rels[links.back().rel]), links.back().inv, 0, c.p, b.p, nullptr, sums + k};
        if (op.K.n) put(std::max(c.at, b.at), op);
      }
      if (k != 5 && k != steps) continue;
      // the first few steps alone may show the end, or that there are many
      for (; done < launches.size(); done++)
        for (size_t q = 0; q < launches[done].size(); q += kWalkOps) {
          WalkOps W{};
          W.code = codes();
          const unsigned m = (unsigned)std::min<size_t>(kWalkOps, launches[done].size() - q);
          u64 most = 0;
          for (unsigned i = 0; i < m; i++) {
            W.op[i] = launches[done][q + i];
            most = std::max(most, W.op[i].K.n);
          }
          ProfScope ps("bit_walks", 0, e.stream);
          k_bit_walks<<<dim3(elem_grid(most), m), 256, 0, e.stream>>>(W);
          launch_check("walks");
        }
      WalkRows fresh{};
      std::copy(rows.x + live_done, rows.x + k + 1, fresh.x);
      k_bit_walk_rows<<<dim3(elem_grid(n) / 4 + 1, k + 1 - live_done), 256, 0, e.stream>>>(fresh, (u32)n,
                                                                                       sums + kWalkSteps + 1 + live_done);
      launch_check("walks");
      live_done = k + 1;
      e.check(cudaMemcpyAsync(e.pinned, sums, s.size() * 8, cudaMemcpyDeviceToHost, e.stream), "walks");
      e.sync();
      std::memcpy(s.data(), e.pinned, s.size() * 8);
      ran = k;
      if (s[k] == 0.0 || !(std::accumulate(s.begin(), s.begin() + k + 1, 0.0) <= many)) break;
      a.at = b.at = live.at = (int)done;  // what follows goes to launches of its own
    }
    // iterations, derivations and live rows to the end; past the last step as if their
    // decline over the last four went on to zero, 64 steps at most
    double its = 0, total = 0, touched = 0;
    for (int k = 0; k <= ran; k++) {
      its += k == 0 || s[k] > 0.0;
      total += s[k];
      touched += std::min(s[k], s[kWalkSteps + 1 + k]);
    }
    if (!(total <= many)) return true;
    if (ran > 4 && s[ran] > 0.0) {
      if (s[ran] > 1.1 * s[ran - 4]) return true;
      const double fall = (s[ran - 4] - s[ran]) / 4;
      const double tail = s[ran] < 64.0 * fall ? s[ran] / fall : 64.0;
      its += tail;
      total += s[ran] * tail / 2;
      touched += std::min(s[ran], s[kWalkSteps + 1 + ran]) * tail / 2;
    }
    // Seconds.  Matrices: clearing, scanning, reading out (and turning back), launches,
    // and each live row read and written by each product.  The general path: its
    // launches and host waits, its derivations, and for keys of 32 bits a filter's
    // clearing, which spares it a sort in every iteration.
    const double row = B.words * 4.0 / 6.8e12;  // a row's time at the copy rate
    const double products = rec ? rec->links.size() - 1.0 : 1.0;
    const double on_bits = (B.transposed ? 13.0 : 7.5) * B.rows * row + (3.0 + products) * touched * row +
                           its * (15e-6 + 18e-6 * products);
    const double general = (B.rows > 65536 ? its * 160e-6 : 200e-6 + its * 120e-6) + total * 50e-12;
    return on_bits < general;
  }

  // a link as the stored orientation reads it
  Link oriented(const Link& l) const { return B.transposed ? Link{l.rel, !l.inv, l.atom} : l; }
  std::vector<Link> links_of(const Chain& C) const {
    std::vector<Link> v;
    for (auto& l : C.links) v.push_back(oriented(l));
    if (B.transposed) std::reverse(v.begin(), v.end());
    return v;
  }
  bool stored_way(const Link& l) const { return l.inv == (B.transposed ? 1 : 0); }

  BCsr csr(const Link& l) const {
    const BitRel& R = B.rel[l.rel];
    const BitCsr& C = R.csr[l.inv];
    BCsr c{};
    c.ptr = C.ptr;
    c.col = C.col.as<u32>();
    c.heavy = C.heavy;
    c.n_heavy = C.heavy + C.heavy_cap;
    return c;
  }
  void build_csr(const Link& l) {
    BitCsr& C = B.rel[l.rel].csr[l.inv];
    if (C.built) return;
    C.built = true;
    const KeyCols K = key_cols(e.rels[l.rel]);
    const u64 D = B.rows;
    C.heavy_cap = (u32)(K.n / kHeavyRow + 1);
    // lengths (their scan: ptr), fill positions, column flags, heavy rows and their number
    const u64 words = (D + 1) + D + D + C.heavy_cap + 1;
    e.ensure(C.zeroed, words * 4);
    e.ensure(C.col, std::max<u64>(K.n, 1) * 4);
    e.check(cudaMemsetAsync(C.zeroed.p, 0, words * 4, e.stream), "rows");
    C.ptr = C.zeroed.as<u32>();
    C.used = C.ptr + D + 1;
    C.colflag = C.used + D;
    C.heavy = C.colflag + D;
    if (!K.n) return;
    ProfScope ps("bit_rows", K.n * (K.key64 ? 8.0 : 4.0) * 2.0 + K.n * 4.0 + D * 12.0, e.stream);
    k_csr_count<<<elem_grid(K.n), 256, 0, e.stream>>>(K, codes(), l.inv, C.ptr, C.colflag);
    launch_check("rows");
    e.ensure(e.scratch, scan_scratch_elems(D + 1) * 4 + 64);
    exclusive_scan<u32, u32>(C.ptr, C.ptr, D + 1, nullptr, e.scratch.as<u32>(), e.stream);
    e.after_launch("rows");
    e.launches += scan_launches(D + 1);
    k_csr_fill<<<elem_grid(K.n), 256, 0, e.stream>>>(K, codes(), l.inv, C.ptr, C.used, C.col.as<u32>(),
                                                     C.heavy, C.heavy + C.heavy_cap);
    launch_check("rows");
  }

  void build_filled(const Link& l) {
    BitCsr& C = B.rel[l.rel].csr[l.inv];
    if (C.filled.p) return;
    e.ensure(C.filled, (u64)B.words * 4);
    k_filled_rows<<<warp_grid(B.words), 256, 0, e.stream>>>(C.ptr, B.rows, B.words, C.filled.as<u32>());
    launch_check("rows");
  }

  u64 mat_bytes() const { return (u64)B.rows * B.words * 4; }

  void allocate() {
    const u64 mb = mat_bytes(), D = B.rows;
    for (size_t r = 0; r < e.rels.size(); r++) {
      BitRel& R = B.rel[r];
      if (!e.rels[r].idb) continue;
      e.ensure(R.full, mb);
      e.check(cudaMemsetAsync(R.full.p, 0, mb, e.stream), "bit matrix");
      for (int b = 0; b < 2; b++) e.ensure(R.recent[b], mb);
      // row counts of F, D, D' (and the transposed copies), flags: cleared as one
      const int n_counts = 3 + (accumulates[r] ? 1 : 0) + (R.need_t ? (linear ? 1 : 2) : 0);
      e.ensure(R.counts, n_counts * D * 4);
      e.check(cudaMemsetAsync(R.counts.p, 0, n_counts * D * 4, e.stream), "bit matrix");
      u32* c = R.counts.as<u32>();
      R.fcnt = c;
      R.rcnt[0] = c + D;
      R.rcnt[1] = c + 2 * D;
      c += 3 * D;
      if (accumulates[r]) {
        e.ensure(R.acc, mb);
        e.check(cudaMemsetAsync(R.acc.p, 0, mb, e.stream), "bit matrix");
        R.aflag = c;
        c += D;
      }
      if (R.need_t) {
        e.ensure(R.trecent, mb);
        R.trcnt = c;
        c += D;
        if (!linear) {
          e.ensure(R.tfull, mb);
          e.check(cudaMemsetAsync(R.tfull.p, 0, mb, e.stream), "bit matrix");
          R.tfcnt = c;
        }
      }
    }
    for (int i = 0; i < n_temp; i++) {
      e.ensure(B.temp[i], mb);
      e.ensure(B.tbag[i], D * 8);
    }
    // what finish() needs is taken here as well: a request refused after the
    // iterations would throw their work away
    for (size_t r = 0; r < e.rels.size(); r++)
      if (e.rels[r].idb) e.ensure(B.rel[r].off, (D + 1) * 8);
    e.ensure(e.scratch, scan_scratch_elems(D) * 8 + 64);
    e.ensure(B.state, kAllSlots * 8);
    e.check(cudaMemsetAsync(B.state.p, 0, kAllSlots * 8, e.stream), "bit state");
    if (listed()) {
      e.ensure(B.list, D * 4);
      e.ensure(B.hlist, D * 4);
      e.ensure(B.slist, D * 4);
    }
  }

  // rows x 128-word chunks beyond about two waves of warps: products list the
  // rows they have work for first
  bool listed() const { return (u64)B.rows * ((B.words + 127) / 128) > 152ull * 8 * kGatherWarps * 2; }


  // the operand of a link: derived relations by which set the arm reads
  BMat matrix(const Link& l, bool recent, int cur) const {
    const BitRel& R = B.rel[l.rel];
    BMat m{};
    const bool st = stored_way(l);
    const DevBuf& bits = recent ? (st ? R.recent[cur] : R.trecent) : (st ? R.full : R.tfull);
    m.bits = bits.as<u32>();
    m.cnt = recent ? (st ? R.rcnt[cur] : R.trcnt) : (st ? R.fcnt : R.tfcnt);
    return m;
  }

  double words_before = 0;
  void profile_before() {
    if (g_prof) words_before = (double)e.read_u64(B.state.as<u64>() + B_WORDS);
  }
  void profile_after() {
    if (g_prof) g_prof->add_last_bytes(4.0 * ((double)e.read_u64(B.state.as<u64>() + B_WORDS) - words_before));
  }

  // One arm: the chain's product with the recent set at link `delta` (body
  // position), full sets at the other derived atoms (recent ones too in a
  // linear program, where there are none).  `commit`: it is the last product
  // into its head and no product of this iteration reads F.
  void run_arm(const Chain& C, int delta, bool all_full, bool commit, int cur) {
    const std::vector<Link> L = links_of(C);
    const int m = (int)L.size();
    BOp base{};
    base.rows = B.rows;
    base.words = B.words;
    base.state = B.state.as<u64>();
    if (!all_full)
      for (const Link& l : L)
        if (e.rels[l.rel].idb && l.atom < delta) base.skip[base.n_skip++] = (int)l.rel;
    auto recent = [&](const Link& l) { return linear || (!all_full && l.atom == delta); };
    BMat cur_m{};
    BCsr cur_c{};
    bool bits = e.rels[L[m - 1].rel].idb;
    if (bits) cur_m = matrix(L[m - 1], recent(L[m - 1]), cur);
    else cur_c = csr(L[m - 1]);
    for (int i = m - 2; i >= -1; i--) {  // i == -1: a single atom, copied
      if (i == -1 && m > 1) break;
      BOp P = base;
      P.mb = cur_m;
      P.mc = cur_c;
      int ik = I_IDENT;
      if (i >= 0) {
        if (e.rels[L[i].rel].idb) {
          ik = I_BITS;
          P.ib = matrix(L[i], recent(L[i]), cur);
        } else {
          ik = I_CSR;
          P.ic = csr(L[i]);
        }
      }
      const bool last = i <= 0;
      if (!last) {
        const int t = i % 2;
        P.out = B.temp[t].as<u32>();
        P.obag = B.tbag[t].as<u64>();
        // rows that the next index matrix never lists need not be formed
        if (!e.rels[L[i - 1].rel].idb) P.need = B.rel[L[i - 1].rel].csr[L[i - 1].inv].colflag;
      } else {
        set_head(P, C.head, cur, commit);
        P.diag = C.diag;
      }
      if (!bits && ik == I_BITS) {
        P.filled = B.rel[L[m - 1].rel].csr[L[m - 1].inv].filled.as<u32>();
      }
      product(P, ik, bits);
      cur_m = BMat{};
      cur_m.bits = P.out;
      cur_m.bag = P.obag;
      bits = true;
    }
  }

  void set_head(BOp& P, u32 head, int cur, bool commit) {
    BitRel& H = B.rel[head];
    P.acc = H.acc.as<u32>();
    P.aflag = H.aflag;
    P.commit = commit;
    P.full = H.full.as<u32>();
    P.next = H.recent[cur ^ 1].as<u32>();
    P.ncnt = H.rcnt[cur ^ 1];
    P.fcnt = H.fcnt;
    P.n_new = B.state.as<u64>() + rel_slot((int)head, 2);
  }

  int n_lists = 0;  // products of the current iteration that listed their rows
  std::vector<BStep>* record = nullptr;  // the loop's steps are being collected, not launched
  void add_step(int kind, int ik, const BOp* P, const BTrans* X) {
    BStep S;
    std::memset(&S, 0, sizeof(S));
    S.kind = kind;
    S.ik = ik;
    if (P) S.P = *P;
    if (X) S.X = *X;
    record->push_back(S);
  }

  void product(BOp P, int ik, bool bits) {
    const u32 chunks = (P.words + 127) / 128;
    if (record) {
      add_step(bits ? K_GATHER : K_SCATTER, ik, &P, nullptr);
      return;
    }
    profile_before();
    if (listed() && n_lists < kMaxLists) {
      P.list = B.list.as<u32>();
      P.hlist = B.hlist.as<u32>();
      if (bits && ik == I_CSR && P.words > kWide * 128) P.slist = B.slist.as<u32>();
      P.n_list = B.state.as<u64>() + kStateSlots + 3 * n_lists++;
      {
        ProfScope ps("bit_active", P.rows * 12.0, e.stream);
        const unsigned g = warp_grid((P.rows + 31) / 32);
        if (ik == I_IDENT) k_bit_active<I_IDENT><<<g, 256, 0, e.stream>>>(P, bits);
        else if (ik == I_CSR) k_bit_active<I_CSR><<<g, 256, 0, e.stream>>>(P, bits);
        else k_bit_active<I_BITS><<<g, 256, 0, e.stream>>>(P, bits);
      }
      launch_check("bit rows");
    }
    if (bits) {
      {
        ProfScope ps("bit_gather", 0, e.stream);
        if (ik == I_IDENT) k_bit_gather<I_IDENT><<<warp_grid((u64)P.rows * chunks), 256, 0, e.stream>>>(P);
        else if (ik == I_CSR) {
          if (P.slist) {
            k_bit_gather_wide<<<warp_grid((u64)P.rows * chunks), 256, 0, e.stream>>>(P);
            e.launches++;
          }
          k_bit_gather<I_CSR><<<warp_grid((u64)P.rows * chunks), 256, 0, e.stream>>>(P);
        } else k_bit_gather<I_BITS><<<block_grid((u64)P.rows * chunks), 256, 0, e.stream>>>(P);
      }
      launch_check("bit gather");
    } else {
      {
        ProfScope ps("bit_scatter", 0, e.stream);
        const size_t sm = (size_t)P.words * 4;
        if (ik == I_IDENT) k_bit_scatter<I_IDENT><<<block_grid(P.rows), 256, sm, e.stream>>>(P);
        else if (ik == I_CSR) k_bit_scatter<I_CSR><<<block_grid(P.rows), 256, sm, e.stream>>>(P);
        else k_bit_scatter<I_BITS><<<block_grid(P.rows), 256, sm, e.stream>>>(P);
      }
      launch_check("bit scatter");
    }
    profile_after();
  }

  void transpose(const BTrans& X) {
    {
      ProfScope ps("bit_transpose", 2.0 * mat_bytes(), e.stream);
      const u64 tiles = (u64)((B.rows + 255) / 256) * ((B.words + 7) / 8);
      k_bit_transpose<<<block_grid(tiles), 256, 0, e.stream>>>(X);
    }
    launch_check("bit transpose");
  }

  void transpose_recent(int cur, u64* state) {
    for (size_t r = 0; r < e.rels.size(); r++) {
      BitRel& R = B.rel[r];
      if (!e.rels[r].idb || !R.need_t) continue;
      BTrans X{};
      X.src.bits = R.recent[cur].as<u32>();
      X.src.cnt = R.rcnt[cur];
      X.rows = B.rows;
      X.words = B.words;
      X.dst = R.trecent.as<u32>();
      X.dcnt = R.trcnt;
      X.full = R.tfull.as<u32>();
      X.fcnt = R.tfcnt;
      X.state = state;
      if (record) add_step(K_TRANSPOSE, 0, nullptr, &X);
      else transpose(X);
    }
  }

  BEnd end_of(u32 max_iters, int cur) {
    BEnd E{};
    E.rows = B.rows;
    E.max_iters = max_iters;
    E.state = B.state.as<u64>();
    for (size_t r = 0; r < e.rels.size(); r++) {
      if (!e.rels[r].idb) continue;
      const int i = E.n_rel++;
      BitRel& R = B.rel[r];
      E.rel[i] = (int)r;
      E.old_cnt[i] = R.rcnt[cur];
      E.aflag[i] = R.aflag;
      E.tcnt[i] = R.need_t ? R.trcnt : nullptr;
    }
    return E;
  }

  // the products of one iteration (k >= 1) on recent buffers `cur`; their results
  // go to cur ^ 1
  void products(u32 k, int cur) {
    // the arms of this iteration: in the first, every loaded fact is recent, so
    // the arm of each rule's first atom covers the rule; later only derived
    // atoms have recent facts
    struct ArmRef { const Chain* c; int delta; };
    std::vector<ArmRef> arms;
    for (auto& C : chains) {
      if (k == 1) {
        bool empty = false;
        for (auto& l : C.links) empty = empty || !e.rels[l.rel].views[0].n;
        if (!empty) arms.push_back({&C, 0});
        continue;
      }
      for (size_t a = 0; a < C.order.size(); a++)
        if (e.rels[C.links[C.order[a]].rel].idb) arms.push_back({&C, (int)a});
    }
    std::vector<int> left(e.rels.size(), 0);
    n_lists = 0;
    for (auto& a : arms) left[a.c->head]++;
    for (auto& a : arms) {
      const bool commit = linear && --left[a.c->head] == 0;
      run_arm(*a.c, a.delta, k == 1, commit, cur);
    }
    if (!linear) {
      std::vector<char> has(e.rels.size(), 0);
      for (auto& a : arms) has[a.c->head] = 1;
      for (size_t r = 0; r < e.rels.size(); r++) {
        if (!has[r]) continue;
        BOp P{};
        P.rows = B.rows;
        P.words = B.words;
        P.state = B.state.as<u64>();
        set_head(P, (u32)r, cur, true);
        const u32 chunks = (P.words + 127) / 128;
        if (record) {
          add_step(K_COMMIT, 0, &P, nullptr);
          continue;
        }
        profile_before();
        {
          ProfScope ps("bit_commit", 0, e.stream);
          k_bit_commit<<<warp_grid((u64)P.rows * chunks), 256, 0, e.stream>>>(P);
        }
        launch_check("bit commit");
        profile_after();
      }
    }
  }

  void iteration(u32 k, u32 max_iters, int cur) {
    products(k, cur);
    const BEnd E = end_of(max_iters, cur);
    k_bit_end<<<std::min(elem_grid(B.rows), 152u), 256, 0, e.stream>>>(E);
    launch_check("bit end");
    transpose_recent(cur ^ 1, B.state.as<u64>());
  }

  bool run(u32 max_iters, u32& k, u64& new_facts, int* rc) {
    if (!chains_of(e, chains)) return false;
    B.transposed = store_transposed(e, chains);
    B.rel.clear();
    B.rel.resize(e.rels.size());
    accumulates.assign(e.rels.size(), 0);
    std::vector<int> first(e.rels.size(), 0), later(e.rels.size(), 0);
    for (auto& C : chains) {
      int idb = 0;
      for (auto& l : C.links)
        if (e.rels[l.rel].idb) {
          idb++;
          if (!stored_way(oriented(l))) B.rel[l.rel].need_t = true;
        }
      if (idb > 1) linear = false;
      first[C.head]++;
      later[C.head] += idb;
      if ((int)C.links.size() > 2) n_temp = std::max(n_temp, std::min(2, (int)C.links.size() - 2));
    }
    if (n_temp) n_temp = 2;
    for (size_t r = 0; r < e.rels.size(); r++) {
      // the first iteration's rules that have facts, and each later iteration's arms
      int f = 0;
      for (auto& C : chains) {
        bool empty = false;
        for (auto& l : C.links) empty = empty || !e.rels[l.rel].views[0].n;
        f += C.head == r && !empty;
      }
      accumulates[r] = e.rels[r].idb && (!linear || f > 1 || later[r] > 1);
    }
    if (!domain()) return false;
    allocate();
    for (auto& C : chains)
      for (size_t i = 0; i < C.links.size(); i++) {
        const Link l = oriented(C.links[i]);
        if (e.rels[l.rel].idb) continue;
        build_csr(l);
        // the operand of a scatter by bits: which of its rows hold something
        const size_t n = C.links.size(), before = B.transposed ? i + 1 : i - 1;
        if (n > 1 && i == (B.transposed ? 0 : n - 1) && e.rels[C.links[before].rel].idb) build_filled(l);
      }
    std::vector<u64> h(kStateSlots, 0);
    bool loaded = false;
    for (size_t r = 0; r < e.rels.size(); r++) {
      if (!e.rels[r].idb || !e.rels[r].views[0].n) continue;
      loaded = true;
      BitRel& R = B.rel[r];
      const KeyCols K = key_cols(e.rels[r]);
      e.check(cudaMemsetAsync(R.recent[0].p, 0, mat_bytes(), e.stream), "bit matrix");
      k_set_facts<<<elem_grid(K.n), 256, 0, e.stream>>>(K, codes(), B.transposed, B.words, R.full.as<u32>(),
                                                        R.recent[0].as<u32>(), R.rcnt[0], R.fcnt);
      launch_check("bit facts");
      h[rel_slot((int)r, 0)] = h[rel_slot((int)r, 1)] = K.n;
    }
    if (loaded) {
      e.check(cudaMemcpyAsync(B.state.p, h.data(), h.size() * 8, cudaMemcpyHostToDevice, e.stream), "bit state");
      e.sync();  // h goes out of scope with the run; the copy is from pageable memory
      transpose_recent(0, nullptr);
    }
    if ((u64)B.rows * ((B.words + 127) / 128) <= kLoopTasks && !g_prof) {
      loop_launch(max_iters);
      read_state();
      return done(k, new_facts, rc);
    }
    // Iterations are queued in groups without waiting: one that follows the
    // fixpoint sees the done flag and does nothing (about 2 us a launch), which
    // is cheaper than a host wait per iteration (about 10 us).
    u32 queued = 0;
    for (u32 group = 4;; group = std::min(16u, group * 2)) {
      for (u32 i = 0; i < group && queued < max_iters; i++, queued++) iteration(queued + 1, max_iters, (int)(queued & 1));
      read_state();
      if (e.pinned[B_DONE] || queued >= max_iters) break;
    }
    return done(k, new_facts, rc);
  }

  void read_state() {
    e.check(cudaMemcpyAsync(e.pinned, B.state.p, kReadSlots * 8, cudaMemcpyDeviceToHost, e.stream), "bit state");
    e.sync();
    if (e.pinned[kStateSlots] >> 32)
      throw LobError(LOB_E_TIMEOUT, "a bounded wait of the bit-matrix loop gave up; the run's results are invalid");
  }

  // the first iteration's steps, then those of later ones by recent buffer, and the
  // transposes after them
  void loop_launch(u32 max_iters) {
    std::vector<BStep> steps, after;
    BLoop L;
    std::memset(&L, 0, sizeof(L));
    record = &steps;
    for (int i = 0; i < 3; i++) {
      L.first[i] = (int)steps.size();
      products(i == 0 ? 1 : 2, i == 1 ? 1 : 0);
    }
    L.first[3] = (int)steps.size();
    record = &after;
    for (int b = 0; b < 2; b++) {
      L.after_first[b] = (int)after.size();
      transpose_recent(b, B.state.as<u64>());
    }
    L.after_first[2] = (int)after.size();
    record = nullptr;
    const size_t n_steps = steps.size();
    steps.insert(steps.end(), after.begin(), after.end());
    e.ensure(B.steps, std::max<size_t>(steps.size(), 1) * sizeof(BStep));
    e.check(cudaMemcpyAsync(B.steps.p, steps.data(), steps.size() * sizeof(BStep), cudaMemcpyHostToDevice, e.stream), "steps");
    L.steps = B.steps.as<BStep>();
    L.after = B.steps.as<BStep>() + n_steps;
    for (int b = 0; b < 2; b++) L.end[b] = end_of(max_iters, b);
    L.state = B.state.as<u64>();
    L.bar = reinterpret_cast<u32*>(B.state.as<u64>() + kStateSlots);
    const u64 tasks = (u64)B.rows * ((B.words + 127) / 128);
    const unsigned blocks = (unsigned)std::max<u64>(1, std::min<u64>((tasks + kGatherWarps - 1) / kGatherWarps, 4ull * e.sms));
    const size_t sm = (size_t)B.words * 4;
    void* args[] = {&L};
    {
      ProfScope ps("bit_loop", 0, e.stream);
      e.check(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_bit_loop), dim3(blocks), dim3(256), args, sm, e.stream),
              "bit loop");
    }
    launch_check("bit loop");
  }

  // The run's results become the engine's only after the last step that can fail:
  // until then the relations hold their loaded facts, which the general path starts
  // from when this one gives up.
  bool done(u32& k, u64& new_facts, int* rc) {
    const std::vector<u64> s(e.pinned, e.pinned + kStateSlots);
    finish();
    *rc = s[B_DONE] == 1 ? LOB_OK : LOB_E_MAXITER;
    k = (u32)s[B_ITER];
    new_facts = s[B_NEW];
    e.cand_emitted = s[B_CAND];
    for (size_t r = 0; r < e.rels.size(); r++)
      if (e.rels[r].idb) e.rels[r].views[0].n = s[rel_slot((int)r, 0)];
    return true;
  }

  // results in row order, with each row's offset
  void finish() {
    const u64 D = B.rows;
    for (size_t r = 0; r < e.rels.size(); r++) {
      BitRel& R = B.rel[r];
      if (!e.rels[r].idb) continue;
      if (B.transposed) {
        BTrans X{};
        X.src.bits = R.full.as<u32>();
        X.src.cnt = R.fcnt;
        X.rows = B.rows;
        X.words = B.words;
        X.dst = R.recent[0].as<u32>();
        transpose(X);
        std::swap(R.full, R.recent[0]);
        {
          ProfScope ps("bit_counts", (double)mat_bytes(), e.stream);
          k_row_counts<<<warp_grid(D), 256, 0, e.stream>>>(R.full.as<u32>(), B.rows, B.words, R.fcnt);
        }
        launch_check("bit counts");
      }
      exclusive_scan<u32, u64>(R.fcnt, R.off.as<u64>(), D, R.off.as<u64>() + D, e.scratch.as<u64>(), e.stream);
      e.after_launch("bit offsets");
      e.launches += scan_launches(D);
      for (DevBuf* b : {&R.recent[0], &R.recent[1], &R.counts, &R.acc, &R.trecent, &R.tfull}) e.release(*b);
    }
    for (int i = 0; i < 2; i++) {
      e.release(B.temp[i]);
      e.release(B.tbag[i]);
    }
  }
};

}  // namespace

bool bit_run(lob_engine& e, u32 max_iters, u32& k, u64& new_facts, int* rc) {
  e.bit.reset(new BitRun());
  e.bit_watch = 0;
  try {
    Run R(e);
    if (R.run(max_iters, k, new_facts, rc)) {
      e.bit->on = true;
      return true;
    }
  } catch (const LobError& x) {
    bit_release(e);
    if (x.code != LOB_E_OOM) throw;
    return false;  // the general path may need less
  }
  bit_release(e);
  return false;
}

bool bit_blow_up(const lob_engine& e) {
  const double n = (double)e.bit_watch;
  double next = 0.0;
  for (auto& p : e.plans)
    for (auto& A : p.arms) {
      const auto& body = p.ast.body;
      if (!e.rels[body[A.delta].rel].idb) continue;
      double d = (double)e.rels[body[A.delta].rel].n_recent;
      for (size_t i = 0; i < body.size(); i++)
        if ((int)i != A.delta) d *= (double)e.rels[body[i].rel].views[0].n / n;
      next += d;
    }
  return next > n * n / 32.0;
}

void bit_release(lob_engine& e) {
  if (!e.bit) return;
  BitRun& B = *e.bit;
  for (DevBuf* b : {&B.pres, &B.pref, &B.dict, &B.state, &B.steps, &B.list, &B.hlist, &B.slist, &B.temp[0], &B.temp[1], &B.tbag[0], &B.tbag[1]}) e.release(*b);
  for (BitRel& R : B.rel) {
    for (DevBuf* b : {&R.full, &R.recent[0], &R.recent[1], &R.counts, &R.acc, &R.trecent, &R.tfull, &R.off}) e.release(*b);
    for (BitCsr& C : R.csr)
      for (DevBuf* b : {&C.zeroed, &C.col, &C.filled}) e.release(*b);
  }
  e.bit.reset();
}

void bit_read(lob_engine& e, u32 rel, u32* cols, u64 stride, float* tags, u32* samples) {
  BitRun& B = *e.bit;
  BitRel& R = B.rel[rel];
  const u64 n = e.rels[rel].views[0].n;
  ProfScope ps("bit_read", (double)B.rows * B.words * 4 + n * (8.0 + (tags ? 4.0 : 0.0) + (samples ? 4.0 : 0.0)), e.stream);
  k_bit_read<<<warp_grid(B.rows), 256, 0, e.stream>>>(R.full.as<u32>(), B.rows, B.words, R.off.as<u64>(),
                                                      B.mapped ? B.dict.as<u32>() : nullptr, cols, cols + stride, tags,
                                                      samples);
}
