// Linear recursion of tagged programs: every iteration after the first in one
// cooperative launch.
//
// A derived relation whose recursive rules read one derived atom and one input
// atom -- reach(y) :- reach(x), edge(x,y), the shape of the Pathfinder and grid
// programs -- spends its time on launches: a 64 x 64 grid takes 187 iterations of
// about 900 candidates each, and count / scan / partition / emit / read-out /
// merge as separate kernels cost 45 to 80 us an iteration, whatever the number
// of facts.  Such a relation needs none of the sorted arrays while it grows,
// because nothing probes it.  Here it lives in dense arrays over its key space
// (tag, first-appearance stamp, membership bitmap), an iteration's candidates
// are (+)-added into an accumulator slot each and listed once when first
// touched, and one step of the loop takes the list of iteration k:
//     commit   candidate tag against the stored one (the relation's policy),
//     expand   if new or improved, probe the input relation and (+)-add the
//              products as candidates of iteration k + 1,
// with accumulators and lists of alternating parity, so that a single grid
// barrier separates the steps and the facts of each iteration are exactly those
// of Algorithm 1's.  A key is listed once, so its commit has one owner.
//
// What bounds it: the chain of dependent accesses of a step (list entry,
// accumulator, stored tag, offsets, matched fact, membership, accumulator) and
// its barrier.  Relations of a few thousand keys therefore run in one block with
// every array but the input relation in shared memory, where a step's barrier is
// __syncthreads; larger ones in up to one block per SM on arrays in L2.  A
// step's facts are spread over all warps before a warp takes a second one.
//
// Measured (GB300): 64 x 64 grid, diff-add-mult, fixpoint of 128 iterations 8.6
// -> 0.76 ms; diff-max-min, forward and backward 13.5 -> 1.7 ms; top-1-proofs over 64
// grids of side 16, forward and backward 9.1 -> 2.0 ms.  A step takes 4 us (12 with the
// arrays in L2), an iteration of the graph of kernels 67.  In shared memory a step
// has one barrier, the arrays of either parity are one array (an indexed pair of
// pointers would be generic ones: a step took 5.1 us), new facts are counted per
// warp, and a match's key and tag are loaded together.
#include "linear.h"

#include <algorithm>
#include <cstring>

#include "engine.h"
#include "pjoin.h"
#include "scan.cuh"

namespace {

constexpr int kLinThreads = 512;        // arrays in global memory
constexpr int kLinShThreads = 1024;     // one block, arrays in shared memory
constexpr u32 kLinShBytes = 210 * 1024; // shared memory those may take
constexpr int kLinMaxArms = 8;
constexpr int kLinMaxRels = 8;
constexpr u64 kLinRelSlots = 1ull << 24;  // keys of one relation (dense arrays)
constexpr u64 kLinMaxSlots = 1ull << 25;
constexpr u32 kLinSpin = 1u << 26;     // barrier polls before giving up

// LS_FULLARENA: top-1-proofs, one more than the first step that found the proof
// arena full
enum : int { LS_STOP = 0, LS_ITER, LS_CAND, LS_NEW, LS_ERR, LS_BAR, LS_FULLARENA, LS_LIST = 8, LS_FRESH = 12 };
// LS_LIST + i: length of the list of step i mod 3; LS_FRESH + i * kLinMaxRels +
// rel: the step's new facts (low half) and improved ones (high half); then per
// relation |F| and |recent| at the end
constexpr int LS_FULL = LS_FRESH + 3 * kLinMaxRels, LS_LAST = LS_FULL + kLinMaxRels;
constexpr int kLinSlots = LS_LAST + kLinMaxRels;
enum : u64 { LIN_FIXPOINT = 1, LIN_MAXITER = 2, LIN_ARENA = 3 };

struct LinArm {
  PStep P;
  int drel, hrel;  // relation indexes within the component
};
struct LinArgs {
  int n_rel, n_arm;
  u32 slots;
  u32 base[kLinMaxRels];   // a relation's first slot
  const LinArm* arms;
  // of either parity, one after the other:
  void* acc;               // candidate tags by slot, all zero between uses
  u32* touched;            // slots listed already
  u32* list;
  void* ftag;
  u32* fstamp;             // add-mult: iteration of first appearance | clamped << 31
  u32* fbits;              // membership
  const u32* start;        // slots recent after iteration k0
  u64 n_start;
  u64 fcount[kLinMaxRels];  // |F| after iteration k0
  u32 k0, max_iters;
  u64* state;
  Top1Arena top1;          // top-1-proofs
  u32* rec;                // add-mult: |recent| after iteration k at [(k - k0 - 1) * n_rel + rel]
};

LOB_DEV u64 lin_word(const void* p, int w64, u64 i) {
  return w64 ? reinterpret_cast<const u64*>(p)[i] : (u64)reinterpret_cast<const u32*>(p)[i];
}
LOB_DEV u64 lin_pick(const POperand& o, u64 wi, u64 wv) {
  if (o.word == 2) return o.cval;
  return ((o.word ? wv : wi) >> o.shift) & (o.width >= 64 ? ~0ull : ((1ull << o.width) - 1ull));
}
LOB_DEV bool lin_checks(const PCheck* c, int n, u64 wi, u64 wv) {
  bool ok = true;
  for (int q = 0; q < n; q++) ok = ok && ((lin_pick(c[q].a, wi, wv) == lin_pick(c[q].b, wi, wv)) == (c[q].eq != 0));
  return ok;
}
LOB_DEV u64 lin_lower(const void* keys, int key64, u64 n, u64 x) {
  if (key64) return lower_bound_dev<u64>(reinterpret_cast<const u64*>(keys), 0, n, x);
  if (x > 0xFFFFFFFFull) return n;
  return lower_bound_dev<u32>(reinterpret_cast<const u32*>(keys), 0, n, (u32)x);
}
// the matches of input word wi in the arm's input relation
LOB_DEV u32 lin_probe(const PStep& P, u64 wi, u32& lo) {
  lo = 0;
  if (P.n_in_checks && !lin_checks(P.in_checks, P.n_in_checks, wi, 0)) return 0;
  u64 pv = 0;
  for (int q = 0; q < P.n_prefix; q++) {
    const u64 x = lin_pick(P.prefix[q].op, wi, 0);
    if (P.prefix[q].limit_bits < 64 && (x >> P.prefix[q].limit_bits)) return 0;
    pv |= x << P.prefix[q].shift;
  }
  u64 l, h;
  if (P.index_mode == INDEX_DENSE) {
    l = P.dense_offs[pv];
    h = P.dense_offs[pv + 1];
  } else if (P.index_mode == INDEX_HASH) {
    hash_find(reinterpret_cast<const HashSlot*>(P.dense_offs), P.hash_bits, pv, l, h);
  } else if (P.whole_view) {
    l = 0;
    h = P.v_n;
  } else {
    const u64 klo = pv << P.rest_shift, khi = klo + (1ull << P.rest_shift);
    l = lin_lower(P.v_keys, P.v_key64, P.v_n, klo);
    h = khi < klo ? P.v_n : lin_lower(P.v_keys, P.v_key64, P.v_n, khi);
  }
  lo = (u32)l;
  return (u32)(h - l);
}

// All blocks of the launch, or false when one of them gave up waiting.  The
// count only grows, so a late block can never see it reset.  Thread 0's own writes
// before the call, and its warp's before a __syncwarp, are among those ordered.
LOB_DEV bool lin_barrier_warp0(u64* state, u32& gen) {
  volatile u64* s = state;
  __threadfence();
  gen++;
  atomicAdd(reinterpret_cast<unsigned long long*>(state) + LS_BAR, 1ull);
  const u64 want = (u64)gen * gridDim.x;
  u32 n = 0;
  while (s[LS_BAR] < want && !s[LS_ERR] && n < kLinSpin) n++;
  if (s[LS_BAR] < want) s[LS_ERR] = 1;
  __threadfence();
  return s[LS_ERR] == 0;
}
LOB_DEV bool lin_barrier(u64* state, u32& gen) {
  __shared__ u32 ok;
  __syncthreads();
  if (gridDim.x == 1) return true;
  if (threadIdx.x == 0) ok = lin_barrier_warp0(state, gen);
  __syncthreads();
  return ok != 0;
}

template <class T> LOB_DEV T lin_ld(const T* p) { return *reinterpret_cast<const volatile T*>(p); }

// the loop's arrays, in global or shared memory
template <class Sem>
struct LinArrays {
  typename Sem::Cand* acc;
  u32 *touched, *list;
  typename Sem::Stored* ftag;
  u32 *fstamp, *fbits;
  u64* state;
};
// bytes of the shared form, per slot and fixed (the state block)
template <class Sem> constexpr u32 lin_slot_bytes() {
  return 2 * (u32)sizeof(typename Sem::Cand) + (u32)sizeof(typename Sem::Stored) + 4 + 8;
}
LOB_HD u32 lin_shared_bytes(u32 slot_bytes, u32 slots) { return slots * slot_bytes + 3 * (slots / 8) + kLinSlots * 8; }

// ---------------------------------------------------------------------------
// top-1-proofs: (x) of a derived fact's proof and an input fact's, which is one
// id or empty.  Candidates that cannot win are not formed (a stored proof only
// gets likelier): the proof {p_1 .. p_n} and one more fact x has probability at
// most p max(1, p_x), and about p p_x once x is known not to be among them.  A
// union with a fact of the proof is the proof itself.  What is left reads the
// proof in eight lanes, four candidates a warp, and forms the product as
// top1_union does: ascending ids, FP64, rounded once.  Bound by the chain of
// loads (tag, length, ids, probabilities) and the FP64 products.  64 grids of side
// 16, 44 iterations of 3,500 candidates: the general steps took 190 us an
// iteration (53 of them for unions by single threads), a step here takes 20.
// ---------------------------------------------------------------------------
constexpr float kTopSlack = 1.000001f;  // f32 rounding of p, of p_x and of their product, with room to spare
// probability bits of a candidate that cannot beat `best` (bits; ~0: nothing there)
LOB_DEV bool top_loses(u32 p, u32 px, bool together, u32 best) {
  if (p > 0x7F800000u || px > 0x7F800000u || best > 0x7F800000u) return false;  // a sign, a NaN, nothing to beat
  const float fp = __uint_as_float(p), fx = __uint_as_float(px);
  const float u = together ? fp * fx : fp * fmaxf(fx, 1.0f);
  return fp >= 1e-30f && u >= 1e-30f && u * kTopSlack <= __uint_as_float(best);
}
// One union for each group of eight lanes with live set (all lanes of the warp
// call).  Returns its tag to the whole group, 0 when it is dropped.
LOB_DEV u64 top_union(const Top1Arena& T, bool live, u64 a, u64 b, u32 best, unsigned long long* full, u32 step) {
  const int lane = threadIdx.x & 31, g0 = lane & 24, l8 = lane & 7;
  const u32 ra = (u32)a, rb = (u32)b;
  u64 out = 0;
  u32 la = live ? __ldcg(T.words + ra) : 0u;
  if (live && la == 0) out = b;  // the empty proof is the identity
  else if (live && (rb == 0 || ra == rb)) out = a;
  bool work = live && !out;
  if (!work) la = 0;
  const u32 x = (rb - 1) >> 1, px = (u32)(b >> 32);
  const u32 lmax = __reduce_max_sync(0xFFFFFFFFu, la);
  u32 below = 0, id0[4];
  bool has = false;
#pragma unroll
  for (int c = 0; c < 4; c++) {
    const u32 i = 8 * c + l8;
    id0[c] = i < la ? __ldcg(T.words + ra + 1 + i) : 0xFFFFFFFFu;
    below += id0[c] < x;
    has = has || (i < la && id0[c] == x);
  }
  for (u32 i = 32 + l8; i < lmax + l8; i += 8) {
    const u32 id = i < la ? __ldcg(T.words + ra + 1 + i) : 0xFFFFFFFFu;
    below += id < x;
    has = has || (i < la && id == x);
  }
  has = (__ballot_sync(0xFFFFFFFFu, has) >> g0) & 0xFFu;
#pragma unroll
  for (int o = 4; o; o >>= 1) below += __shfl_xor_sync(0xFFFFFFFFu, below, o);
  if (work && has) {
    out = a;
    work = false;
  }
  if (out && best != ~0u && (u32)(out >> 32) <= best) out = 0;
  if (work && la + 1 > T.proof_cap) {
    if (l8 == 0) atomicOr(T.err, 1u);
    work = false;
  }
  if (work && top_loses((u32)(a >> 32), px, true, best)) work = false;
  if (!__any_sync(0xFFFFFFFFu, work)) return out;
  double p = 1.0;
  const double fx = (double)__uint_as_float(px);
  if (!work) la = 0;
  const u32 pmax = __reduce_max_sync(0xFFFFFFFFu, la);
  for (u32 i0 = 0; i0 < pmax; i0 += 8) {
    const u32 i = i0 + l8;
    u32 id = i0 < 32 ? id0[0] : 0u;
    if (i0 == 8) id = id0[1];
    if (i0 == 16) id = id0[2];
    if (i0 == 24) id = id0[3];
    if (i0 >= 32 && i < la) id = __ldcg(T.words + ra + 1 + i);
    const float pr = i < la ? __ldg(T.prob + id) : 1.0f;
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const float q = __shfl_sync(0xFFFFFFFFu, pr, g0 + j);
      if (i0 + j == below) p *= fx;
      if (i0 + j < la) p *= (double)q;
    }
  }
  if (below >= ((pmax + 7) & ~7u)) p *= fx;
  const u32 bits = __float_as_uint((float)p);
  if (best != ~0u && bits <= best) work = false;
  unsigned long long at = 0;
  const u32 need = la + 2;
  if (work && l8 == 0) at = atomicAdd(T.tail, (unsigned long long)need);
  at = __shfl_sync(0xFFFFFFFFu, at, g0);
  if (work && at + need > T.cap) {
    if (l8 == 0) atomicCAS(full, 0ull, (unsigned long long)step + 1);
    work = false;
  }
  if (!work) return out;
  u32* w = T.words + at;
  if (l8 == 0) {
    w[0] = la + 1;
    w[1 + below] = x;
  }
#pragma unroll
  for (int c = 0; c < 4; c++)
    if (8 * c + l8 < la) w[1 + 8 * c + l8 + (id0[c] > x)] = id0[c];
  for (u32 i = 32 + l8; i < la; i += 8) {
    const u32 id = __ldcg(T.words + ra + 1 + i);
    w[1 + i + (id > x)] = id;
  }
  return ((u64)bits << 32) | at;
}

template <class Sem, bool kSh>
__global__ void __launch_bounds__(kSh ? kLinShThreads : kLinThreads) k_linear(const __grid_constant__ LinArgs A) {
  constexpr int kT = kSh ? kLinShThreads : kLinThreads;
  typedef typename Sem::Stored S;
  typedef typename Sem::Cand C;
  constexpr bool kTop1 = std::is_same<Sem, SemTop1>::value;
  __shared__ LinArm arms[kLinMaxArms];
  __shared__ u32 fresh_sh[2][2][kLinMaxRels];  // by parity: new, improved (several blocks)
  __shared__ u32 go;
  __shared__ unsigned long long cand_sh;
  LinArrays<Sem> X;
  if constexpr (kSh) {
    extern __shared__ __align__(16) unsigned char sh[];
    unsigned char* q = sh;
    const u32 n = A.slots;
    X.state = reinterpret_cast<u64*>(q); q += kLinSlots * 8;
    X.acc = reinterpret_cast<C*>(q); q += 2 * (u64)n * sizeof(C);
    X.ftag = reinterpret_cast<S*>(q); q += (u64)n * sizeof(S);
    X.fstamp = reinterpret_cast<u32*>(q); q += (u64)n * 4;
    X.list = reinterpret_cast<u32*>(q); q += 2 * (u64)n * 4;
    X.touched = reinterpret_cast<u32*>(q); q += 2 * (n / 8);
    X.fbits = reinterpret_cast<u32*>(q);
    for (u32 i = threadIdx.x; i < n; i += kT) {
      X.acc[i] = X.acc[n + i] = C(0);
      X.ftag[i] = reinterpret_cast<const S*>(A.ftag)[i];
      X.fstamp[i] = A.fstamp ? A.fstamp[i] : 0u;
    }
    for (u32 i = threadIdx.x; i < n / 32; i += kT) {
      X.touched[i] = X.touched[n / 32 + i] = 0u;
      X.fbits[i] = A.fbits[i];
    }
    for (u32 i = threadIdx.x; i < (u32)kLinSlots; i += kT) X.state[i] = 0;
  } else {
    X.acc = reinterpret_cast<C*>(A.acc);
    X.touched = A.touched;
    X.list = A.list;
    X.ftag = reinterpret_cast<S*>(A.ftag);
    X.fstamp = A.fstamp;
    X.fbits = A.fbits;
    X.state = A.state;
  }
  for (u32 i = threadIdx.x; i < A.n_arm * sizeof(LinArm) / 4; i += kT)
    reinterpret_cast<u32*>(arms)[i] = reinterpret_cast<const u32*>(A.arms)[i];
  if (threadIdx.x == 0) cand_sh = 0;
  if (threadIdx.x < 4 * kLinMaxRels) (&fresh_sh[0][0][0])[threadIdx.x] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const u32 warp = blockIdx.x * (kT / 32) + (threadIdx.x >> 5), nwarps = gridDim.x * (kT / 32);
  u64* st = X.state;
  unsigned long long* ast = reinterpret_cast<unsigned long long*>(st);
  // the last warp, least likely to hold facts, keeps the counters
  const bool keeper = blockIdx.x == 0 && (threadIdx.x >> 5) == kT / 32 - 1;
  u32 gen = 0;
  u64 cand = 0, new_facts = 0;
  u64 fcount[kLinMaxRels];
#pragma unroll
  for (int r = 0; r < kLinMaxRels; r++) fcount[r] = r < A.n_rel ? A.fcount[r] : 0;
  // step 0 expands the facts recent after iteration k0; step j > 0 commits the
  // candidates of iteration k0 + j and expands what is new
  u32 rot = 0, rot1 = 1, rot2 = 2;  // step, step + 1, step + 2 mod 3
  for (u32 step = 0;; step++, rot = rot1, rot1 = rot2, rot2 = rot == 0 ? 2 : rot - 1) {
    const u32 k = A.k0 + step;
    const int par = step & 1;
    const bool commit = step > 0;
    // this step's arrays, and those of the next
    C *acc = X.acc + (par ? A.slots : 0u), *next_acc = X.acc + (par ? 0u : A.slots);
    u32 *touched = X.touched + (par ? A.slots / 32 : 0u), *next_touched = X.touched + (par ? 0u : A.slots / 32);
    const u32* list = X.list + (par ? A.slots : 0u);
    u32* out_list = X.list + (par ? 0u : A.slots);
    const u32 n = commit ? (u32)lin_ld(st + LS_LIST + rot) : (u32)A.n_start;
    // Counters of steps to come.  The list length read in the last step is done
    // with; the new-fact counts of the last step may still be read by a slow
    // warp, those of the step before may not.
    if (keeper && lane <= kLinMaxRels) {
      if (lane == kLinMaxRels) st[LS_LIST + rot2] = 0;
      else st[LS_FRESH + rot1 * kLinMaxRels + lane] = 0;
    }
    u32 n_fresh = 0, n_better = 0;  // one relation: this warp's new and improved facts
    const bool expand = k < A.max_iters;
    const u32 per = min(32u, (n + nwarps - 1) / nwarps);  // facts a warp takes at a time
    for (u32 i0 = warp * per; i0 < n; i0 += nwarps * per) {
      const bool in = lane < (int)per && i0 + lane < n;
      u32 slot = 0;
      int rel = -1;
      S tag{};
      bool fresh = false;
      if (in) {
        slot = commit ? lin_ld(list + i0 + lane) : A.start[i0 + lane];
        rel = 0;
        while (rel + 1 < A.n_rel && slot >= A.base[rel + 1]) rel++;
        S* f = X.ftag + slot;
        if (commit) {
          C* a = acc + slot;
          const u32 bit = 1u << (slot & 31u);
          const C c = lin_ld(a);
          const bool present = lin_ld(X.fbits + (slot >> 5)) & bit;
          S old{};
          if constexpr (Sem::kIdempotent) old = lin_ld(f);  // not written yet: 0
          *reinterpret_cast<volatile C*>(a) = C(0);
          atomicAnd(touched + (slot >> 5), ~bit);
          tag = Sem::store(c);
          if (!present) {
            fresh = true;
            if constexpr (std::is_same<Sem, SemAddMult>::value)
              *reinterpret_cast<volatile u32*>(X.fstamp + slot) = k | (c > 1.0 ? 0x80000000u : 0u);
            *reinterpret_cast<volatile S*>(f) = tag;
            atomicOr(X.fbits + (slot >> 5), bit);
            if (A.n_rel == 1) n_fresh++;
            else atomicAdd(kSh ? reinterpret_cast<u32*>(st + LS_FRESH + rot * kLinMaxRels + rel) : &fresh_sh[par][0][rel], 1u);
          } else if (Sem::kIdempotent && Sem::better(tag, old)) {
            fresh = true;
            *reinterpret_cast<volatile S*>(f) = tag;
            if (A.n_rel == 1) n_better++;
            else atomicAdd(kSh ? reinterpret_cast<u32*>(st + LS_FRESH + rot * kLinMaxRels + rel) + 1 : &fresh_sh[par][1][rel], 1u);
          }
        } else {
          tag = lin_ld(f);
          fresh = true;
        }
      }
      if (!expand) continue;
      const u64 wi = in ? (u64)slot - A.base[rel] : 0ull;
      const C ct = Sem::from_stored(tag);
      u32 plen = 0;  // top-1-proofs: the length of the fact's proof
      if constexpr (kTop1) plen = fresh ? __ldcg(A.top1.words + (u32)tag) : 0u;
      for (int a = 0; a < A.n_arm; a++) {
        const LinArm& arm = arms[a];
        const PStep& P = arm.P;
        u32 lo = 0;
        const u32 c = fresh && arm.drel == rel ? lin_probe(P, wi, lo) : 0u;
        const u32 inc = warp_inclusive_sum(c);
        const u32 tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
        if (!tot) continue;
        cand += tot;
        const u32 ex = inc - c;
        const u32 hbase = A.base[arm.hrel];
        for (u32 t0 = 0; t0 < tot; t0 += 32) {
          const u32 t = t0 + lane;
          int src = 0;  // the last lane whose outputs start at or before t
#pragma unroll
          for (int s = 16; s; s >>= 1) {
            const u32 x = __shfl_sync(0xFFFFFFFFu, ex, src + s);
            if (x <= t) src += s;
          }
          const u64 wr = __shfl_sync(0xFFFFFFFFu, wi, src);
          const u32 lr = __shfl_sync(0xFFFFFFFFu, lo, src);
          const u32 er = __shfl_sync(0xFFFFFFFFu, ex, src);
          const C tr = __shfl_sync(0xFFFFFFFFu, ct, src);
          bool add = false;
          u32 hs = 0;
          if constexpr (kTop1) {
            u64 edge = 0;
            u32 best = ~0u;
            bool want = false;
            const u32 len = __shfl_sync(0xFFFFFFFFu, plen, src);
            if (t < tot) {
              const u64 v = (u64)lr + (t - er);
              const u64 wv = lin_word(P.v_keys, P.v_key64, v);
              edge = reinterpret_cast<const S*>(P.v_tags)[v];
              if (lin_checks(P.checks, P.n_checks, wr, wv)) {
                u64 w = 0;
                for (int q = 0; q < P.n_out; q++) w |= lin_pick(P.out[q].op, wr, wv) << P.out[q].shift;
                hs = hbase + (u32)w;
                // the likelier of the stored proof and the candidate there already
                const u64 c = lin_ld(next_acc + hs);
                if (c) best = (u32)(c >> 32);
                if (lin_ld(X.fbits + (hs >> 5)) & (1u << (hs & 31u))) {
                  const u32 f = (u32)(lin_ld(X.ftag + hs) >> 32);
                  best = best == ~0u ? f : max(best, f);
                }
                want = len >= A.top1.proof_cap || !top_loses((u32)(tr >> 32), (u32)(edge >> 32), false, best);
              }
            }
            u64 made = 0;
            for (u32 todo = __ballot_sync(0xFFFFFFFFu, want); todo;) {
              u32 m = todo;
              for (int q = 0; q < (lane >> 3); q++) m &= m - 1;
              const int of = m ? __ffs(m) - 1 : 0;
              const u64 ta = __shfl_sync(0xFFFFFFFFu, (u64)tr, of), te = __shfl_sync(0xFFFFFFFFu, edge, of);
              const u32 tb = __shfl_sync(0xFFFFFFFFu, best, of);
              const u64 u = top_union(A.top1, m != 0, ta, te, tb, ast + LS_FULLARENA, step);
              const int mine = __popc(todo & ((1u << lane) - 1u));
              const u64 back = __shfl_sync(0xFFFFFFFFu, u, (mine & 3) * 8);
              if (((todo >> lane) & 1u) && mine < 4) made = back;
              for (int q = 0; q < 4; q++) todo &= todo - 1;
            }
            if (made) {
              dense_add<Sem>(next_acc, hs, made);
              const u32 bit = 1u << (hs & 31u);
              u32* tw = next_touched + (hs >> 5);
              if (!(lin_ld(tw) & bit)) add = !(atomicOr(tw, bit) & bit);
            }
          } else if (t < tot) {
            const u64 v = (u64)lr + (t - er);
            const u64 wv = lin_word(P.v_keys, P.v_key64, v);
            const S vtag = reinterpret_cast<const S*>(P.v_tags)[v];  // both loads in flight at once
            if (lin_checks(P.checks, P.n_checks, wr, wv)) {
              u64 w = 0;
              for (int q = 0; q < P.n_out; q++) w |= lin_pick(P.out[q].op, wr, wv) << P.out[q].shift;
              hs = hbase + (u32)w;
              const u32 bit = 1u << (hs & 31u);
              const C prod = Sem::mul(tr, Sem::from_stored(vtag));
              // A candidate that cannot change the stored tag is dropped here: a
              // fact that is present stays present, and a tag only grows.  Facts
              // being committed in this step may be seen or not (a tag not yet
              // seen reads 0): their own commit of this candidate decides then.
              bool useless = lin_ld(X.fbits + (hs >> 5)) & bit;
              if constexpr (Sem::kIdempotent) useless = useless && lin_ld(X.ftag + hs) >= Sem::store(prod);
              if (!useless) {
                dense_add<Sem>(next_acc, hs, prod);
                u32* tw = next_touched + (hs >> 5);
                if (!(lin_ld(tw) & bit)) add = !(atomicOr(tw, bit) & bit);
              }
            }
          }
          const u32 m = __ballot_sync(0xFFFFFFFFu, add);
          if (m) {
            u64 at = 0;
            if (lane == 0) at = atomicAdd(ast + LS_LIST + rot1, (unsigned long long)__popc(m));
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            if (add) *reinterpret_cast<volatile u32*>(out_list + at + __popc(m & ((1u << lane) - 1u))) = hs;
          }
        }
      }
    }
    if (A.n_rel == 1) {
      n_fresh = __reduce_add_sync(0xFFFFFFFFu, n_fresh);
      n_better = __reduce_add_sync(0xFFFFFFFFu, n_better);
      if (lane == 0 && (n_fresh | n_better)) {
        u32* to = kSh ? reinterpret_cast<u32*>(st + LS_FRESH + rot * kLinMaxRels) : &fresh_sh[par][0][0];
        if (n_fresh) atomicAdd(to, n_fresh);
        if (n_better) atomicAdd(kSh ? to + 1 : &fresh_sh[par][1][0], n_better);
      }
    }
    __syncthreads();
    if constexpr (!kSh) {
      if (threadIdx.x < 32) {
        if (lane < A.n_rel && (fresh_sh[par][0][lane] | fresh_sh[par][1][lane])) {
          atomicAdd(ast + LS_FRESH + rot * kLinMaxRels + lane,
                    ((unsigned long long)fresh_sh[par][1][lane] << 32) | fresh_sh[par][0][lane]);
          fresh_sh[par][0][lane] = fresh_sh[par][1][lane] = 0;
          __threadfence();
        }
        __syncwarp();
        if (lane == 0) go = gridDim.x == 1 || lin_barrier_warp0(st, gen);
      }
      __syncthreads();
      if (!go) break;
    }
    if constexpr (kTop1) {  // a faster block's next step may have found it full already
      const u64 f = lin_ld(st + LS_FULLARENA);
      if (f && f <= step + 1) {
        if (keeper && lane == 0) st[LS_STOP] = LIN_ARENA;
        break;
      }
    }
    if (!commit) continue;
    u64 total = 0;
#pragma unroll
    for (int r = 0; r < kLinMaxRels; r++) {
      if (r >= A.n_rel) break;
      const u64 v = lin_ld(st + LS_FRESH + rot * kLinMaxRels + r);
      const u64 added = v & 0xFFFFFFFFull, improved = v >> 32;
      fcount[r] += added;
      total += added + improved;
      if (keeper && lane == 0) {
        if (A.rec) A.rec[(u64)(step - 1) * A.n_rel + r] = (u32)added;
        st[LS_FULL + r] = fcount[r];  // (read by the host, after the last step)
        st[LS_LAST + r] = added + improved;
      }
    }
    const u64 stop = !total ? LIN_FIXPOINT : k >= A.max_iters ? LIN_MAXITER : 0;
    new_facts += total;
    if (stop) {
      if (keeper && lane == 0) {
        st[LS_NEW] = new_facts;
        st[LS_ITER] = k;
        st[LS_STOP] = stop;
      }
      break;
    }
  }
  // join outputs, summed per warp (every lane holds its warp's count)
  __syncthreads();
  if (lane == 0 && cand) atomicAdd(&cand_sh, (unsigned long long)cand);
  __syncthreads();
  if (threadIdx.x == 0 && cand_sh) atomicAdd(ast + LS_CAND, cand_sh);
  if constexpr (kSh) {
    __syncthreads();
    for (u32 i = threadIdx.x; i < A.slots; i += kT) {
      reinterpret_cast<S*>(A.ftag)[i] = X.ftag[i];
      if (A.fstamp) A.fstamp[i] = X.fstamp[i];
    }
    for (u32 i = threadIdx.x; i < A.slots / 32; i += kT) A.fbits[i] = X.fbits[i];
    for (u32 i = threadIdx.x; i < (u32)kLinSlots; i += kT) A.state[i] = X.state[i];
  }
}

// ---------------------------------------------------------------------------
// Backward pass of diff-add-mult over the linear components.  A fact first
// derived in iteration s is the recent fact of its groundings in iteration s +
// 1 only, so the facts sorted by stamp are the replay: one step per stamp, from
// the last to 1, expands the facts of stamp s and takes from each head of stamp
// s + 1 (whose adjoint is complete) its share, with a grid barrier between the
// steps.  The replay of one iteration as count / scan / partition / emit with a
// host wait took 55 us whatever its size; a step takes about 3.
// ---------------------------------------------------------------------------
struct LinBwdArm {
  PStep P;
  int drel, hrel;
  const u32* prow;  // probed view row -> primary row (null: the primary view)
  double* vadj;     // adjoints of the probed relation (null: none needed)
};
struct LinBwdRel {
  const void* keys;
  int key64;
  const float* tags;
  const u32* stamps;
  const u32* hrow;  // key -> row
  double* adj;
  u32 base;         // the relation's first entry number
};
struct LinBwdArgs {
  int n_rel, n_arm;
  LinBwdRel rel[kLinMaxRels];
  const LinBwdArm* arms;
  const u32* entries;  // base + row, by stamp
  const u32* off;      // a stamp's first entry
  u32 last;            // iterations of the run
  u64* state;
};

__global__ void __launch_bounds__(kLinThreads) k_linear_backward(const __grid_constant__ LinBwdArgs A) {
  __shared__ LinBwdArm arms[kLinMaxArms];
  for (u32 i = threadIdx.x; i < A.n_arm * sizeof(LinBwdArm) / 4; i += kLinThreads)
    reinterpret_cast<u32*>(arms)[i] = reinterpret_cast<const u32*>(A.arms)[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const u64 warp = (u64)blockIdx.x * (kLinThreads / 32) + (threadIdx.x >> 5), nwarps = (u64)gridDim.x * (kLinThreads / 32);
  u32 gen = 0;
  for (u32 s = A.last - 1; s >= 1; s--) {
    const u32 first = A.off[s];
    const u64 n = A.off[s + 1] - first;
    if (!n) continue;
    const u64 per = min(32ull, (n + nwarps - 1) / nwarps);
    for (u64 i0 = warp * per; i0 < n; i0 += nwarps * per) {
      const bool in = lane < (int)per && i0 + lane < n;
      int rel = -1;
      u32 row = 0;
      u64 wi = 0;
      double tag = 0.0;
      if (in) {
        const u32 x = A.entries[first + i0 + lane];
        rel = 0;
        while (rel + 1 < A.n_rel && x >= A.rel[rel + 1].base) rel++;
        row = x - A.rel[rel].base;
        wi = lin_word(A.rel[rel].keys, A.rel[rel].key64, row);
        tag = (double)A.rel[rel].tags[row];
      }
      for (int a = 0; a < A.n_arm; a++) {
        const LinBwdArm& arm = arms[a];
        const PStep& P = arm.P;
        const LinBwdRel& H = A.rel[arm.hrel];
        double* dadj = A.rel[arm.drel].adj;
        u32 lo = 0;
        const u32 c = in && arm.drel == rel ? lin_probe(P, wi, lo) : 0u;
        const u32 inc = warp_inclusive_sum(c);
        const u32 tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
        const u32 ex = inc - c;
        for (u32 t0 = 0; t0 < tot; t0 += 32) {
          const u32 t = t0 + lane;
          int src = 0;  // the last lane whose outputs start at or before t
#pragma unroll
          for (int q = 16; q; q >>= 1) {
            const u32 x = __shfl_sync(0xFFFFFFFFu, ex, src + q);
            if (x <= t) src += q;
          }
          const u64 wr = __shfl_sync(0xFFFFFFFFu, wi, src);
          const u32 lr = __shfl_sync(0xFFFFFFFFu, lo, src);
          const u32 er = __shfl_sync(0xFFFFFFFFu, ex, src);
          const u32 rr = __shfl_sync(0xFFFFFFFFu, row, src);
          const double tr = __shfl_sync(0xFFFFFFFFu, tag, src);
          if (t >= tot) continue;
          const u64 v = (u64)lr + (t - er);
          const u64 wv = lin_word(P.v_keys, P.v_key64, v);
          if (!lin_checks(P.checks, P.n_checks, wr, wv)) continue;
          u64 w = 0;
          for (int q = 0; q < P.n_out; q++) w |= lin_pick(P.out[q].op, wr, wv) << P.out[q].shift;
          const u32 h = H.hrow[w];
          // not new in iteration s + 1, or its sum was clamped (bit 31)
          if (h == 0xFFFFFFFFu || H.stamps[h] != s + 1) continue;
          const double adj = lin_ld(H.adj + h);
          if (adj == 0.0) continue;
          atomicAdd(dadj + rr, adj * (double)reinterpret_cast<const float*>(P.v_tags)[v]);
          if (arm.vadj) atomicAdd(arm.vadj + (arm.prow ? arm.prow[v] : (u32)v), adj * tr);
        }
      }
    }
    if (!lin_barrier(A.state, gen)) return;
  }
}

// facts by stamp: stamps 1 .. last - 1 (later ones are never a recent fact)
__global__ void k_lin_stamp_count(const u32* __restrict__ stamps, u64 n, u32 last, u32* __restrict__ cnt) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const u32 s = stamps[i] & 0x7FFFFFFFu;
    if (s >= 1 && s < last) atomicAdd(cnt + s, 1u);
  }
}
__global__ void k_lin_stamp_fill(const u32* __restrict__ stamps, u64 n, u32 last, u32 base, const u32* __restrict__ off,
                                 u32* __restrict__ used, u32* __restrict__ out) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const u32 s = stamps[i] & 0x7FFFFFFFu;
    if (s >= 1 && s < last) out[off[s] + atomicAdd(used + s, 1u)] = base + (u32)i;
  }
}

// facts present after iteration 1: tag, stamp and membership by slot
template <class S>
__global__ void k_lin_init(const void* __restrict__ keys, int key64, const S* __restrict__ tags,
                           const u32* __restrict__ stamps, u64 n, u32 base, S* __restrict__ ftag, u32* __restrict__ fstamp,
                           u32* __restrict__ fbits) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const u32 s = base + (u32)load_key(keys, key64, i);
    ftag[s] = tags[i];
    if (stamps) fstamp[s] = stamps[i];
    atomicOr(fbits + (s >> 5), 1u << (s & 31u));
  }
}
__global__ void k_lin_slots(const void* __restrict__ keys, int key64, u64 n, u32 base, u32* __restrict__ out) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[i] = base + (u32)load_key(keys, key64, i);
}
// tags and stamps of the sorted keys
template <class S>
__global__ void k_lin_collect(const void* __restrict__ keys, int key64, u64 n, u32 base, const S* __restrict__ ftag,
                              const u32* __restrict__ fstamp, S* __restrict__ tags, u32* __restrict__ stamps) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const u32 s = base + (u32)load_key(keys, key64, i);
    tags[i] = ftag[s];
    if (stamps) stamps[i] = fstamp[s];
  }
}

// Slots of a relation's key space: one more than its largest possible key, in
// whole 16-byte pieces of the bitmaps.
u64 lin_slots(const lob_engine& e, const RelSt& r) {
  const Layout& L = r.views[0].lay;
  if (L.bits > 40) return ~0ull >> 8;
  u64 top = L.swidth ? (u64)e.max_sample << L.sshift : 0ull;
  for (int j = 0; j < L.arity; j++) top += (u64)r.maxv[j] << L.shift[j];
  return (top + 128) & ~127ull;
}
unsigned lin_grid(u64 n) { return (unsigned)std::max<u64>(1, std::min<u64>((n + 255) / 256, 152ull * 16)); }

struct LinRun {
  lob_engine& e;
  std::vector<u32> rels;
  std::vector<int> index;  // relation id -> index in rels, or -1
  explicit LinRun(lob_engine& en) : e(en) {}
  DevBuf arms, acc, touched, list, used, ftag, fstamp, fbits, start, state, rec;
  ~LinRun() {
    for (DevBuf* b : {&arms, &acc, &touched, &list, &used, &ftag, &fstamp, &fbits, &start,
                      &state, &rec})
      e.release(*b);
  }

  template <class Sem>
  void launch(const LinArgs& A, unsigned blocks) {
    void* args[] = {const_cast<LinArgs*>(&A)};
    const u32 sh = lin_shared_bytes(lin_slot_bytes<Sem>(), A.slots);
    if (sh <= kLinShBytes && blocks == 1) {
      e.check(allow_dynamic_smem(k_linear<Sem, true>, (int)sh), "linear loop");
      ProfScope ps("linear_loop", 0, e.stream);
      k_linear<Sem, true><<<1, kLinShThreads, sh, e.stream>>>(A);
    } else {
      ProfScope ps("linear_loop", 0, e.stream);
      e.check(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_linear<Sem, false>), dim3(blocks), dim3(kLinThreads), args, 0,
                                          e.stream), "linear loop");
    }
    e.after_launch("linear loop");
    e.launches++;
  }
  template <class S>
  void init(const RelSt& R, u32 base) {
    const ViewSt& V = R.views[0];
    if (V.n)
      k_lin_init<S><<<lin_grid(V.n), 256, 0, e.stream>>>(V.keys.p, V.lay.key64, V.tags.as<S>(),
                                                         fstamp.p ? V.stamps.as<u32>() : nullptr, V.n, base, ftag.as<S>(),
                                                         fstamp.as<u32>(), fbits.as<u32>());
    e.after_launch("linear facts");
    e.launches++;
  }
  template <class S>
  void collect(RelSt& R, u32 base) {
    ViewSt& V = R.views[0];
    k_lin_collect<S><<<lin_grid(V.n), 256, 0, e.stream>>>(V.keys.p, V.lay.key64, V.n, base, ftag.as<S>(), fstamp.as<u32>(),
                                                          V.tags.as<S>(), fstamp.p ? V.stamps.as<u32>() : nullptr);
    e.after_launch("linear result");
    e.launches++;
  }
};

}  // namespace

// The derived relations whose component (relations that rules connect) is
// linear: dense, in all their rules at most one derived atom, which is then
// joined with one input relation by a packed step, and, where views carry
// stamps, no secondary view to keep.  False when there are none.
bool linear_component(const lob_engine& e, std::vector<char>& in) {
  const size_t n = e.rels.size();
  in.assign(n, 0);
  if (e.semiring == SR_UNIT || e.n_strata != 1) return false;
  // top-1-proofs runs keep no dense accumulators outside this loop
  const bool top1 = sem_top1(e.semiring);
  std::vector<int> comp(n);
  for (size_t r = 0; r < n; r++) comp[r] = (int)r;
  std::vector<char> bad(n, 0);
  std::vector<int> n_arms(n, 0);
  auto join = [&](int a, int b) {
    const int x = comp[a], y = comp[b];
    for (auto& c : comp)
      if (c == y) c = x;
  };
  for (auto& p : e.plans)
    for (auto& a : p.ast.body)
      if (e.rels[a.rel].idb) join((int)p.ast.head.rel, (int)a.rel);
  for (size_t r = 0; r < n; r++) {
    const RelSt& R = e.rels[r];
    if (!R.idb) continue;
    const bool dense = top1 ? e.opt_acc_dense && R.views[0].lay.bits <= e.opt_acc_bits : R.dense;
    if (!dense || lin_slots(e, R) > kLinRelSlots || (sem_stamps(e.semiring) && R.views.size() > 1)) bad[comp[r]] = 1;
  }
  for (auto& p : e.plans) {
    int derived = 0;
    for (auto& a : p.ast.body) derived += e.rels[a.rel].idb;
    if (!derived) continue;
    const int c = comp[p.ast.head.rel];
    if (derived > 1 || p.ast.body.size() != 2) bad[c] = 1;
    for (auto& A : p.arms)
      if (e.rels[p.ast.body[A.delta].rel].idb) {
        n_arms[c]++;
        if (!(top1 ? A.packed.linear_only : A.packed.ok) || A.steps.size() != 2) bad[c] = 1;
      }
  }
  bool any = false;
  int rels = 0, arms = 0;
  u64 slots = 0;
  for (size_t c = 0; c < n; c++) {
    if (bad[c] || !n_arms[c]) continue;
    u64 s = 0;
    int m = 0;
    for (size_t r = 0; r < n; r++)
      if (e.rels[r].idb && comp[r] == (int)c) {
        s += lin_slots(e, e.rels[r]);
        m++;
      }
    if (rels + m > kLinMaxRels || arms + n_arms[c] > kLinMaxArms || slots + s > kLinMaxSlots) continue;
    rels += m;
    arms += n_arms[c];
    slots += s;
    for (size_t r = 0; r < n; r++)
      if (e.rels[r].idb && comp[r] == (int)c) in[r] = any = true;
  }
  return any;
}

void run_linear(lob_engine& e, u32 max_iters, lob_stats& s, LinearOut& out) {
  const u32 k0 = 1;
  std::vector<char> in;
  if (!e.opt_driver || e.lean || k0 >= max_iters || !linear_component(e, in)) return;
  if (e.opt_driver == 1 && !e.loop_caps.count("linear_history")) {
    // as for the device-driven graph: the first run of an engine is host-driven
    e.loop_caps["linear_history"] = 1;
    return;
  }
  LinRun L(e);
  L.index.assign(e.rels.size(), -1);
  LinArgs A;
  std::memset(&A, 0, sizeof(A));
  u64 slots = 0, recent = 0, probed = 0;
  for (size_t r = 0; r < e.rels.size(); r++) {
    if (!in[r]) continue;
    L.index[r] = A.n_rel;
    A.base[A.n_rel] = (u32)slots;
    A.fcount[A.n_rel++] = e.rels[r].views[0].n;
    slots += lin_slots(e, e.rels[r]);
    recent += e.rels[r].n_recent;
    L.rels.push_back((u32)r);
  }
  if (!recent) return;
  std::vector<LinArm> arms;
  for (auto& p : e.plans)
    for (auto& Ar : p.arms) {
      const u32 drel = p.ast.body[Ar.delta].rel;
      if (L.index[p.ast.head.rel] < 0 || !e.rels[drel].idb) continue;
      const StepPlan& S = Ar.steps[1];
      ViewSt& W = e.rels[p.ast.body[S.atom].rel].views[S.view];
      if (W.n > 0x7FFFFFFull) return;  // 32 rows' outputs stay below 2^32
      LinArm a;
      std::memset(&a, 0, sizeof(a));
      a.P = Ar.packed.steps[0];
      a.drel = L.index[drel];
      a.hrel = L.index[p.ast.head.rel];
      if (!W.n) continue;
      engine_ensure_index(e, W, S.prefix_len);
      a.P.v_keys = W.keys.p;
      a.P.v_key64 = W.lay.key64;
      a.P.v_tags = W.tags.p;
      a.P.v_n = W.n;
      const IndexSt& I = W.index[S.prefix_len];
      a.P.index_mode = I.mode;
      a.P.dense_offs = I.offs.as<u64>();
      a.P.hash_bits = I.hash_bits;
      probed += W.n;
      arms.push_back(a);
    }
  const int ks = sem_kernel(e.semiring);
  const int sb = stored_bytes(e.semiring), cb = cand_bytes(e.semiring);
  const bool stamps = sem_stamps(e.semiring), top1 = sem_top1(e.semiring);
  e.extra = true;
  e.ensure(L.arms, std::max<size_t>(arms.size(), 1) * sizeof(LinArm));
  if (!arms.empty())
    e.check(cudaMemcpyAsync(L.arms.p, arms.data(), arms.size() * sizeof(LinArm), cudaMemcpyHostToDevice, e.stream), "arms");
  e.ensure(L.acc, 2 * slots * cb);
  e.ensure(L.touched, 2 * (slots / 8));
  e.ensure(L.list, 2 * slots * 4);
  e.ensure(L.ftag, slots * sb);
  if (stamps) e.ensure(L.fstamp, slots * 4);
  e.ensure(L.fbits, slots / 8);
  e.ensure(L.start, recent * 4);
  e.ensure(L.state, kLinSlots * 8);
  // an add-mult iteration that is not the last adds a fact, so there are at most
  // as many as slots; the other semirings' backward passes need no record
  if (stamps) e.ensure(L.rec, (slots + 1) * A.n_rel * 4);
  u64 at = 0;
  for (int q = 0; q < A.n_rel; q++) {
    const RelSt& R = e.rels[L.rels[q]];
    if (R.n_recent) {
      k_lin_slots<<<lin_grid(R.n_recent), 256, 0, e.stream>>>(R.rkeys.p, R.views[0].lay.key64, R.n_recent, A.base[q],
                                                              L.start.as<u32>() + at);
      e.after_launch("linear facts");
      e.launches++;
    }
    at += R.n_recent;
  }
  A.n_arm = (int)arms.size();
  A.arms = L.arms.as<LinArm>();
  A.acc = L.acc.p;
  A.touched = L.touched.as<u32>();
  A.list = L.list.as<u32>();
  A.ftag = L.ftag.p;
  A.fstamp = L.fstamp.as<u32>();
  A.fbits = L.fbits.as<u32>();
  A.start = L.start.as<u32>();
  A.n_start = recent;
  A.max_iters = max_iters;
  A.state = L.state.as<u64>();
  A.rec = L.rec.as<u32>();
  // A block per 16,384 probed rows: a grid of side 64 has about 200 recent facts
  // in an iteration, which one block expands in a round or two without a grid
  // barrier.  Unions of proofs are worth more blocks: the loop over 64 grids of
  // side 16 (65,000 rows) takes 1.61 / 1.19 / 0.98 / 0.90 / 0.87 ms with a block
  // per 4,096 / 2,048 / 1,024 / 512 / 256 rows.
  const u64 share = top1 ? 512 : 16384;
  const unsigned blocks = (unsigned)std::max<u64>(1, std::min<u64>(e.sms, probed / share));
  A.k0 = k0;
  A.slots = (u32)slots;
  std::vector<u64> h(kLinSlots, 0);
  do {  // again when the proof arena ran out: the loop changes only arrays of its own
    e.check(cudaMemsetAsync(L.acc.p, 0, 2 * slots * cb, e.stream), "accumulators");
    e.check(cudaMemsetAsync(L.touched.p, 0, 2 * (slots / 8), e.stream), "accumulators");
    e.check(cudaMemsetAsync(L.ftag.p, 0, slots * sb, e.stream), "tags");
    e.check(cudaMemsetAsync(L.fbits.p, 0, slots / 8, e.stream), "membership");
    e.check(cudaMemsetAsync(L.state.p, 0, kLinSlots * 8, e.stream), "linear state");
    for (int q = 0; q < A.n_rel; q++) {
      if (sb == 8) L.init<u64>(e.rels[L.rels[q]], A.base[q]);
      else L.init<float>(e.rels[L.rels[q]], A.base[q]);
    }
    if (top1) A.top1 = top1_desc(e);
    switch (ks) {
      case SR_MAX_MIN: L.launch<SemMaxMin>(A, blocks); break;
      case SR_DIFF_MAX_MIN: L.launch<SemDiffMaxMin>(A, blocks); break;
      case SR_TOP1: L.launch<SemTop1>(A, blocks); break;
      default: L.launch<SemAddMult>(A, blocks); break;
    }
  } while (top1 && !top1_settle(e));
  e.check(cudaMemcpyAsync(h.data(), L.state.p, kLinSlots * 8, cudaMemcpyDeviceToHost, e.stream), "linear state");
  e.sync();
  if (h[LS_ERR]) throw LobError(LOB_E_TIMEOUT, "a bounded wait of the linear loop gave up; the run's results are invalid");
  if (h[LS_STOP] != LIN_FIXPOINT && h[LS_STOP] != LIN_MAXITER)
    throw LobError(LOB_E_CUDA, "internal error: linear loop stopped without a reason");
  const u32 ran = (u32)h[LS_ITER] - k0;
  std::vector<u32> rec(stamps ? (u64)ran * A.n_rel : 0);
  if (stamps)
    e.check(cudaMemcpyAsync(rec.data(), L.rec.p, rec.size() * 4, cudaMemcpyDeviceToHost, e.stream), "linear record");
  if (stamps) e.sync();
  out.first = k0 + 1;
  out.last = k0 + ran;
  out.max_iter = h[LS_STOP] == LIN_MAXITER;
  for (u32 i = 0; i < ran; i++) {  // counts at the start of iteration k0 + 1 + i
    out.counts.emplace_back();
    for (int q = 0; q < A.n_rel; q++) {
      const u64 last = i ? (stamps ? rec[(u64)(i - 1) * A.n_rel + q] : 0) : e.rels[L.rels[q]].n_recent;
      const u64 full = i ? out.counts[i - 1][q].first + (stamps ? last : 0) : A.fcount[q];
      out.counts.back().emplace_back(full, last);
    }
  }
  s.graph_launches++;
  s.device_iterations += ran;
  s.new_facts += h[LS_NEW];
  e.cand_emitted += h[LS_CAND];
  // the relations in key order again
  for (int q = 0; q < A.n_rel; q++) {
    RelSt& R = e.rels[L.rels[q]];
    ViewSt& V = R.views[0];
    const u64 n = h[LS_FULL + q], nbits = lin_slots(e, R);
    out.rels.push_back(L.rels[q]);
    out.n_recent.push_back(h[LS_LAST + q]);
    R.n_recent = 0;
    R.finished = true;
    for (auto& kv : V.index) kv.second.valid = false;
    for (size_t vi = 1; vi < R.views.size(); vi++) R.views[vi].stale = true;
    const u32* bits = L.fbits.as<u32>() + A.base[q] / 32;
    const int kb = V.lay.key64 ? 8 : 4;
    e.ensure(e.scratch, bits_scratch_bytes(nbits));
    e.launches += bits_count(bits, nullptr, nbits, e.scratch.p, e.counts.as<u64>() + 1, e.stream);
    e.after_launch("linear result");
    e.ensure(V.keys, n * kb);
    e.ensure(V.tags, n * sb);
    if (stamps) e.ensure(V.stamps, n * 4);
    bits_extract(bits, nullptr, nbits, V.lay.key64, V.keys.p, n, e.scratch.p, e.stream);
    e.after_launch("linear result");
    e.launches++;
    V.n = n;
    if (sb == 8) L.collect<u64>(R, A.base[q]);
    else L.collect<float>(R, A.base[q]);
  }
  out.taken = true;
}

void linear_merge(lob_engine& e, u32 k, const LinearOut& out) {
  if (!out.taken) return;
  const size_t nrel = e.rels.size();
  while (e.iter_counts.size() < k) {  // iterations only the linear components ran: the rest is at rest
    e.iter_counts.emplace_back();
    for (size_t r = 0; r < nrel; r++) e.iter_counts.back().emplace_back(e.rels[r].views[0].n, 0);
  }
  for (size_t q = 0; q < out.rels.size(); q++) {
    const u32 r = out.rels[q];
    for (u32 it = out.first; it <= k; it++)
      e.iter_counts[it - 1][r] = it <= out.last ? out.counts[it - out.first][q]
                                                : std::make_pair((u64)e.rels[r].views[0].n, (u64)0);
    e.rels[r].n_recent = out.max_iter ? out.n_recent[q] : 0;
  }
}

bool linear_backward(lob_engine& e, const LinearAdjoints& J, const std::vector<char>& needed, std::vector<char>& in,
                     bool& extra) {
  if (!e.opt_packed_backward || !linear_component(e, in)) return false;
  // a rule's head is needed only if its body is, so what is needed of a component
  // takes its adjoints from needed heads alone
  bool any = false;
  for (size_t r = 0; r < in.size(); r++) any = (in[r] = in[r] && needed[r]) || any;
  if (!any) return false;
  const u32 last = e.last_iter;
  LinRun L(e);
  L.index.assign(e.rels.size(), -1);
  LinBwdArgs A;
  std::memset(&A, 0, sizeof(A));
  u64 rows = 0, probed = 0;
  for (size_t r = 0; r < e.rels.size(); r++) {
    if (!in[r]) continue;
    const ViewSt& V = e.rels[r].views[0];
    if (V.n && !J.hrow[r]) return false;
    L.index[r] = A.n_rel;
    LinBwdRel& B = A.rel[A.n_rel++];
    B.keys = V.keys.p;
    B.key64 = V.lay.key64;
    B.tags = V.tags.as<float>();
    B.stamps = V.stamps.as<u32>();
    B.hrow = J.hrow[r];
    B.adj = J.adj[r];
    B.base = (u32)rows;
    rows += V.n;
    L.rels.push_back((u32)r);
  }
  if (rows >= 0xFFFFFFFFull) return false;
  std::vector<LinBwdArm> arms;
  for (auto& p : e.plans)
    for (auto& Ar : p.arms) {
      const u32 drel = p.ast.body[Ar.delta].rel;
      if (L.index[p.ast.head.rel] < 0 || !e.rels[drel].idb) continue;
      const StepPlan& S = Ar.steps[1];
      const u32 vrel = p.ast.body[S.atom].rel;
      ViewSt& W = e.rels[vrel].views[S.view];
      if (W.n > 0x7FFFFFFull) return false;
      if (!W.n) continue;
      engine_ensure_index(e, W, S.prefix_len);
      LinBwdArm a;
      std::memset(&a, 0, sizeof(a));
      a.P = Ar.packed.steps[0];
      a.drel = L.index[drel];
      a.hrel = L.index[p.ast.head.rel];
      a.P.v_keys = W.keys.p;
      a.P.v_key64 = W.lay.key64;
      a.P.v_tags = W.tags.p;
      a.P.v_n = W.n;
      const IndexSt& I = W.index[S.prefix_len];
      a.P.index_mode = I.mode;
      a.P.dense_offs = I.offs.as<u64>();
      a.P.hash_bits = I.hash_bits;
      a.prow = S.view ? J.prow[vrel][S.view] : nullptr;
      a.vadj = e.rels[vrel].in_has_tags ? J.adj[vrel] : nullptr;
      probed += W.n;
      arms.push_back(a);
    }
  if (last < 2 || arms.empty() || !rows) return true;  // iterations after the first derived nothing
  extra = true;
  e.ensure(L.arms, arms.size() * sizeof(LinBwdArm));
  e.check(cudaMemcpyAsync(L.arms.p, arms.data(), arms.size() * sizeof(LinBwdArm), cudaMemcpyHostToDevice, e.stream), "arms");
  // entries by stamp: counts (scanned in place), fill positions
  DevBuf &off = L.list, &used = L.used, &entries = L.start;
  const u64 ns = (u64)last + 1;
  e.ensure(off, (ns + 1) * 4);
  e.ensure(used, ns * 4);
  e.ensure(entries, rows * 4);
  e.ensure(L.state, kLinSlots * 8);
  e.check(cudaMemsetAsync(off.p, 0, (ns + 1) * 4, e.stream), "stamps");
  e.check(cudaMemsetAsync(used.p, 0, ns * 4, e.stream), "stamps");
  e.check(cudaMemsetAsync(L.state.p, 0, kLinSlots * 8, e.stream), "stamps");
  for (int q = 0; q < A.n_rel; q++) {
    const u64 n = e.rels[L.rels[q]].views[0].n;
    if (n) k_lin_stamp_count<<<lin_grid(n), 256, 0, e.stream>>>(A.rel[q].stamps, n, last, off.as<u32>());
  }
  e.after_launch("stamps");
  e.ensure(e.scratch, scan_scratch_elems(ns + 1) * 4 + 64);
  exclusive_scan<u32, u32>(off.as<u32>(), off.as<u32>(), ns + 1, nullptr, e.scratch.as<u32>(), e.stream);
  e.after_launch("stamps");
  for (int q = 0; q < A.n_rel; q++) {
    const u64 n = e.rels[L.rels[q]].views[0].n;
    if (n)
      k_lin_stamp_fill<<<lin_grid(n), 256, 0, e.stream>>>(A.rel[q].stamps, n, last, A.rel[q].base, off.as<u32>(),
                                                         used.as<u32>(), entries.as<u32>());
  }
  e.after_launch("stamps");
  A.n_arm = (int)arms.size();
  A.arms = L.arms.as<LinBwdArm>();
  A.entries = entries.as<u32>();
  A.off = off.as<u32>();
  A.last = last;
  A.state = L.state.as<u64>();
  const unsigned blocks = (unsigned)std::max<u64>(1, std::min<u64>(e.sms, probed / 16384));
  void* args[] = {&A};
  {
    ProfScope ps("linear_backward", 0, e.stream);
    e.check(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_linear_backward), dim3(blocks), dim3(kLinThreads), args, 0,
                                        e.stream), "linear backward");
  }
  e.after_launch("linear backward");
  if (e.read_u64(L.state.as<u64>() + LS_ERR))
    throw LobError(LOB_E_TIMEOUT, "a bounded wait of the backward pass gave up; its gradients are invalid");
  return true;
}
