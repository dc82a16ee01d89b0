// lob_unique_rows_noalloc: sort and deduplicate a small batch of rows without
// allocating any device memory.
//
// Some callers cannot allocate device memory at the point where they need this
// step: latency-critical serving paths where cudaMalloc / cudaFree would
// synchronise the device or wait on the driver, plug-ins that run inside a host
// application which owns and budgets all device memory itself, and processes
// that have split the GPU's memory among tenants ahead of time.  For them this
// entry point works entirely in one fixed scratch array that is part of the
// library image: every GPU that loads the library holds it (kScratchBytes,
// about 4.3 MB) until the process exits.
//
// The scratch array is shared by every call on a device and keeps whatever the
// last call left in it.  Everything a call reads from it is written earlier in
// the same call: keys, digit counts, the blocks' maxima and row counts, and the
// barrier words, which a memset before the launch clears (about 2 us).  Two calls
// whose work overlaps on the GPU (for example on two streams at once) race on the
// array, and callers must order them; should they not, those two results are wrong
// and no later call's.  The calls of a process take turns at kHeads sets of barrier
// words, so that one of the two cannot clear what the other's blocks wait for.
//
// One cooperative launch does it all: the columns' largest values (a barrier), keys
// packed into as few bits as those need, the radix passes over them
// (sort_fused.cuh), and the distinct keys counted (a barrier) and written out.
// What bounds it: the barriers and the chain within a pass, about 9 us for each
// 8 bits of key.  Pack, 40 sort launches, three for the distinct rows and unpack
// took 219 us for 100,003 rows of two columns; one launch takes 53.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "../../include/lobster.h"
#include "kernels.h"
#include "sort_fused.cuh"

namespace {

constexpr u64 kMaxRows = LOB_NOALLOC_MAX_ROWS;
constexpr u64 kKeyBytes = kMaxRows * sizeof(u64);
// digit counts, then per block its columns' maxima and row count; barrier words
constexpr u64 kCountWords = fused_count_words(kFTiles) + 4 * kFTiles;
constexpr u32 kHeads = 64;
constexpr u64 kScratchBytes = 2 * kKeyBytes + kCountWords * 4 + (u64)kHeads * kFHead * 4;
static_assert(kScratchBytes <= 4600000, "scratch budget");
static_assert(512ull * kFItems * kFTiles >= kMaxRows, "the largest batch fits the launch");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
std::atomic<u32> g_calls{0};
unsigned char* g_scratch_ptr[kMaxDevices] = {nullptr};

// Host code must not use g_noalloc_scratch directly: on the host that name is
// only a stand-in for the device symbol.  The device address comes from
// cudaGetSymbolAddress, once per device, with that device current.
int scratch_for_current_device(unsigned char** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return LOB_E_CUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) return LOB_E_ARG;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return LOB_E_CUDA;
    }
    g_scratch_ptr[dev] = reinterpret_cast<unsigned char*>(p);
  }
  *out = g_scratch_ptr[dev];
  return LOB_OK;
}

LOB_DEV int bit_count(u32 x) { return 32 - __clz(x); }

template <int NT>
__global__ void __launch_bounds__(NT, 1) k_unique_rows(const u32* __restrict__ cols, u32 arity, u64 n, u32* __restrict__ out,
                                                       u64* __restrict__ n_out, u64* keys_a, u64* keys_b, u32* counts, u32* head) {
  typedef FusedSmem<u64, NoPay, NT> Smem;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem& S = *reinterpret_cast<Smem*>(smem_raw);
  __shared__ u32 red[2][NT / 32];
  __shared__ u64 sm64[NT / 32 + 1];
  u32* per_block = counts + fused_count_words(kFTiles);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  FusedTile<u64, NoPay, NT> T;
  T.place(n);
  T.src_k = keys_a;
  T.dst_k = keys_b;
  u32 gen = 0;
  bool good = true;
  // the rows, and the largest value of each column
  u32 c0[kFItems], c1[kFItems], m0 = 0, m1 = 0;
#pragma unroll
  for (int r = 0; r < kFItems; r++) {
    const bool v = T.valid(r);
    c0[r] = v ? cols[T.at(r)] : 0u;
    c1[r] = v && arity == 2 ? cols[n + T.at(r)] : 0u;
    m0 = max(m0, c0[r]);
    m1 = max(m1, c1[r]);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    m0 = max(m0, __shfl_xor_sync(0xFFFFFFFFu, m0, o));
    m1 = max(m1, __shfl_xor_sync(0xFFFFFFFFu, m1, o));
  }
  if (lane == 0) { red[0][warp] = m0; red[1][warp] = m1; }
  __syncthreads();
  for (int w = 0; w < NT / 32; w++) { m0 = max(m0, red[0][w]); m1 = max(m1, red[1][w]); }
  if (gridDim.x > 1) {
    if (threadIdx.x == 0) { per_block[2 * blockIdx.x] = m0; per_block[2 * blockIdx.x + 1] = m1; }
    good = fused_barrier(head, gen);
    m0 = m1 = 0;
    for (u32 b = lane; b < gridDim.x; b += 32) {
      m0 = max(m0, __ldcg(per_block + 2 * b));
      m1 = max(m1, __ldcg(per_block + 2 * b + 1));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      m0 = max(m0, __shfl_xor_sync(0xFFFFFFFFu, m0, o));
      m1 = max(m1, __shfl_xor_sync(0xFFFFFFFFu, m1, o));
    }
  }
  const int b1 = arity == 2 ? bit_count(m1) : 0, bits = bit_count(m0) + b1;
#pragma unroll
  for (int r = 0; r < kFItems; r++)
    if (T.valid(r)) {
      T.k[r] = ((u64)c0[r] << b1) | c1[r];
      keys_a[T.at(r)] = T.k[r];
    }
  // (a pass's count barrier comes before anything reads the keys of another block)
  good = good && fused_passes(T, S, n, bits, head, counts, gen);
  // distinct keys: those that differ from the one before; a row of all ones is dropped
  if (good) {
#pragma unroll
    for (int r = 0; r < kFItems; r++)
      if (T.valid(r)) S.keys[T.wofs + r * 32 + lane] = T.k[r];
    if (gridDim.x > 1 && bits == 0) good = fused_barrier(head, gen);  // no pass had one
    __syncthreads();
  }
  u32 heads[kFItems], mine = 0;
  if (good) {
#pragma unroll
    for (int r = 0; r < kFItems; r++) {
      const int o = T.wofs + r * 32 + lane;
      bool h = T.valid(r);
      if (h) {
        const u32 x = (u32)(T.k[r] >> b1), y = arity == 2 ? (u32)(T.k[r] & ((1ull << b1) - 1)) : 0xFFFFFFFFu;
        if (x == 0xFFFFFFFFu && y == 0xFFFFFFFFu) h = false;
        else if (o) h = S.keys[o - 1] != T.k[r];
        else if (T.tbase) h = __ldcg(T.src_k + T.tbase - 1) != T.k[r];
      }
      heads[r] = __ballot_sync(0xFFFFFFFFu, h);
      mine += __popc(heads[r]);
    }
  }
  u64 tile_count;
  const u64 wbase = block_exclusive_sum<u64>(lane == 0 ? (u64)mine : 0ull, sm64, &tile_count);
  u64 pos = __shfl_sync(0xFFFFFFFFu, wbase, 0), all = tile_count;
  if (gridDim.x > 1) {
    u32* rows = per_block + 2 * kFTiles;
    if (good) {
      if (threadIdx.x == 0) rows[blockIdx.x] = (u32)tile_count;
      good = fused_barrier(head, gen);
    }
    u64 before = 0;
    all = 0;
    for (u32 b = lane; b < gridDim.x; b += 32) {
      const u32 c = good ? __ldcg(rows + b) : 0u;
      all += c;
      if (b < blockIdx.x) before += c;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      all += __shfl_xor_sync(0xFFFFFFFFu, all, o);
      before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
    }
    pos += before;
  }
  if (good) {
#pragma unroll
    for (int r = 0; r < kFItems; r++) {
      if ((heads[r] >> lane) & 1u) {
        const u64 o = pos + __popc(heads[r] & ((1u << lane) - 1u));
        out[o] = (u32)(T.k[r] >> b1);
        if (arity == 2) out[n + o] = (u32)(T.k[r] & ((1ull << b1) - 1));
      }
      pos += __popc(heads[r]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_out = all;
  }
  if (gridDim.x > 1 && threadIdx.x == 0) {  // the last block to leave: did some block give up?
    __threadfence();
    if (atomicAdd(head + 2, 1u) + 1 == gridDim.x && *reinterpret_cast<volatile u32*>(head + 1)) *n_out = ~0ull;
  }
}

template <int NT>
cudaError_t launch_unique_rows(const u32* cols, u32 arity, u64 n, u32* out, u64* n_out, unsigned char* s, cudaStream_t st) {
  u64* a = reinterpret_cast<u64*>(s);
  u64* b = reinterpret_cast<u64*>(s + kKeyBytes);
  u32* counts = reinterpret_cast<u32*>(s + 2 * kKeyBytes);
  u32* head = counts + kCountWords + kFHead * (g_calls.fetch_add(1, std::memory_order_relaxed) % kHeads);
  constexpr int kSm = (int)sizeof(FusedSmem<u64, NoPay, NT>);
  if (kSm > 48 * 1024) allow_dynamic_smem(k_unique_rows<NT>, kSm);
  const unsigned tiles = (unsigned)std::max<u64>(1, (n + NT * kFItems - 1) / (NT * kFItems));
  if (tiles == 1) {
    k_unique_rows<NT><<<1, NT, kSm, st>>>(cols, arity, n, out, n_out, a, b, counts, head);
    return cudaGetLastError();
  }
  const cudaError_t cleared = cudaMemsetAsync(head, 0, kFHead * sizeof(u32), st);
  if (cleared != cudaSuccess) return cleared;
  void* args[] = {&cols, &arity, &n, &out, &n_out, &a, &b, &counts, &head};
  return cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_unique_rows<NT>), dim3(tiles), dim3(NT), args, kSm, st);
}

}  // namespace

extern "C" int lob_unique_rows_noalloc(const uint32_t* cols, uint32_t arity, uint64_t n, uint32_t* out_cols,
                                       uint64_t* n_out, void* cuda_stream) {
  if (!n_out || (arity != 1 && arity != 2) || (n && (!cols || !out_cols))) return LOB_E_ARG;
  if (n > kMaxRows) return LOB_E_CAPACITY;
  unsigned char* s = nullptr;
  int rc = scratch_for_current_device(&s);
  if (rc != LOB_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = n <= 256ull * kFItems * kFTiles
                      ? launch_unique_rows<256>(cols, arity, n, out_cols, reinterpret_cast<u64*>(n_out), s, st)
                      : launch_unique_rows<512>(cols, arity, n, out_cols, reinterpret_cast<u64*>(n_out), s, st);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess ? LOB_OK : LOB_E_CUDA;
}
