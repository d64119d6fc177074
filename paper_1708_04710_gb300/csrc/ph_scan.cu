// Device scans and the LSD radix sort used to order simplices by squared diameter.
//
// Both are tile based: a tile is kThreads * kItems consecutive elements handled by one block. Tiles
// take their turns from a ticket and wait for earlier ones (with a bound).
#include <utility>

#include "ph_internal.cuh"

namespace ph {

constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;

// ---------------------------------------------------------------------------------------------
// exclusive scans of one or two int32 arrays into int64 (n + 1 values each, the total last), in one
// kernel: tiles in order from a ticket, each publishing its sum and looking back over the tiles
// before it (decoupled look-back). state: per array one word per tile, zeroed before
// ---------------------------------------------------------------------------------------------
__global__ void k_scan_counts(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int64_t n,
                              int64_t* oa, int64_t* ob, unsigned long long* state,
                              int64_t ntiles, unsigned int* ticket, int32_t* fault) {
  __shared__ int64_t sh[kWarps + 1];
  __shared__ int64_t s_prefix[2];
  __shared__ unsigned int s_tile;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  __syncthreads();
  const int64_t t = s_tile;
  const int64_t i0 = t * kTile + threadIdx.x * kItems;
  for (int k = 0; k < (b ? 2 : 1); k++) {
    const int32_t* in = k ? b : a;
    int64_t* out = k ? ob : oa;
    int32_t x[kItems];
    int64_t sum = 0;
#pragma unroll
    for (int i = 0; i < kItems; i++) {
      x[i] = i0 + i < n ? in[i0 + i] : 0;
      sum += x[i];
    }
    int64_t tot;
    int64_t run = block_excl_sum<int64_t>(sum, sh, tot);
    if (threadIdx.x < 32) {
      const int64_t p = tile_prefix(state + k * ntiles, t, tot, fault);
      if (threadIdx.x == 0) s_prefix[k] = p;
    }
    __syncthreads();
    run += s_prefix[k];
#pragma unroll
    for (int i = 0; i < kItems; i++) {
      if (i0 + i < n) out[i0 + i] = run;
      run += x[i];
      if (i0 + i == n - 1) out[n] = run;
    }
  }
}

// a (and b, unless null): n counts each; n >= 1. fault: set when a bounded wait ran out
void scan_counts(ph_ctx* ctx, const int32_t* a, const int32_t* b, int64_t n, int64_t* oa,
                 int64_t* ob, int32_t* fault) {
  const int64_t ntiles = (n + kTile - 1) / kTile;
  unsigned long long* state = alloc_n<unsigned long long>(ctx, 2 * ntiles + 1);
  PH_CUDA(cudaMemsetAsync(state, 0, (2 * ntiles + 1) * sizeof(unsigned long long), ctx->stream));
  k_scan_counts<<<(unsigned)ntiles, kThreads, 0, ctx->stream>>>(
      a, b, n, oa, ob, state, ntiles, (unsigned int*)(state + 2 * ntiles), fault);
  PH_CHECK_LAUNCH();
  ctx->dfree(state);
}

// ---------------------------------------------------------------------------------------------
// LSD radix sort of (uint64 key, uint64 value) pairs by key bits [lo_bit, hi_bit), stable.
// 8-bit digits, one kernel per digit: a tile ranks its elements per digit value in shared memory,
// publishes its 256 counts and looks back for those of the tiles before it, one thread per
// digit value, and scatters. One kernel before them counts every digit over all keys. Up to 8192 pairs
// are sorted by one block, all digits in one kernel (k_radix_tiles). Bound by the scattered 16-byte
// writes, by latency for short lists. With separate count, scan and scatter kernels per digit the
// sorts of a 400-point cloud's edges and triangles took 0.75 ms; its edges take 55 us now. A block
// of 8192 pairs takes as long as the kernels over the whole device (7140 pairs, 5 digits: 39 against
// 43 us) but is one launch, and a batch's clouds sort side by side: the edges of 512 clouds of 20 to
// 120 points 290 -> 130 us.
// ---------------------------------------------------------------------------------------------
constexpr int kMaxDigits = 8;

__global__ void k_radix_count(const uint64_t* __restrict__ keys, int64_t n, int lo_bit, int digits,
                              unsigned long long* hist) {
  __shared__ unsigned cnt[kMaxDigits][256];
  for (int d = 0; d < digits; d++) cnt[d][threadIdx.x] = 0;
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = keys[i] >> lo_bit;
    for (int d = 0; d < digits; d++) atomicAdd(&cnt[d][(k >> (8 * d)) & 255u], 1u);
  }
  __syncthreads();
  for (int d = 0; d < digits; d++)
    if (cnt[d][threadIdx.x])
      atomicAdd(&hist[d * 256 + threadIdx.x], (unsigned long long)cnt[d][threadIdx.x]);
}

// Ranks of a tile's elements: element i of a thread is the tile's element warp * 256 + 32 i + lane.
// cnt[w][d] becomes the number of the tile's elements with digit d in warps before w; returns this
// thread's digit value's (threadIdx.x) number in the tile.
template <int NW>
__device__ __forceinline__ unsigned tile_ranks(const unsigned (&digit)[kItems],
                                               unsigned (&rank)[kItems],
                                               unsigned (*cnt)[257]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int d = lane; d < 257; d += 32) cnt[w][d] = 0;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < kItems; i++) {
    const unsigned peers = __match_any_sync(0xffffffffu, digit[i]);
    const unsigned old = cnt[w][digit[i]];
    rank[i] = old + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
    if (lane == __ffs(peers) - 1) cnt[w][digit[i]] = old + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  unsigned run = 0;
  if (NW > kWarps && threadIdx.x >= 256) return run;
#pragma unroll
  for (int v = 0; v < NW; v++) {
    const unsigned c = cnt[v][threadIdx.x];
    cnt[v][threadIdx.x] = run;
    run += c;
  }
  return run;
}

__global__ void __launch_bounds__(kThreads) k_radix_pass(
    const uint64_t* __restrict__ kin, const uint64_t* __restrict__ vin,
    uint64_t* __restrict__ kout, uint64_t* __restrict__ vout, int64_t n, int shift,
    const unsigned long long* __restrict__ hist, unsigned long long* state, unsigned int* ticket,
    int32_t* fault) {
  __shared__ unsigned cnt[kWarps][257];
  __shared__ int64_t base[256];
  __shared__ int64_t sh[kWarps + 1];
  __shared__ unsigned int s_tile;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);  // tiles in order: the look-back waits
  __syncthreads();
  const int64_t t = s_tile;
  const int64_t i0 = t * kTile + (threadIdx.x >> 5) * (32 * kItems) + (threadIdx.x & 31);
  uint64_t k[kItems], v[kItems];
  unsigned digit[kItems], rank[kItems];
#pragma unroll
  for (int i = 0; i < kItems; i++) {
    const bool in = i0 + 32 * i < n;
    k[i] = in ? kin[i0 + 32 * i] : 0;
    v[i] = in ? vin[i0 + 32 * i] : 0;
    digit[i] = in ? (unsigned)((k[i] >> shift) & 255u) : 256u;
  }
  const unsigned mine = tile_ranks<kWarps>(digit, rank, cnt);
  int64_t tot;
  int64_t b = block_excl_sum<int64_t>((int64_t)hist[threadIdx.x], sh, tot);
  unsigned long long* st = state + t * 256 + threadIdx.x;
  atomicExch(st, (t == 0 ? kIncl : kAgg) | mine);
  if (t > 0) {
    int64_t prefix = 0;
    bool done = false;
    for (int64_t p = t - 1; !done; p -= 8) {  // eight states in flight
      unsigned long long w[8];
#pragma unroll
      for (int q = 0; q < 8; q++)
        w[q] = p >= q ? *(const volatile unsigned long long*)(st - (t - p + q) * 256) : kIncl;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        if (done) continue;
        if (!(w[q] & kFlags)) w[q] = wait_state(st - (t - p + q) * 256, fault);
        prefix += (int64_t)(w[q] & ~kFlags);
        done = (w[q] & kFlags) == kIncl;
      }
    }
    atomicExch(st, kIncl | (unsigned long long)(prefix + mine));
    b += prefix;
  }
  base[threadIdx.x] = b;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kItems; i++) {
    if (digit[i] == 256u) continue;
    const int64_t pos = base[digit[i]] + cnt[threadIdx.x >> 5][digit[i]] + rank[i];
    if (pos >= n) continue;  // (only after a wait that gave up)
    kout[pos] = k[i];
    vout[pos] = v[i];
  }
}

// All digits of one tile per block: elements stay in registers and change places in shared memory.
// Tile b: elements off[b] .. off[b + 1], or all n without off; at most NW * 256. largest (device):
// the keys have one bit more than this value, instead of `digits`
template <int NW>
__global__ void __launch_bounds__(NW * 32) k_radix_tiles(uint64_t* keys, uint64_t* vals,
                                                         const int64_t* __restrict__ off, int64_t n,
                                                         int lo_bit, int digits,
                                                         const unsigned long long* largest) {
  extern __shared__ uint64_t sm[];
  uint64_t* xk = sm;
  uint64_t* xv = xk + NW * 256;
  unsigned (*cnt)[257] = reinterpret_cast<unsigned (*)[257]>(xv + NW * 256);
  __shared__ unsigned base[256], sums[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t first = off ? off[blockIdx.x] : 0;
  if (largest) digits = (min(64, 65 - __clzll((long long)*largest)) + 7) / 8;
  const int len = (int)(off ? off[blockIdx.x + 1] - first : n);
  keys += first;
  vals += first;
  const int i0 = w * 256 + lane;
  uint64_t k[8], v[8];
  unsigned digit[8], rank[8];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    k[i] = i0 + 32 * i < len ? keys[i0 + 32 * i] : 0;
    v[i] = i0 + 32 * i < len ? vals[i0 + 32 * i] : 0;
  }
  for (int p = 0; p < digits; p++) {
#pragma unroll
    for (int i = 0; i < 8; i++)
      digit[i] = i0 + 32 * i < len ? (unsigned)((k[i] >> (lo_bit + 8 * p)) & 255u) : 256u;
    const unsigned mine = tile_ranks<NW>(digit, rank, cnt);
    unsigned inc = warp_incl_sum(mine);
    if (threadIdx.x < 256 && lane == 31) sums[w] = inc;
    // (also the barrier before the sums are read) one value for all: nothing moves
    if (__syncthreads_or(threadIdx.x < 256 && (int)mine == len)) continue;
    if (threadIdx.x < 256) {
      for (int q = 0; q < w; q++) inc += sums[q];
      base[threadIdx.x] = inc - mine;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; i++) {
      if (digit[i] == 256u) continue;
      const unsigned pos = base[digit[i]] + cnt[w][digit[i]] + rank[i];
      xk[pos] = k[i];
      xv[pos] = v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; i++) {
      if (i0 + 32 * i < len) {
        k[i] = xk[i0 + 32 * i];
        v[i] = xv[i0 + 32 * i];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; i++) {
    if (i0 + 32 * i < len) {
      keys[i0 + 32 * i] = k[i];
      vals[i0 + 32 * i] = v[i];
    }
  }
}

template <int NW>
static void launch_tiles(ph_ctx* ctx, uint64_t* keys, uint64_t* vals, const int64_t* off,
                         int ntiles, int64_t n, int lo_bit, int digits,
                         const unsigned long long* largest) {
  constexpr size_t bytes = NW * 256 * 16 + NW * 257 * sizeof(unsigned);
  if (bytes > 48 * 1024)
    PH_CUDA(cudaFuncSetAttribute(k_radix_tiles<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)bytes));
  k_radix_tiles<NW><<<ntiles, NW * 32, bytes, ctx->stream>>>(keys, vals, off, n, lo_bit, digits,
                                                             largest);
  PH_CHECK_LAUNCH();
}

// sorts each of ntiles ranges (off[t] .. off[t + 1], device) of at most longest <= kSortTile pairs
// by itself, in one kernel; off null: one range of longest pairs. largest: see k_radix_tiles
void radix_sort_tiles(ph_ctx* ctx, uint64_t* keys, uint64_t* vals, const int64_t* off, int ntiles,
                      int64_t longest, int lo_bit, int hi_bit, const unsigned long long* largest) {
  if (longest <= 1 || (!largest && hi_bit <= lo_bit)) return;
  const int digits = (hi_bit - lo_bit + 7) / 8;
  if (longest <= 2048) launch_tiles<8>(ctx, keys, vals, off, ntiles, longest, lo_bit, digits,
                                        largest);
  else if (longest <= 4096) launch_tiles<16>(ctx, keys, vals, off, ntiles, longest, lo_bit, digits,
                                        largest);
  else launch_tiles<32>(ctx, keys, vals, off, ntiles, longest, lo_bit, digits,
                                        largest);
}

// fault: device word, set when a bounded wait ran out (the order is then incomplete)
void radix_sort_u64(ph_ctx* ctx, uint64_t* keys, uint64_t* vals, int64_t n, int lo_bit,
                    int hi_bit, uint64_t* tmp_keys, uint64_t* tmp_vals, int32_t* fault) {
  if (n <= 1 || hi_bit <= lo_bit) return;
  cudaStream_t st = ctx->stream;
  const int digits = (hi_bit - lo_bit + 7) / 8;
  if (n <= kSortTile) {
    radix_sort_tiles(ctx, keys, vals, nullptr, 1, n, lo_bit, hi_bit);
    return;
  }
  const int64_t ntiles = (n + kTile - 1) / kTile;
  // per digit: its counts, its ticket, its tiles' states (long sorts: one digit's, cleared in between)
  constexpr int64_t kManyStates = 4 << 20;
  const int64_t states = 256 * ntiles;
  const bool again = states * digits > kManyStates;
  const int64_t words = 257 * digits + states * (again ? 1 : digits);
  unsigned long long* buf = alloc_n<unsigned long long>(ctx, words);
  unsigned long long* ticket = buf + 256 * digits;
  unsigned long long* state = ticket + digits;
  PH_CUDA(cudaMemsetAsync(buf, 0, words * sizeof(unsigned long long), st));
  k_radix_count<<<grid_for(ctx, n, kThreads * 4), kThreads, 0, st>>>(keys, n, lo_bit, digits, buf);
  PH_CHECK_LAUNCH();
  uint64_t *ka = keys, *va = vals, *kb = tmp_keys, *vb = tmp_vals;
  for (int p = 0; p < digits; p++) {
    if (again && p > 0)
      PH_CUDA(cudaMemsetAsync(state, 0, states * sizeof(unsigned long long), st));
    k_radix_pass<<<(unsigned)ntiles, kThreads, 0, st>>>(
        ka, va, kb, vb, n, lo_bit + 8 * p, buf + 256 * p, state + (again ? 0 : states * p),
        (unsigned int*)(ticket + p), fault);
    PH_CHECK_LAUNCH();
    std::swap(ka, kb);
    std::swap(va, vb);
  }
  if (ka != keys) {
    PH_CUDA(cudaMemcpyAsync(keys, ka, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
    PH_CUDA(cudaMemcpyAsync(vals, va, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
  }
  ctx->dfree(buf);
}

}  // namespace ph
