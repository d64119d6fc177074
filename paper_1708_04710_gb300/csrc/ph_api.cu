// C ABI of the library: context life cycle, device memory, extraction of pairs and essential
// simplices (Lemma 1, Eq. paired), and inspection of the filtration.
#include <algorithm>
#include <cstring>
#include <functional>
#include <new>

#include "ph_internal.cuh"

// ---------------------------------------------------------------------------------------------
// device memory of a context
// ---------------------------------------------------------------------------------------------
// Blocks of up to kKeepBlock bytes that a context is done with are kept for its next allocations
// (kKeepTotal bytes in all), so that a program that builds and reduces small complexes again and
// again does not go through its allocator some sixty times per call. All use is in the order of
// the context's stream, so a kept block can be handed out at once. Blocks that no build since the
// one before last has used go back, and all do when an allocation fails.
constexpr size_t kKeepBlock = size_t(32) << 20, kKeepTotal = size_t(256) << 20;

void ph_ctx::give_back(const Block& b) {
  if (has_alloc) alloc.free(b.p, b.bytes, alloc.user, (void*)stream);
  else cudaFreeAsync(b.p, stream);
}

void ph_ctx::drop_kept(int64_t before) {
  size_t n = 0;
  for (const Kept& k : kept) {
    if (k.build < before) {
      give_back(k.b);
      kept_bytes -= k.b.bytes;
    } else {
      kept[n++] = k;
    }
  }
  kept.resize(n);
}

void* ph_ctx::dalloc(size_t bytes) {
  bytes = bytes <= 256 ? 256 : (bytes + 255) & ~size_t(255);
  // the smallest kept block that fits without much waste, the first in memory of several: builds of
  // one size then get the same blocks again, and find their pass graphs made (60 us each)
  size_t best = kept.size();
  for (size_t i = 0; i < kept.size(); i++) {
    const Block& b = kept[i].b;
    if (b.bytes < bytes || b.bytes > 2 * bytes + 65536) continue;
    if (best == kept.size() || b.bytes < kept[best].b.bytes ||
        (b.bytes == kept[best].b.bytes && std::less<void*>()(b.p, kept[best].b.p)))
      best = i;
  }
  if (best < kept.size()) {
    const Block b = kept[best].b;
    kept_bytes -= b.bytes;
    kept[best] = kept.back();
    kept.pop_back();
    blocks.push_back(b);
    return b.p;
  }
  void* p = nullptr;
  for (int attempt = 0; attempt < 3 && !p; attempt++) {
    if (attempt > 0) {  // make room: the kept blocks, then those a reduction can do without
      if (attempt > 1 && !ph::give_up_ahead(this)) break;
      if (attempt == 1 && kept.empty()) continue;
      drop_kept(INT64_MAX);
    }
    if (has_alloc) {
      p = alloc.alloc(bytes, alloc.user, (void*)stream);
    } else if (cudaMallocAsync(&p, bytes, stream) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
  }
  if (!p) {
    err = "device allocation of " + std::to_string(bytes) + " bytes failed";
    throw ph::Fail{PH_ERR_ALLOC};
  }
  if (reinterpret_cast<uintptr_t>(p) % 256 != 0) {  // the kernels copy in 16-byte units
    give_back({p, bytes});
    err = "the device allocator returned memory that is not 256-byte aligned";
    throw ph::Fail{PH_ERR_ALLOC};
  }
  blocks.push_back({p, bytes});
  return p;
}

void ph_ctx::keep_or_give_back(const Block& b) {
  if (b.bytes <= kKeepBlock && kept_bytes + b.bytes <= kKeepTotal) {
    kept.push_back({b, builds});
    kept_bytes += b.bytes;
  } else {
    give_back(b);
  }
}

void ph_ctx::dfree(void* p) {
  if (!p) return;
  for (size_t i = blocks.size(); i-- > 0;) {
    if (blocks[i].p == p) {
      const Block b = blocks[i];
      blocks[i] = blocks.back();
      blocks.pop_back();
      keep_or_give_back(b);
      return;
    }
  }
}

void* ph_ctx::pinned(size_t bytes) {
  if (bytes > h_pinned_bytes) {
    if (h_pinned) cudaFreeHost(h_pinned);
    h_pinned = nullptr;
    h_pinned_bytes = 0;
    if (cudaMallocHost(&h_pinned, bytes) != cudaSuccess) {
      cudaGetLastError();
      h_pinned = nullptr;
      err = "page-locked host allocation failed";
      throw ph::Fail{PH_ERR_ALLOC};
    }
    h_pinned_bytes = bytes;
  }
  return h_pinned;
}

void ph_ctx::free_all() {
  ph::free_reduce_state(this);
  builds++;
  drop_kept(builds - 1);
  for (auto& b : blocks) keep_or_give_back(b);
  blocks.clear();
  built = reduced = extracted = is_vr = false;
  // every pointer into the freed blocks must go: a stale one handed to dfree later could match
  // a new allocation at the same address and free it while it is in use
  p_birth = p_death = p_bd2 = p_dd2 = e_idx = e_d2 = out_delta = nullptr;
  p_dim = e_dim = nullptr;
  is_low = nullptr;
  out_before = nullptr;
  seg = low = beta = key = rows0 = nullptr;
  col_off = nullptr;
  gidx = nullptr;
  verts = nullptr;
  d2tab = nullptr;
  d_pt_off = nullptr;
  d_seg_start = nullptr;
  m = nnz = 0;
  D = 0;
  n_points = 0;
}

namespace ph {

// ---------------------------------------------------------------------------------------------
// extraction: pairs (low(j), j) for low(j) >= 0 and essential simplices (low(j) = -1 and j not
// the low of any column), written per cloud, ordered by (dimension, index)
// ---------------------------------------------------------------------------------------------
__global__ void k_mark_image(int64_t m, const int32_t* __restrict__ low, uint8_t* is_low) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < m;
       x += (int64_t)gridDim.x * blockDim.x) {
    int32_t l = low[x];
    if (l >= 0) is_low[l] = 1;
  }
}

// Extraction reads low twice and moves each result once. One scan counts, per tile of ids, the
// pairs and the essentials up to its end (one 64-bit state per tile, one kernel) and, at
// each segment's first id, how many come before it; the writers count again within a tile and
// write straight into the caller's arrays when these take all clouds' results on this device.
// Bound by memory for long complexes (per id 5 bytes in each kernel, plus the results with one
// gathered birth each), by the two waits of a request for short ones. With two flag arrays, six scan
// kernels and a copy of every result the pairs and essentials of 512 clouds of 20 to 120 points (42.7 M
// simplices) took 1.51 + 0.29 ms, now 0.38 + 0.39 ms; of 400 points 0.49 + 0.12 ms, now 0.16 + 0.14;
// of 40 points 183 + 37 us, now 67 + 28 us.
constexpr int kScanTile = 4096, kOutTile = 1024;  // ids per block of the scan; per counted place
// a writer's round takes kScanTile ids of a long complex (a round of 1024 held 39 pairs of a 512-cloud
// batch's and waited on each in turn: 256 us), kOutTile of a short one, whose rounds run side by side
constexpr int64_t kLongOut = 1 << 21;

// state: pairs << 31 | essentials (each total is below 2^31, that of the pairs below 2^30)
__device__ __forceinline__ int64_t pack_counts(unsigned pairs, unsigned ess) {
  return (int64_t)pairs << 31 | ess;
}

__device__ __forceinline__ int first_at_least(const int64_t* __restrict__ v, int n, int64_t x) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (v[mid] >= x) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// before: per kOutTile ids, the packed counts before them; seg_before: per segment (and the end)
__global__ void __launch_bounds__(kThreads) k_out_scan(
    int64_t m, int nseg, const int32_t* __restrict__ low, const uint8_t* __restrict__ is_low,
    const int64_t* __restrict__ seg_start, unsigned long long* state, int64_t ntiles,
    unsigned long long* before, int64_t* seg_before, unsigned int* ticket, int32_t* fault) {
  constexpr int kWords = kScanTile / 32, kPer = kWords / kWarps;
  // per word of 32 ids: its flags, and the tile's counts before it
  __shared__ uint32_t s_pair[kWords + 1], s_ess[kWords + 1];
  __shared__ int64_t s_before[kWords + 1];
  __shared__ unsigned s_tile;
  __shared__ int64_t s_prefix;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);  // tiles in order: the look-back waits
  __syncthreads();
  const int64_t t = s_tile, tile0 = t * kScanTile;
  int32_t l[kPer];
  uint8_t il[kPer];
#pragma unroll
  for (int i = 0; i < kPer; i++) {
    const int64_t x = tile0 + (w * kPer + i) * 32 + lane;
    l[i] = x < m ? low[x] : -1;
    il[i] = x < m ? is_low[x] : 1;
  }
#pragma unroll
  for (int i = 0; i < kPer; i++) {
    const unsigned pm = __ballot_sync(0xffffffffu, l[i] >= 0);
    const unsigned em = __ballot_sync(0xffffffffu, l[i] < 0 && !il[i]);
    if (lane == 0) {
      s_pair[w * kPer + i] = pm;
      s_ess[w * kPer + i] = em;
    }
  }
  __syncthreads();
  if (w == 0) {
    int64_t run = 0;
    for (int q = 0; q < kWords; q += 32) {
      const int64_t c = pack_counts(__popc(s_pair[q + lane]), __popc(s_ess[q + lane]));
      const int64_t inc = warp_incl_sum(c);
      s_before[q + lane] = run + inc - c;
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
    const int64_t p = tile_prefix(state, t, run, fault);
    if (lane == 0) {
      s_before[kWords] = run;
      s_pair[kWords] = s_ess[kWords] = 0;
      s_prefix = p;
    }
  }
  __syncthreads();
  if (threadIdx.x < kScanTile / kOutTile && tile0 + threadIdx.x * kOutTile < m)
    before[tile0 / kOutTile + threadIdx.x] =
        (unsigned long long)(s_prefix + s_before[threadIdx.x * (kOutTile / 32)]);
  // segments that start in this tile (at m: after the last)
  const int64_t end = t == ntiles - 1 ? m + 1 : tile0 + kScanTile;
  const int s1 = first_at_least(seg_start, nseg + 1, end);
  for (int s = first_at_least(seg_start, nseg + 1, tile0) + threadIdx.x; s < s1; s += blockDim.x) {
    const int i = (int)(seg_start[s] - tile0);
    const unsigned below = (1u << (i & 31)) - 1u;
    const int64_t v = s_prefix + s_before[i >> 5] +
                      pack_counts(__popc(s_pair[i >> 5] & below), __popc(s_ess[i >> 5] & below));
    seg_before[2 * s] = v >> 31;
    seg_before[2 * s + 1] = v & 0x7fffffff;
  }
}

__device__ __forceinline__ int64_t diam2_of(const int32_t* key, const int64_t* d2tab, int32_t x) {
  int32_t k = key[x];
  return k >= 0 ? d2tab[k] : 0;
}

struct OutArrays {  // the caller's or the internal arrays; null: not asked for
  int64_t *birth, *death, *bd2, *dd2;
  int32_t* dim;
};

// kEss: idx in death, its dimension in dim, its squared diameter in dd2. A round lists its pairs
// (or essentials) in shared memory first, so neighbouring threads take neighbouring results: of 42.7 M
// ids 1.6 M are pairs, and a lane per id left most lanes idle (380 us).
template <bool kEss, int kRound>
__global__ void __launch_bounds__(kThreads) k_write_out(
    int64_t m, int nc, const int32_t* __restrict__ seg, const int32_t* __restrict__ low,
    const uint8_t* __restrict__ is_low, const int64_t* __restrict__ gidx,
    const int32_t* __restrict__ key, const int64_t* __restrict__ d2tab,
    const unsigned long long* __restrict__ before, const int64_t* __restrict__ delta, OutArrays o,
    int64_t n, int32_t* bad) {
  constexpr int kPer = kRound / kThreads, kWordsPerLane = kRound / 1024;
  __shared__ uint16_t s_list[kRound];
  __shared__ unsigned s_cnt[kRound / 32];
  __shared__ int s_total;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t ntiles = (m + kRound - 1) / kRound;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t tile0 = t * kRound;
    const int64_t pre = (int64_t)before[tile0 / kOutTile];
    const int64_t base = kEss ? pre & 0x7fffffff : pre >> 31;
    bool f[kPer];
    unsigned mask[kPer];
#pragma unroll
    for (int i = 0; i < kPer; i++) {
      const int64_t x = tile0 + (w * kPer + i) * 32 + lane;
      f[i] = x < m && (kEss ? low[x] < 0 : low[x] >= 0);
      if (kEss) f[i] = f[i] & (x < m && !is_low[x]);
    }
    __syncthreads();  // the list of the round before is done with
#pragma unroll
    for (int i = 0; i < kPer; i++) {
      mask[i] = __ballot_sync(0xffffffffu, f[i]);
      if (lane == 0) s_cnt[w * kPer + i] = __popc(mask[i]);
    }
    __syncthreads();
    if (w == 0) {  // counts to places
      unsigned c[kWordsPerLane], sum = 0;
#pragma unroll
      for (int i = 0; i < kWordsPerLane; i++) sum += c[i] = s_cnt[lane * kWordsPerLane + i];
      unsigned run = warp_incl_sum(sum);
      if (lane == 31) s_total = (int)run;
      run -= sum;
#pragma unroll
      for (int i = 0; i < kWordsPerLane; i++) {
        s_cnt[lane * kWordsPerLane + i] = run;
        run += c[i];
      }
    }
    __syncthreads();
    const int cnt = s_total;
#pragma unroll
    for (int i = 0; i < kPer; i++) {
      const int q = w * kPer + i;
      if (f[i]) s_list[s_cnt[q] + __popc(mask[i] & ((1u << lane) - 1u))] = (uint16_t)(q * 32 + lane);
    }
    __syncthreads();
    for (int k0 = threadIdx.x; k0 < cnt; k0 += 2 * kThreads) {  // two results in flight
      int64_t x[2], p[2], ix[2];
      int32_t s[2], kx[2];
#pragma unroll
      for (int u = 0; u < 2; u++) {
        const int k = k0 + u * kThreads;
        x[u] = k < cnt ? tile0 + s_list[k] : -1;
        if (x[u] < 0) continue;
        s[u] = seg[x[u]];
        ix[u] = gidx[x[u]];
        kx[u] = key[x[u]];
      }
#pragma unroll
      for (int u = 0; u < 2; u++) {
        if (x[u] < 0) continue;
        p[u] = delta[2 * s[u] + kEss] + base + k0 + u * kThreads;
        if (p[u] < 0 || p[u] >= n) {
          *bad = 1;
          x[u] = -1;
        }
      }
#pragma unroll
      for (int u = 0; u < 2; u++) {
        if (x[u] < 0) continue;
        if (o.death) o.death[p[u]] = ix[u];
        if (o.dim) o.dim[p[u]] = s[u] / nc - (kEss ? 0 : 1);
        if (o.dd2) o.dd2[p[u]] = kx[u] >= 0 ? d2tab[kx[u]] : 0;
      }
      if (!kEss) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
          if (x[u] < 0) continue;
          const int32_t l = low[x[u]];
          if (o.birth) o.birth[p[u]] = gidx[l];
          if (o.bd2) o.bd2[p[u]] = diam2_of(key, d2tab, l);
        }
      }
    }
  }
}

static void drop_extraction(ph_ctx* ctx) {
  for (void* p : {(void*)ctx->p_birth, (void*)ctx->p_death, (void*)ctx->p_dim, (void*)ctx->p_bd2,
                  (void*)ctx->p_dd2, (void*)ctx->e_idx, (void*)ctx->e_dim, (void*)ctx->e_d2,
                  (void*)ctx->out_before, (void*)ctx->out_delta})
    ctx->dfree(p);
  ctx->p_birth = ctx->p_death = ctx->p_bd2 = ctx->p_dd2 = ctx->e_idx = ctx->e_d2 = nullptr;
  ctx->p_dim = ctx->e_dim = nullptr;
  ctx->is_low = nullptr;
  ctx->out_before = nullptr;
  ctx->out_delta = nullptr;
  ctx->extracted = false;
}

// the places of every pair and essential simplex: counts per cloud, tile states, segment shifts
static void extract_places(ph_ctx* ctx) {
  if (ctx->extracted) return;
  drop_extraction(ctx);
  cudaStream_t st = ctx->stream;
  const int64_t m = ctx->m, ntiles = (m + kScanTile - 1) / kScanTile;
  const int64_t nout = (m + kOutTile - 1) / kOutTile;
  const int nc = ctx->n_clouds;
  const int nseg = (int)ctx->seg_start.size() - 1;
  // counts before each tile, the scan's ticket and tile states, the image of low
  ctx->out_before = alloc_n<unsigned long long>(ctx, nout + 1 + ntiles + (m + 7) / 8);
  ctx->out_delta = alloc_n<int64_t>(ctx, 2 * nseg);
  unsigned long long* words = ctx->out_before + nout;
  ctx->is_low = reinterpret_cast<uint8_t*>(words + 1 + ntiles);
  PH_CUDA(cudaMemsetAsync(words, 0, (1 + ntiles) * sizeof(unsigned long long) + m, st));
  // the segments' counts and the fault word: written by the scan into page-locked memory (a copy back
  // would be two more operations to wait for)
  int64_t* sg = static_cast<int64_t*>(ctx->pinned((2 * (nseg + 1) + 1) * sizeof(int64_t)));
  int32_t* fault = reinterpret_cast<int32_t*>(sg + 2 * (nseg + 1));
  *fault = 0;
  k_mark_image<<<grid_for(ctx, m, kThreads), kThreads, 0, st>>>(m, ctx->low, ctx->is_low);
  PH_CHECK_LAUNCH();
  k_out_scan<<<(unsigned)ntiles, kThreads, 0, st>>>(
      m, nseg, ctx->low, ctx->is_low, ctx->d_seg_start, words + 1, ntiles, ctx->out_before, sg,
      (unsigned int*)words, fault);
  PH_CHECK_LAUNCH();
  PH_CUDA(cudaStreamSynchronize(st));
  PH_REQUIRE(*fault == 0, PH_ERR_CUDA, "a bounded wait of the extraction ran out");
  // output bases: clouds in order, inside a cloud dimensions in order
  const int ndim = ctx->max_dim + 1;
  std::vector<int64_t> delta(2 * nseg);
  ctx->pair_off.assign(nc + 1, 0);
  ctx->ess_off.assign(nc + 1, 0);
  int64_t bp = 0, be = 0;
  for (int c = 0; c < nc; c++) {
    ctx->pair_off[c] = bp;
    ctx->ess_off[c] = be;
    for (int d = 0; d < ndim; d++) {
      int s = d * nc + c;
      delta[2 * s] = bp - sg[2 * s];
      delta[2 * s + 1] = be - sg[2 * s + 1];
      bp += sg[2 * (s + 1)] - sg[2 * s];
      be += sg[2 * (s + 1) + 1] - sg[2 * s + 1];
    }
  }
  ctx->pair_off[nc] = bp;
  ctx->ess_off[nc] = be;
  ctx->n_pairs = bp;
  ctx->n_ess = be;
  PH_CUDA(cudaMemcpyAsync(ctx->out_delta, delta.data(), delta.size() * sizeof(int64_t),
                          cudaMemcpyHostToDevice, st));
  ctx->extracted = true;
}

// the writers' error word is page-locked memory as well (finish_out reads it)
template <bool kEss>
static void write_out(ph_ctx* ctx, const OutArrays& o) {
  int32_t* bad = static_cast<int32_t*>(ctx->pinned(sizeof(int32_t)));
  *bad = 0;
  const int64_t nout = (ctx->m + kOutTile - 1) / kOutTile;
  const bool lng = ctx->m >= kLongOut;
  const unsigned grid = grid_for(ctx, lng ? (ctx->m + kScanTile - 1) / kScanTile : nout, 1);
  (lng ? k_write_out<kEss, kScanTile> : k_write_out<kEss, kOutTile>)<<<grid, kThreads, 0,
                                                                       ctx->stream>>>(
      ctx->m, ctx->n_clouds, ctx->seg, ctx->low, ctx->is_low, ctx->gidx, ctx->key, ctx->d2tab,
      ctx->out_before, ctx->out_delta, o, kEss ? ctx->n_ess : ctx->n_pairs,
      bad);
  PH_CHECK_LAUNCH();
}

// after the results were written (and copied): waits, and checks the writers' error word
static void finish_out(ph_ctx* ctx, bool written) {
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  const int32_t bad = written ? *static_cast<int32_t*>(ctx->pinned(sizeof(int32_t))) : 0;
  if (bad) ctx->extracted = false;
  PH_REQUIRE(bad == 0, PH_ERR_INVALID, "internal error: extraction index out of range");
}

template <typename T>
static void renew(ph_ctx* ctx, T*& p, int64_t n) {
  ctx->dfree(p);
  p = nullptr;
  p = ph::alloc_n<T>(ctx, n);
}

// whether a kernel of this context may write the array (a copy takes more: another device's
// memory, any alignment)
static bool writable(ph_ctx* ctx, const void* p, size_t align, bool on_device) {
  if (!p) return true;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const bool there = on_device ? at.type == cudaMemoryTypeDevice && at.device == ctx->device
                               : at.type == cudaMemoryTypeHost && at.devicePointer == p;
  return there && reinterpret_cast<uintptr_t>(p) % align == 0;
}
// A few results go straight into page-locked host arrays too, without internal arrays and copies: 780
// pairs 84 -> 78 us, 9140 essentials 35 -> 31 us; from 18,000 on both ways measure alike.
constexpr int64_t kHostDirect = 16384;

__global__ void k_inspect(CloudIds ids, const int32_t* __restrict__ seg, int nc,
                          const int64_t* __restrict__ gidx, const int32_t* __restrict__ key,
                          const int64_t* __restrict__ d2tab, const uint64_t* __restrict__ verts,
                          const int32_t* __restrict__ beta, const int32_t* __restrict__ low,
                          int32_t* o_dim, int64_t* o_d2, int32_t* o_v, int32_t* o_beta,
                          int32_t* o_low, int64_t n, int vbits, int32_t* bad) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ids.n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = ids.id(t);
    int64_t g = gidx[x];
    if (g < 0 || g >= n) {
      *bad = 1;
      continue;
    }
    int d = seg[x] / nc;
    o_dim[g] = d;
    o_d2[g] = diam2_of(key, d2tab, (int32_t)x);
    uint64_t p = verts[x];
    for (int q = 0; q < kVrSlots; q++)
      o_v[kVrSlots * g + q] = (p == ~0ull || q > d) ? -1 : packed_vert_at(p, q, vbits);
    o_beta[g] = beta[x] >= 0 ? (int32_t)gidx[beta[x]] : -1;
    o_low[g] = low[x] >= 0 ? (int32_t)gidx[low[x]] : -1;
  }
}

}  // namespace ph

// ---------------------------------------------------------------------------------------------
// ABI
// ---------------------------------------------------------------------------------------------
#define PH_API_BEGIN                  \
  if (!ctx) return PH_ERR_INVALID;    \
  ctx->err.clear();                   \
  ph::NvtxRange nvtx_range_(__func__); \
  try {
#define PH_API_END                                    \
  }                                                   \
  catch (const ph::Fail& f) {                         \
    return f.code;                                    \
  }                                                   \
  catch (const std::bad_alloc&) {                     \
    ctx->err = "host allocation failed";              \
    return PH_ERR_ALLOC;                              \
  }                                                   \
  catch (...) {                                       \
    ctx->err = "unexpected failure";                  \
    return PH_ERR_INVALID;                            \
  }

extern "C" {

void ph_default_opts(ph_opts* o) {
  if (!o) return;
  std::memset(o, 0, sizeof(*o));
  o->strict_phase2 = 0;
  o->use_cor10 = 1;
  o->lane_merge_words = 0;
  o->staged_merge_max = 0;
  o->merge_items = 0;
  o->collect_stats = 0;
  o->use_graph = 1;
  o->time_kernels = 0;
  o->add_blocks_per_sm = 0;
  o->timeout_ms = 0;
  o->predict_pairs = 0;
  o->dense_threshold = 0;
  o->warp_chunks_below = 0;
  o->warp_chunk_words = 0;
  o->narrow_chunks_below = 0;
  o->phase2_sets = 0;
  o->phase2_priority = 0;
  o->arena_words = 0;
}

int ph_create(ph_ctx** out, const ph_opts* opts, const ph_allocator* alloc, void* stream) {
  if (!out) return PH_ERR_INVALID;
  *out = nullptr;
  ph_ctx* ctx = new (std::nothrow) ph_ctx();
  if (!ctx) return PH_ERR_ALLOC;
  if (opts) ctx->opts = *opts;
  else ph_default_opts(&ctx->opts);
  if (ctx->opts.phase2_priority < 0 || ctx->opts.phase2_priority > 1) {
    delete ctx;
    return PH_ERR_INVALID;
  }
  if (alloc && alloc->alloc && alloc->free) {
    ctx->alloc = *alloc;
    ctx->has_alloc = true;
  }
  ctx->stream = (cudaStream_t)stream;
  if (cudaGetDevice(&ctx->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, ctx->device) !=
          cudaSuccess) {
    cudaGetLastError();
    delete ctx;
    return PH_ERR_CUDA;
  }
  *out = ctx;
  return PH_OK;
}

void ph_destroy(ph_ctx* ctx) {
  if (!ctx) return;
  cudaStreamSynchronize(ctx->stream);
  ctx->free_all();
  ctx->drop_kept(INT64_MAX);
  ph::free_graphs(ctx);
  if (ctx->rs.hstate) cudaFreeHost(ctx->rs.hstate);
  if (ctx->h_pinned) cudaFreeHost(ctx->h_pinned);
  cudaStreamSynchronize(ctx->stream);
  delete ctx;
}

int ph_build_filtration(ph_ctx* ctx, const int32_t* coords, const int64_t* cloud_offsets,
                        int32_t n_clouds, int64_t n_points, int32_t D, int32_t max_dim,
                        int64_t max_diam2, int64_t* m_out) {
  PH_API_BEGIN
  ctx->free_all();
  ph::build_vr(ctx, coords, cloud_offsets, n_clouds, n_points, D, max_dim, max_diam2);
  ctx->built = true;
  ctx->is_vr = true;
  if (m_out) *m_out = ctx->m;
  return PH_OK;
  PH_API_END
}

int ph_build_filtration_scales(ph_ctx* ctx, const int32_t* coords, const int64_t* cloud_offsets,
                               int32_t n_clouds, int64_t n_points, int32_t D, int32_t max_dim,
                               int64_t scale_step, int32_t n_scales, int64_t* m_out) {
  PH_API_BEGIN
  PH_REQUIRE(scale_step >= 1, PH_ERR_INVALID, "scale_step must be >= 1 grid unit");
  ctx->free_all();
  ph::build_vr(ctx, coords, cloud_offsets, n_clouds, n_points, D, max_dim, -1, scale_step,
               n_scales);
  ctx->built = true;
  ctx->is_vr = true;
  if (m_out) *m_out = ctx->m;
  return PH_OK;
  PH_API_END
}

int ph_load_boundary(ph_ctx* ctx, int64_t m, const int32_t* dims, const int64_t* colptr,
                     const int32_t* rows) {
  PH_API_BEGIN
  ctx->free_all();
  ph::load_boundary(ctx, m, dims, colptr, rows);
  ctx->built = true;
  return PH_OK;
  PH_API_END
}

int ph_reduce(ph_ctx* ctx, int32_t max_passes, ph_stats* out) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->built, PH_ERR_INVALID, "no filtration: call ph_build_filtration first");
  // the places of the results belong to the lows as they are: they go before any pass changes these,
  // since the call may also end part-way (time bound, refused allocation)
  ctx->extracted = false;
  if (!ctx->rs.init) ph::reduce_init(ctx, max_passes);
  int rc = ctx->rs.status;
  if (!(ctx->rs.done && ctx->rs.status == PH_OK)) rc = ph::reduce_run(ctx, max_passes);
  ctx->reduced = true;
  if (out) {
    std::memset(out, 0, sizeof(*out));
    out->passes = ctx->rs.passes;
    out->status = rc;
    out->m = ctx->m;
    const auto& hs = ctx->rs.h_stats;
    for (size_t r = 0; r + PH_PS_N <= hs.size(); r += PH_PS_N) {
      out->col_adds += hs[r + PH_PS_ADDS];
      out->xors += hs[r + PH_PS_XORS];
      // algorithmic bytes: per active column per pass 4 (low) + 4 (table atomic) + 4 (table
      // read) + 1 (flags) + 8 (active list) + 8 (scan) = 29; per addition 8 bytes per XOR
      // (4 * (|src| + |tgt| + |out|) = 8 * |src union tgt|)
      out->alg_bytes += 29 * hs[r + PH_PS_ACTIVE] + 8 * hs[r + PH_PS_XORS];
      out->add_bytes += 8 * hs[r + PH_PS_XORS] + 8 * hs[r + PH_PS_COPIED] +
                        40 * hs[r + PH_PS_ACTIVE];
    }
    out->add_launches = ctx->rs.add_launches;
    out->ms_add = ctx->rs.ms_add;
  }
  return rc;
  PH_API_END
}

int ph_reset_reduction(ph_ctx* ctx) {
  PH_API_BEGIN
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  ph::free_reduce_state(ctx);
  ph::drop_extraction(ctx);
  ctx->reduced = false;
  return PH_OK;
  PH_API_END
}

int ph_get_pass_stats(ph_ctx* ctx, int64_t* out, int32_t max_rows, int32_t* rows_out) {
  PH_API_BEGIN
  const auto& hs = ctx->rs.h_stats;
  int32_t rows = (int32_t)(hs.size() / PH_PS_N);
  if (rows_out) *rows_out = rows;
  if (out) std::memcpy(out, hs.data(), (size_t)std::min(rows, max_rows) * PH_PS_N * 8);
  return PH_OK;
  PH_API_END
}

int ph_get_add_times(ph_ctx* ctx, float* out, int32_t max_n, int32_t* n_out) {
  PH_API_BEGIN
  const auto& v = ctx->rs.add_ms;
  if (n_out) *n_out = (int32_t)v.size();
  if (out) std::memcpy(out, v.data(), sizeof(float) * std::min<size_t>(v.size(), (size_t)max_n));
  return PH_OK;
  PH_API_END
}

static void copy_out(ph_ctx* ctx, void* dst, const void* src, size_t bytes, int on_device) {
  if (!dst || bytes == 0) return;
  PH_CUDA(cudaMemcpyAsync(dst, src, bytes,
                          on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                          ctx->stream));
}

int ph_get_pairs(ph_ctx* ctx, int32_t cloud, int64_t* birth, int64_t* death, int32_t* dim,
                 int64_t* birth_diam2, int64_t* death_diam2, int64_t capacity, int64_t* count,
                 int32_t on_device) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->reduced, PH_ERR_INVALID, "call ph_reduce first");
  PH_REQUIRE(cloud >= -1 && cloud < ctx->n_clouds, PH_ERR_INVALID, "cloud out of range");
  ph::extract_places(ctx);
  int64_t a = cloud < 0 ? 0 : ctx->pair_off[cloud];
  int64_t n = (cloud < 0 ? ctx->pair_off[ctx->n_clouds] : ctx->pair_off[cloud + 1]) - a;
  if (count) *count = n;
  if (!birth && !death && !dim && !birth_diam2 && !death_diam2) return PH_OK;
  PH_REQUIRE(capacity >= n, PH_ERR_CAPACITY, "output capacity too small");
  if (n == ctx->n_pairs && !ctx->p_birth && (on_device || n <= ph::kHostDirect) &&
      ph::writable(ctx, birth, 8, on_device) && ph::writable(ctx, death, 8, on_device) &&
      ph::writable(ctx, dim, 4, on_device) && ph::writable(ctx, birth_diam2, 8, on_device) &&
      ph::writable(ctx, death_diam2, 8, on_device)) {
    ph::write_out<false>(ctx, ph::OutArrays{birth, death, birth_diam2, death_diam2, dim});
    ph::finish_out(ctx, true);
    return PH_OK;
  }
  const bool written = !ctx->p_birth;
  if (written) {
    const int64_t all = ctx->n_pairs;
    ph::renew(ctx, ctx->p_death, all);
    ph::renew(ctx, ctx->p_dim, all);
    ph::renew(ctx, ctx->p_bd2, all);
    ph::renew(ctx, ctx->p_dd2, all);
    ph::renew(ctx, ctx->p_birth, all);  // last: with it all five are there
    ph::write_out<false>(
        ctx, ph::OutArrays{ctx->p_birth, ctx->p_death, ctx->p_bd2, ctx->p_dd2, ctx->p_dim});
  }
  copy_out(ctx, birth, ctx->p_birth + a, n * 8, on_device);
  copy_out(ctx, death, ctx->p_death + a, n * 8, on_device);
  copy_out(ctx, dim, ctx->p_dim + a, n * 4, on_device);
  copy_out(ctx, birth_diam2, ctx->p_bd2 + a, n * 8, on_device);
  copy_out(ctx, death_diam2, ctx->p_dd2 + a, n * 8, on_device);
  ph::finish_out(ctx, written);
  return PH_OK;
  PH_API_END
}

int ph_get_essential(ph_ctx* ctx, int32_t cloud, int64_t* idx, int32_t* dim, int64_t* diam2,
                     int64_t capacity, int64_t* count, int32_t on_device) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->reduced, PH_ERR_INVALID, "call ph_reduce first");
  PH_REQUIRE(cloud >= -1 && cloud < ctx->n_clouds, PH_ERR_INVALID, "cloud out of range");
  ph::extract_places(ctx);
  int64_t a = cloud < 0 ? 0 : ctx->ess_off[cloud];
  int64_t n = (cloud < 0 ? ctx->ess_off[ctx->n_clouds] : ctx->ess_off[cloud + 1]) - a;
  if (count) *count = n;
  if (!idx && !dim && !diam2) return PH_OK;
  PH_REQUIRE(capacity >= n, PH_ERR_CAPACITY, "output capacity too small");
  if (n == ctx->n_ess && !ctx->e_idx && (on_device || n <= ph::kHostDirect) &&
      ph::writable(ctx, idx, 8, on_device) && ph::writable(ctx, dim, 4, on_device) &&
      ph::writable(ctx, diam2, 8, on_device)) {
    ph::write_out<true>(ctx, ph::OutArrays{nullptr, idx, nullptr, diam2, dim});
    ph::finish_out(ctx, true);
    return PH_OK;
  }
  const bool written = !ctx->e_idx;
  if (written) {
    const int64_t all = ctx->n_ess;
    ph::renew(ctx, ctx->e_dim, all);
    ph::renew(ctx, ctx->e_d2, all);
    ph::renew(ctx, ctx->e_idx, all);  // last: with it all three are there
    ph::write_out<true>(ctx, ph::OutArrays{nullptr, ctx->e_idx, nullptr, ctx->e_d2, ctx->e_dim});
  }
  copy_out(ctx, idx, ctx->e_idx + a, n * 8, on_device);
  copy_out(ctx, dim, ctx->e_dim + a, n * 4, on_device);
  copy_out(ctx, diam2, ctx->e_d2 + a, n * 8, on_device);
  ph::finish_out(ctx, written);
  return PH_OK;
  PH_API_END
}

int ph_get_essential_estimate(ph_ctx* ctx, int32_t cloud, uint8_t* in_e, int64_t* count) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->reduced && ctx->rs.init, PH_ERR_INVALID, "call ph_reduce first");
  PH_REQUIRE(cloud >= 0 && cloud < ctx->n_clouds, PH_ERR_INVALID, "cloud out of range");
  const int nc = ctx->n_clouds;
  int64_t n = 0;
  for (int d = 0; d <= ctx->max_dim; d++)
    n += ctx->seg_start[d * nc + cloud + 1] - ctx->seg_start[d * nc + cloud];
  if (count) *count = n;
  if (!in_e) return PH_OK;
  ph::essential_estimate(ctx, cloud, in_e, n);
  return PH_OK;
  PH_API_END
}

int ph_get_columns(ph_ctx* ctx, int32_t cloud, int64_t* colptr, int32_t* rows, int64_t capacity,
                   int64_t* nnz) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->reduced && ctx->rs.init, PH_ERR_INVALID, "call ph_reduce first");
  PH_REQUIRE(cloud >= 0 && cloud < ctx->n_clouds, PH_ERR_INVALID, "cloud out of range");
  PH_REQUIRE(colptr != nullptr, PH_ERR_INVALID, "colptr is required");
  const int nc = ctx->n_clouds;
  int64_t n = 0;
  for (int d = 0; d <= ctx->max_dim; d++)
    n += ctx->seg_start[d * nc + cloud + 1] - ctx->seg_start[d * nc + cloud];
  ph::reduced_columns(ctx, cloud, n, colptr, rows, capacity, nnz);
  return PH_OK;
  PH_API_END
}

int ph_get_predicted_lows(ph_ctx* ctx, int32_t cloud, int32_t* pred, int64_t* count) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->reduced && ctx->rs.init, PH_ERR_INVALID, "call ph_reduce first");
  PH_REQUIRE(ctx->opts.predict_pairs, PH_ERR_INVALID, "the context was made without predict_pairs");
  PH_REQUIRE(cloud >= 0 && cloud < ctx->n_clouds, PH_ERR_INVALID, "cloud out of range");
  const int nc = ctx->n_clouds;
  int64_t n = 0;
  for (int d = 0; d <= ctx->max_dim; d++)
    n += ctx->seg_start[d * nc + cloud + 1] - ctx->seg_start[d * nc + cloud];
  if (count) *count = n;
  if (!pred) return PH_OK;
  ph::predicted_lows(ctx, cloud, pred, n);
  return PH_OK;
  PH_API_END
}

int ph_get_filtration(ph_ctx* ctx, int32_t cloud, int32_t* dim, int64_t* diam2, int32_t* verts,
                      int32_t* beta, int32_t* low, int64_t* count) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->built, PH_ERR_INVALID, "no filtration");
  PH_REQUIRE(cloud >= 0 && cloud < ctx->n_clouds, PH_ERR_INVALID, "cloud out of range");
  const int nc = ctx->n_clouds;
  int64_t n = 0;
  for (int d = 0; d <= ctx->max_dim; d++)
    n += ctx->seg_start[d * nc + cloud + 1] - ctx->seg_start[d * nc + cloud];
  if (count) *count = n;
  if (!dim) return PH_OK;
  int32_t* o_dim = ph::alloc_n<int32_t>(ctx, n);
  int64_t* o_d2 = ph::alloc_n<int64_t>(ctx, n);
  int32_t* o_v = ph::alloc_n<int32_t>(ctx, ph::kVrSlots * n);
  int32_t* o_beta = ph::alloc_n<int32_t>(ctx, n);
  int32_t* o_low = ph::alloc_n<int32_t>(ctx, n);
  int32_t* d_bad = ph::alloc_n<int32_t>(ctx, 1);
  PH_CUDA(cudaMemsetAsync(d_bad, 0, sizeof(int32_t), ctx->stream));
  const ph::CloudIds ids = ph::cloud_ids(ctx, cloud);
  ph::k_inspect<<<ph::grid_for(ctx, ids.n, ph::kThreads), ph::kThreads, 0, ctx->stream>>>(
      ids, ctx->seg, nc, ctx->gidx, ctx->key, ctx->d2tab, ctx->verts, ctx->beta, ctx->low, o_dim, o_d2,
      o_v, o_beta, o_low, n, ctx->vbits, d_bad);
  PH_CHECK_LAUNCH();
  int32_t* bad = static_cast<int32_t*>(ctx->pinned(sizeof(int32_t)));
  PH_CUDA(cudaMemcpyAsync(bad, d_bad, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
  copy_out(ctx, dim, o_dim, n * 4, 0);
  copy_out(ctx, diam2, o_d2, n * 8, 0);
  copy_out(ctx, verts, o_v, n * 4 * ph::kVrSlots, 0);
  copy_out(ctx, beta, o_beta, n * 4, 0);
  copy_out(ctx, low, o_low, n * 4, 0);
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  for (void* p : {(void*)o_dim, (void*)o_d2, (void*)o_v, (void*)o_beta, (void*)o_low,
                  (void*)d_bad})
    ctx->dfree(p);
  PH_REQUIRE(*bad == 0, PH_ERR_INVALID, "internal error: filtration index out of range");
  return PH_OK;
  PH_API_END
}

int64_t ph_kernel_launches(const ph_ctx* ctx) { return ctx ? ctx->launches : 0; }

const char* ph_last_error(const ph_ctx* ctx) { return ctx ? ctx->err.c_str() : "NULL context"; }

}  // extern "C"
