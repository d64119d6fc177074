// Differentiable persistence diagrams: a loss over the finite pairs of one dimension and its
// gradient with respect to the point coordinates.
//
// The pairing (which simplex kills which, Lemma 1) is computed exactly from grid-rounded
// coordinates and is piecewise constant in the coordinates, so it carries no gradient. The
// birth and death values of a pair are Euclidean diameters (Sec. 2.2, VR: f_r(sigma) =
// 1{diam(sigma) <= 2r}); a simplex's diameter is the length of one of its edges, its realising
// edge: an edge realises itself, a higher simplex is realised by the realising edge of its last
// face in the filtration (the largest row of its boundary column), which has the same diameter.
// For a pair with realising edges (p, q) at birth and (r, s) at death,
//   b = |x_p - x_q|, d = |x_r - x_s|, loss = sum over pairs of (d - b)^2,
//   dloss/dx_r = 2 (d - b) (x_r - x_s) / d,  dloss/dx_s = -dloss/dx_r,
//   dloss/dx_p = -2 (d - b) (x_p - x_q) / b, dloss/dx_q = -dloss/dx_p,
// with the term of a zero-length edge left out (its direction is undefined).
#include <cmath>

#include "ph_internal.cuh"

namespace ph {

struct DiagLayout {
  int64_t dimoff[kMaxDim + 2];
  int64_t rowbase[kMaxDim + 2];
  int maxd;
  int nc;
  int vbits;  // bits per packed vertex of the build
};

__global__ void k_to_grid(const float* __restrict__ x, int64_t n, int32_t* g, int32_t* bad) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float v = x[i] * 65536.0f;  // exact: a power-of-two scaling
    if (!(fabsf(v) <= 16777216.0f)) {  // also catches NaN
      *bad = 1;
      g[i] = 0;
    } else {
      g[i] = __float2int_rn(v);  // round half to even
    }
  }
}

// the realising edge of simplex x (an id of dimension >= 1): follow the last face down to an
// edge; returns the two point indices (global rows of the coordinate array)
__device__ __forceinline__ void realising_edge(const DiagLayout& L, const int32_t* __restrict__ rows0,
                                               const uint64_t* __restrict__ verts,
                                               const int64_t* __restrict__ pt_off, int64_t x,
                                               int64_t& p, int64_t& q) {
  int d = 0;
  while (d < L.maxd && x >= L.dimoff[d + 1]) d++;
  while (d > 1) {
    x = rows0[L.rowbase[d] + (int64_t)(d + 1) * (x - L.dimoff[d]) + d];  // largest row
    d--;
  }
  const uint64_t v = verts[x];
  const int64_t base = pt_off[(int)(v >> 48)];
  p = base + (int64_t)packed_vert_at(v, 0, L.vbits);
  q = base + (int64_t)packed_vert_at(v, 1, L.vbits);
}

__device__ __forceinline__ float edge_len(const float* __restrict__ x, int D, int64_t p,
                                          int64_t q) {
  float s = 0.f;
  for (int k = 0; k < D; k++) {
    const float t = x[p * D + k] - x[q * D + k];
    s += t * t;
  }
  return sqrtf(s);
}

// Calls f(j, low) by one thread for every column j of [lo, hi) with a low, by one block. One column
// in twenty is paired, and a pair takes a chain of gathers: the block lists the pairs of 2048 columns
// at a time in shared memory, in order, and its threads take neighbours of the list once there are
// enough for all (pair k goes to thread k mod kThreads). Bound by those chains. With a column per
// thread every warp waited for its one or two pairs: loss and gradient of 256 clouds of 64 points
// (10.7 M triangles, 500,000 pairs) took 277 + 208 us, now 54 + 67 us.
constexpr int kPairRound = 2048;
template <class F>
__device__ __forceinline__ void for_each_pair(const int32_t* __restrict__ low, int64_t lo, int64_t hi,
                                              F f) {
  constexpr int kPer = kPairRound / kThreads, kWords = kPairRound / 32;
  __shared__ int64_t s_j[kPairRound + kThreads];
  __shared__ int32_t s_low[kPairRound + kThreads];
  __shared__ int s_cnt[kWords], s_total;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int n = 0;  // listed, the same in every thread
  for (int64_t j0 = lo; j0 < hi; j0 += kPairRound) {
    int32_t b[kPer];
    unsigned mask[kPer];
#pragma unroll
    for (int i = 0; i < kPer; i++) {
      const int64_t j = j0 + (w * kPer + i) * 32 + lane;
      b[i] = j < hi ? low[j] : -1;
    }
#pragma unroll
    for (int i = 0; i < kPer; i++) {
      mask[i] = __ballot_sync(0xffffffffu, b[i] >= 0);
      if (lane == 0) s_cnt[w * kPer + i] = __popc(mask[i]);
    }
    __syncthreads();
    if (w == 0) {  // counts to places
      const int a = s_cnt[2 * lane], c = s_cnt[2 * lane + 1];
      const int inc = warp_incl_sum(a + c);
      s_cnt[2 * lane] = inc - a - c;
      s_cnt[2 * lane + 1] = inc - c;
      if (lane == 31) s_total = inc;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; i++) {
      if (b[i] < 0) continue;
      const int q = w * kPer + i, p = n + s_cnt[q] + __popc(mask[i] & ((1u << lane) - 1u));
      s_j[p] = j0 + q * 32 + lane;
      s_low[p] = b[i];
    }
    n += s_total;
    __syncthreads();
    const int take = j0 + kPairRound < hi ? n & ~(kThreads - 1) : n;
    for (int k = threadIdx.x; k < take; k += kThreads) f(s_j[k], s_low[k]);
    n -= take;
    if (take > 0 && n > 0) {  // the rest, fewer than there are threads, to the front
      __syncthreads();
      const int64_t j = threadIdx.x < n ? s_j[take + threadIdx.x] : 0;
      const int32_t l = threadIdx.x < n ? s_low[take + threadIdx.x] : 0;
      __syncthreads();
      if (threadIdx.x < n) {
        s_j[threadIdx.x] = j;
        s_low[threadIdx.x] = l;
      }
    }
  }
}

// one block per cloud: the finite pairs whose death simplex has dimension dd = dim + 1 are the
// columns of segment (dd, cloud) with a low; the block sums their terms in a fixed order
__global__ void k_diag_loss(DiagLayout L, int dd, const int64_t* __restrict__ seg_start,
                            const int32_t* __restrict__ low, const int32_t* __restrict__ rows0,
                            const uint64_t* __restrict__ verts, const int64_t* __restrict__ pt_off,
                            const float* __restrict__ x, int D, float* loss,
                            unsigned long long* npairs) {
  __shared__ double sh[kThreads];
  const int c = blockIdx.x;
  const int64_t lo = seg_start[dd * L.nc + c], hi = seg_start[dd * L.nc + c + 1];
  double acc = 0.;  // (with several terms per thread a float sum would round more often)
  unsigned long long cnt = 0;
  for_each_pair(low, lo, hi, [&](int64_t j, int32_t b) {
    int64_t r, s;
    realising_edge(L, rows0, verts, pt_off, j, r, s);
    const float dlen = edge_len(x, D, r, s);
    float blen = 0.f;
    if (dd >= 2) {
      int64_t p, q;
      realising_edge(L, rows0, verts, pt_off, b, p, q);
      blen = edge_len(x, D, p, q);
    }
    const float t = dlen - blen;
    acc += (double)t * t;
    cnt++;
  });
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss[c] = (float)sh[0];
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(npairs, cnt);
}

__global__ void k_diag_total(const float* __restrict__ loss, int nc, float* total) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    float s = 0.f;
    for (int c = 0; c < nc; c++) s += loss[c];
    *total = s;
  }
}

__global__ void k_diag_bwd(DiagLayout L, int dd, int64_t lo, int64_t hi,
                           const int32_t* __restrict__ seg, const int32_t* __restrict__ low,
                           const int32_t* __restrict__ rows0, const uint64_t* __restrict__ verts,
                           const int64_t* __restrict__ pt_off, const float* __restrict__ x, int D,
                           const float* __restrict__ gloss, float* grad) {
  // a run of whole rounds per block
  const int64_t rounds = (hi - lo + kPairRound - 1) / kPairRound;
  const int64_t per = (rounds + gridDim.x - 1) / gridDim.x * kPairRound;
  const int64_t first = lo + blockIdx.x * per, end = first + per < hi ? first + per : hi;
  for_each_pair(low, first, end, [&](int64_t j, int32_t b) {
    const int c = seg[j] % L.nc;
    int64_t r, s, p = -1, q = -1;
    realising_edge(L, rows0, verts, pt_off, j, r, s);
    const float dlen = edge_len(x, D, r, s);
    float blen = 0.f;
    if (dd >= 2) {
      realising_edge(L, rows0, verts, pt_off, b, p, q);
      blen = edge_len(x, D, p, q);
    }
    const float g = 2.f * (dlen - blen) * gloss[c];
    if (dlen > 0.f) {
      const float f = g / dlen;
      for (int k = 0; k < D; k++) {
        const float t = f * (x[r * D + k] - x[s * D + k]);
        atomicAdd(&grad[r * D + k], t);
        atomicAdd(&grad[s * D + k], -t);
      }
    }
    if (p >= 0 && blen > 0.f) {
      const float f = g / blen;
      for (int k = 0; k < D; k++) {
        const float t = f * (x[p * D + k] - x[q * D + k]);
        atomicAdd(&grad[p * D + k], -t);
        atomicAdd(&grad[q * D + k], t);
      }
    }
  });
}

static DiagLayout layout_of(ph_ctx* ctx) {
  DiagLayout L{};
  L.maxd = ctx->max_dim;
  L.vbits = ctx->vbits;
  L.nc = ctx->n_clouds;
  int64_t rb = 0;
  for (int d = 0; d <= ctx->max_dim + 1; d++) L.dimoff[d] = ctx->dimoff[d];
  for (int d = 0; d <= ctx->max_dim; d++) {
    L.rowbase[d] = rb;
    rb += (d > 0 ? d + 1 : 0) * (ctx->dimoff[d + 1] - ctx->dimoff[d]);
  }
  return L;
}

}  // namespace ph

#define PH_API_BEGIN \
  if (!ctx) return PH_ERR_INVALID; \
  ctx->err.clear();                \
  try {
#define PH_API_END                                    \
  }                                                   \
  catch (const ph::Fail& f) {                         \
    return f.code;                                    \
  }                                                   \
  catch (...) {                                       \
    ctx->err = "unexpected failure";                  \
    return PH_ERR_INVALID;                            \
  }

extern "C" {

int ph_build_filtration_f32(ph_ctx* ctx, const float* coords, const int64_t* cloud_offsets,
                            int32_t n_clouds, int64_t n_points, int32_t D, int32_t max_dim,
                            int64_t max_diam2, int64_t* m_out) {
  PH_API_BEGIN
  PH_REQUIRE(coords != nullptr && n_points >= 1 && D >= 1 && D <= 16, PH_ERR_INVALID,
             "bad coordinates");
  ctx->free_all();
  const int64_t n = n_points * D;
  // the rounded copy lives with the filtration (freed with it)
  int32_t* g = ph::alloc_n<int32_t>(ctx, n);
  int32_t* bad = static_cast<int32_t*>(ctx->pinned(sizeof(int32_t)));  // written by the kernel
  *bad = 0;
  ph::k_to_grid<<<ph::grid_for(ctx, n, ph::kThreads), ph::kThreads, 0, ctx->stream>>>(coords, n,
                                                                                     g, bad);
  PH_CHECK_LAUNCH();
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  PH_REQUIRE(*bad == 0, PH_ERR_INVALID, "coordinates must be finite with |x| <= 256");
  ph::build_vr(ctx, g, cloud_offsets, n_clouds, n_points, D, max_dim, max_diam2);
  ctx->built = true;
  ctx->is_vr = true;
  if (m_out) *m_out = ctx->m;
  return PH_OK;
  PH_API_END
}

int ph_diagram_loss(ph_ctx* ctx, const float* coords, int32_t D, int32_t dim, float* loss,
                    int64_t* n_pairs) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->reduced, PH_ERR_INVALID, "call ph_reduce first");
  PH_REQUIRE(ctx->is_vr, PH_ERR_INVALID, "diagram losses need a filtration built from points");
  PH_REQUIRE(coords && loss, PH_ERR_INVALID, "NULL argument");
  PH_REQUIRE(dim >= 0 && dim + 1 <= ctx->max_dim, PH_ERR_INVALID,
             "dim + 1 must not exceed the filtration's max_dim");
  // the kernels index coords by the build's point rows: any other shape reads out of bounds
  PH_REQUIRE(D == ctx->D, PH_ERR_INVALID,
             "D must equal the D of the build (" + std::to_string(ctx->D) + ")");
  const ph::DiagLayout L = ph::layout_of(ctx);
  unsigned long long* cnt = ph::alloc_n<unsigned long long>(ctx, 1);
  const int64_t* d_pt = ctx->d_pt_off;
  PH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), ctx->stream));
  ph::k_diag_loss<<<ctx->n_clouds, ph::kThreads, 0, ctx->stream>>>(
      L, dim + 1, ctx->d_seg_start, ctx->low, ctx->rows0, ctx->verts, d_pt, coords, D, loss, cnt);
  PH_CHECK_LAUNCH();
  ph::k_diag_total<<<1, 32, 0, ctx->stream>>>(loss, ctx->n_clouds, loss + ctx->n_clouds);
  PH_CHECK_LAUNCH();
  auto* h = static_cast<unsigned long long*>(ctx->pinned(sizeof(*cnt)));
  PH_CUDA(cudaMemcpyAsync(h, cnt, sizeof(*cnt), cudaMemcpyDeviceToHost, ctx->stream));
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  ctx->dfree(cnt);
  if (n_pairs) *n_pairs = (int64_t)*h;
  return PH_OK;
  PH_API_END
}

int ph_diagram_backward(ph_ctx* ctx, const float* coords, int32_t D, int32_t dim,
                        const float* grad_loss, float* grad_coords) {
  PH_API_BEGIN
  PH_REQUIRE(ctx->reduced, PH_ERR_INVALID, "call ph_reduce first");
  PH_REQUIRE(ctx->is_vr, PH_ERR_INVALID, "diagram losses need a filtration built from points");
  PH_REQUIRE(coords && grad_loss && grad_coords, PH_ERR_INVALID, "NULL argument");
  PH_REQUIRE(dim >= 0 && dim + 1 <= ctx->max_dim, PH_ERR_INVALID,
             "dim + 1 must not exceed the filtration's max_dim");
  PH_REQUIRE(D == ctx->D, PH_ERR_INVALID,
             "D must equal the D of the build (" + std::to_string(ctx->D) + ")");
  const ph::DiagLayout L = ph::layout_of(ctx);
  const int64_t* d_pt = ctx->d_pt_off;
  const int64_t lo = ctx->dimoff[dim + 1], hi = ctx->dimoff[dim + 2];
  ph::k_diag_bwd<<<ph::grid_for(ctx, hi - lo, ph::kPairRound), ph::kThreads, 0, ctx->stream>>>(
      L, dim + 1, lo, hi, ctx->seg, ctx->low, ctx->rows0, ctx->verts, d_pt, coords, D, grad_loss,
      grad_coords);
  PH_CHECK_LAUNCH();
  return PH_OK;
  PH_API_END
}

}  // extern "C"
