// Filtration and boundary-matrix construction on the device (Sec. 2.2-2.3, Definition 4).
//
// Vietoris-Rips: a simplex enters at its diameter (f_r(sigma) = 1{diam(sigma) <= 2r}); its
// squared diameter is the largest squared edge length among its vertices, an exact int64 on
// the 2^-16 grid. The compatible ordering is (squared diameter, dimension, vertex tuple in
// lexicographic order). Rather than sorting 64-bit diameters for every dimension, edges are
// sorted once by (cloud, diameter, lex) and given the dense rank of their squared diameter; a
// higher simplex's key is the largest rank among its edges, which orders exactly like its
// squared diameter. Candidates are enumerated in (cloud, lex) order, so a stable sort by that
// key yields (cloud, diameter, lex) directly: dense ranks grow with the cloud index. Without ties
// among the edges, triangles and tetrahedra are listed per edge instead, with no sort.
#include <algorithm>
#include <memory>

#include "ph_internal.cuh"

namespace ph {

// cloud in the top 16 bits, then 48 / vbits vertex slots of vbits bits (unused: all ones)
__host__ __device__ __forceinline__ uint64_t pack_simplex(uint32_t cloud, int k, const int* v,
                                                          int vbits) {
  uint64_t p = (uint64_t)cloud << 48;
  const int slots = 48 / vbits;
  const uint64_t none = (1ull << vbits) - 1ull;
  for (int i = 0; i < slots; i++) {
    uint64_t x = i < k ? (uint64_t)v[i] : none;
    p |= x << (48 - vbits * (i + 1));
  }
  return p;
}
__device__ __forceinline__ uint32_t packed_cloud(uint64_t p) { return (uint32_t)(p >> 48); }

// C(n, k) for the small k of a VR build (k <= 6); exact in int64 for n < 2^12. A product of k
// consecutive integers divided by k!, each case a division by a constant (a multiply and a
// shift), so the unranking's binary searches carry no run-time 64-bit division
__host__ __device__ __forceinline__ int64_t binom_small(int64_t n, int k) {
  if (n < k || n < 0 || k < 0) return 0;
  switch (k) {
    case 0: return 1;
    case 1: return n;
    case 2: return n * (n - 1) / 2;
    case 3: return n * (n - 1) * (n - 2) / 6;
    case 4: return n * (n - 1) * (n - 2) * (n - 3) / 24;
    case 5: return n * (n - 1) * (n - 2) * (n - 3) * (n - 4) / 120;
    default: {
      int64_t r = 1;
      for (int i = 0; i < k; i++) r = r * (n - i) / (i + 1);  // each prefix is a binomial
      return r;
    }
  }
}

// k-subset of [n] with lexicographic rank r (0-based). Uses the complement map
// v -> n-1-v, which turns lexicographic order into reversed colexicographic order, where a
// subset's rank is sum_i C(u_i, i+1) and can be peeled off greedily.
__device__ __forceinline__ void lex_unrank(int64_t r, int n, int k, int* v) {
  int64_t R = binom_small(n, k) - 1 - r;
  int u[kVrSlots];
  int hi = n - 1;
  for (int i = k - 1; i >= 0; i--) {
    int lo = i, h = hi;
    while (lo < h) {
      int mid = (lo + h + 1) >> 1;
      if (binom_small(mid, i + 1) <= R) lo = mid; else h = mid - 1;
    }
    u[i] = lo;
    R -= binom_small(lo, i + 1);
    hi = lo - 1;
  }
  for (int i = 0; i < k; i++) v[i] = n - 1 - u[k - 1 - i];
}

__device__ __forceinline__ int64_t lex_rank(const int* v, int n, int k) {
  int64_t R = 0;
  for (int i = 0; i < k; i++) R += binom_small(n - 1 - v[k - 1 - i], i + 1);
  return binom_small(n, k) - 1 - R;
}

__device__ __forceinline__ int find_cloud(const int64_t* __restrict__ off, int nc, int64_t t) {
  int lo = 0, hi = nc - 1;  // last c with off[c] <= t
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

struct CloudTabs {
  const int64_t* pt_off;  // [nc+1] point offsets
  const int64_t* mo;      // [nc+1] offsets of the n_c x n_c tables
  int nc;
  int vbits;              // bits per packed vertex
};

__device__ __forceinline__ int packed_vert(const CloudTabs& ct, uint64_t p, int i) {
  return packed_vert_at(p, i, ct.vbits);
}

// ------------------------------------------------------------------------------------------
// squared distances of every ordered pair of each cloud; block row y = cloud. The points are
// checked with their own pair; one atomic per warp that raises the maximum
__global__ void k_pairwise(const int32_t* __restrict__ x, int D, CloudTabs ct, int64_t* d2,
                           unsigned long long* maxd2, int32_t* bad) {
  int c = blockIdx.y;
  int64_t p0 = ct.pt_off[c];
  int n = (int)(ct.pt_off[c + 1] - p0);
  int64_t nn = (int64_t)n * n;
  unsigned long long mx = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nn;
       t += (int64_t)gridDim.x * blockDim.x) {
    const unsigned a = (unsigned)t / (unsigned)n, b = (unsigned)t % (unsigned)n;  // n < 2^12
    const int32_t* xa = x + (p0 + a) * D;
    const int32_t* xb = x + (p0 + b) * D;
    int64_t s = 0;
    for (int k = 0; k < D; k++) {
      int64_t dd = (int64_t)xa[k] - (int64_t)xb[k];
      s += dd * dd;
      if (a == b && (xa[k] > (1 << 24) || xa[k] < -(1 << 24))) *bad = 1;
    }
    d2[ct.mo[c] + t] = s;
    mx = s > (int64_t)mx ? (unsigned long long)s : mx;
  }
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long y = __shfl_down_sync(0xffffffffu, mx, o);
    mx = y > mx ? y : mx;
  }
  if ((threadIdx.x & 31) == 0 && mx > *(volatile unsigned long long*)maxd2) atomicMax(maxd2, mx);
}

// Index of the first scale r_i = i * step with d <= 2 r_i for a squared distance d2 (Sec. 2.2:
// a simplex is in the complex at scale r when its diameter is at most 2r), by exact integer
// comparison: the smallest i >= 0 with d2 <= (2 i step)^2.
__host__ __device__ __forceinline__ int64_t scale_index_of(int64_t d2, int64_t step) {
  if (d2 <= 0) return 0;
  int64_t i = (int64_t)ceil(sqrt((double)d2) / (2.0 * (double)step));
  while (i > 0 && (2 * (i - 1) * step) * (2 * (i - 1) * step) >= d2) i--;
  while ((2 * i * step) * (2 * i * step) < d2) i++;
  return i;
}

__global__ void k_scale_index(int64_t* d2, int64_t n, int64_t step) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    d2[t] = scale_index_of(d2[t], step);
}

// count one kept candidate for cloud c with one atomic per group of lanes sharing c
__device__ __forceinline__ void count_kept(int64_t* count_per_cloud, int c, bool keep) {
  const unsigned peers = __match_any_sync(__activemask(), keep ? c : -1);
  if (keep && (threadIdx.x & 31) == __ffs(peers) - 1)
    atomicAdd((unsigned long long*)&count_per_cloud[c], (unsigned long long)__popc(peers));
}

// edge candidates in (cloud, lex) order; truncated edges get key = sent, or, if given, a key of one
// bit more than *largest. Kept ones are counted if some may be truncated
__global__ void k_edge_cand(CloudTabs ct, const int64_t* __restrict__ cand, int64_t ncand,
                            const int64_t* __restrict__ d2, int64_t max_d2, uint64_t sent,
                            const unsigned long long* largest, uint64_t* keys, uint64_t* vals,
                            int64_t* count_per_cloud) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ncand;
       t += (int64_t)gridDim.x * blockDim.x) {
    int c = find_cloud(cand, ct.nc, t);
    int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    int v[2];
    lex_unrank(t - cand[c], n, 2, v);
    int64_t e = d2[ct.mo[c] + (int64_t)v[0] * n + v[1]];
    bool keep = max_d2 < 0 || e <= max_d2;
    if (largest && !keep) sent = (2ull << (64 - __clzll((long long)*largest))) - 1ull;
    keys[t] = keep ? (uint64_t)e : sent;
    vals[t] = pack_simplex((uint32_t)c, 2, v, ct.vbits);
    if (max_d2 >= 0) count_kept(count_per_cloud, c, keep);
  }
}

__global__ void k_rekey_cloud(const uint64_t* __restrict__ vals, uint64_t* keys, int64_t n,
                              uint64_t sent, uint64_t nc) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    keys[t] = keys[t] == sent ? nc : (uint64_t)packed_cloud(vals[t]);
}

// first element of each distinct (cloud, squared diameter) among the sorted edges
__global__ void k_edge_newflag(const uint64_t* __restrict__ vals, int64_t E, CloudTabs ct,
                               const int64_t* __restrict__ d2, int32_t* flag, int64_t* ed2,
                               const int32_t* fault) {
  if (*fault) return;  // (a wait of the sort ran out)
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < E;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t p = vals[i];
    int c = (int)packed_cloud(p);
    int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    int64_t e = d2[ct.mo[c] + (int64_t)packed_vert(ct, p, 0) * n + packed_vert(ct, p, 1)];
    ed2[i] = e;
    int32_t f = 1;
    if (i > 0) {
      uint64_t q = vals[i - 1];
      int cq = (int)packed_cloud(q);
      if (cq == c) {
        int64_t eq = d2[ct.mo[c] + (int64_t)packed_vert(ct, q, 0) * n + packed_vert(ct, q, 1)];
        f = (eq != e);
      }
    }
    flag[i] = f;
  }
}

struct IdOut {
  int32_t* seg;
  int32_t* key;
  int32_t* low;
  uint64_t* verts;
  int32_t* rows0;
};

__global__ void k_edge_finish(const uint64_t* __restrict__ vals, int64_t E, CloudTabs ct,
                              const int32_t* __restrict__ flag, const int64_t* __restrict__ excl,
                              const int64_t* __restrict__ ed2, int64_t id0, int32_t* eid,
                              int32_t* erank, int64_t* d2tab, IdOut o, int64_t rowbase,
                              const int64_t* __restrict__ status, int64_t* host) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // for the host, in page-locked memory
    host[0] = *status;  // bad coordinates (low half), a wait of the sort that ran out (high half)
    host[1] = excl[E];  // distinct lengths
  }
  if (*status >> 32) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < E;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t p = vals[i];
    int c = (int)packed_cloud(p);
    int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    int a = packed_vert(ct, p, 0), b = packed_vert(ct, p, 1);
    int32_t rank = (int32_t)(excl[i] + flag[i] - 1);
    if (flag[i]) d2tab[rank] = ed2[i];
    int64_t id = id0 + i;
    int64_t mo = ct.mo[c];
    eid[mo + (int64_t)a * n + b] = (int32_t)id;
    eid[mo + (int64_t)b * n + a] = (int32_t)id;
    erank[mo + (int64_t)a * n + b] = rank;
    erank[mo + (int64_t)b * n + a] = rank;
    o.seg[id] = ct.nc + c;
    o.key[id] = rank;
    o.verts[id] = p;
    int32_t r0 = (int32_t)(ct.pt_off[c] + a), r1 = (int32_t)(ct.pt_off[c] + b);
    o.rows0[rowbase + 2 * i] = r0;
    o.rows0[rowbase + 2 * i + 1] = r1;
    o.low[id] = r1;
  }
}

// candidates of dimension k-1 (k vertices, 3 <= k <= 6): key = largest edge rank
__global__ void k_simplex_cand(CloudTabs ct, const int64_t* __restrict__ cand, int64_t ncand,
                               int k, const int32_t* __restrict__ erank, uint64_t sent,
                               uint64_t* keys, uint64_t* vals, int64_t* count_per_cloud) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ncand;
       t += (int64_t)gridDim.x * blockDim.x) {
    int c = find_cloud(cand, ct.nc, t);
    int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    int v[kVrSlots];
    lex_unrank(t - cand[c], n, k, v);
    const int32_t* er = erank + ct.mo[c];
    int32_t mx = -1;
    bool keep = true;
    for (int p = 0; p < k; p++)
      for (int q = p + 1; q < k; q++) {
        int32_t r = er[(int64_t)v[p] * n + v[q]];
        if (r < 0) keep = false;
        mx = r > mx ? r : mx;
      }
    keys[t] = keep ? (uint64_t)mx : sent;
    vals[t] = pack_simplex((uint32_t)c, k, v, ct.vbits);
    count_kept(count_per_cloud, c, keep);
  }
}

__device__ __forceinline__ void sort_small(int32_t* r, int k) {
  for (int i = 1; i < k; i++) {
    int32_t x = r[i];
    int j = i - 1;
    while (j >= 0 && r[j] > x) {
      r[j + 1] = r[j];
      j--;
    }
    r[j + 1] = x;
  }
}

// Where a dimension's simplices go: known on the device before the host reads the counts
struct DimPlace {
  int64_t n, id0, rowbase;
};
// by one block: the place of a dimension (k vertices) of count[0..nc) simplices after the one before
// (nothing is written after a sort whose wait ran out)
__global__ void k_dim_place(const int64_t* __restrict__ count, int nc, int k, DimPlace* place,
                            const int32_t* fault) {
  __shared__ int64_t sh[kWarps + 1];
  int64_t n = 0;
  for (int c = threadIdx.x; c < nc; c += kThreads) n += count[c];
  int64_t total;
  block_excl_sum<int64_t>(n, sh, total);
  if (threadIdx.x == 0) {
    const DimPlace before = place[-1];
    *place = DimPlace{*fault ? 0 : total, before.id0 + before.n, before.rowbase + (k - 1) * before.n};
  }
}

__global__ void k_tri_finish(const uint64_t* __restrict__ keys, const uint64_t* __restrict__ vals,
                             const DimPlace* __restrict__ place, CloudTabs ct,
                             const int32_t* __restrict__ eid, IdOut o, int32_t* tid_tab,
                             const int64_t* __restrict__ tri_lex_off) {
  const int64_t T = place->n, id0 = place->id0, rowbase = place->rowbase;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < T;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t p = vals[i];
    int c = (int)packed_cloud(p);
    int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    int v[3] = {packed_vert(ct, p, 0), packed_vert(ct, p, 1), packed_vert(ct, p, 2)};
    const int32_t* e = eid + ct.mo[c];
    int32_t r[3] = {e[(int64_t)v[1] * n + v[2]], e[(int64_t)v[0] * n + v[2]],
                    e[(int64_t)v[0] * n + v[1]]};
    sort_small(r, 3);
    int64_t id = id0 + i;
    for (int q = 0; q < 3; q++) o.rows0[rowbase + 3 * i + q] = r[q];
    o.low[id] = r[2];
    o.seg[id] = 2 * ct.nc + c;
    o.key[id] = (int32_t)keys[i];
    o.verts[id] = p;
    if (tid_tab) tid_tab[tri_lex_off[c] + lex_rank(v, n, 3)] = (int32_t)id;
  }
}

// simplices of k >= 4 vertices (dimension >= 3): faces are the (k-1)-subsets, found by their
// lexicographic rank in the table the previous dimension filled; this dimension fills its own
// table when a higher one follows
__global__ void k_high_finish(const uint64_t* __restrict__ keys, const uint64_t* __restrict__ vals,
                              const DimPlace* __restrict__ place, int k, CloudTabs ct,
                              const int32_t* __restrict__ face_tab,
                              const int64_t* __restrict__ face_lex_off, int32_t* self_tab,
                              const int64_t* __restrict__ self_lex_off, IdOut o) {
  const int64_t Q = place->n, id0 = place->id0, rowbase = place->rowbase;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Q;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t p = vals[i];
    int c = (int)packed_cloud(p);
    int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    int v[kVrSlots];
    for (int q = 0; q < k; q++) v[q] = packed_vert(ct, p, q);
    int32_t r[kVrSlots];
    for (int drop = 0; drop < k; drop++) {
      int f[kVrSlots], m = 0;
      for (int q = 0; q < k; q++)
        if (q != drop) f[m++] = v[q];
      r[drop] = face_tab[face_lex_off[c] + lex_rank(f, n, k - 1)];
    }
    sort_small(r, k);
    int64_t id = id0 + i;
    for (int q = 0; q < k; q++) o.rows0[rowbase + (int64_t)k * i + q] = r[q];
    o.low[id] = r[k - 1];
    o.seg[id] = (k - 1) * ct.nc + c;
    o.key[id] = (int32_t)keys[i];
    o.verts[id] = p;
    if (self_tab) self_tab[self_lex_off[c] + lex_rank(v, n, k)] = (int32_t)id;
  }
}

// ------------------------------------------------------------------------------------------
// triangles and tetrahedra without a sort
// ------------------------------------------------------------------------------------------
// When no two edges of a cloud have the same length, every simplex of dimension 2 or more has one
// longest edge, and the filtration lists the simplices of a dimension by that edge, those of
// one edge ab in the lexicographic order of their other vertices (two sorted tuples that share a
// and b compare like the rest). So one warp per edge writes its simplices straight to their places:
// L(ab), the vertices c whose edges to a and b are both shorter, gives the triangles abc, and
// the pairs c < d of L(ab) whose edge is shorter than ab the tetrahedra abcd, in order. The
// counts per edge, scanned, are the places, and the filtration indices and left(i) (Definition 3)
// of edges follow from them. With sorted candidates (each unranked by binary searches, five
// kernels per 8-bit digit, then an atomic per row for left and two searches per simplex for the
// index) the build of a 400-point cloud took 2.1 ms and now takes 0.46 ms, that of 120 points in
// 8-d to dimension 3 with a cut 1.24 -> 0.31 ms, of 512 clouds of 20 to 120 points 6.4 -> 1.43 ms.
// Counting is bound by instruction issue (225 warp instructions an edge of 80 points), listing by
// issue and by its writes of 40 bytes a triangle.
// The direct listing is taken whenever it applies: it is faster at every size measured (40
// points: 470 -> 128 us, the one-block sort of the edges included). With ties, and in dimensions 4
// and 5, candidates are sorted.
constexpr int kDirectPoints = 512;   // points per cloud with tetrahedra (a warp's list of L(ab))
constexpr int kDirectWarps = 4;
static_assert(kVertBits == 12, "packed simplices are written here");

struct Direct {
  const uint64_t* edge;   // sorted edges (packed), E of them; edge e has id N + e
  int64_t E, N;
  const int32_t* eid;     // per cloud n x n: edge id, -1 if not in the complex
  const int64_t* es;      // per cloud: first edge
  const int64_t* off2;    // [E + 1] triangles before each edge's
  const int64_t* off3;    // [E + 1] tetrahedra, null without them
  const uint32_t* mask;   // [E][words] L(ab) as bits
  int words;
  int32_t* left;          // per row id
  int64_t* gidx;
};

__global__ void __launch_bounds__(32 * kDirectWarps) k_link_count(CloudTabs ct, Direct g,
                                                                  int32_t* cnt2, int32_t* cnt3,
                                                                  uint32_t* mask) {
  __shared__ uint16_t s_list[kDirectWarps][kDirectPoints];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t e = (int64_t)blockIdx.x * kDirectWarps + w; e < g.E;
       e += (int64_t)gridDim.x * kDirectWarps) {
    const uint64_t p = g.edge[e];
    const int c = (int)packed_cloud(p), a = packed_vert(ct, p, 0), b = packed_vert(ct, p, 1);
    const int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    const int32_t* tab = g.eid + ct.mo[c];
    const int32_t id = (int32_t)(g.N + e);
    int n2 = 0;
    const int32_t* ra = tab + (int64_t)a * n;
    const int32_t* rb = tab + (int64_t)b * n;
    uint32_t mine = 0;  // mask word lane of the current 32
    for (int c0 = 0; c0 < n; c0 += 64) {
      int32_t ac[2], bc[2];
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const int x = c0 + 32 * q + lane;
        ac[q] = x < n ? ra[x] : -1;
        bc[q] = x < n ? rb[x] : -1;
      }
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const bool f = (uint32_t)ac[q] < (uint32_t)id && (uint32_t)bc[q] < (uint32_t)id;
        const unsigned m = __ballot_sync(0xffffffffu, f);
        if (lane == (((c0 >> 5) + q) & 31)) mine = m;
        if (cnt3 && f) s_list[w][n2 + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(c0 + 32 * q + lane);
        n2 += __popc(m);
      }
      if ((c0 & 1023) == 960 || c0 + 64 >= n) {
        const int word = ((c0 >> 5) & ~31) + lane;
        if (word < g.words) mask[e * g.words + word] = mine;
        mine = 0;
      }
    }
    if (lane == 0) cnt2[e] = n2;
    if (!cnt3) continue;
    __syncwarp();
    int n3 = 0;
    for (int i = 0; i + 1 < n2; i++) {
      const int32_t* rc = tab + (int64_t)s_list[w][i] * n;
      for (int j = i + 1 + lane; j < n2; j += 32) {
        const int32_t cd = rc[s_list[w][j]];
        n3 += cd >= 0 && cd < id ? 1 : 0;
      }
    }
    n3 = (int)__reduce_add_sync(0xffffffffu, (unsigned)n3);
    if (lane == 0) cnt3[e] = n3;
    __syncwarp();
  }
}

// per cloud (and the end): triangles and tetrahedra before its first edge, then whether a wait ran out;
// into page-locked memory
__global__ void k_cloud_bounds(Direct g, int nc, int64_t* out, const int32_t* fault) {
  if (blockIdx.x == 0 && threadIdx.x == 0) out[2 * (nc + 1)] = *fault;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= nc; c += gridDim.x * blockDim.x) {
    out[c] = g.off2[g.es[c]];
    out[nc + 1 + c] = g.off3 ? g.off3[g.es[c]] : 0;
  }
}

__device__ __forceinline__ void lower_left(int32_t* left, int32_t row, int32_t col) {
  if (left[row] > col) atomicMin(&left[row], col);
}

// lists the vertices of up to kListWords mask words from word q0 on (in order) by one warp
constexpr int kListWords = kDirectPoints / 32;
__device__ __forceinline__ int list_mask(const uint32_t* mask, int q0, int words, uint16_t* list) {
  const int lane = threadIdx.x & 31;
  const int nq = min(kListWords, words - q0);
  const uint32_t mine = lane < nq ? mask[q0 + lane] : 0;
  int n = 0;
  for (int q = 0; q < nq; q++) {
    const uint32_t m = __shfl_sync(0xffffffffu, mine, q);
    if ((m >> lane) & 1u) list[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)((q0 + q) * 32 + lane);
    n += __popc(m);
  }
  __syncwarp();
  return n;
}

// id of the triangle on three vertices of one cloud: its longest edge's place plus the number of
// smaller vertices in that edge's L
__device__ __forceinline__ int32_t triangle_id(const Direct& g, const int32_t* tab, int n, int u,
                                               int v, int x) {
  const int32_t uv = tab[(int64_t)u * n + v], ux = tab[(int64_t)u * n + x],
                vx = tab[(int64_t)v * n + x];
  int32_t e = uv;
  int third = x;
  if (ux > e) {
    e = ux;
    third = v;
  }
  if (vx > e) {
    e = vx;
    third = u;
  }
  const int64_t ei = e - g.N;
  const uint32_t* m = g.mask + ei * g.words;
  int k = __popc(m[third >> 5] & ((1u << (third & 31)) - 1u));
  for (int q = 0; q < (third >> 5); q++) k += __popc(m[q]);
  return (int32_t)(g.N + g.E + g.off2[ei] + k);
}

// A warp takes `group` consecutive edges (a power of two, up to 32; as many as leave every warp of the
// machine some): what an edge needs is loaded by one lane each, and their triangles are one run that
// the lanes share, 32 at a time. A lane finds its edge by a search over the group's places and its
// vertex by a search in the edge's mask. With a warp per edge 645 instructions went into an edge of 26
// triangles: 10.7 M triangles in 256 clouds of 64 points took 384 us, now 139; 42 M in 512 clouds 1178,
// now 569; 10.6 M of 400 points 176, now 161 (their writes alone take 62 us at the copy rate).
__global__ void __launch_bounds__(32 * kDirectWarps) k_tri_emit(CloudTabs ct, Direct g, IdOut o,
                                                                int64_t rowbase, int group) {
  __shared__ int32_t s_rows[kDirectWarps][96];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.N;
       i += (int64_t)gridDim.x * blockDim.x)  // a vertex's index is its place in its cloud
    g.gidx[i] = i - ct.pt_off[find_cloud(ct.pt_off, ct.nc, i)];
  for (int64_t e0 = ((int64_t)blockIdx.x * kDirectWarps + w) * group; e0 < g.E;
       e0 += (int64_t)gridDim.x * kDirectWarps * group) {
    const int64_t e = e0 + lane;
    const bool mine = lane < group && e < g.E;
    int c = 0, a = 0, b = 0, n = 0;
    int64_t t0 = 0, t1 = 0, gi = 0;
    if (mine) {
      const uint64_t p = g.edge[e];
      t0 = g.off2[e];
      t1 = g.off2[e + 1];
      c = (int)packed_cloud(p);
      a = packed_vert(ct, p, 0);
      b = packed_vert(ct, p, 1);
      const int64_t v0 = ct.pt_off[c], es = g.es[c];
      n = (int)(ct.pt_off[c + 1] - v0);
      const int32_t id = (int32_t)(g.N + e);
      gi = n + (e - es) + (t0 - g.off2[es]) + (g.off3 ? g.off3[e] - g.off3[es] : 0);
      g.gidx[id] = gi;
      lower_left(g.left, (int32_t)(v0 + a), id);
      lower_left(g.left, (int32_t)(v0 + b), id);
      // an edge's first column is its own first triangle: it is shorter than the longest edge of
      // any other triangle that holds it
      if (t1 > t0) g.left[id] = (int32_t)(g.N + g.E + t0);
    }
    // Without one (the edges of the relative neighbourhood graph) it is the triangle on it whose
    // longest edge is least: no two share that edge
    for (unsigned none = __ballot_sync(0xffffffffu, mine && t1 == t0); none; none &= none - 1) {
      const int src = __ffs(none) - 1;
      const int ea = __shfl_sync(0xffffffffu, a, src), eb = __shfl_sync(0xffffffffu, b, src);
      const int en = __shfl_sync(0xffffffffu, n, src);
      const int32_t* tab = g.eid + ct.mo[__shfl_sync(0xffffffffu, c, src)];
      const int32_t* ra = tab + (int64_t)ea * en;
      const int32_t* rb = tab + (int64_t)eb * en;
      uint32_t least = 0x7f7f7f7fu;
      int third = -1;
      for (int x = lane; x < en; x += 32) {
        const int32_t ac = ra[x], bc = rb[x];
        const uint32_t longest = ac < 0 || bc < 0 ? 0x7f7f7f7fu : (uint32_t)max(ac, bc);
        if (longest < least) {
          least = longest;
          third = x;
        }
      }
      const uint32_t all = __reduce_min_sync(0xffffffffu, least);
      if (third >= 0 && least == all)
        g.left[g.N + e0 + src] = triangle_id(g, tab, en, ea, eb, third);
    }
    // the group's triangles, as places from its first one's on
    const int last = (int)min((int64_t)group, g.E - e0) - 1;
    const int64_t first = __shfl_sync(0xffffffffu, t0, 0);
    const int total = (int)(__shfl_sync(0xffffffffu, t1, last) - first);
    const int place = mine ? (int)(t0 - first) : INT32_MAX;
    const int ab = a | b << 16;
    for (int r0 = 0; r0 < total; r0 += 32) {
      const int r = r0 + lane;
      int i = 0;  // the last edge of the group whose place is not above r
      for (int step = group >> 1; step > 0; step >>= 1)
        if (__shfl_sync(0xffffffffu, place, i + step) <= r) i += step;
      int k = r - __shfl_sync(0xffffffffu, place, i);
      const int eab = __shfl_sync(0xffffffffu, ab, i), ec = __shfl_sync(0xffffffffu, c, i);
      const int en = __shfl_sync(0xffffffffu, n, i);
      const int64_t index = __shfl_sync(0xffffffffu, gi, i) + 1 + k;
      if (r < total) {
        const int64_t ee = e0 + i, t = g.N + g.E + first + r;
        const int ea = eab & 0xffff, eb = eab >> 16;
        const int32_t id = (int32_t)(g.N + ee);
        // vertex k of L(ab)
        const uint32_t* m = g.mask + ee * g.words;
        uint32_t bits = *m;
        int x = 0;
        for (int pc = __popc(bits); pc <= k; pc = __popc(bits)) {
          k -= pc;
          bits = *++m;
          x += 32;
        }
#pragma unroll
        for (int half = 16; half > 0; half >>= 1) {
          const uint32_t low = bits & ((1u << half) - 1u);
          const int pc = __popc(low);
          const bool up = k >= pc;
          k -= up ? pc : 0;
          x += up ? half : 0;
          bits = up ? bits >> half : low;
        }
        const int32_t* tab = g.eid + ct.mo[ec];
        const int32_t ac = tab[ea * en + x], bc = tab[eb * en + x];
        o.verts[t] = (uint64_t)ec << 48 | (uint64_t)min(ea, x) << 36 |
                     (uint64_t)(x < ea ? ea : min(x, eb)) << 24 | (uint64_t)max(eb, x) << 12 |
                     ((1u << 12) - 1u);  // the last slot is empty
        o.seg[t] = 2 * ct.nc + ec;
        o.key[t] = (int32_t)ee;
        o.low[t] = id;
        g.gidx[t] = index;
        s_rows[w][3 * lane] = min(ac, bc);
        s_rows[w][3 * lane + 1] = max(ac, bc);
        s_rows[w][3 * lane + 2] = id;
      }
      __syncwarp();
      const int have = 3 * min(32, total - r0);
      int32_t* rows = o.rows0 + rowbase + 3 * (first + r0);
#pragma unroll
      for (int q = 0; q < 3; q++)
        if (q * 32 + lane < have) rows[q * 32 + lane] = s_rows[w][q * 32 + lane];
      __syncwarp();
    }
  }
}

// One block per edge: its rows of pairs are counted, then written, by all warps. The edges with the
// longest lists bound it: with a warp per edge the 920,000 tetrahedra of 120 points took 198 us, with
// eight warps 87 us.
constexpr int kTetThreads = 256, kTetWarps = kTetThreads / 32;

__global__ void __launch_bounds__(kTetThreads) k_tet_emit(CloudTabs ct, Direct g, IdOut o,
                                                          int64_t id0, int64_t rowbase) {
  __shared__ uint16_t s_list[kDirectPoints];
  __shared__ int32_t s_row[kDirectPoints];
  __shared__ int s_n2;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t e = blockIdx.x; e < g.E; e += gridDim.x) {
    const int64_t q0 = g.off3[e];
    if (g.off3[e + 1] == q0) continue;
    const uint64_t p = g.edge[e];
    const int c = (int)packed_cloud(p), a = packed_vert(ct, p, 0), b = packed_vert(ct, p, 1);
    const int n = (int)(ct.pt_off[c + 1] - ct.pt_off[c]);
    const int32_t* tab = g.eid + ct.mo[c];
    const int32_t id = (int32_t)(g.N + e);
    const int64_t es = g.es[c];
    const int64_t gi = n + (e - es) + 1 + (g.off2[e + 1] - g.off2[es]) + (q0 - g.off3[es]);
    const int32_t tri0 = (int32_t)(g.N + g.E + g.off2[e]);
    __syncthreads();  // the lists of the edge before are done with
    if (w == 0) {
      const int k = list_mask(g.mask + e * g.words, 0, (n + 31) >> 5, s_list);
      if (lane == 0) s_n2 = k;
    }
    __syncthreads();
    const int n2 = s_n2;
    for (int i = w; i < n2; i += kTetWarps) {
      const int32_t* rc = tab + (int64_t)s_list[i] * n;
      int k = 0;
      for (int j = i + 1 + lane; j < n2; j += 32) {
        const int32_t cd = rc[s_list[j]];
        k += cd >= 0 && cd < id ? 1 : 0;
      }
      k = (int)__reduce_add_sync(0xffffffffu, (unsigned)k);
      if (lane == 0) s_row[i] = k;
    }
    __syncthreads();
    if (w == 0) {
      int run = 0;
      for (int i = 0; i < n2; i += 32) {
        const int k = i + lane < n2 ? s_row[i + lane] : 0;
        const int inc = warp_incl_sum(k);
        if (i + lane < n2) s_row[i + lane] = run + inc - k;
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
    }
    __syncthreads();
    for (int i = w; i < n2; i += kTetWarps) {
      const int x = s_list[i];
      const int32_t* rc = tab + (int64_t)x * n;
      int run = s_row[i];
      for (int j0 = i + 1; j0 < n2; j0 += 32) {
        const int j = j0 + lane;
        const int y = j < n2 ? s_list[j] : 0;
        const int32_t cd = j < n2 ? rc[y] : -1;
        const bool f = cd >= 0 && cd < id;
        const unsigned m = __ballot_sync(0xffffffffu, f);
        if (f) {
          const int k = run + __popc(m & ((1u << lane) - 1u));
          const int64_t t = id0 + q0 + k;
          int32_t v[4] = {a, b, x, y};
          sort_small(v, 4);
          const uint64_t packed = (uint64_t)c << 48 | (uint64_t)v[0] << 36 | (uint64_t)v[1] << 24 |
                                  (uint64_t)v[2] << 12 | (uint64_t)v[3];
          int32_t r[4] = {tri0 + i, tri0 + j, triangle_id(g, tab, n, a, x, y),
                          triangle_id(g, tab, n, b, x, y)};
          sort_small(r, 4);
          o.verts[t] = packed;
          o.seg[t] = 3 * ct.nc + c;
          o.key[t] = (int32_t)e;
          o.low[t] = r[3];
          g.gidx[t] = gi + k;
          int32_t* ro = o.rows0 + rowbase + 4 * (q0 + k);
          for (int q = 0; q < 4; q++) {
            ro[q] = r[q];
            lower_left(g.left, r[q], (int32_t)t);
          }
        }
        run += __popc(m);
      }
    }
  }
}

__global__ void k_vertex_init(CloudTabs ct, int64_t N, IdOut o) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
    int c = find_cloud(ct.pt_off, ct.nc, i);
    int v = (int)(i - ct.pt_off[c]);
    o.seg[i] = c;
    o.key[i] = -1;
    o.low[i] = -1;
    o.verts[i] = pack_simplex((uint32_t)c, 1, &v, ct.vbits);
  }
}

// ------------------------------------------------------------------------------------------
// left(i) (Definition 3) by atomicMin over the columns holding row i, then
// beta_j = max{ i : left(i) = j } (Definition 4) by atomicMax.
// ------------------------------------------------------------------------------------------
struct ColLayout {  // initial column storage: dim d column x at rowbase[d] + (d+1)(x - dimoff[d])
  int64_t dimoff[kMaxDim + 2];
  int64_t rowbase[kMaxDim + 2];
  int maxd;
};

__device__ __forceinline__ int id_dim(const ColLayout& L, int64_t x) {
  int d = 0;
  while (d < L.maxd && x >= L.dimoff[d + 1]) d++;
  return d;
}

// col_off: the columns of a loaded matrix (any length); null: d + 1 rows at a fixed stride
__global__ void k_left(ColLayout L, const int32_t* __restrict__ rows0,
                       const int64_t* __restrict__ col_off, int32_t* left) {
  int64_t n = L.dimoff[L.maxd + 1] - L.dimoff[1];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t j = L.dimoff[1] + t;
    int d = id_dim(L, j);
    const int32_t* r = col_off ? rows0 + col_off[j]
                               : rows0 + L.rowbase[d] + (int64_t)(d + 1) * (j - L.dimoff[d]);
    const int64_t len = col_off ? col_off[j + 1] - col_off[j] : d + 1;
    for (int64_t q = 0; q < len; q++) lower_left(left, r[q], (int32_t)j);
  }
}

__global__ void k_beta(int64_t nrows, int64_t m, const int32_t* __restrict__ left, int32_t* beta) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nrows;
       i += (int64_t)gridDim.x * blockDim.x) {
    int32_t j = left[i];
    if (j < m) atomicMax(&beta[j], (int32_t)i);  // rows without a coface keep the fill
  }
}

// filtration index of every simplex within its cloud: simplices of other dimensions that
// precede it are those of lower dimension with diameter <= its own and of higher dimension with
// diameter < its own (ties are broken by dimension); all vertices (diameter 0) come first.
__global__ void k_gidx(int64_t m, int nc, int maxd, const int32_t* __restrict__ seg,
                       const int32_t* __restrict__ key, const int64_t* __restrict__ seg_start,
                       const int64_t* __restrict__ pt_off, int64_t* gidx) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < m;
       x += (int64_t)gridDim.x * blockDim.x) {
    int s = seg[x];
    int d = s / nc, c = s % nc;
    int64_t g = x - seg_start[s];
    if (d > 0) {
      int32_t k = key[x];
      g += pt_off[c + 1] - pt_off[c];
      for (int dd = 1; dd <= maxd; dd++) {
        if (dd == d) continue;
        int64_t lo = seg_start[dd * nc + c], hi = seg_start[dd * nc + c + 1];
        int64_t a = lo, b = hi;
        if (dd < d) {  // count key <= k
          while (a < b) {
            int64_t mid = (a + b) >> 1;
            if (key[mid] <= k) a = mid + 1; else b = mid;
          }
        } else {  // count key < k
          while (a < b) {
            int64_t mid = (a + b) >> 1;
            if (key[mid] < k) a = mid + 1; else b = mid;
          }
        }
        g += a - lo;
      }
    }
    gidx[x] = g;
  }
}

static int bitlen(uint64_t v) {
  int b = 0;
  while (v) {
    b++;
    v >>= 1;
  }
  return b;
}

// segments and initial lows of a loaded matrix
__global__ void k_loaded(ColLayout L, int64_t m, const int32_t* __restrict__ rows0,
                         const int64_t* __restrict__ col_off, int32_t* seg, int32_t* low) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < m;
       x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t end = col_off[x + 1];
    seg[x] = id_dim(L, x);
    low[x] = end > col_off[x] ? rows0[end - 1] : -1;
  }
}

// common tail of build_vr and load_boundary: segment table, per-id arrays already filled
static void finish_layout(ph_ctx* ctx) {
  ctx->d_seg_start = alloc_n<int64_t>(ctx, (int64_t)ctx->seg_start.size());
  PH_CUDA(cudaMemcpyAsync(ctx->d_seg_start, ctx->seg_start.data(),
                          ctx->seg_start.size() * sizeof(int64_t), cudaMemcpyHostToDevice,
                          ctx->stream));
}

// beta of every column (Definition 4): left(i) first, then the largest row per left column
void compute_beta(ph_ctx* ctx) {
  cudaStream_t st = ctx->stream;
  ColLayout L{};
  L.maxd = ctx->max_dim;
  for (int d = 0; d <= ctx->max_dim + 1; d++) L.dimoff[d] = ctx->dimoff[d];
  int64_t rb = 0;
  for (int d = 0; d <= ctx->max_dim; d++) {
    L.rowbase[d] = rb;
    rb += (d > 0 ? d + 1 : 0) * (ctx->dimoff[d + 1] - ctx->dimoff[d]);
  }
  int32_t* left = alloc_n<int32_t>(ctx, ctx->m);
  ctx->beta = alloc_n<int32_t>(ctx, ctx->m);
  PH_CUDA(cudaMemsetAsync(left, 0x7f, ctx->m * sizeof(int32_t), st));  // > every id
  PH_CUDA(cudaMemsetAsync(ctx->beta, 0xff, ctx->m * sizeof(int32_t), st));
  k_left<<<grid_for(ctx, ctx->m, kThreads), kThreads, 0, st>>>(L, ctx->rows0, ctx->col_off,
                                                               left);
  PH_CHECK_LAUNCH();
  k_beta<<<grid_for(ctx, ctx->m, kThreads), kThreads, 0, st>>>(ctx->m, ctx->m, left, ctx->beta);
  PH_CHECK_LAUNCH();
  ctx->dfree(left);
}

// An explicit complex given in filtration order: re-index it dim-major (stable inside each
// dimension, which keeps every order the reduction compares) and store its boundary. A column
// may hold any number of rows of the dimension below (a simplicial, cubical or cellular
// boundary over F2, or a partially reduced matrix R = D V), so columns are kept with offsets.
void load_boundary(ph_ctx* ctx, int64_t m, const int32_t* dims, const int64_t* colptr,
                   const int32_t* rows) {
  cudaStream_t st = ctx->stream;
  PH_REQUIRE(m >= 1 && m < 0x7f000000LL, PH_ERR_INVALID, "m out of range");
  PH_REQUIRE(dims && colptr && rows, PH_ERR_INVALID, "NULL argument");
  int maxd = 0;
  std::vector<int64_t> cnt(kMaxDim + 1, 0);
  for (int64_t j = 0; j < m; j++) {
    PH_REQUIRE(dims[j] >= 0 && dims[j] <= kMaxDim, PH_ERR_INVALID, "dimension out of range");
    maxd = std::max(maxd, (int)dims[j]);
    cnt[dims[j]]++;
  }
  std::vector<int64_t> dimoff(maxd + 2, 0);
  for (int d = 0; d <= maxd; d++) dimoff[d + 1] = dimoff[d] + cnt[d];
  PH_REQUIRE(colptr[0] == 0, PH_ERR_INVALID, "colptr[0] must be 0");
  int64_t nnz = 0;
  for (int64_t j = 0; j < m; j++) {
    const int64_t n = colptr[j + 1] - colptr[j];
    PH_REQUIRE(n >= 0 && (dims[j] > 0 || n == 0), PH_ERR_INVALID,
               "column lengths must be >= 0, and 0 in dimension 0");
    nnz += n;
  }
  // One host buffer, copied at once: the filtration index and the column's end per id, the columns'
  // rows as ids; then, not copied, the id per index. Kept page-locked memory up to a size (fresh pages
  // and seven copies were a fifth of the 374 us of a 96 x 80 image grid's 30,369 simplices; 300 us now).
  constexpr int64_t kLoadPinned = 16 << 20;
  const int64_t copied = (2 * m + 1) * 8 + (nnz + (nnz & 1)) * 4, bytes = copied + 4 * m;
  std::unique_ptr<char[]> pageable;
  char* host = nullptr;
  if (bytes <= kLoadPinned) {
    try {
      host = static_cast<char*>(ctx->pinned(bytes));
    } catch (const Fail&) {  // pageable memory does as well
      ctx->err.clear();
    }
  }
  if (!host) {
    pageable.reset(new char[bytes]);
    host = pageable.get();
  }
  int64_t* h_gidx = reinterpret_cast<int64_t*>(host);
  int64_t* h_off = h_gidx + m;  // column offsets in id order
  int32_t* h_rows = reinterpret_cast<int32_t*>(h_off + m + 1);
  int32_t* id_of = reinterpret_cast<int32_t*>(host + copied);
  std::vector<int64_t> fill(dimoff.begin(), dimoff.end());
  for (int64_t j = 0; j < m; j++) {
    const int64_t x = fill[dims[j]]++;
    id_of[j] = (int32_t)x;
    h_gidx[x] = j;
    h_off[x + 1] = colptr[j + 1] - colptr[j];
  }
  h_off[0] = 0;
  for (int64_t x = 0; x < m; x++) h_off[x + 1] += h_off[x];
  for (int64_t j = 0; j < m; j++) {
    const int d = dims[j];
    const int64_t n = colptr[j + 1] - colptr[j];
    const int32_t* r = rows + colptr[j];
    int32_t* o = h_rows + h_off[id_of[j]];
    int32_t prev = -1;
    for (int64_t p = 0; p < n; p++) {
      PH_REQUIRE(r[p] >= 0 && r[p] < j && dims[r[p]] == d - 1, PH_ERR_INVALID,
                 "rows must be earlier simplices of dimension d - 1");
      PH_REQUIRE(r[p] > prev, PH_ERR_INVALID, "rows must be strictly ascending");
      prev = r[p];
      o[p] = id_of[r[p]];
    }
  }
  ctx->n_clouds = 1;
  ctx->max_dim = maxd;
  ctx->m = m;
  ctx->nnz = nnz;
  ctx->pt_off = {0, cnt[0]};
  for (int d = 0; d <= maxd + 1; d++) ctx->dimoff[d] = dimoff[d];
  ctx->seg_start.assign(dimoff.begin(), dimoff.end());
  ctx->seg = alloc_n<int32_t>(ctx, m);
  ctx->key = alloc_n<int32_t>(ctx, m);
  ctx->low = alloc_n<int32_t>(ctx, m);
  ctx->gidx = reinterpret_cast<int64_t*>(ctx->dalloc(copied + kColSlack * sizeof(int32_t)));
  ctx->col_off = ctx->gidx + m;
  ctx->rows0 = reinterpret_cast<int32_t*>(ctx->col_off + m + 1);
  ctx->verts = alloc_n<uint64_t>(ctx, m);
  ctx->d2tab = alloc_n<int64_t>(ctx, 1);
  ctx->n_d2 = 0;
  PH_CUDA(cudaMemcpyAsync(ctx->gidx, host, copied, cudaMemcpyHostToDevice, st));
  PH_CUDA(cudaMemsetAsync(ctx->key, 0xff, m * sizeof(int32_t), st));      // no key
  PH_CUDA(cudaMemsetAsync(ctx->verts, 0xff, m * sizeof(uint64_t), st));  // no vertices
  ColLayout L{};
  L.maxd = maxd;
  for (int d = 0; d <= maxd + 1; d++) L.dimoff[d] = dimoff[d];
  k_loaded<<<grid_for(ctx, m, kThreads), kThreads, 0, st>>>(L, m, ctx->rows0, ctx->col_off, ctx->seg,
                                                            ctx->low);
  PH_CHECK_LAUNCH();
  finish_layout(ctx);
  compute_beta(ctx);
  PH_CUDA(cudaStreamSynchronize(st));
}

static const char* const kSortFault = "a bounded wait of the filtration build ran out";

// triangles and tetrahedra of a complex without ties, with beta and the filtration indices of
// every dimension; fills the counts of dimensions 2 and 3 (per cloud in h_cnt). scratch: page-locked,
// 3 (nc + 1) + 3 words
static void build_direct(ph_ctx* ctx, const CloudTabs& ct, Direct g, const IdOut& o,
                         std::vector<int64_t>& h_cnt, std::vector<int64_t>& cnts, int words,
                         int64_t* scratch, int32_t* d_fault) {
  cudaStream_t st = ctx->stream;
  const int nc = ct.nc;
  const bool tets = ctx->max_dim == 3;
  // per cloud: first edge; then, from the device, triangles and tetrahedra before it
  int64_t* d_es = alloc_n<int64_t>(ctx, nc + 1);
  scratch[0] = 0;
  for (int c = 0; c < nc; c++) scratch[c + 1] = scratch[c] + h_cnt[c];
  PH_CUDA(cudaMemcpyAsync(d_es, scratch, (nc + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, st));
  int32_t* cnt2 = alloc_n<int32_t>(ctx, g.E);
  int32_t* cnt3 = tets ? alloc_n<int32_t>(ctx, g.E) : nullptr;
  int64_t* off2 = alloc_n<int64_t>(ctx, g.E + 1);
  int64_t* off3 = tets ? alloc_n<int64_t>(ctx, g.E + 1) : nullptr;
  uint32_t* mask = alloc_n<uint32_t>(ctx, g.E * words);
  g.es = d_es;
  g.off2 = off2;
  g.off3 = off3;
  g.mask = mask;
  g.words = words;
  const unsigned grid = grid_for(ctx, g.E, kDirectWarps, 16);
  k_link_count<<<grid, 32 * kDirectWarps, 0, st>>>(ct, g, cnt2, cnt3, mask);
  PH_CHECK_LAUNCH();
  scan_counts(ctx, cnt2, cnt3, g.E, off2, off3, d_fault);
  int64_t* h_bounds = scratch + nc + 1;
  k_cloud_bounds<<<grid_for(ctx, nc + 1, kThreads), kThreads, 0, st>>>(g, nc, h_bounds, d_fault);
  PH_CHECK_LAUNCH();
  PH_CUDA(cudaStreamSynchronize(st));
  PH_REQUIRE(h_bounds[2 * (nc + 1)] == 0, PH_ERR_CUDA, kSortFault);
  for (int d = 2; d <= ctx->max_dim; d++) {
    const int64_t* b = h_bounds + (d - 2) * (nc + 1);
    for (int c = 0; c < nc; c++) h_cnt[(int64_t)(d - 1) * nc + c] = b[c + 1] - b[c];
    cnts[d] = b[nc];
  }
  const int64_t id3 = g.N + g.E + cnts[2], m = id3 + (tets ? cnts[3] : 0);
  const int64_t rows = tets ? id3 : g.N + g.E;  // simplices below the top dimension
  int32_t* left = alloc_n<int32_t>(ctx, rows);
  ctx->gidx = alloc_n<int64_t>(ctx, m);
  ctx->beta = alloc_n<int32_t>(ctx, m);
  g.left = left;
  g.gidx = ctx->gidx;
  PH_CUDA(cudaMemsetAsync(left, 0x7f, rows * sizeof(int32_t), st));  // > every id
  PH_CUDA(cudaMemsetAsync(ctx->beta, 0xff, m * sizeof(int32_t), st));
  int group = 1;
  while (group < 32 && g.E / (2 * group) >= (int64_t)ctx->num_sms * 64) group *= 2;
  k_tri_emit<<<grid_for(ctx, (g.E + group - 1) / group, kDirectWarps, 16), 32 * kDirectWarps, 0, st>>>(
      ct, g, o, 2 * g.E, group);
  PH_CHECK_LAUNCH();
  if (tets && cnts[3] > 0) {
    k_tet_emit<<<grid_for(ctx, g.E, 1, 16), kTetThreads, 0, st>>>(ct, g, o, id3, 2 * g.E + 3 * cnts[2]);
    PH_CHECK_LAUNCH();
  }
  k_beta<<<grid_for(ctx, rows, kThreads), kThreads, 0, st>>>(rows, m, left, ctx->beta);
  PH_CHECK_LAUNCH();
  for (void* p : {(void*)d_es, (void*)cnt2, (void*)cnt3, (void*)off2, (void*)off3, (void*)mask,
                  (void*)left})
    ctx->dfree(p);
}

void build_vr(ph_ctx* ctx, const int32_t* coords, const int64_t* cloud_offsets, int32_t nc,
              int64_t n_points, int32_t D, int32_t max_dim, int64_t max_diam2,
              int64_t scale_step, int32_t n_scales) {
  cudaStream_t st = ctx->stream;
  PH_REQUIRE(coords != nullptr, PH_ERR_INVALID, "coords is NULL");
  PH_REQUIRE(nc >= 1 && nc <= kMaxClouds, PH_ERR_INVALID, "n_clouds out of range");
  PH_REQUIRE(D >= 1 && D <= 16, PH_ERR_INVALID, "D must be in 1..16");
  PH_REQUIRE(max_dim >= 1 && max_dim <= kMaxVrDim, PH_ERR_INVALID, "max_dim must be 1..5");
  const int vbits = vert_bits_for(max_dim);
  std::vector<int64_t> off(nc + 1);
  if (cloud_offsets) {
    for (int c = 0; c <= nc; c++) off[c] = cloud_offsets[c];
  } else {
    PH_REQUIRE(nc == 1, PH_ERR_INVALID, "cloud_offsets required for several clouds");
    off[0] = 0;
    off[1] = n_points;
  }
  PH_REQUIRE(off[0] == 0 && off[nc] == n_points, PH_ERR_INVALID,
             "cloud_offsets must start at 0 and end at n_points");
  // per cloud: n x n table offsets and, for k = 2..max_dim+1 vertices, the candidate offsets
  const int K = max_dim + 1;  // largest vertex count
  std::vector<int64_t> mo(nc + 1, 0);
  std::vector<std::vector<int64_t>> cand(kVrSlots + 1, std::vector<int64_t>(nc + 1, 0));
  int64_t ncand_all = 0;
  for (int c = 0; c < nc; c++) {
    int64_t n = off[c + 1] - off[c];
    PH_REQUIRE(n >= 1 && n < (1 << vbits) - 1, PH_ERR_CAPACITY,
               max_dim <= 3 ? "each cloud needs 1..4094 points"
                            : "each cloud needs 1..254 points above dimension 3");
    mo[c + 1] = mo[c] + n * n;
    for (int k = 2; k <= kVrSlots; k++)
      cand[k][c + 1] = cand[k][c] + (k <= K ? binom_small(n, k) : 0);
  }
  for (int k = 2; k <= K; k++) ncand_all += cand[k][nc];
  PH_REQUIRE(n_points + ncand_all < INT32_MAX, PH_ERR_CAPACITY,
             "more than 2^31 - 1 candidate simplices");
  ctx->n_clouds = nc;
  ctx->max_dim = max_dim;
  ctx->vbits = vbits;
  ctx->pt_off = off;
  ctx->D = D;
  ctx->n_points = n_points;

  // device copies of the small tables: off, mo, cand[2..kVrSlots]
  const int ntab = 2 + (kVrSlots - 1);
  int64_t* d_tabs = alloc_n<int64_t>(ctx, ntab * (nc + 1));
  std::vector<int64_t> h_tabs;
  h_tabs.insert(h_tabs.end(), off.begin(), off.end());
  h_tabs.insert(h_tabs.end(), mo.begin(), mo.end());
  for (int k = 2; k <= kVrSlots; k++) h_tabs.insert(h_tabs.end(), cand[k].begin(), cand[k].end());
  PH_CUDA(cudaMemcpyAsync(d_tabs, h_tabs.data(), h_tabs.size() * sizeof(int64_t),
                          cudaMemcpyHostToDevice, st));
  CloudTabs ct{d_tabs, d_tabs + (nc + 1), nc, vbits};
  ctx->d_pt_off = d_tabs;
  auto d_cand = [&](int k) -> const int64_t* { return d_tabs + (int64_t)k * (nc + 1); };

  // scratch: status words [0] bad coords, [1] max d2, then per-cloud counts of every dimension
  int64_t* d_misc = alloc_n<int64_t>(ctx, 2 + (int64_t)kMaxVrDim * nc);
  PH_CUDA(cudaMemsetAsync(d_misc, 0, (2 + (int64_t)kMaxVrDim * nc) * sizeof(int64_t), st));
  auto cnt_dim = [&](int d) { return d_misc + 2 + (int64_t)(d - 1) * nc; };  // d >= 1

  int64_t nn = mo[nc];
  int64_t* d2 = alloc_n<int64_t>(ctx, nn);
  int32_t* eid = alloc_n<int32_t>(ctx, nn);
  int32_t* erank = alloc_n<int32_t>(ctx, nn);
  PH_CUDA(cudaMemsetAsync(eid, 0xff, nn * sizeof(int32_t), st));
  PH_CUDA(cudaMemsetAsync(erank, 0xff, nn * sizeof(int32_t), st));
  int64_t nmax = 0;
  for (int c = 0; c < nc; c++) nmax = std::max(nmax, off[c + 1] - off[c]);
  {
    dim3 g((unsigned)std::max<int64_t>(1, std::min<int64_t>((nmax * nmax + 255) / 256, 4096)),
           (unsigned)nc);
    k_pairwise<<<g, kThreads, 0, st>>>(coords, D, ct, d2, (unsigned long long*)(d_misc + 1),
                                     (int32_t*)d_misc);
    PH_CHECK_LAUNCH();
  }
  // page-locked scratch: status words and per-cloud counts come back through it
  int64_t* h_misc = static_cast<int64_t*>(ctx->pinned(
      (3 + kMaxVrDim * ((int64_t)nc + 1)) * sizeof(int64_t)));
  static const char* const kBadCoords = "coordinates must lie in [-2^24, 2^24] grid units";
  // Every cloud's edges are sorted by one block, if they fit (truncated ones of several clouds have
  // to come after all clouds' edges). That sort finds the largest squared distance by itself;
  // otherwise the host needs it, to choose the digits or to put it on the grid of scales
  int64_t longest = 0;
  for (int c = 0; c < nc; c++) longest = std::max(longest, cand[2][c + 1] - cand[2][c]);
  const bool tiles = longest <= kSortTile && (nc == 1 || (max_diam2 < 0 && scale_step == 0));
  const unsigned long long* largest = nullptr;
  int d2bits = 0;
  if (tiles && scale_step == 0) {
    largest = (const unsigned long long*)(d_misc + 1);
  } else {
    PH_CUDA(cudaMemcpyAsync(h_misc, d_misc, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    PH_CUDA(cudaStreamSynchronize(st));
    PH_REQUIRE(h_misc[0] == 0, PH_ERR_INVALID, kBadCoords);
    int64_t maxkey = h_misc[1];
    if (scale_step > 0) {  // filtration values on the grid of scales: d2 -> scale index
      PH_REQUIRE(n_scales >= 1 && scale_step <= (int64_t)1 << 26, PH_ERR_INVALID,
                 "the scale grid needs n_scales >= 1 and a step of at most 2^26 grid units");
      k_scale_index<<<grid_for(ctx, nn, kThreads), kThreads, 0, st>>>(d2, nn, scale_step);
      PH_CHECK_LAUNCH();
      maxkey = scale_index_of(h_misc[1], scale_step);
      max_diam2 = n_scales;  // simplices above the largest scale are left out
    }
    d2bits = bitlen((uint64_t)maxkey) + 1;  // one extra bit for the sentinel
  }

  // ---------------- edges ----------------
  const int64_t ncand2 = cand[2][nc];
  uint64_t* kbuf = alloc_n<uint64_t>(ctx, ncand2);
  uint64_t* vbuf = alloc_n<uint64_t>(ctx, ncand2);
  uint64_t* ktmp = alloc_n<uint64_t>(ctx, ncand2);
  uint64_t* vtmp = alloc_n<uint64_t>(ctx, ncand2);
  int32_t* d_fault = reinterpret_cast<int32_t*>(d_misc) + 1;  // beside the bad-coordinate word
  const uint64_t sent_e = (1ull << d2bits) - 1ull;
  std::vector<int64_t> cnts(K, 0);  // simplices per dimension
  cnts[0] = n_points;
  std::vector<int64_t> h_cnt((int64_t)kMaxVrDim * nc, 0);  // per (dimension >= 1, cloud)
  if (cand[2][nc] > 0) {
    k_edge_cand<<<grid_for(ctx, cand[2][nc], kThreads), kThreads, 0, st>>>(
        ct, d_cand(2), cand[2][nc], d2, max_diam2, sent_e, largest, kbuf, vbuf, cnt_dim(1));
    PH_CHECK_LAUNCH();
    if (tiles)
      radix_sort_tiles(ctx, kbuf, vbuf, d_cand(2), nc, longest, 0, d2bits, largest);
    else
      radix_sort_u64(ctx, kbuf, vbuf, cand[2][nc], 0, d2bits, ktmp, vtmp, d_fault);
    if (nc > 1 && !tiles) {
      k_rekey_cloud<<<grid_for(ctx, cand[2][nc], kThreads), kThreads, 0, st>>>(
          vbuf, kbuf, cand[2][nc], sent_e, (uint64_t)nc);
      PH_CHECK_LAUNCH();
      radix_sort_u64(ctx, kbuf, vbuf, cand[2][nc], 0, bitlen((uint64_t)nc), ktmp, vtmp, d_fault);
    }
  }

  // edges per cloud: all candidates, unless some were truncated
  if (max_diam2 >= 0) {
    PH_CUDA(cudaMemcpyAsync(h_misc, cnt_dim(1), nc * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    PH_CUDA(cudaStreamSynchronize(st));
  }
  for (int c = 0; c < nc; c++)
    cnts[1] += h_cnt[c] = max_diam2 >= 0 ? h_misc[c] : cand[2][c + 1] - cand[2][c];
  const int64_t E = cnts[1];

  // ids and initial storage of dims 0 and 1 now, higher dims after their candidate counts are
  // known. Provisional allocation uses candidate counts as bounds.
  const int64_t N = n_points;
  int64_t m_bound = N + E, nnz_bound = 2 * E;
  for (int k = 3; k <= K; k++) {
    m_bound += cand[k][nc];
    nnz_bound += (int64_t)k * cand[k][nc];
  }
  ctx->seg = alloc_n<int32_t>(ctx, m_bound);
  ctx->key = alloc_n<int32_t>(ctx, m_bound);
  ctx->low = alloc_n<int32_t>(ctx, m_bound);
  ctx->verts = alloc_n<uint64_t>(ctx, m_bound);
  ctx->rows0 = alloc_n<int32_t>(ctx, nnz_bound + kColSlack);
  IdOut o{ctx->seg, ctx->key, ctx->low, ctx->verts, ctx->rows0};

  k_vertex_init<<<grid_for(ctx, N, kThreads), kThreads, 0, st>>>(ct, N, o);
  PH_CHECK_LAUNCH();

  ctx->d2tab = alloc_n<int64_t>(ctx, std::max<int64_t>(E, 1));
  int64_t n_d2 = 0;
  if (E == 0 && largest) {
    PH_CUDA(cudaMemcpyAsync(h_misc, d_misc, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    PH_CUDA(cudaStreamSynchronize(st));
    PH_REQUIRE(*(int32_t*)h_misc == 0, PH_ERR_INVALID, kBadCoords);
  }
  if (E > 0) {
    int32_t* flag = alloc_n<int32_t>(ctx, E);
    int64_t* excl = alloc_n<int64_t>(ctx, E + 1);
    int64_t* ed2 = alloc_n<int64_t>(ctx, E);
    k_edge_newflag<<<grid_for(ctx, E, kThreads), kThreads, 0, st>>>(vbuf, E, ct, d2, flag, ed2,
                                                                  d_fault);
    PH_CHECK_LAUNCH();
    scan_counts(ctx, flag, nullptr, E, excl, nullptr, d_fault);
    k_edge_finish<<<grid_for(ctx, E, kThreads), kThreads, 0, st>>>(
        vbuf, E, ct, flag, excl, ed2, N, eid, erank, ctx->d2tab, o, 0, d_misc, h_misc);
    PH_CHECK_LAUNCH();
    PH_CUDA(cudaStreamSynchronize(st));
    PH_REQUIRE(*(int32_t*)h_misc == 0, PH_ERR_INVALID, kBadCoords);
    PH_REQUIRE(h_misc[0] == 0, PH_ERR_CUDA, kSortFault);
    n_d2 = h_misc[1];
    ctx->dfree(flag);
    ctx->dfree(excl);
    ctx->dfree(ed2);
  }
  ctx->n_d2 = n_d2;
  const int rbits = bitlen((uint64_t)n_d2);  // keys 0..n_d2-1, sentinel n_d2

  // ---------------- dimensions 2..max_dim ----------------
  // id of each simplex by the lexicographic rank of its vertex set, for the next dimension's
  // faces (edges use the n x n table eid instead)
  std::vector<int32_t*> lex_tab(kVrSlots + 1, nullptr);
  // no two edges of a cloud of one length: triangles and tetrahedra need no sort
  const bool direct = (max_dim == 2 || (max_dim == 3 && nmax <= kDirectPoints)) && E > 0 && n_d2 == E;
  if (direct) {
    build_direct(ctx, ct, Direct{vbuf, E, N, eid}, o, h_cnt, cnts, (int)((nmax + 31) / 32),
                 h_misc, d_fault);
  } else if (max_dim >= 2) {  // buffers for the largest dimension's candidates
    int64_t most = 0;
    for (int k = 3; k <= K; k++) most = std::max(most, cand[k][nc]);
    for (uint64_t** b : {&kbuf, &vbuf, &ktmp, &vtmp}) {
      ctx->dfree(*b);
      *b = nullptr;
      *b = alloc_n<uint64_t>(ctx, most);
    }
  }
  if (!direct && max_dim >= 2) {
    // every dimension is sorted and written before the host reads a count
    DimPlace* place = alloc_n<DimPlace>(ctx, K);  // per dimension
    DimPlace* h_place = reinterpret_cast<DimPlace*>(h_misc);
    *h_place = DimPlace{E, N, 0};
    PH_CUDA(cudaMemcpyAsync(place + 1, h_place, sizeof(DimPlace), cudaMemcpyHostToDevice, st));
    for (int k = 3; k <= K; k++) {
      const int d = k - 1;
      const int64_t n_cand = cand[k][nc];
      if (k < K) {  // the next dimension looks its faces up here
        lex_tab[k] = alloc_n<int32_t>(ctx, std::max<int64_t>(n_cand, 1));
        PH_CUDA(cudaMemsetAsync(lex_tab[k], 0xff, std::max<int64_t>(n_cand, 1) * sizeof(int32_t), st));
      }
      if (n_cand > 0) {
        k_simplex_cand<<<grid_for(ctx, n_cand, kThreads), kThreads, 0, st>>>(
            ct, d_cand(k), n_cand, k, erank, (uint64_t)n_d2, kbuf, vbuf, cnt_dim(d));
        PH_CHECK_LAUNCH();
        radix_sort_u64(ctx, kbuf, vbuf, n_cand, 0, rbits, ktmp, vtmp, d_fault);
      }
      k_dim_place<<<1, kThreads, 0, st>>>(cnt_dim(d), nc, k, place + d, d_fault);
      PH_CHECK_LAUNCH();
      if (n_cand > 0) {
        const unsigned grid = grid_for(ctx, n_cand, kThreads);
        if (k == 3)
          k_tri_finish<<<grid, kThreads, 0, st>>>(kbuf, vbuf, place + d, ct, eid, o, lex_tab[3],
                                                  d_cand(3));
        else
          k_high_finish<<<grid, kThreads, 0, st>>>(kbuf, vbuf, place + d, k, ct, lex_tab[k - 1],
                                                   d_cand(k - 1), lex_tab[k], d_cand(k), o);
        PH_CHECK_LAUNCH();
      }
    }
    PH_CUDA(cudaMemcpyAsync(h_misc, d_misc, (2 + (int64_t)max_dim * nc) * sizeof(int64_t),
                            cudaMemcpyDeviceToHost, st));
    PH_CUDA(cudaStreamSynchronize(st));
    PH_REQUIRE(h_misc[0] == 0, PH_ERR_CUDA, kSortFault);
    for (int d = 2; d <= max_dim; d++)
      for (int c = 0; c < nc; c++)
        cnts[d] += h_cnt[(int64_t)(d - 1) * nc + c] = h_misc[2 + (int64_t)(d - 1) * nc + c];
    ctx->dfree(place);
  }

  // ---------------- layout ----------------
  ctx->m = 0;
  ctx->nnz = 0;
  for (int d = 0; d <= max_dim; d++) {
    ctx->m += cnts[d];
    if (d > 0) ctx->nnz += (int64_t)(d + 1) * cnts[d];
  }
  ctx->dimoff[0] = 0;
  for (int d = 0; d <= max_dim; d++) ctx->dimoff[d + 1] = ctx->dimoff[d] + cnts[d];
  ctx->seg_start.assign((max_dim + 1) * nc + 1, 0);
  int64_t pos = 0;
  for (int d = 0; d <= max_dim; d++)
    for (int c = 0; c < nc; c++) {
      ctx->seg_start[d * nc + c] = pos;
      pos += d == 0 ? off[c + 1] - off[c] : h_cnt[(int64_t)(d - 1) * nc + c];
    }
  ctx->seg_start[(max_dim + 1) * nc] = pos;
  finish_layout(ctx);

  if (!direct) {
    compute_beta(ctx);
    ctx->gidx = alloc_n<int64_t>(ctx, ctx->m);
    k_gidx<<<grid_for(ctx, ctx->m, kThreads), kThreads, 0, st>>>(
        ctx->m, nc, max_dim, ctx->seg, ctx->key, ctx->d_seg_start, d_tabs, ctx->gidx);
    PH_CHECK_LAUNCH();
  }
  PH_CUDA(cudaStreamSynchronize(st));

  ctx->dfree(kbuf);
  ctx->dfree(vbuf);
  ctx->dfree(ktmp);
  ctx->dfree(vtmp);
  ctx->dfree(d2);
  ctx->dfree(eid);
  ctx->dfree(erank);
  for (int32_t* t : lex_tab)
    if (t) ctx->dfree(t);
  ctx->dfree(d_misc);
  // (d_tabs stays: the diagram losses read pt_off)
}

}  // namespace ph
