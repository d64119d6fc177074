// Parallel multi-scale reduction (Algorithm 2, Sec. 3.1) on the device.
//
// One pass = one cycle of the outer loop of Algorithm 2. Every decision of a pass is taken from
// the state at its start, so the result of a pass does not depend on thread scheduling:
//   (table)      tab[low(j)] = min j over the active columns and the pivots: the left-most
//                column with each low, which defines the neighbour sets N(j) (Eq. neighbours).
//                One 64-bit word per row whose high half falls from pass to pass, so the entries
//                of a pass beat those of earlier ones in an atomicMin and nothing is reset (a
//                proven pivot's entry has high half 0 and stays); the survivors of a pass enter
//                the next one's as their new lows appear, so no kernel gathers the lows
//                again; k_first fills the first pass's at set-up. With it, the first row of each
//                (cloud, dim) that is not known to be paired (for Corollary 10).
//   k_phase1     Phase I (Algorithm 5) as a segmented exclusive prefix-max over the active
//                columns of each (cloud, dim), P_j = largest low of an earlier colliding column,
//                in one pass over tiles with a decoupled look-back; then the marks: j is proven
//                if it is left-most for its low and low(j) = beta_j (Thm 5) or low(j) > P_j
//                (Thms 6-7); empty columns become final; the zero case of Corollary 10 zeroes a
//                column whose candidate rows are all paired; each new pivot clears column
//                low(j) (Lemma 1); each active slot's source candidate is stored for Phase II.
//                Also upper bounds of the space Phase II can need: the grid's last block stops
//                the pass after its marks if they exceed what the host provided (the host grows
//                it and continues the pass at Phase II).
//   k_add        Phase II: every colliding column l gets column tab[low(l)] added (XOR of two
//                sorted row lists, or of bitmaps once a column fills in). Sources are
//                left-most, hence never targets, so additions are independent. Survivors take
//                their place in the next active list by a decoupled look-back and their slot in
//                the other arena by one atomic per chunk; new pivots move to the pivot store
//                (their columns never change again). Blocks of 128 threads take 128-slot chunks
//                from a device work queue (64 and 64 once the lanes share merge pieces), or
//                each warp 32 slots once the list is short and its jobs long, and 8 slots in
//                the last, short passes. While jobs are short
//                each lane merges its own job; later the lanes share every job's merge-path
//                pieces. Ten specialisations (row lists / bitmaps x block / 32-slot warp
//                chunks x lane / piece merges, and 8-slot warp chunks with pieces); the loop
//                switches between them at most four times per reduction.
//   k_visit,     Phase II for long lists of triangles (look-ahead): nineteen of twenty additions
//   k_merge      have a proven pivot as their source, which will not change any more, so a visit
//                runs up to eight passes of a column at once as long as its low meets proven
//                pivots of few rows; the lows on the way are stored for the passes they belong
//                to. What was added is kept beside the column's list (its delta) and merged into
//                it every eighth pass. Lows, marks, pass counts and the reduced matrix are those
//                of the pass-by-pass run.
//   (p sets)     With Phase II limited to p neighbour sets (Sec. 3.4), k_set_* rank the sets
//                between k_phase1 and k_add and hold back the other targets.
//   k_commit     publishes the new locations of the columns other jobs may have been reading
//                and moves on the first unpaired row of the segments where it was paired; its last
//                block ends the pass: the next active list, convergence (no collision left,
//                Thm 8), the pass cap and time bound, and inside a CUDA graph the conditional
//                that repeats the pass.
// All per-pass state lives in device memory (DevState), so the same kernel sequence runs either
// from a host loop or as the body of a graph's conditional while node. Each kernel may start
// while its predecessor drains (programmatic dependent launch) and waits for it first. Short lists of
// short columns run in k_loop, one cooperative kernel for all their passes.
#include <algorithm>
#include <cstring>
#include <utility>

#include "ph_internal.cuh"

namespace ph {


enum : int32_t { ST_RUN = 0, ST_DONE = 1, ST_CAPPED = 2, ST_HOST = 3, ST_FAULT = 4,
                 ST_TIMEOUT = 5, ST_SWITCH = 6 };
constexpr int kSpinLimit = 1 << 22;  // iterations of a look-back wait before it gives up
constexpr int kBarrierLimit = 1 << 24;  // ... of a grid barrier's (some seconds)

struct DevState {
  int32_t* act;   // active ids, ascending
  int32_t* act2;  // next active list
  int32_t* alen;   // per slot of act: its column's stored length (ColMeta::len)
  int32_t* alen2;  // the same for act2
  int64_t n_act;
  int32_t* arena[2];  // survivors are written into arena[arena_cur]
  int64_t arena_cap[2];
  int32_t* piv_base;  // current chunk of the pivot store
  int64_t piv_cap;
  // counters that many blocks update by atomics each sit on their own 128-byte line, so that
  // different L2 slices serve them
  alignas(128) unsigned long long piv_used;
  int64_t* stats;  // [stats_rows][PH_PS_N] or nullptr
  int32_t stats_rows;
  int32_t pass;
  int32_t max_passes;
  int32_t status;
  int32_t passes;
  int32_t host_reason;  // 1 arena, 2 pivot store, 4 counter rows
  unsigned int blocks_done;       // blocks of the current grid that have finished (last-block)
  unsigned long long t_start;     // global timer (ns) when this ph_reduce's loop began
  unsigned long long t_limit;     // ns the loop may run before it stops with ST_TIMEOUT
  alignas(128) unsigned long long targets;  // of the current pass
  unsigned long long bound_words, bound_piv;
  alignas(128) unsigned long long arena_used;  // words taken in the arena of the current pass
  alignas(128) unsigned int queue;             // next chunk for k_add
  alignas(128) unsigned int tile_queue;        // next tile for k_phase1
  alignas(128) int32_t n_deferred;             // entries of dlist
  alignas(128) unsigned int n_work;            // entries of work
  alignas(128) unsigned int n_dirty;           // entries of dirty
  // between horizons: the due columns of the top dimension (listed in newpos), those that will be due
  // in the next pass (in act2), and the slots that the visits have to look through themselves
  alignas(128) unsigned int n_due;
  alignas(128) unsigned int n_enter;
  alignas(128) unsigned int scan_end;
  alignas(128) unsigned int bar_count;         // grid barriers of k_loop: blocks arrived, and
  alignas(128) unsigned int bar_gen;           // barriers done
  alignas(128) int32_t fault;                  // a bounded wait ran out
  int32_t debug_fault;  // the first failed bounds check of the debug build (PH_DCHECK), 0 if none
  // bit-packed columns: the passes after the first one that saw a target that may reach its
  // threshold run the additions kernel that handles them (and converts columns); the pass loop
  // stops once there (ST_SWITCH) so that the host continues it with that kernel
  int32_t dense_on;
  int32_t dense_want;
  // Phase II work shape: 128-slot chunks per block while the active list is long or its jobs
  // short, 32-slot chunks per warp (no block barriers, more queue atomics) once it holds fewer
  // than warp_below columns whose survivors reserve warp_words or more arena words on
  // average; this switches once per reduction (ST_SWITCH)
  int32_t warp_on;
  int64_t warp_below;
  int64_t warp_words;  // the mean arena words per survivor the switch needs
  // Phase II merges each job in its own lane while jobs are short (lane_on), and merge pieces
  // spread over the lanes once the mean arena words per survivor reach lane_words; this
  // switches once per reduction (ST_SWITCH)
  int32_t lane_on;
  int64_t lane_words;
  unsigned int loop_blocks;  // blocks of the loop kernel still at work
  int64_t loop_below;  // the loop kernel takes over from the graph at this many columns (-1: never)
  // ... and once merge pieces are on and fewer than narrow_below columns are active, rounds of
  // 8 columns per warp, so that the short late passes spread over more warps (ST_SWITCH, once)
  int32_t narrow_on;
  int64_t narrow_below;
  int32_t chunk_slots;  // slots per chunk of this pass's k_add (8, 32, 64 or 128)
  // Look-ahead (see look_ahead): a column visited by the additions of pass p may run up to
  // `ahead` passes at once, but never past the pass `horizon`, where every column is up to date
  // again, the active list is compacted and the columns move to the other arena
  int32_t ahead;       // 1: every pass's additions are k_add's, all columns, as in Algorithm 2
  int64_t ahead_above; // ... from the first horizon with fewer columns than this
  int32_t horizon;
  int32_t compact;    // this pass compacts the active list (its columns are all up to date)
  int32_t arena_cur;  // the arena this pass writes into
  int32_t drain;      // past the time bound: no more look-ahead, stop after the horizon's pass
  int32_t leave;      // the last pass of look-ahead
  // (at the end: among the words that every pass's last block reads it cost the passes 0.7 %)
  int64_t pass_words;  // arena words of the last pass before a switch
};

struct RArgs {
  DevState* ds;
  int32_t* low;
  const int32_t* beta;
  ColMeta* meta;      // per id: the column's rows, length, flags and clearing mark
  int32_t** nxt_ptr;
  int32_t* nxt_len;
  int32_t* owner;
  unsigned long long* tab;  // per row: the left-most column with that low (tab_key_of)
  int32_t* first_unp;       // per segment: its first row not known to be paired
  int32_t* next_unp;        // ... while it is searched for (INT32_MAX otherwise)
  int32_t* dirty;           // segments whose first_unp became paired in this pass,
  int32_t* dirty_on;        // and per segment whether it is among them
  const int32_t* seg;
  int64_t rows_end;
  int nseg;           // (cloud, dim) segments
  int nc;
  int strict;
  int cor10;
  unsigned long long* tile_st;  // per Phase I tile: look-back state of its aggregate / prefix
  unsigned long long* loop_tile_st;  // the same for the loop kernel's tiles
  unsigned long long* look;  // per Phase II chunk: look-back state of the survivor count
  int32_t* dlist;     // columns whose update (nxt_ptr, nxt_len) waits for k_commit
  int32_t* newpos;    // per active slot, in a pass that compacts: its place in the next list, -1
  int32_t* src_e;     // per active slot: the colliding column's left-most column, -1 if none
  // look-ahead: lows[(q & ring) * m + e] is the low of slot e's column at the start of pass q,
  // for the passes up to due[e], the pass whose additions visit the column next
  int32_t* lows;
  int32_t* due;
  int64_t lows_stride;
  int32_t ring;       // rows of `lows` less one (a power of two less one)
  int4* prec;         // per row: its proven pivot's other rows (rec_of)
  int32_t* delta;     // per id: rows added to the column that are not in its list yet
  uint8_t* kind;      // per slot, and
  int32_t* work;      // the slots, of the columns that k_visit leaves to k_merge
  // bit-packed columns: a job's result is a bitmap over its row segment when the sum of the two
  // row counts exceeds the threshold, max(the stored bitmap's words, t0) with t0 = dense_mode
  // when > 0, else 32 (dense_mode < 0: never), or when either column is already a bitmap
  int dense_mode;
  int32_t dense_floor;             // no addition of at most this many rows goes bit-packed
  int32_t dense_min[kMaxDim + 1];  // per column dimension: smallest threshold of its segments
  int32_t dim_start[kMaxDim + 1];  // first column id of each dimension (m above the top one)
  const int64_t* seg_start;        // device copy of the segment table
  int predict;        // 1: Corollary 10 non-zero case (pair predictions)
  uint32_t* unp_bits; // per row, bit: not known to be paired at the start of the pass
  int32_t* unp_words; // [nwords + 1] exclusive prefix of unpaired rows per 32-row word
  int32_t* pred;      // per id: predicted lowstar (Corollary 10), -1
  int staged_max;     // merges of more rows than this run from global memory
  int force_km;       // > 0: merge-path positions per lane for every warp
  // Phase II limited to p neighbour sets per pass (Sec. 3.4): per row of the boundary
  int32_t* set_n;     // eligible targets of the row's set
  int32_t* set_neg;   // those known to be negative
  uint8_t* set_on;    // the set is acted on this pass
};

// per-pass values, read once at kernel start (no kernel changes them while others read them)
struct PV {
  int32_t* act;
  int32_t* act2;
  int32_t* alen;
  int32_t* alen2;
  int64_t n_act;
  int do_adds;
  int64_t* stats;
  int32_t* arena_next;
  int32_t* piv_base;
  int dense_on;
  int64_t arena_next_cap;  // words of arena_next and of the pivot store's chunk (bounds checks)
  int64_t piv_cap;
  unsigned long long tab_key;  // tab_key_of the next pass, whose table is built during this one
  int32_t compact;
  int32_t limit;      // the last pass a column visited now may run ahead to
  int32_t ahead;      // passes a visit may run ahead; 1: every pass visits every column
  int32_t whole;      // ... and the lists must be whole there (the pass cap, or the time bound)
};

// The left-most-column table holds, per row, a column below the pass it was entered for, counted
// down: an atomicMin lets later passes' entries replace earlier ones, and the left-most
// column win within a pass, so the table is never reset. A proven pivot is the left-most column of
// its low for good: its entry has no pass and wins for ever.
__device__ __forceinline__ unsigned long long tab_key_of(int32_t pass) {
  return (unsigned long long)(0x7fffffff - pass) << 32;
}

__device__ __forceinline__ PV pass_view(const DevState* ds) {
  PV v;
  v.act = ds->act;
  v.act2 = ds->act2;
  v.alen = ds->alen;
  v.alen2 = ds->alen2;
  v.n_act = ds->n_act;
  v.do_adds = ds->pass < ds->max_passes;
  v.stats = ds->stats ? ds->stats + (int64_t)ds->pass * PH_PS_N : nullptr;
  v.arena_next = ds->arena[ds->arena_cur];
  v.piv_base = ds->piv_base;
  v.dense_on = ds->dense_on;
  v.arena_next_cap = ds->arena_cap[ds->arena_cur];
  v.piv_cap = ds->piv_cap;
  v.tab_key = tab_key_of(ds->pass + 1);
  v.compact = ds->compact;
  v.ahead = ds->ahead;
  v.limit = ds->drain || ds->leave ? ds->pass + 1
                      : min(min(ds->pass + ds->ahead, ds->horizon), ds->max_passes);
  v.whole = ds->drain || v.limit == ds->max_passes;
  return v;
}

__device__ __forceinline__ void stat_add(int64_t* stats, int k, int64_t v) {
  // warp-aggregated counter update
  int64_t s = v;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane_id() == 0 && s != 0) atomicAdd((unsigned long long*)&stats[k], (unsigned long long)s);
}


__device__ __forceinline__ int64_t warp_sum64(int64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Programmatic dependent launch. The kernels of a pass are launched so that each may start
// while the one before it in the stream drains (its blocks fill the SMs that kernel frees): every
// pass kernel first waits here until the previous kernel has completed and its writes are
// visible, before it reads or writes anything. Without such a predecessor the wait returns at
// once. The trigger, given once a kernel's blocks run, lets the next kernel's launch begin.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// True in the one block that finishes the grid last; it then sees every other block's writes.
// Only the first `participants` blocks of the grid may call it (the others have no work and
// may leave at once).
__device__ __forceinline__ bool last_block(unsigned int* done, unsigned int participants) {
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == participants - 1;
  __syncthreads();
  return s_last;
}

// ------------------------------------------------------------------------------------------
// The row state of the next pass, from the pivots, flags and beta as they stand: at set-up the
// first row of each (cloud, dim) segment that is not known to be paired (Corollary 10; later
// passes move it on in next_unpaired), and for every pass the unpaired bitmap (pair predictions).
// Every block of the grid takes part; the last block then finishes it with rows_of_pass_last.
__device__ __forceinline__ bool is_unpaired(const RArgs& a, int64_t x) {
  const uint8_t flags = a.meta[x].flags;  // (all three loads at once)
  const int32_t beta = a.beta[x], owner = a.owner[x];
  return !(flags & F_PROVEN) && beta < 0 && owner < 0;
}
template <bool kFirst>
__device__ void rows_of_pass(const RArgs& a, unsigned blocks) {
  // warp-uniform loop: each iteration a warp covers 32 consecutive rows, one bitmap word
  const int64_t stride = (int64_t)blocks * blockDim.x;
  for (int64_t x0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); x0 < a.rows_end;
       x0 += stride) {
    const int64_t x = x0 + (threadIdx.x & 31);
    const bool unpaired = x < a.rows_end && is_unpaired(a, x);
    const unsigned w = __ballot_sync(0xffffffffu, unpaired);
    if (kFirst && unpaired) {  // one atomic per segment among the warp's unpaired rows: its first
      const int32_t sg = a.seg[x];
      const unsigned same = __match_any_sync(w, sg);
      if ((threadIdx.x & 31) == __ffs(same) - 1) atomicMin(&a.first_unp[sg], (int32_t)x);
    }
    if (a.predict && (threadIdx.x & 31) == 0) a.unp_bits[x0 >> 5] = w;
  }
}

// by the last block: the bitmap's prefix counts per word
__device__ void rows_of_pass_last(const RArgs& a) {
  if (!a.predict) return;
  __shared__ int64_t sh[kWarps + 1];
  const int64_t nwords = (a.rows_end + 31) / 32;
  int64_t carry = 0;
  for (int64_t base = 0; base < nwords; base += kThreads) {
    const int64_t w = base + threadIdx.x;
    const int64_t c = w < nwords ? __popc(__ldcg(a.unp_bits + w)) : 0;
    int64_t tot;
    const int64_t ex = block_excl_sum<int64_t>(c, sh, tot);
    if (w < nwords) a.unp_words[w] = (int32_t)(carry + ex);
    carry += tot;
  }
  if (threadIdx.x == 0) a.unp_words[nwords] = (int32_t)carry;
}

// The segments whose first unpaired row became paired in this pass get their next one. Rows stay
// paired, so the search starts at the old one; it ends some rows on as a rule, but far away after
// the first pass, or when the row that held up a long run of paired ones is paired at last.
// A few segments are searched by all blocks together, in strides that end once a lower row is
// found, and next_unpaired_last, by the last block, takes over the result; many (of a batch, or
// by a single block) by one block each. (One block alone took 455 us over all passes of 120 points in
// 8-d, whose next row is far.)
constexpr unsigned kSearchTogether = 4;
__device__ __forceinline__ void next_unpaired(const RArgs& a, unsigned blocks) {
  const unsigned nd = a.ds->n_dirty;
  if (nd == 0) return;
  if (nd <= kSearchTogether && blocks > 1) {
    for (unsigned i = 0; i < nd; i++) {
      const int32_t s = a.dirty[i];
      const int64_t end = a.seg_start[s + 1];
      int64_t x0 = (int64_t)a.first_unp[s] + blockIdx.x * blockDim.x + (threadIdx.x & ~31);
      for (; x0 < end && x0 < *(volatile int32_t*)&a.next_unp[s];
           x0 += (int64_t)blocks * blockDim.x) {  // by whole warps
        const int64_t x = x0 + (threadIdx.x & 31);
        const unsigned w = __ballot_sync(0xffffffffu, x < end && is_unpaired(a, x));
        if (w) {
          if ((threadIdx.x & 31) == __ffs(w) - 1) atomicMin(&a.next_unp[s], (int32_t)x);
          break;
        }
      }
    }
    return;
  }
  if (nd > blocks) {  // more segments than blocks: a warp each
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    for (unsigned i = blockIdx.x * warps + (threadIdx.x >> 5); i < nd; i += blocks * warps) {
      const int32_t s = a.dirty[i];
      const int64_t end = a.seg_start[s + 1];
      int32_t first = INT32_MAX;
      for (int64_t x0 = a.first_unp[s]; x0 < end && first == INT32_MAX; x0 += 128) {
        bool u[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int64_t x = x0 + 32 * q + lane;
          u[q] = x < end && is_unpaired(a, x);
        }
#pragma unroll
        for (int q = 3; q >= 0; q--) {
          const unsigned w = __ballot_sync(0xffffffffu, u[q]);
          if (w) first = (int32_t)(x0 + 32 * q + __ffs(w) - 1);
        }
      }
      if (lane == 0) {
        a.first_unp[s] = first;
        a.dirty_on[s] = 0;
      }
    }
    return;
  }
  __shared__ int32_t s_first;
  for (unsigned i = blockIdx.x; i < nd; i += blocks) {
    const int32_t s = a.dirty[i];
    const int64_t end = a.seg_start[s + 1];
    int32_t first = INT32_MAX;
    for (int64_t x0 = a.first_unp[s]; x0 < end && first == INT32_MAX; x0 += blockDim.x) {
      if (threadIdx.x == 0) s_first = INT32_MAX;
      __syncthreads();
      const int64_t x = x0 + threadIdx.x;
      const unsigned w = __ballot_sync(0xffffffffu, x < end && is_unpaired(a, x));
      if (w && (threadIdx.x & 31) == __ffs(w) - 1) atomicMin(&s_first, (int32_t)x);
      __syncthreads();
      first = s_first;
      __syncthreads();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      a.first_unp[s] = first;
      a.dirty_on[s] = 0;
    }
  }
}
__device__ __forceinline__ void next_unpaired_last(const RArgs& a, unsigned blocks) {
  const unsigned nd = a.ds->n_dirty;
  if (nd > kSearchTogether || blocks == 1) return;
  for (unsigned i = threadIdx.x; i < nd; i += blockDim.x) {
    const int32_t s = a.dirty[i];
    a.first_unp[s] = *(volatile int32_t*)&a.next_unp[s];
    a.next_unp[s] = INT32_MAX;
    a.dirty_on[s] = 0;
  }
}

__device__ __forceinline__ void first_tab(const RArgs& a);

// set-up: the first pass's table and row state (independent of each other)
__global__ void k_first(RArgs a) {
  first_tab(a);
  rows_of_pass<true>(a, gridDim.x);
  if (last_block(&a.ds->blocks_done, gridDim.x)) {
    rows_of_pass_last(a);
    if (threadIdx.x == 0) a.ds->blocks_done = 0;
  }
}

// rows of the start-of-pass unpaired bitmap before row x
__device__ __forceinline__ int32_t unpaired_before(const RArgs& a, int64_t x) {
  const int64_t w = x >> 5;
  const unsigned low_bits = (x & 31) ? (0xffffffffu >> (32 - (x & 31))) : 0u;
  return a.unp_words[w] + ((x & 31) ? __popc(a.unp_bits[w] & low_bits) : 0);
}

// Corollary 10, non-zero case: beta_j >= 0 makes j negative (Thm 5), so its candidate set L_j
// holds the unpaired rows of K_{d-1} in [beta_j, low(j)] only (rows of one cloud's segment are
// contiguous ids). One candidate is lowstar(j) (Lemma 9). Returns it, -1 if there are several,
// -2 if there is none (impossible; counted as a check).
__device__ __forceinline__ int32_t predicted_low(const RArgs& a, int32_t b, int32_t l) {
  const int32_t c0 = unpaired_before(a, b);
  const int32_t n = unpaired_before(a, (int64_t)l + 1) - c0;
  if (n != 1) return n == 0 ? -2 : -1;
  int64_t lo = b >> 5, hi = l >> 5;  // last word whose prefix is <= c0
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (a.unp_words[mid] <= c0) lo = mid; else hi = mid - 1;
  }
  unsigned bits = a.unp_bits[lo];
  for (int32_t k = c0 - a.unp_words[lo]; k > 0; k--) bits &= bits - 1;  // skip k set bits
  return (int32_t)(lo * 32 + __ffs(bits) - 1);
}

// The first pass's left-most-column table (at set-up; every later pass's table is filled by the
// pass before it): tab[low(j)] = min j over all columns by atomicMin, and every low marked as seen
// for the essential estimate. In a run of columns with one low the first has the least id. Eight
// columns per thread in two 16-byte loads (42.7 M columns: 236 us with the ids read from the active
// list, four at a time).
constexpr int kTabItems = 8;
__device__ __forceinline__ void first_tab(const RArgs& a) {
  const PV v = pass_view(a.ds);
  const unsigned long long tag = tab_key_of(a.ds->pass);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * kTabItems;
  for (int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * kTabItems; i0 < v.n_act;
       i0 += stride) {
    int32_t l[kTabItems];
    if (i0 + kTabItems <= v.n_act) {
      const int4 x = *reinterpret_cast<const int4*>(a.low + i0);
      const int4 y = *reinterpret_cast<const int4*>(a.low + i0 + 4);
      l[0] = x.x, l[1] = x.y, l[2] = x.z, l[3] = x.w;
      l[4] = y.x, l[5] = y.y, l[6] = y.z, l[7] = y.w;
    } else {
#pragma unroll
      for (int k = 0; k < kTabItems; k++) l[k] = i0 + k < v.n_act ? a.low[i0 + k] : -1;
    }
    int32_t before = i0 > 0 ? a.low[i0 - 1] : -1;
#pragma unroll
    for (int k = 0; k < kTabItems; k++) {
      if (l[k] != before && l[k] >= 0 && PH_DCHECK(&a.ds->debug_fault, l[k] < a.rows_end, 1)) {
        const unsigned long long key = tag | (unsigned)(i0 + k);
        if (a.tab[l[k]] > key) atomicMin(&a.tab[l[k]], key);
        if (!a.meta[l[k]].low_seen) a.meta[l[k]].low_seen = 1;
      }
      before = l[k];
    }
  }
}

// ------------------------------------------------------------------------------------------
// bit-packed columns
// ------------------------------------------------------------------------------------------
// the smallest threshold over the segments of column j's dimension (fixed indices only: a
// kernel parameter array indexed at run time would be copied out)
__device__ __forceinline__ int32_t dense_min_of(const RArgs& a, int32_t j) {
  int32_t t = a.dense_min[0];
#pragma unroll
  for (int k = 1; k <= kMaxDim; k++) t = j >= a.dim_start[k] ? a.dense_min[k] : t;
  return t;
}

// the (cloud, dim) segment of column j, seg[j] = dim * clouds + cloud: with one cloud the
// dimension, found from the dimension starts (no load); else loaded
__device__ __forceinline__ int32_t seg_of(const RArgs& a, int32_t j) {
  if (a.nc != 1) return a.seg[j];
  int32_t d = 0;
#pragma unroll
  for (int k = 1; k <= kMaxDim; k++) d += j >= a.dim_start[k] ? 1 : 0;
  return d;
}

// first column id of column j's dimension
__device__ __forceinline__ int32_t dim_start_of(const RArgs& a, int32_t j) {
  int32_t b = 0;
#pragma unroll
  for (int k = 1; k <= kMaxDim; k++) b = j >= a.dim_start[k] ? a.dim_start[k] : b;
  return b;
}
// the smallest threshold over the dimensions of the columns j0..j1 (none: INT32_MAX)
__device__ __forceinline__ int32_t dense_min_between(const RArgs& a, int32_t j0, int32_t j1) {
  int32_t t = INT32_MAX;
#pragma unroll
  for (int k = 0; k <= kMaxDim; k++) {
    const int32_t end = k < kMaxDim ? a.dim_start[k + 1] : INT32_MAX;
    if (j0 <= j1 && a.dim_start[k] <= j1 && end > j0) t = min(t, a.dense_min[k]);
  }
  return t;
}

// row segment of column j: first row id and bitmap words
__device__ __forceinline__ void row_segment(const RArgs& a, int32_t j, int64_t& base,
                                            int32_t& words) {
  const int rs = a.seg[j] - a.nc;
  base = a.seg_start[rs];
  words = (int32_t)((a.seg_start[rs + 1] - base + 31) / 32);
}

// A bit-packed column is stored as one header word (its row count) followed by the bitmap, bit
// r - base of word (r - base) / 32 for row r of the segment. Its length field holds
// -(stored words) - 1, so a plain length load tells the two forms apart, and the stored words of
// either form are what a move of the column takes: Phase I reserves that much for it.
constexpr int kDenseHead = 1;
__device__ __forceinline__ int32_t stored_words(int32_t len) { return len < 0 ? -len - 1 : len; }
__device__ __forceinline__ int32_t dense_len(int32_t words) { return -words - 1; }

// does an addition of n rows in all (target + source) into column j produce a bitmap? The
// stored bitmap is smaller than n, so it fits the n words Phase I reserved for the result
__device__ __noinline__ bool goes_dense_slow(const RArgs& a, int32_t j, int64_t n) {
  int64_t base;
  int32_t words;
  row_segment(a, j, base, words);
  return n > max(words + kDenseHead, a.dense_mode > 0 ? a.dense_mode : 32);
}
// the cheap part first: no bitmap at or below the floor, nor below every segment of j's dimension
__device__ __forceinline__ bool goes_dense(const RArgs& a, int32_t j, int64_t n) {
  return n > a.dense_floor && n > dense_min_of(a, j) && goes_dense_slow(a, j, n);
}


// ------------------------------------------------------------------------------------------
// look-ahead
// ------------------------------------------------------------------------------------------
// Nearly every addition's source is a proven pivot (95-99 % on Vietoris-Rips complexes), and
// nearly every pivot is an unreduced column of d + 1 rows. A proven pivot is the left-most
// column of its low for good and never changes, so as long as a column's low belongs to one, its
// next additions depend on nothing else: the additions kernel runs them for several passes in
// one visit (look_ahead) and stores the low of each pass. The passes in between read the stored
// lows (k_phase1: Phase I, Corollary 10) and leave the column alone. Only the low of a column is
// ever seen by other columns while it collides with a pivot, so every pass decides as if the
// columns had been added one pass at a time. A column is visited again when its stored lows end
// (due[e]), at the latest at the horizon, where all are up to date: then the active list is
// compacted, its slots fixed until the next horizon (a slot whose column left holds dead_slot).
constexpr int kAheadMax = 8;  // passes per visit (a power of two: rows of stored lows)
// What visits add to a column gathers in a block of its own (its delta) until it is merged into
// the column's list: up to kOld rows are kept from visit to visit, and a visit adds up to R rows
// per pass: R = 2, the rows of a triangle's boundary beside its low. (Look-ahead is for complexes
// whose top columns are triangles' three rows; with R = 3, for tetrahedra, it lost: 8 Gaussian
// dimensions, 120 points, 0.9 M simplices, 1.8 -> 2.8 ms. So it did on the two rows of edges:
// 4.5 M of 3000 points without triangles 3.9 -> 7.5 ms, 8 M of 4000 points 6.4 -> 13.6 ms.)
constexpr int kSourceRows = 2;
constexpr int kOld = 8;
// Look-ahead spends instructions (4,360 warp instructions per round of 32 columns in a pass of 2.2 M, some
// 230 of them per pass that a visit runs ahead; issue active 56 %, DRAM 13 %) where pass-by-pass
// additions are bound by memory traffic: every pass rewrites every column and reads its source.
// Pass by pass -> look-ahead: 10.67 M columns (400 points on a torus) 48.8 -> 36.9 ms, 4.5 M
// on a torus 29.2 -> 22.6 ms, on a sphere 12.8 -> 8.7 ms, 42.7 M in 512 clouds 45.5 -> 41.8 ms; on
// 2.6 M columns 11.9 -> 11.8 ms, on 1.3 M 6.5 -> 6.2 ms, on 0.9 M 4.4 -> 4.3 ms: little to gain
// below kAheadFrom, where a visit's two kernels and the larger tables also cost memory. Lists that
// shrink under kAheadAbove go on pass by pass (10.67 M columns: 34.3 ms with twice as many, 33.7 with
// 100,000; 3.7 M in 48 clouds: 5.85 and 5.95 ms; here 34.1 and 5.85).
constexpr int64_t kAheadFrom = 3000000;   // triangles from which look-ahead pays, and columns
constexpr int64_t kAheadAbove = 250000;   // down to which it goes on
constexpr int kLonger = 12;  // the longest source inside a visit: kRecRows + this many rows
constexpr int kDeltaRows = kOld + kSourceRows * kAheadMax;
// words per row of stored lows, and of due words: threads read eight slots in two 16-byte loads
__host__ __device__ inline int64_t lows_stride_of(int64_t m) { return (m + 7) & ~int64_t(7); }

// The rows of a row's proven pivot, one 16-byte record: x is its length (0: no pivot yet), y, z
// and w its rows below the low, then INT32_MAX (length <= kRecRows), or y and z the address of its
// rows. A bit-packed pivot's record holds kRecLong alone.
constexpr int32_t kRecRows = 4;
constexpr int32_t kRecLong = INT32_MAX;

// The word of a slot that says when its column is visited next: the pass itself, ~pass for a column
// without beta, which Corollary 10 may zero, kDeadDue for a slot whose column left. A pass before the
// horizon needs no more of a column ahead of it than this word and the stored low.
constexpr int32_t kDeadDue = INT32_MAX;
__device__ __forceinline__ int32_t due_pass(int32_t d) { return d < 0 ? ~d : d; }

__device__ __forceinline__ int32_t dead_slot(int32_t j) { return -2 - j; }
__device__ __forceinline__ int32_t slot_id(int32_t a) { return a >= 0 ? a : -2 - a; }

__device__ __forceinline__ int4 rec_of(const int32_t* rows, int32_t len) {
  int4 r = make_int4(len, INT32_MAX, INT32_MAX, INT32_MAX);
  if (len < 0) {
    r.x = kRecLong;
  } else if (len <= kRecRows) {
    if (len > 1) r.y = rows[0];
    if (len > 2) r.z = rows[1];
    if (len > 3) r.w = rows[2];
  } else {
    r.y = (int32_t)(unsigned)((unsigned long long)rows & 0xffffffffu);
    r.z = (int32_t)(unsigned)((unsigned long long)rows >> 32);
  }
  return r;
}
__device__ __forceinline__ const int32_t* rec_rows(const int4& r) {
  return reinterpret_cast<const int32_t*>((unsigned long long)(unsigned)r.y |
                                          ((unsigned long long)(unsigned)r.z << 32));
}

// ------------------------------------------------------------------------------------------
// Phase I scan
// ------------------------------------------------------------------------------------------
// exclusive block scan with carry-in; returns the exclusive prefix, sets the running total
__device__ __forceinline__ SegMax block_scan_segmax(SegMax v, SegMax carry, SegMax* sh,
                                                    SegMax& total) {
  const int lane = lane_id(), w = threadIdx.x >> 5;
  SegMax inc = warp_incl_segmax(v);
  if (lane == 31) sh[w] = inc;
  __syncthreads();
  if (w == 0) {
    SegMax x = lane < kWarps ? sh[lane] : SegMax{INT32_MAX, -1};
    SegMax xi = warp_incl_segmax(x);
    SegMax xe;
    xe.seg = __shfl_up_sync(0xffffffffu, xi.seg, 1);
    xe.val = __shfl_up_sync(0xffffffffu, xi.val, 1);
    xe = lane == 0 ? carry : segmax_combine(carry, xe);
    if (lane < kWarps) sh[lane] = xe;
    if (lane == kWarps - 1) sh[kWarps] = segmax_combine(carry, xi);
  }
  __syncthreads();
  SegMax pre = sh[w];
  SegMax ex;
  ex.seg = __shfl_up_sync(0xffffffffu, inc.seg, 1);
  ex.val = __shfl_up_sync(0xffffffffu, inc.val, 1);
  ex = lane == 0 ? pre : segmax_combine(pre, ex);
  total = sh[kWarps];
  __syncthreads();
  return ex;
}


constexpr unsigned long long kLookAgg = 1ull << 38, kLookIncl = 2ull << 38;
constexpr unsigned long long kLookFlags = 3ull << 38, kLookVal = (1ull << 38) - 1;

// Decoupled look-back over the tiles before `chunk`: the number of places kept by all earlier
// tiles. A tile publishes its own count (an aggregate state), then its inclusive prefix. Each
// state word holds its value, so no fence is needed; states carry the pass number and never
// need resetting within one reduction. Tiles are claimed in order from the work queue, so every
// predecessor belongs to a running or finished block. A wait that runs past its bound records a
// fault (reported as an error) and counts as zero.
__device__ __forceinline__ unsigned long long look_tag(int32_t pass) {
  return (unsigned long long)(pass & 0xffffff) << 40;
}

__device__ __forceinline__ void look_publish(const RArgs& a, int32_t pass, int64_t chunk,
                                             int64_t agg) {
  atomicExch(a.look + chunk,
             look_tag(pass) | (chunk == 0 ? kLookIncl : kLookAgg) | (unsigned long long)agg);
}

// by one full warp; returns the exclusive prefix of `chunk` and publishes its inclusive one
__device__ __forceinline__ int64_t look_back(const RArgs& a, int32_t pass, int64_t chunk,
                                             int64_t agg) {
  if (chunk == 0) return 0;
  const int lane = lane_id();
  const unsigned long long tag = look_tag(pass);
  const unsigned long long* st = a.look;
  int64_t prefix = 0;
  bool fault = false;
  for (int64_t p = chunk - 1;; p -= 32) {
    const int64_t q = p - lane;
    unsigned long long w = tag | kLookIncl;  // before chunk 0: nothing
    if (q >= 0) {
      for (int it = 0;; it++) {
        w = *(const volatile unsigned long long*)(st + q);
        if ((w >> 40) == (tag >> 40) && (w & kLookFlags)) break;
        if (it > kSpinLimit) {
          fault = true;
          w = tag | kLookIncl;
          break;
        }
        __nanosleep(32);
      }
    }
    const bool incl = (w & kLookFlags) == kLookIncl;
    const unsigned im = __ballot_sync(0xffffffffu, incl);
    const int stop = im ? __ffs(im) - 1 : 32;  // nearest inclusive state
    const int64_t val = lane <= stop ? (int64_t)(w & kLookVal) : 0;
    prefix += __shfl_sync(0xffffffffu, warp_incl_sum(val), 31);
    if (im || p < 32) break;
  }
  if (lane == 0) atomicExch(a.look + chunk, tag | kLookIncl | (unsigned long long)(prefix + agg));
  if (__any_sync(0xffffffffu, fault) && lane == 0) a.ds->fault = 1;
  return prefix;
}

// the space this pass's Phase II can need (arena, pivot store) against what the host provided;
// no column has changed yet, and the marks made depend only on the pass's starting state, so a
// pass stopped here continues at Phase II once the host has grown the buffers
struct Space {
  unsigned long long arena_used, arena_cap, piv_used, piv_cap;
};
__device__ __forceinline__ Space space_of(const DevState* ds) {
  return Space{*(const volatile unsigned long long*)&ds->arena_used,
               (unsigned long long)*(const volatile int64_t*)&ds->arena_cap[ds->arena_cur],
               *(const volatile unsigned long long*)&ds->piv_used,
               (unsigned long long)*(const volatile int64_t*)&ds->piv_cap};
}
__device__ __forceinline__ int lacks_space(const DevState* ds, const Space& s) {
  const unsigned long long words = *(const volatile unsigned long long*)&ds->bound_words;
  const unsigned long long piv = *(const volatile unsigned long long*)&ds->bound_piv;
  return (s.arena_used + words > s.arena_cap ? 1 : 0) | (piv + s.piv_used > s.piv_cap ? 2 : 0);
}
__device__ __forceinline__ void stop_for_space(DevState* ds, int reason) {
  ds->host_reason = reason;
  ds->status = ST_HOST;
}
__device__ __forceinline__ void check_capacity(DevState* ds) {
  if (const int reason = lacks_space(ds, space_of(ds))) stop_for_space(ds, reason);
}

// Phase I and the marks in one kernel, a single-pass scan over tiles of kFTile active slots
// (kFItems consecutive slots per thread), claimed in order from a work queue. A tile loads its
// slots' columns, lows, sources and lengths once; takes its Phase I aggregate and each thread's
// prefix within the tile from one block scan; publishes the aggregate and looks back over the
// tiles before it for its prefix (decoupled look-back, as the additions kernel's survivor
// count); then applies the marks. The space bounds of the pass are summed on the way, and the
// grid's last block checks them against what the host provided: a pass that does not fit stops
// after its marks (which depend only on the state at the pass's start) and the host continues it
// at Phase II once the buffers have grown.
constexpr int kFItems = 4;
constexpr int kFTile = kThreads * kFItems;
// tile state word: pass tag (8 bits) | flags (2) | segment (23) | val + 1 (31). Eight bits of
// tag tell this pass from the previous ones: the active list never grows within a reduction, so a
// tile in use in pass p was published in pass p - 1, or, by look-ahead's larger tiles between horizons,
// eight passes before at most. Set-up clears every state, and a pass after k_loop, which has states of
// its own, those that it left alone
constexpr unsigned long long kTAgg = 1ull << 54, kTIncl = 2ull << 54, kTFlags = 3ull << 54;
__device__ __forceinline__ unsigned long long tile_word(unsigned long long tag, unsigned long long flag,
                                                       SegMax x) {
  return tag | flag | ((unsigned long long)(x.seg & 0x7fffff) << 31) |
         (unsigned long long)((uint32_t)(x.val + 1) & 0x7fffffffu);
}
__device__ __forceinline__ SegMax tile_value(unsigned long long w) {
  return SegMax{(int32_t)((w >> 31) & 0x7fffff), (int32_t)(w & 0x7fffffffu) - 1};
}

__device__ __forceinline__ void tile_publish(unsigned long long* st, int32_t pass, int64_t t,
                                             SegMax agg) {
  const unsigned long long tag = (unsigned long long)(pass & 0xff) << 56;
  atomicExch(st + t, tile_word(tag, t == 0 ? kTIncl : kTAgg, agg));
}

// by warp 0: publishes tile t's aggregate, returns the Phase I value of every tile before it
// (SegMax{-1, -1}, a left identity of segmax_combine, for none) and publishes t's inclusive state
__device__ __forceinline__ SegMax tile_look_back(unsigned long long* st, int32_t pass, int64_t t,
                                                 SegMax agg, bool& fault) {
  const int lane = lane_id();
  const unsigned long long tag = (unsigned long long)(pass & 0xff) << 56;
  const SegMax none{-1, -1};
  if (lane == 0) tile_publish(st, pass, t, agg);
  if (t == 0) return none;
  SegMax acc = none;
  bool have = false;
  for (int64_t p = t - 1;; p -= 32) {
    const int64_t q = p - lane;  // lane 0 the nearest tile
    SegMax x = none;
    bool incl = true;  // before tile 0: an inclusive state of nothing
    if (q >= 0) {
      unsigned long long w = 0;
      for (int it = 0;; it++) {
        w = *(const volatile unsigned long long*)(st + q);
        if ((w >> 56) == (tag >> 56) && (w & kTFlags)) break;
        if (it > kSpinLimit) {
          fault = true;
          w = tag | kTIncl;
          break;
        }
        __nanosleep(32);
      }
      x = tile_value(w);
      incl = (w & kTFlags) == kTIncl;
    }
    const unsigned im = __ballot_sync(0xffffffffu, incl);
    const int stop = im ? __ffs(im) - 1 : 32;
    // the window in order, farthest (highest lane) first; lanes past the stop are left identities
    SegMax val = lane <= stop ? x : none;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      SegMax u;
      u.seg = __shfl_down_sync(0xffffffffu, val.seg, o);
      u.val = __shfl_down_sync(0xffffffffu, val.val, o);
      if (lane + o < 32) val = segmax_combine(u, val);
    }
    SegMax win;
    win.seg = __shfl_sync(0xffffffffu, val.seg, 0);
    win.val = __shfl_sync(0xffffffffu, val.val, 0);
    acc = have ? segmax_combine(win, acc) : win;  // this window comes before the later ones
    have = true;
    if (im) break;
  }
  if (lane == 0) atomicExch(st + t, tile_word(tag, kTIncl, segmax_combine(acc, agg)));
  return acc;
}

// A pass that compacts also gives every slot whose column may survive its place in the next active
// list (newpos), by a second look-back over the tiles: a column that left all the same (proven
// by its P_j, or cleared) leaves a dead place there.
//
// kLoop: in the loop kernel (every block resident) tiles of one slot per thread are dealt out in
// order instead, to all `parts` blocks.
template <bool kLookAhead, bool kLoop>
__device__ __forceinline__ void phase1_pass(const RArgs& a, unsigned parts) {
  __shared__ SegMax sh[kWarps + 1];
  __shared__ int64_t shs[kWarps + 1];
  __shared__ int64_t s_tile;
  __shared__ SegMax s_pre;
  __shared__ int s_keep[kWarps + 1];
  __shared__ int64_t s_place;
  constexpr int kFI = kLoop ? 1 : kFItems;
  constexpr int64_t kFTile = kThreads * kFI;
  if (blockIdx.x >= parts) return;
  DevState* ds = a.ds;
  const PV v = pass_view(ds);
  const int32_t pass = ds->pass;
  const int32_t* fu = a.first_unp;
  const int32_t* lows = a.lows + (int64_t)(pass & a.ring) * a.lows_stride;
  constexpr int32_t ahead = kLookAhead ? kAheadMax : 1;
  const int32_t visit_rows = ahead > 1 ? kDeltaRows : 0;  // rows a visit may add to a column
  const int64_t ntiles = (v.n_act + kFTile - 1) / kFTile;
  int64_t bw = 0, bp = 0;
  int64_t n_zero = 0, n_piv = 0, n_c10 = 0, n_pred = 0, n_empty = 0;
  bool want = false;  // a target whose addition may reach its dimension's bit-packing threshold
  bool fault = false;
  for (int64_t t = blockIdx.x;; t += parts) {
    if constexpr (!kLoop) {  // a tile is claimed only when its work begins: later tiles wait for it
      if (threadIdx.x == 0) s_tile = atomicAdd(&ds->tile_queue, 1u);
      __syncthreads();
      t = s_tile;
    }
    if (t >= ntiles) break;
    const int64_t tile0 = t * kFTile;
    // bit-packing thresholds of the tile's columns (ascending ids, so dimensions too): exact in
    // the top dimension (ids from t_b on), the smallest of the others below it
    int32_t t_b = 0, t_hi = INT32_MAX, t_lo = INT32_MAX;
    if (a.dense_floor != INT32_MAX) {
      const int32_t j0 = slot_id(v.act[tile0]);
      const int32_t j1 = slot_id(v.act[min(tile0 + kFTile, v.n_act) - 1]);
      t_b = dim_start_of(a, j1);
      t_hi = dense_min_of(a, j1);
      t_lo = dense_min_between(a, j0, t_b - 1);
    }
    const int64_t e0 = tile0 + (int64_t)threadIdx.x * kFI;
    // a column ahead of this pass (its additions run up to a later one) collides with a pivot
    // here; of it only the stored low matters
    constexpr int32_t kAhead = -2;  // in place of its source
    int32_t j[kFI], l[kFI], sg[kFI], n[kFI], b[kFI], s[kFI];
#pragma unroll
    for (int i = 0; i < kFI; i++) {
      j[i] = e0 + i < v.n_act ? v.act[e0 + i] : INT32_MIN;
      s[i] = l[i] = -1;
      if (ahead > 1 && e0 + i < v.n_act) {
        if (due_pass(a.due[e0 + i]) > pass) s[i] = kAhead;
        l[i] = lows[e0 + i];
      }
    }
#pragma unroll
    for (int i = 0; i < kFI; i++) {
      // (a slot whose column left keeps its segment, so the scan's runs stay whole)
      sg[i] = j[i] != INT32_MIN ? seg_of(a, slot_id(j[i])) : INT32_MAX;
      if (j[i] < 0) j[i] = l[i] = -1;
      else if (ahead == 1) l[i] = a.low[j[i]];
      n[i] = j[i] >= 0 && s[i] != kAhead ? v.alen[e0 + i] : 0;
      b[i] = j[i] >= 0 ? a.beta[j[i]] : -1;
    }
#pragma unroll
    for (int i = 0; i < kFI; i++) {
      if (!PH_DCHECK(&ds->debug_fault, l[i] < a.rows_end, 2)) l[i] = -1, j[i] = -1;
      if (s[i] != kAhead) s[i] = l[i] >= 0 ? (int32_t)(unsigned)a.tab[l[i]] : -1;
    }
    // Phase I values (the low of a colliding column, in its (cloud, dim) segment) and the space
    // bounds: a column's reservation is its stored words (its rows, or its bitmap with the
    // header); a target's source may be added; a left-most column may be proven and move
    SegMax x[kFI];
#pragma unroll
    for (int i = 0; i < kFI; i++) {
      const bool collide = l[i] >= 0 && s[i] != j[i];
      bw += stored_words(n[i]);
      if (collide && s[i] != kAhead) {
        const int32_t ns = stored_words(a.meta[s[i]].len);
        bw += max(ns, visit_rows);
        want |= n[i] + ns > (j[i] >= t_b ? t_hi : t_lo);
      } else if (l[i] >= 0 && !collide) {
        bp += stored_words(n[i]);
      }
      x[i] = SegMax{sg[i], collide ? l[i] : -1};
    }
    SegMax agg = x[0];
#pragma unroll
    for (int i = 1; i < kFI; i++) agg = segmax_combine(agg, x[i]);
    SegMax tot;
    const SegMax pre_t = block_scan_segmax(agg, SegMax{-1, -1}, sh, tot);  // within the tile
    // a tile without a mark that needs P_j only publishes its value (every 16th its prefix, so that
    // walks stay short): 24 clouds, 2.28 M columns 3250 -> 3165 us, 10,700 columns 468 -> 448 us
    bool needs = false;
#pragma unroll
    for (int i = 0; i < kFI; i++) needs |= l[i] >= 0 && s[i] == j[i] && l[i] != b[i];
    unsigned long long* tile_st = kLoop ? a.loop_tile_st : a.tile_st;
    needs = __syncthreads_or(needs) || (t & 15) == 0;
    if (!needs) {
      if (threadIdx.x == 0) tile_publish(tile_st, pass, t, tot);
    } else if (threadIdx.x < 32) {
      const SegMax P = tile_look_back(tile_st, pass, t, tot, fault);
      if (threadIdx.x == 0) s_pre = P;
    }
    // the marks: a new pivot proven by Thm 5 (left-most, low = beta) or by Phase I (left-most,
    // low > P_j); else the zero case of Corollary 10, else a pair prediction. Every active
    // column carries no flag (proven, final and cleared columns leave the active list in the
    // pass that marks them; the new-pivot mark goes with them), so marks are stored without a
    // load. Only a left-most column whose low is not its beta needs P_j: the others are marked
    // while warp 0 looks back, the rest after the tile's prefix is known.
    auto dirty = [&](int32_t seg) {
      if (atomicExch(&a.dirty_on[seg], 1) == 0) a.dirty[atomicAdd(&ds->n_dirty, 1u)] = seg;
    };
    auto pivot = [&](int i) {
      if (ahead > 1) {
        const ColMeta mj = load_meta(a.meta + j[i]);
        a.prec[l[i]] = rec_of(mj.ptr, mj.len);
      }
      a.meta[j[i]].flags = F_PROVEN | F_NEWPIV;
      a.owner[l[i]] = j[i];
      a.tab[l[i]] = (unsigned)j[i];  // its row's left-most column from now on (as it is now)
      // a paired row: its segment's first unpaired one?
      if (l[i] == fu[sg[i] - a.nc]) dirty(sg[i] - a.nc);
      if (j[i] == fu[sg[i]]) dirty(sg[i]);
      a.meta[l[i]].cleared = 1;  // clearing (Lemma 1): column l is positive and paired with j
      n_piv++;
    };
    // a zeroed column: one ahead of the pass leaves its slot at once (it is nobody's source); one
    // that is up to date in the additions kernel, where others may be reading it
    auto zero = [&](int i) {
      a.meta[j[i]].flags = F_FINAL;
      if (s[i] == kAhead) {
        a.meta[j[i]].len = 0;
        a.low[j[i]] = -1;
        v.act[e0 + i] = dead_slot(j[i]);
        a.due[e0 + i] = kDeadDue;
      }
    };
    auto unproven = [&](int i) {  // true: zeroed
      if (a.cor10 && b[i] < 0 && l[i] < fu[sg[i] - a.nc]) {
        zero(i);  // Corollary 10, zero case
        n_c10++;
        return true;
      }
      if (a.predict && b[i] >= 0 && a.pred[j[i]] < 0) {
        const int32_t pi = predicted_low(a, b[i], l[i]);
        if (pi >= 0) {
          a.pred[j[i]] = pi;
          n_pred++;
        } else if (pi == -2) {
          n_empty++;
        }
      }
      return false;
    };
    unsigned waits = 0;  // items whose mark needs P_j
    unsigned keeps = 0;  // items whose column may stay active
#pragma unroll
    for (int i = 0; i < kFI; i++) {
      if (j[i] < 0) {
        if (e0 + i < v.n_act) a.src_e[e0 + i] = -1;
        continue;
      }
      if (s[i] != kAhead)
        a.src_e[e0 + i] = s[i] != j[i] ? s[i] : -1;  // Phase II reads it in list order
      (void)PH_DCHECK(&ds->debug_fault, a.meta[j[i]].flags == 0, 7);
      if (l[i] < 0) {
        zero(i);
        n_zero++;
      } else if (s[i] != j[i]) {
        if (!unproven(i)) keeps |= 1u << i;
      } else if (l[i] == b[i]) {
        pivot(i);
      } else {
        waits |= 1u << i;
        keeps |= 1u << i;
      }
    }
    int place = 0;  // of this thread's first kept item among the tile's
    if (v.compact && ahead > 1) {
      int kept;
      place = block_excl_sum<int>(__popc(keeps), s_keep, kept);
      if (threadIdx.x < 32) {
        if (threadIdx.x == 0) look_publish(a, pass, t, kept);
        const int64_t before = look_back(a, pass, t, kept);
        if (threadIdx.x == 0) s_place = before;
      }
    }
    __syncthreads();
    if (v.compact && ahead > 1) {
#pragma unroll
      for (int i = 0; i < kFI; i++) {
        if (j[i] < 0) continue;
        const bool kept = (keeps >> i) & 1u;
        a.newpos[e0 + i] =
            kept ? (int32_t)(s_place + place + __popc(keeps & ((1u << i) - 1u))) : -1;
      }
    }
    if (waits) {
      SegMax run = threadIdx.x == 0 ? s_pre : segmax_combine(s_pre, pre_t);
#pragma unroll
      for (int i = 0; i < kFI; i++) {
        const SegMax pre = run;
        run = segmax_combine(run, x[i]);
        if (!((waits >> i) & 1u)) continue;
        const int32_t P = (pre.seg == x[i].seg) ? pre.val : -1;
        if (l[i] > P) pivot(i); else unproven(i);
      }
    }
  }
  if (v.stats) {
    stat_add(v.stats, PH_PS_ZERO_FINAL, n_zero);
    stat_add(v.stats, PH_PS_NEW_PIVOTS, n_piv);
    stat_add(v.stats, PH_PS_PREDICTED, n_pred);
    stat_add(v.stats, PH_PS_EMPTY_L, n_empty);
    stat_add(v.stats, PH_PS_COR10, n_c10);
  }
  if (want && !v.dense_on) ds->dense_want = 1;  // bit-packed additions from the next pass
  if (__any_sync(0xffffffffu, fault) && lane_id() == 0) ds->fault = 1;
  if constexpr (kLoop) {
    const int64_t ww = warp_sum64(bw), wp = warp_sum64(bp);
    if (lane_id() == 0 && (ww || wp)) {
      atomicAdd(&ds->bound_words, (unsigned long long)ww);
      atomicAdd(&ds->bound_piv, (unsigned long long)wp);
    }
    return;
  }
  int64_t tw, tp;
  block_excl_sum<int64_t>(bw, shs, tw);
  block_excl_sum<int64_t>(bp, shs, tp);
  if (threadIdx.x == 0 && (tw || tp)) {
    atomicAdd(&ds->bound_words, (unsigned long long)tw);
    atomicAdd(&ds->bound_piv, (unsigned long long)tp);
  }
}

// Phase I of a look-ahead pass before the horizon (no pair predictions). Nineteen of twenty columns
// are ahead of it: their due word and stored low are all there is to read, eight slots per thread in
// four loads, and what is left to do for one is the zero case of Corollary 10. The others' slots are
// listed in shared memory and taken by one thread each. Bound by the chain of waits of each tile:
// phase1_pass, which reads every slot's column, segment and beta, took 95 to 130 us for such a pass of
// 10.67 M columns, this takes 50 to 100 us (the 85 MB of due words and lows would take 13 us). The
// reduction of 10.67 M columns 36.0 -> 34.8 ms, of 42.7 M in 512 clouds 41.5 -> 39.7 ms.
constexpr int kMidItems = 8, kMidTile = kThreads * kMidItems;
__device__ __forceinline__ void mark_pivot(const RArgs& a, const int32_t* fu, int32_t j, int32_t l,
                                           int32_t sg) {
  auto dirty = [&](int32_t seg) {
    if (atomicExch(&a.dirty_on[seg], 1) == 0) a.dirty[atomicAdd(&a.ds->n_dirty, 1u)] = seg;
  };
  const ColMeta mj = load_meta(a.meta + j);
  a.prec[l] = rec_of(mj.ptr, mj.len);
  a.meta[j].flags = F_PROVEN | F_NEWPIV;
  a.owner[l] = j;
  a.tab[l] = (unsigned)j;  // its row's left-most column from now on (as it is now)
  if (l == fu[sg - a.nc]) dirty(sg - a.nc);
  if (j == fu[sg]) dirty(sg);
  a.meta[l].cleared = 1;  // clearing (Lemma 1)
}

__device__ __forceinline__ void phase1_mid(const RArgs& a) {
  __shared__ SegMax sh[kWarps + 1];
  __shared__ int64_t s_tile;
  __shared__ SegMax s_pre;
  __shared__ int s_n, s_ne;
  __shared__ unsigned int s_due, s_enter;
  __shared__ uint16_t s_slot[kMidTile];
  __shared__ int32_t s_val[kMidTile];   // of a listed slot: its Phase I value,
  __shared__ int32_t s_wait[kMidTile];  // its column if the mark needs P_j, else -1
  DevState* ds = a.ds;
  const PV v = pass_view(ds);
  const int32_t pass = ds->pass;
  const int32_t* fu = a.first_unp;
  const int32_t* lows = a.lows + (int64_t)(pass & a.ring) * a.lows_stride;
  const int64_t ntiles = (v.n_act + kMidTile - 1) / kMidTile;
  int64_t bw = 0, bp = 0;
  int64_t n_ahead = 0;
  bool want = false, fault = false;
  for (;;) {
    if (threadIdx.x == 0) {
      s_tile = atomicAdd(&ds->tile_queue, 1u);
      s_n = s_ne = 0;
    }
    __syncthreads();
    const int64_t t = s_tile;
    if (t >= ntiles) break;
    const int64_t tile0 = t * kMidTile, e0 = tile0 + (int64_t)threadIdx.x * kMidItems;
    int32_t d[kMidItems], l[kMidItems];
    {
      const int64_t r0 = min(e0, a.lows_stride - kMidItems);  // (threads past the list read its end)
      const int4 d0 = *reinterpret_cast<const int4*>(a.due + r0);
      const int4 d1 = *reinterpret_cast<const int4*>(a.due + r0 + 4);
      const int4 l0 = *reinterpret_cast<const int4*>(lows + r0);
      const int4 l1 = *reinterpret_cast<const int4*>(lows + r0 + 4);
      d[0] = d0.x, d[1] = d0.y, d[2] = d0.z, d[3] = d0.w;
      d[4] = d1.x, d[5] = d1.y, d[6] = d1.z, d[7] = d1.w;
      l[0] = l0.x, l[1] = l0.y, l[2] = l0.z, l[3] = l0.w;
      l[4] = l1.x, l[5] = l1.y, l[6] = l1.z, l[7] = l1.w;
    }
    // one segment for the whole tile, as a rule (ids, and so segments, ascend)
    const int32_t id0 = slot_id(v.act[tile0]);
    const int32_t sg0 = seg_of(a, id0);
    const int32_t sg1 = seg_of(a, slot_id(v.act[min(tile0 + kMidTile, v.n_act) - 1]));
    const bool one = sg0 == sg1;
    // the visits look through slots below the top dimension themselves (a pass may clear those)
    const bool top = id0 >= a.rows_end;
    if (!top && threadIdx.x == 0)
      atomicMax(&ds->scan_end, (unsigned int)min(tile0 + kMidTile, v.n_act));
    int32_t sg[kMidItems];
#pragma unroll
    for (int i = 0; i < kMidItems; i++)
      sg[i] = e0 + i >= v.n_act ? INT32_MAX : one ? sg0 : seg_of(a, slot_id(v.act[e0 + i]));
    const int32_t fu0 = sg0 >= a.nc ? fu[sg0 - a.nc] : INT32_MIN;
    unsigned listed = 0, enter = 0;
#pragma unroll
    for (int i = 0; i < kMidItems; i++) {
      const int32_t dp = due_pass(d[i]);
      const bool dead = e0 + i >= v.n_act || d[i] == kDeadDue;
      if (dead) {
        l[i] = -1;
      } else if (dp <= pass) {
        listed |= 1u << i;
      } else if (l[i] < 0 || (d[i] < 0 && l[i] < (one ? fu0 : fu[sg[i] - a.nc]))) {
        const int32_t j = v.act[e0 + i];  // zeroed: it leaves its slot at once
        a.meta[j].flags = F_FINAL;
        a.meta[j].len = 0;
        a.low[j] = -1;
        v.act[e0 + i] = dead_slot(j);
        a.due[e0 + i] = kDeadDue;
      } else if (top) {
        n_ahead++;
        enter |= dp == pass + 1 ? 1u << i : 0u;
      }
    }
    const int my_enter = enter ? atomicAdd(&s_ne, __popc(enter)) : 0;
    if (listed) {
      int p = atomicAdd(&s_n, __popc(listed));
#pragma unroll
      for (int i = 0; i < kMidItems; i++)
        if ((listed >> i) & 1u) {
          s_slot[p++] = (uint16_t)(threadIdx.x * kMidItems + i);
          s_val[threadIdx.x * kMidItems + i] = l[i];
        }
    }
    __syncthreads();
    const int n_list = s_n;
    if (top && threadIdx.x == 0) {  // (read after the scan's barriers)
      if (n_list) s_due = atomicAdd(&ds->n_due, (unsigned int)n_list);
      if (s_ne) s_enter = atomicAdd(&ds->n_enter, (unsigned int)s_ne);
    }
    if (n_list > 0) {
      // bit-packing thresholds, as in phase1_pass
      int32_t t_b = 0, t_hi = INT32_MAX, t_lo = INT32_MAX;
      if (a.dense_floor != INT32_MAX) {
        const int32_t j0 = slot_id(v.act[tile0]);
        const int32_t j1 = slot_id(v.act[min(tile0 + kMidTile, v.n_act) - 1]);
        t_b = dim_start_of(a, j1);
        t_hi = dense_min_of(a, j1);
        t_lo = dense_min_between(a, j0, t_b - 1);
      }
      for (int k = threadIdx.x; k < n_list; k += kThreads) {
        const int x = s_slot[k];
        const int64_t e = tile0 + x;
        const int32_t lj = s_val[x];
        const int32_t s = lj >= 0 ? (int32_t)(unsigned)a.tab[lj] : -1;
        const int32_t j = v.act[e], nj = v.alen[e];
        int32_t wait = -1, val = -1, src = -1;
        if (PH_DCHECK(&ds->debug_fault, j >= 0 && lj < a.rows_end, 2)) {
          const int32_t b = a.beta[j], sj = one ? sg0 : seg_of(a, j);
          (void)PH_DCHECK(&ds->debug_fault, a.meta[j].flags == 0, 7);
          bw += stored_words(nj);
          if (lj < 0) {
            a.meta[j].flags = F_FINAL;
          } else if (s != j) {
            const int32_t ns = stored_words(a.meta[s].len);
            bw += max(ns, kDeltaRows);
            want |= nj + ns > (j >= t_b ? t_hi : t_lo);
            val = lj;
            src = s;
            if (a.cor10 && b < 0 && lj < fu[sj - a.nc]) a.meta[j].flags = F_FINAL;
          } else {
            bp += stored_words(nj);
            if (lj == b) mark_pivot(a, fu, j, lj, sj);
            else wait = j;
          }
          a.src_e[e] = src;
        }
        s_val[x] = val;
        s_wait[x] = wait;
      }
      __syncthreads();
    }
    unsigned waits = 0;
    SegMax agg{-1, -1};
#pragma unroll
    for (int i = 0; i < kMidItems; i++) {
      if ((listed >> i) & 1u) {
        const int x = threadIdx.x * kMidItems + i;
        if (s_wait[x] >= 0) waits |= 1u << i;
        else l[i] = s_val[x];
      }
      const SegMax xi{sg[i], (waits >> i) & 1u ? -1 : l[i]};
      agg = i == 0 ? xi : segmax_combine(agg, xi);
    }
    SegMax tot;
    const SegMax pre_t = block_scan_segmax(agg, SegMax{-1, -1}, sh, tot);  // within the tile
    if (top) {
      for (int k = threadIdx.x; k < n_list; k += kThreads)
        a.newpos[s_due + k] = (int32_t)(tile0 + s_slot[k]);
      if (enter) {
        int32_t* o = v.act2 + s_enter + my_enter;
#pragma unroll
        for (int i = 0; i < kMidItems; i++)
          if ((enter >> i) & 1u) *o++ = (int32_t)(e0 + i);
      }
    }
    // a tile without such a mark only publishes its value (every 16th its prefix, so walks stay short)
    if (!__syncthreads_or(waits) && (t & 15)) {
      if (threadIdx.x == 0) tile_publish(a.tile_st, pass, t, tot);
      continue;
    }
    if (threadIdx.x < 32) {
      const SegMax P = tile_look_back(a.tile_st, pass, t, tot, fault);
      if (threadIdx.x == 0) s_pre = P;
    }
    __syncthreads();
    if (waits) {
      SegMax run = threadIdx.x == 0 ? s_pre : segmax_combine(s_pre, pre_t);
#pragma unroll
      for (int i = 0; i < kMidItems; i++) {
        const SegMax pre = run;
        const bool w = (waits >> i) & 1u;
        run = segmax_combine(run, SegMax{sg[i], w ? -1 : l[i]});
        if (!w) continue;
        const int32_t j = s_wait[threadIdx.x * kMidItems + i];
        const int32_t P = pre.seg == sg[i] ? pre.val : -1;
        if (l[i] > P) mark_pivot(a, fu, j, l[i], sg[i]);
        else if (a.cor10 && a.beta[j] < 0 && l[i] < fu[sg[i] - a.nc]) a.meta[j].flags = F_FINAL;
      }
    }
    __syncthreads();  // the lists are done with
  }
  if (want && !v.dense_on) ds->dense_want = 1;
  if (__any_sync(0xffffffffu, fault) && lane_id() == 0) ds->fault = 1;
  const int64_t ww = warp_sum64(bw), wp = warp_sum64(bp), wa = warp_sum64(n_ahead);
  if (lane_id() == 0 && (ww || wp)) {
    atomicAdd(&ds->bound_words, (unsigned long long)ww);
    atomicAdd(&ds->bound_piv, (unsigned long long)wp);
  }
  if (lane_id() == 0 && wa) atomicAdd(&ds->targets, (unsigned long long)wa);  // still targets
}

// no more blocks take part in Phase I than there are tiles (the others leave at once: a short
// pass's grid is mostly idle); block 0 always does
__device__ __forceinline__ unsigned phase1_parts(const DevState* ds, unsigned blocks) {
  const int64_t ntiles = (ds->n_act + kFTile - 1) / kFTile;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks, ntiles));
}

template <bool kLookAhead>
__global__ void __launch_bounds__(kThreads, 4) k_phase1(RArgs a) {
  pdl_wait();
  pdl_trigger();
  DevState* ds = a.ds;
  if (ds->status != ST_RUN) return;
  const unsigned parts = phase1_parts(ds, gridDim.x);
  if (blockIdx.x >= parts) return;
  if (kLookAhead && !ds->compact && !a.predict) {
    phase1_mid(a);
  } else {
    if (kLookAhead && !ds->compact && blockIdx.x == 0 && threadIdx.x == 0)
      ds->scan_end = (unsigned int)ds->n_act;
    phase1_pass<kLookAhead, false>(a, parts);
  }
  // the last of the taking-part blocks checks the space this pass's Phase II needs
  if (last_block(&ds->blocks_done, parts)) {
    if (threadIdx.x == 0) {
      ds->blocks_done = 0;
      check_capacity(ds);
    }
  }
}

// ------------------------------------------------------------------------------------------
// Phase II with p processors (Sec. 3.4): the neighbour sets a pass acts on
// ------------------------------------------------------------------------------------------
// every active target whose addition this pass may do is counted in its set (row low(j));
// the tests are those of the additions themselves, applied to the marks of this pass
__global__ void k_set_count(RArgs a) {
  if (a.ds->status != ST_RUN) return;
  const PV v = pass_view(a.ds);
  if (!v.do_adds) return;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < v.n_act; e += stride) {
    const int32_t s = a.src_e[e];
    if (s < 0) continue;
    const int32_t j = v.act[e];
    const ColMeta mj = load_meta(a.meta + j);
    if ((mj.flags & (F_PROVEN | F_FINAL)) || mj.cleared) continue;
    const ColMeta ms = load_meta(a.meta + s);
    if ((ms.flags & F_FINAL) || ms.cleared || (a.strict && !(ms.flags & F_PROVEN))) continue;
    const int32_t i = a.low[j];
    atomicAdd(a.set_n + i, 1);
    if (a.beta[j] >= 0) atomicAdd(a.set_neg + i, 1);
  }
}

// Ties between sets go to the row that comes first in its cloud's filtration (then to the
// lower id): the rows are first sorted by their filtration index, and the stable sort by
// priority below keeps that order among equal keys.
__global__ void k_set_tiekeys(RArgs a, const int64_t* __restrict__ gidx, uint64_t* key,
                              uint64_t* row) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.rows_end; i += stride) {
    key[i] = (uint64_t)gidx[i];
    row[i] = (uint64_t)i;
    a.set_on[i] = 0;
  }
}

// Sort keys of the sets, in the current order of the rows: ascending key order is the priority
// order (priority 0: larger sets first; 1: more known-negative targets first, then larger
// sets); rows without a set sort last. bits: enough for any count.
__global__ void k_set_keys(RArgs a, int priority, int bits, uint64_t* key,
                           const uint64_t* __restrict__ row) {
  const uint64_t top = (1ull << bits) - 1;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.rows_end; t += stride) {
    const int64_t i = (int64_t)row[t];
    const uint64_t n = (uint64_t)a.set_n[i], g = (uint64_t)a.set_neg[i];
    key[t] = priority == 1 ? ((top - g) << bits) | (top - n) : top - n;
  }
}

// the first p sets of the sorted order are acted on
__global__ void k_set_select(RArgs a, int64_t p, const uint64_t* __restrict__ row) {
  const int64_t n = p < a.rows_end ? p : a.rows_end;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += stride) {
    const int64_t i = (int64_t)row[t];
    if (a.set_n[i] > 0) a.set_on[i] = 1;
  }
}

// a target outside the chosen sets keeps its collision (it counts as a target) but skips its
// addition this pass: its slot's source becomes -2 - s
__global__ void k_set_apply(RArgs a) {
  if (a.ds->status != ST_RUN) return;
  const PV v = pass_view(a.ds);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < v.n_act; e += stride) {
    const int32_t s = a.src_e[e];
    if (s >= 0 && !a.set_on[a.low[v.act[e]]]) a.src_e[e] = -2 - s;
  }
}

// ------------------------------------------------------------------------------------------
// what happens to an active column in Phase II
// ------------------------------------------------------------------------------------------
// One job by the whole warp on bitmaps: column A (rows, or a bit-packed column if dense_a) plus
// source B (likewise, dense_b) into the bit-packed column T, the job's reserved slot. Writes
// T's header and returns its row count; its largest row goes to low, its stored words to words.
__device__ __noinline__ int32_t dense_job_warp(const RArgs& a, int32_t j, const int32_t* A,
                                              int na, bool dense_a, const int32_t* B, int nb,
                                              bool dense_b, int32_t* T, int64_t room,
                                              int32_t& low, int32_t& words) {
  const int lane = lane_id();
  int64_t base;
  int32_t W;
  row_segment(a, j, base, W);
#ifdef PH_DEBUG
  // the bitmap fits the slot reserved for the job (room words)
  if (!PH_DCHECK(&a.ds->debug_fault, W + kDenseHead <= room, 6)) {
    low = -1;
    words = 0;
    return 0;
  }
#endif
  uint32_t* bits = reinterpret_cast<uint32_t*>(T + kDenseHead);
  const uint32_t* Ab = reinterpret_cast<const uint32_t*>(A + kDenseHead);
  const uint32_t* Bb = reinterpret_cast<const uint32_t*>(B + kDenseHead);
  const bool wb = B != nullptr && dense_b;
  for (int w = lane; w < W; w += 32) bits[w] = (dense_a ? Ab[w] : 0u) ^ (wb ? Bb[w] : 0u);
  __syncwarp();
  // the row lists, scattered bit by bit (rows of one list are distinct; the lists may share)
  if (!dense_a)
    for (int q = lane; q < na; q += 32) {
      const int64_t r = A[q] - base;
      atomicXor(bits + (r >> 5), 1u << (r & 31));
    }
  if (B != nullptr && !dense_b)
    for (int q = lane; q < nb; q += 32) {
      const int64_t r = B[q] - base;
      atomicXor(bits + (r >> 5), 1u << (r & 31));
    }
  __syncwarp();
  // rows and the largest row of the result (read from L2, where the atomics landed)
  int cnt = 0, top_w = -1;
  uint32_t top_bits = 0;
  for (int w = lane; w < W; w += 32) {
    const uint32_t x = __ldcg(bits + w);
    cnt += __popc(x);
    if (x) {
      top_w = w;
      top_bits = x;
    }
  }
  const int best = __reduce_max_sync(0xffffffffu, (unsigned)(top_w + 1)) - 1;
  const unsigned who = __ballot_sync(0xffffffffu, top_w == best && best >= 0);
  low = -1;
  if (best >= 0) {
    const uint32_t tb = __shfl_sync(0xffffffffu, top_bits, __ffs(who) - 1);
    low = (int32_t)(base + 32 * (int64_t)best + 31 - __clz(tb));
  }
  const int32_t rows = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
  if (lane == 0) T[0] = rows;
  __syncwarp();
  words = W + kDenseHead;
  return rows;
}

struct Job {
  int32_t j;
  int32_t src;    // source column for an addition, -1 if none
  bool surv;      // stays active
  bool newpiv;    // proven this pass: moves to the pivot store
  bool target;    // collides with an earlier column
  int64_t words;  // arena words reserved (survivors only)
  const int32_t* A;  // the column's rows (new pivots and survivors)
  const int32_t* B;  // the source's rows (additions)
  int na, nb;
  bool dense_a, dense_b;  // A / B is a bit-packed column (na / nb are then its stored words)
};

// kDense: columns may be bit-packed (the length field tells); otherwise every column is a row list
template <bool kDense>
__device__ __forceinline__ Job job_of(const RArgs& a, const PV& v, int64_t e) {
  Job jb{-1, -1, false, false, false, 0, nullptr, nullptr, 0, 0, false, false};
  if (e >= v.n_act) return jb;
  // every load is issued up front: the column and its source candidate are known from the
  // active list and k_phase1's per-slot source, so no load waits on another's result
  const int32_t j = v.act[e];
  if (j < 0) return jb;  // (a place that look-ahead left empty)
  const int32_t se = a.src_e[e];  // -1: no collision; <= -2: a target whose set waits
  const int32_t s = se >= 0 ? se : -1;
  const ColMeta mj = load_meta(a.meta + j);  // one 16-byte load per column
  const uint8_t f = mj.flags;
  const uint8_t cj = mj.cleared;
  const int32_t nj = kDense ? stored_words(mj.len) : mj.len;
  const int32_t* pj = mj.ptr;
  uint8_t fs = 0, cs = 0;
  int32_t ns = 0;
  const int32_t* ps = nullptr;
  if (s >= 0) {
    const ColMeta ms = load_meta(a.meta + s);
    fs = ms.flags;
    cs = ms.cleared;
    ns = ms.len;
    ps = ms.ptr;
  }
  jb.j = j;
  jb.newpiv = (f & F_NEWPIV) != 0;
  jb.surv = !(f & (F_PROVEN | F_FINAL)) && !cj;
  if (jb.surv) {
    jb.words = nj;
    jb.target = se != -1;
    if (s >= 0) {
      if (v.do_adds && !(fs & F_FINAL) && !cs && (!a.strict || (fs & F_PROVEN))) {
        jb.src = s;
        jb.dense_b = kDense && ns < 0;
        jb.nb = kDense ? stored_words(ns) : ns;
        jb.words += jb.nb;
        jb.B = ps;
      }
    }
  }
  if (jb.newpiv || jb.surv) {
    jb.A = pj;
    jb.na = nj;
    jb.dense_a = kDense && mj.len < 0;
  }
  return jb;
}

// ------------------------------------------------------------------------------------------
// look_ahead: the additions of several passes on one column, by one lane
// ------------------------------------------------------------------------------------------
// The rows added to a column that are not in its list yet, one per place in any order (every index
// is static): what earlier visits left in the first kOld places, and the rows of this visit's
// sources, R places per pass. A place holds a row negated, or kEmpty. Rows above the column's low
// are spent, and a row may be there several times: the low only falls, so the next low is the
// largest row below it that is there an odd number of times, and nothing has to be taken out on
// the way.
constexpr int32_t kEmpty = -INT32_MAX;
struct Delta {
  int32_t c[kDeltaRows];
};

// odd ^= how many of x[I..] equal l, one instruction per value (the predicate chain stays inside)
__device__ __forceinline__ bool odd_of4(bool odd, int32_t l, int32_t x0, int32_t x1, int32_t x2,
                                        int32_t x3) {
  int32_t r;
  asm("{\n.reg .pred p;\n"
      "setp.ne.s32 p, %1, 0;\n"
      "setp.eq.xor.s32 p, %3, %2, p;\n"
      "setp.eq.xor.s32 p, %4, %2, p;\n"
      "setp.eq.xor.s32 p, %5, %2, p;\n"
      "setp.eq.xor.s32 p, %6, %2, p;\n"
      "selp.s32 %0, 1, 0, p;\n}"
      : "=r"(r)
      : "r"((int32_t)odd), "r"(l), "r"(x0), "r"(x1), "r"(x2), "r"(x3));
  return r != 0;
}

// the next low of a column of which low l was added to: the first kOld places if `old`, N places
// after them, and the column's own rows A[0 .. na), whose end is shortened (top is its last
// row, or -1)
template <int N>
__device__ __forceinline__ int32_t next_low(const Delta& d, bool old, const int32_t* A, int& na,
                                            int32_t& top, int32_t l) {
  for (;;) {
    if (top == l) {
      na--;
      top = na > 0 ? A[na - 1] : -1;
    }
    // the largest row below l, as the smallest unsigned distance from l - 1 (one add-min per
    // place): spent rows and empty places wrap around, and -1 (top at the least) is the farthest
    const int32_t lim = l - 1;
    unsigned best = (unsigned)(lim - top);
    if (old) {
#pragma unroll
      for (int i = 0; i < kOld; i++) best = __viaddmin_u32((unsigned)d.c[i], (unsigned)lim, best);
    }
#pragma unroll
    for (int i = kOld; i < kOld + N; i++)
      best = __viaddmin_u32((unsigned)d.c[i], (unsigned)lim, best);
    l = lim - (int32_t)best;
    if (l < 0) return -1;
    bool odd = top == l;
    if (old) {
#pragma unroll
      for (int i = 0; i < kOld; i += 4)
        odd = odd_of4(odd, -l, d.c[i], d.c[i + 1], d.c[i + 2], d.c[i + 3]);
    }
#pragma unroll
    for (int i = kOld; i < kOld + N; i += 4)
      odd = odd_of4(odd, -l, d.c[i], i + 1 < kOld + N ? d.c[i + 1] : kEmpty,
                    i + 2 < kOld + N ? d.c[i + 2] : kEmpty, i + 3 < kOld + N ? d.c[i + 3] : kEmpty);
    if (odd) return l;
  }
}

// Batcher's odd-even merge sort of N values (any N) as a list of exchanges known at compile time
template <int N>
struct SortNet {
  int n = 0;
  int lo[N * N] = {}, hi[N * N] = {};
  constexpr SortNet() {
    for (int p = 1; p < N; p *= 2)
      for (int k = p; k >= 1; k /= 2)
        for (int j = k % p; j + k < N; j += 2 * k)
          for (int i = 0; i < k && i + j + k < N; i++)
            if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) {
              lo[n] = i + j;
              hi[n] = i + j + k;
              n++;
            }
  }
};
template <int N>
constexpr SortNet<N> kSortNet{};
template <int N, size_t... I>
__device__ __forceinline__ void sort_asc(int32_t (&c)[N], std::index_sequence<I...>) {
  const auto exchange = [&](int32_t& x, int32_t& y) {
    const int32_t m = min(x, y);
    y = max(x, y);
    x = m;
  };
  (exchange(c[std::integral_constant<int, kSortNet<N>.lo[I]>::value],
            c[std::integral_constant<int, kSortNet<N>.hi[I]>::value]),
   ...);
}
// sorts the values, smallest first
template <int N>
__device__ __forceinline__ void sort_asc(int32_t (&c)[N]) {
  sort_asc(c, std::make_index_sequence<(size_t)kSortNet<N>.n>{});
}


// one column's visit, before and after
struct Visit {
  Delta d;             // (after tidy: the rows left, ascending, then INT32_MAX)
  int k;               // rows in d
  const int32_t* A;    // its list
  int na;
  const int32_t* B;    // its first source's rows (nb of them) if that has no short record
  int nb;
  int4 rec;            // that source's record
  int32_t low;
  int32_t due;         // the pass whose additions visit the column next
  bool gone;           // done for: zeroed in pass due - 1 at the latest, its rows needed no more
  bool settle;         // its list has to be whole for the next visit
};

// Runs the additions of passes pass .. v.limit - 1 on the column of each lane that is on (low
// w.low) as far as their sources are known: the first source is given, a later one must be a
// proven pivot (its record in prec, complete after k_phase1's marks). A source of at most R rows
// beside its low takes this pass's places; one longer source per visit fills places from the
// far end, which leaves fewer passes. pos: the slot whose stored lows the run writes. A run ends
// early before another low, and when the column is done for: its low is -1 (k_phase1 of that
// pass makes it final), or lies below fu, the first unpaired row (Corollary 10 zeroes it in that
// pass: the row has a pivot, so the column collides, and fu never falls); that pass itself takes it
// off the list. Returns whether any lane used the places of earlier visits.
__device__ __forceinline__ bool look_ahead(const RArgs& a, const PV& v, int32_t pass, bool on,
                                           int32_t fu, int64_t pos, Visit& w) {
  constexpr int R = kSourceRows, N = R * kAheadMax;
  const int32_t* A = w.A;
  const int32_t* S = w.B;  // the rows of a longer source
  int32_t l = w.low;
  int na = on ? w.na : 0;
  int32_t top = na > 0 ? A[na - 1] : -1;
  int4 q = w.rec;
  const bool visited = on;
  const bool old = __any_sync(0xffffffffu, on && w.k > 0);
  int n_low = 0;
  int most = kAheadMax;  // passes the places suffice for
  bool longer = on && (q.x == 0 || q.x > R + 1);  // this pass's source is a longer one
  bool any_longer = false, in_rec = false;
  int n = longer ? w.nb - 1 : 0;
  auto next = [&](int t) {  // pass + t + 1 starts with low l; is its source known?
    a.lows[(int64_t)((pass + t + 1) & a.ring) * a.lows_stride + pos] = l;
    n_low = t + 1;
    w.gone = l < 0;
    on = false;
    if (l >= 0 && PH_DCHECK(&a.ds->debug_fault, l < a.rows_end && na >= 0, 8)) {
      q = a.prec[l];
      w.gone = q.x > 0 && l < fu;
      w.settle = q.x == 0 || q.x > N + 1;
      on = q.x > 0 && !w.gone && t + 1 < most && pass + t + 1 < v.limit;
      longer = on && q.x > R + 1;
      if (longer) {  // one per visit, of as many rows as leave this pass its place
        n = q.x - 1;
        on = longer = most == kAheadMax && q.x <= kRecRows + kLonger && n <= N - R * (t + 1);
        in_rec = q.x <= kRecRows;
        S = in_rec ? nullptr : rec_rows(q);
      }
    }
  };
  // (one copy of the code for all passes: unrolled, it would not stay in the instruction caches)
#pragma unroll 1
  for (int t = 0; t < kAheadMax && __any_sync(0xffffffffu, on); t++) {
    const bool put = on && !longer;
    const int32_t y = -q.y, z = -q.z;
#pragma unroll
    for (int i = 0; i < kAheadMax; i++) {
      if (t == i && put) {
        w.d.c[kOld + R * i] = y;
        w.d.c[kOld + R * i + 1] = z;
      }
    }
    if (__any_sync(0xffffffffu, longer)) {
      any_longer = true;
#pragma unroll
      for (int i = 0; i < N; i++) {
        if (i >= 4 && i % 4 == 0 && !__any_sync(0xffffffffu, longer && i < n)) break;
        if (longer && i < n)
          w.d.c[kOld + N - 1 - i] = -(i < 3 && in_rec ? (i == 0 ? q.y : i == 1 ? q.z : q.w) : S[i]);
      }
      if (longer) {
        most = max((N - n) / R, t + 1);
        longer = false;
      }
    }
    if (on) {
      if (!any_longer && t < kAheadMax / 2) l = next_low<N / 2>(w.d, old, A, na, top, l);
      else l = next_low<N>(w.d, old, A, na, top, l);
      next(t);
    }
  }
  if (visited) {
    w.low = l;
    w.due = pass + n_low + (w.gone ? 1 : 0);
    w.na = w.gone ? 0 : na;
  }
  return old;
}

// the rows of a visited column's delta that are left, in order from place FROM on (the places
// before it are empty); a row that is there twice cancels
template <int FROM>
__device__ __forceinline__ void tidy(Visit& w, bool on) {
  constexpr int N = kDeltaRows - FROM;
  int32_t c[N];
#pragma unroll
  for (int i = 0; i < N; i++) {
    const int32_t x = -w.d.c[FROM + i];
    c[i] = on && x <= w.low ? x : INT32_MAX;
  }
#pragma unroll 1
  for (int round = 0; round < 2; round++) {
    sort_asc(c);
    if (round == 1) break;
    bool twice = false;
#pragma unroll
    for (int i = 0; i + 1 < N; i++) {
      if (c[i] != INT32_MAX && c[i] == c[i + 1]) {
        c[i] = c[i + 1] = INT32_MAX;
        twice = true;
      }
    }
    if (!__any_sync(0xffffffffu, twice)) break;
  }
  w.k = 0;
#pragma unroll
  for (int i = 0; i < N; i++) {
    w.k += c[i] != INT32_MAX ? 1 : 0;
    w.d.c[i] = c[i];
  }
#pragma unroll
  for (int i = N; i < kDeltaRows; i++) w.d.c[i] = INT32_MAX;
}

// ------------------------------------------------------------------------------------------
// column arithmetic over F2: symmetric difference of two ascending row lists
// ------------------------------------------------------------------------------------------
// merge-path split on diagonal d with ties taken from A first; an equal pair A[x-1] == B[y]
// is kept on the same side of the split so that cancellations never straddle two lanes
__device__ __forceinline__ void merge_split(const int32_t* A, int na,
                                            const int32_t* B, int nb, int d, int& x,
                                            int& y) {
  int lo = d > nb ? d - nb : 0, hi = d < na ? d : na;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (A[mid] <= B[d - 1 - mid]) lo = mid + 1; else hi = mid;
  }
  x = lo;
  y = d - lo;
  if (x > 0 && y < nb && A[x - 1] == B[y]) y++;
}

// warp-cooperative symmetric difference straight from global memory (used for merges too long
// to stage in shared memory); every lane returns the output length and the last row written
__device__ __forceinline__ int warp_symdiff(const int32_t* A, int na, const int32_t* B, int nb,
                                            int32_t* dst, int32_t& last) {
  constexpr int K = 4;
  const int lane = lane_id();
  const int N = na + nb;
  int out = 0;
  last = -1;
  for (int base = 0; base < N; base += 32 * K) {
    int d0 = min(base + lane * K, N), d1 = min(base + (lane + 1) * K, N);
    int x0, y0, x1, y1;
    merge_split(A, na, B, nb, d0, x0, y0);
    merge_split(A, na, B, nb, d1, x1, y1);
    int cnt = 0;
    {
      int i = x0, k = y0;
      while (i < x1 || k < y1) {
        if (k >= y1 || (i < x1 && A[i] < B[k])) {
          cnt++;
          i++;
        } else if (i >= x1 || B[k] < A[i]) {
          cnt++;
          k++;
        } else {
          i++;
          k++;
        }
      }
    }
    int incl = warp_incl_sum(cnt);
    int pos = out + incl - cnt;
    int32_t mylast = -1;
    {
      int i = x0, k = y0;
      while (i < x1 || k < y1) {
        if (k >= y1 || (i < x1 && A[i] < B[k])) {
          mylast = A[i++];
          dst[pos++] = mylast;
        } else if (i >= x1 || B[k] < A[i]) {
          mylast = B[k++];
          dst[pos++] = mylast;
        } else {
          i++;
          k++;
        }
      }
    }
    unsigned has = __ballot_sync(0xffffffffu, cnt > 0);
    if (has) last = __shfl_sync(0xffffffffu, mylast, 31 - __clz(has));
    out += __shfl_sync(0xffffffffu, incl, 31);
  }
  return out;
}

// Per-warp shared staging of a batch of the warp's jobs, and per-job bookkeeping (indexed by
// the job's ordinal among the warp's staged jobs). Each staged list (a job's column A, its source
// B) has a span that starts on a 16-byte boundary: its first row lands at the span's start plus
// the list's misalignment in global memory (0-3 words), so whole 16-byte chunks copy it, and the
// word after its last row holds a sentinel (INT32_MAX), so a merge needs no bounds checks. A
// batch fills at most kStage words; kStageSlack more absorb a merge's reads past the last
// sentinel (at most KM + 1 words, KM <= 16).
constexpr int kStage = 1024;
constexpr int kStageSlack = 32;
constexpr int kScan = 64;  // slots a warp looks through at a time for due ones
struct __align__(16) WarpStage {
  int32_t in[kStage + kStageSlack];
  int32_t* jout[32];  // output slot of the job (its reserved words in the next arena)
  int32_t ia[32];     // index in `in` of the job's first row of A (current batch)
  int32_t ib[32];     // index in `in` of the job's first row of B
  int32_t na[32];
  int32_t nb[32];
  int32_t pc[33];     // first merge piece of the job: exclusive prefix of pieces over the jobs
  int32_t jcnt[32];   // output rows of the job so far
  int32_t jlow[32];   // largest output row (new low), -1 if none
};
constexpr int kAddThreads = 128;
constexpr int kAddWarps = kAddThreads / 32;
constexpr size_t kAddSmem = sizeof(WarpStage) * kAddWarps;
// block chunks with shared merge pieces: 64-thread blocks, whose chunk barriers wait on two warps
constexpr int kPieceBlockThreads = 64;
// the default switch to 8-slot warp chunks: fewer active columns than this many per warp of the
// grid. An 8-slot chunk takes about half as long as a 32-slot one, but pays its fixed costs
// (claim, column records, look-back) on a quarter of the columns: it wins once its chunks fit in
// about two waves of the grid's warps, where the 32-slot chunks leave most warps idle
constexpr int kNarrowColsPerWarp = 16;

// merge the staged rows A[x0..x1), B[y0..y1) of one lane's range; equal rows cancel.
// With WRITE, the surviving rows go to dst; returns their count and the last one in *last.
template <bool WRITE>
__device__ __forceinline__ int lane_symdiff(const int32_t* __restrict__ sA, int x0, int x1,
                                            const int32_t* __restrict__ sB, int y0, int y1,
                                            int32_t* __restrict__ dst, int32_t* last) {
  int cnt = 0;
  int32_t va = x0 < x1 ? sA[x0] : INT32_MAX;
  int32_t vb = y0 < y1 ? sB[y0] : INT32_MAX;
  int i = x0, j = y0;
  int32_t v = -1;
  while (i < x1 || j < y1) {
    if (va == vb) {
      ++i;
      ++j;
      va = i < x1 ? sA[i] : INT32_MAX;
      vb = j < y1 ? sB[j] : INT32_MAX;
    } else if (va < vb) {
      v = va;
      if (WRITE) dst[cnt] = v;
      ++cnt;
      ++i;
      va = i < x1 ? sA[i] : INT32_MAX;
    } else {
      v = vb;
      if (WRITE) dst[cnt] = v;
      ++cnt;
      ++j;
      vb = j < y1 ? sB[j] : INT32_MAX;
    }
  }
  if (WRITE) *last = v;
  return cnt;
}

// Symmetric difference of two short sorted columns (na, nb <= S) by one thread: both are loaded
// into registers, padded with INT32_MAX, B reversed so that the 2S values form a bitonic
// sequence, sorted by a bitonic merge network (static indices: no divergence, no local memory);
// equal rows -- one from each column -- end up adjacent and cancel. Returns the output length
// and the last (largest) row written, -1 if none.
template <int S>
__device__ __forceinline__ int reg_symdiff(const int32_t* A, int na, const int32_t* B, int nb,
                                           int32_t* dst, int32_t& last) {
  int32_t c[2 * S];
#pragma unroll
  for (int i = 0; i < S; i++) c[i] = i < na ? A[i] : INT32_MAX;
#pragma unroll
  for (int i = 0; i < S; i++) c[2 * S - 1 - i] = i < nb ? B[i] : INT32_MAX;
#pragma unroll
  for (int st = S; st >= 1; st >>= 1) {
#pragma unroll
    for (int i = 0; i < 2 * S; i++) {
      if ((i & st) == 0) {
        const int32_t x = c[i], y = c[i + st];
        c[i] = min(x, y);
        c[i + st] = max(x, y);
      }
    }
  }
  int k = 0;
  last = -1;
#pragma unroll
  for (int i = 0; i < 2 * S; i++) {
    const int32_t v = c[i];
    const bool drop = v == INT32_MAX || (i > 0 && c[i - 1] == v) || (i + 1 < 2 * S && c[i + 1] == v);
    if (!drop) {
      dst[k++] = v;
      last = v;
    }
  }
  return k;
}

// waits for all of this thread's asynchronous copies (cp_async16)
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// 16-byte asynchronous copy global -> shared (both addresses 16-byte aligned), cached in L2 only
__device__ __forceinline__ void cp_async16(int32_t* smem_dst, const int32_t* gsrc) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gsrc) : "memory");
}

// merge-path split of the staged lists A = in[ia..ia+na), B = in[ib..ib+nb) on diagonal d, ties
// taken from A first; an equal pair A[x-1] == B[y] is kept on the same side of the split, so that
// cancellations never straddle two pieces
__device__ __forceinline__ void split_staged(const int32_t* __restrict__ in, int ia, int na,
                                             int ib, int nb, int d, int& x, int& y) {
  int lo = d > nb ? d - nb : 0, hi = d < na ? d : na;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (in[ia + mid] <= in[ib + d - 1 - mid]) lo = mid + 1; else hi = mid;
  }
  x = lo;
  y = d - lo;
  if (x > 0 && y < nb && in[ia + x - 1] == in[ib + y]) y++;
}

// Merge rounds over the pieces [P0, P1) of one batch: a job of N staged rows is cut into
// ceil(N / km) pieces of km merge-path positions, and in each round lane l takes piece h0 + l.
// A piece's job is found from a bitmask of the pieces that start a job (each lane of the batch
// owns one job, with its first piece p_first); its end split comes from a binary search, its
// start split from the previous lane (or the previous round). A piece holds at most km + 1 rows
// (a split moves an equal pair to one side). KM > 0 (km = KM): a branch-free merge into
// registers, one shared load per row, the sentinels ending each list; the two copies of a row
// common to both columns come out adjacent and cancel. KM = 0 (any other km): merged
// sequentially, counted first and then merged again to write. Kept rows go to the job's slot
// after the kept rows of its earlier pieces.
template <int KM>
__device__ __forceinline__ void staged_rounds(WarpStage& S_, int P0, int P1, int o0, bool in_batch,
                                              int p_first, int km) {
  constexpr int S = KM > 0 ? KM + 1 : 0;  // register slots: the most rows a piece holds
  const int lane = lane_id();
  const int32_t* __restrict__ in = S_.in;
  int cx = 0, cy = 0;    // end split of the previous round's last piece
  int kprev = o0 - 1;    // job of the piece before the round
  for (int h0 = P0; h0 < P1; h0 += 32) {
    const unsigned start_bit =
        in_batch && p_first >= h0 && p_first < h0 + 32 ? 1u << (p_first - h0) : 0u;
    const unsigned heads = __reduce_or_sync(0xffffffffu, start_bit);
    const int h = h0 + lane;
    const bool valid = h < P1;
    const unsigned upto = 0xffffffffu >> (31 - lane);  // bits 0..lane
    const int o = kprev + __popc(heads & upto);        // this piece's job
    kprev = __shfl_sync(0xffffffffu, o, 31);
    int x0 = 0, y0 = 0, x1 = 0, y1 = 0, d0 = 0, ia = 0, ib = 0, na = 0, nb = 0;
    if (valid) {
      na = S_.na[o];
      nb = S_.nb[o];
      ia = S_.ia[o];
      ib = S_.ib[o];
      d0 = (h - S_.pc[o]) * km;
      const int n = na + nb;
      const int d1 = d0 + km < n ? d0 + km : n;
      if (d1 == n) {
        x1 = na;
        y1 = nb;
      } else {
        split_staged(in, ia, na, ib, nb, d1, x1, y1);
      }
    }
    const int px = __shfl_up_sync(0xffffffffu, x1, 1);
    const int py = __shfl_up_sync(0xffffffffu, y1, 1);
    if (valid && d0 > 0) {  // not a job's first piece: the previous piece is the same job's
      x0 = lane > 0 ? px : cx;
      y0 = lane > 0 ? py : cy;
    }
    cx = __shfl_sync(0xffffffffu, x1, 31);
    cy = __shfl_sync(0xffffffffu, y1, 31);
    const int cnt = valid ? (x1 - x0) + (y1 - y0) : 0;
    unsigned keep = 0;
    int32_t c[S > 0 ? S : 1];
    int kept = 0;
    if constexpr (S > 0) {
      if (valid) {  // branch-free sequential merge; the sentinels end each list
        int i = ia + x0, j = ib + y0;
        int32_t va = in[i], vb = in[j];
#pragma unroll
        for (int t = 0; t < S; t++) {
          const bool ta = va <= vb;
          c[t] = ta ? va : vb;
          if (t + 1 < S) {
            i += ta ? 1 : 0;
            j += ta ? 0 : 1;
            const int32_t nv = in[ta ? i : j];
            va = ta ? nv : va;
            vb = ta ? vb : nv;
          }
        }
        // bit t of eq: row t equals row t + 1 (an equal pair, which cancels); rows past the
        // piece's cnt are masked off, so a pair never reaches past the piece
        const unsigned in_piece = cnt >= 32 ? 0xffffffffu : (1u << cnt) - 1u;
        unsigned eq = 0;
#pragma unroll
        for (int t = 0; t + 1 < S; t++) eq |= (c[t] == c[t + 1] ? 1u : 0u) << t;
        eq &= in_piece >> 1;
        keep = in_piece & ~(eq | (eq << 1));
        kept = __popc(keep);
      }
    } else {
      if (valid) kept = lane_symdiff<false>(in + ia, x0, x1, in + ib, y0, y1, nullptr, nullptr);
    }
    // this piece's place among the kept rows of its job: a scan over the round, restarted at the
    // pieces that start a job (and at lane 0, which continues the previous round's job)
    const unsigned run_heads = __ballot_sync(0xffffffffu, valid && (d0 == 0 || lane == 0));
    const int incl = warp_incl_sum(kept);
    const int rs = 31 - __clz(run_heads & upto);
    const int run_base = __shfl_sync(0xffffffffu, incl - kept, rs);
    const int jc = valid ? S_.jcnt[o] : 0;
    const bool run_last =
        valid && (lane == 31 || ((run_heads >> (lane + 1)) & 1u) || h + 1 >= P1);
    __syncwarp();  // every lane has read its job's count before the run's last lane moves it
    if (kept) {
      int32_t* dst = S_.jout[o] + jc + (incl - kept - run_base);
      int32_t lastv = -1;
      if constexpr (S > 0) {
        int q = 0;
#pragma unroll
        for (int t = 0; t < S; t++) {
          if (keep & (1u << t)) {
            dst[q++] = c[t];
            lastv = c[t];
          }
        }
      } else {
        lane_symdiff<true>(in + ia, x0, x1, in + ib, y0, y1, dst, &lastv);
      }
      atomicMax(&S_.jlow[o], lastv);
    }
    if (run_last) S_.jcnt[o] = jc + (incl - run_base);
    __syncwarp();
  }
}

// One job merged by its own lane, sequentially from the staged lists (the sentinels end each
// list), straight into its slot: a row equal to the one before it cancels that one, so the two
// copies of a row common to both columns never reach the slot. Returns the output length; the
// last row written (the new low) goes to *last, -1 if none.
__device__ __forceinline__ int lane_merge_job(const int32_t* __restrict__ in, int ia, int ib, int n,
                                              int32_t* __restrict__ dst, int32_t* last) {
  int i = ia, j = ib, q = 0;
  int32_t va = in[i], vb = in[j];
  int32_t p = -1, w = -1;
  bool held = false;  // p is a merged row not written yet (it may still cancel)
  for (int t = 0; t < n; t++) {
    const bool ta = va <= vb;
    const int32_t v = ta ? va : vb;
    i += ta ? 1 : 0;
    j += ta ? 0 : 1;
    const int32_t nv = in[ta ? i : j];
    va = ta ? nv : va;
    vb = ta ? vb : nv;
    if (held && v == p) {
      held = false;
    } else {
      if (held) {
        dst[q++] = p;
        w = p;
      }
      p = v;
      held = true;
    }
  }
  if (held) {
    dst[q++] = p;
    w = p;
  }
  *last = w;
  return q;
}

// A survivor j with low l enters the next pass's left-most-column table (and a new low l is
// marked as seen, for the essential estimate; a low that stays was marked when it appeared): the
// table is built while the pass's additions write the new lows, so no kernel of the next pass
// gathers the lows for it
template <bool kNewLow>
__device__ __forceinline__ void next_tab(const RArgs& a, const PV& v, int32_t l, int32_t j) {
  if (l < 0 || !PH_DCHECK(&a.ds->debug_fault, l < a.rows_end, 1)) return;
  const unsigned long long key = v.tab_key | (unsigned)j;
  if (a.tab[l] > key) atomicMin(&a.tab[l], key);
  if (kNewLow && !a.meta[l].low_seen) a.meta[l].low_seen = 1;
}

enum : int {
  kCntTargets, kCntActive, kCntCleared, kCntAdds, kCntXors, kCntCopied, kCntPacked, kNumCnt
};

// Merges by one warp: per lane the column A (rows, or a bit-packed column if dense_a) and the
// source B (likewise, dense_b; null: the column moves) into the lane's slot of the arena (null: no
// job), whose words suffice for all rows. Short columns are merged in registers (one thread per
// job); longer ones are staged in shared memory and merged, each job by its own lane (short
// jobs) or by a merge path over the batch's jobs cut into pieces of km positions (8 unless
// ph_opts.merge_items says otherwise); merges longer than the staging bound run from global
// memory; bit-packed jobs run one at a time by the whole warp. kSlots: lanes with jobs. Returns how
// the lane's job was done (4: bit-packed); o_ptr, o_len, low: the result's place, length and low.
template <bool kDense, int kSlots, bool kLane>
__device__ __forceinline__ int merge_rows(const RArgs& a, const PV& v, WarpStage& S, int32_t j,
                                          int32_t* slot, const int32_t* A, int na, bool dense_a,
                                          const int32_t* B, int nb, bool dense_b, int32_t*& o_ptr,
                                          int& o_len, int32_t& low) {
  const int lane = lane_id();
  const int N = slot != nullptr ? na + nb : 0;
  o_ptr = slot;
  o_len = 0;
  low = -1;
  // short merges: one thread per job, in registers
  // (cls 1: register merge, 3: staged or from global memory). The register path pays off when
  // most of the warp takes it; a few short jobs among long ones would keep the rest of the warp
  // waiting, so they join the staged path instead. One network size serves the whole warp.
  const int need = max(na, nb);
  // cls 4: bit-packed (the column is, or the source is, or the sum exceeds the threshold)
  const bool dense_job =
      kDense && N > 0 && (dense_a || (B != nullptr && (dense_b || (v.dense_on && goes_dense(a, j, N)))));
  // the register network for jobs of up to kRegMax rows per column; the piece kernels keep it
  // small (8), their registers go to the merge pieces
  constexpr int kRegMax = kLane ? 16 : 8;
  int cls = N == 0 ? 0 : (dense_job ? 4 : (need <= kRegMax ? 1 : 3));
  constexpr int kRegMinJobs = 12 * kSlots / 32;  // of the warp's slots
  if (__popc(__ballot_sync(0xffffffffu, cls == 1)) < kRegMinJobs && cls == 1) cls = 3;
  const unsigned wneed = __reduce_max_sync(0xffffffffu, cls == 1 ? (unsigned)need : 0u);
  if (cls == 1) {
    int32_t last;
    int len;
    if constexpr (kRegMax == 16) {
      len = wneed <= 4   ? reg_symdiff<4>(A, na, B, nb, slot, last)
            : wneed <= 8 ? reg_symdiff<8>(A, na, B, nb, slot, last)
                         : reg_symdiff<16>(A, na, B, nb, slot, last);
    } else {
      len = wneed <= 4 ? reg_symdiff<4>(A, na, B, nb, slot, last)
                       : reg_symdiff<8>(A, na, B, nb, slot, last);
    }
    o_ptr = slot;
    o_len = len;
    low = last;
  }
  const unsigned smask = __ballot_sync(0xffffffffu, cls == 3);
  if (smask) {
    // longer merges: staged in shared memory, merge path over the concatenated jobs. Each list
    // takes a 16-byte aligned span (its misalignment, its rows, a sentinel, rounded up to 4 words)
    const int ra = (int)(((uintptr_t)A >> 2) & 3u);
    const int rb = B ? (int)(((uintptr_t)B >> 2) & 3u) : 0;
    const int span_a = (ra + na + 1 + 3) & ~3;
    const int span_b = (rb + nb + 1 + 3) & ~3;
    const bool staged = cls == 3 && N <= a.staged_max && span_a + span_b <= kStage;
    const bool big = cls == 3 && !staged;
    const unsigned stmask = __ballot_sync(0xffffffffu, staged);
    const int ord = __popc(stmask & ((1u << lane) - 1u));  // ordinal among the staged jobs
    const int words = staged ? span_a + span_b : 0;
    const int w_ex = warp_incl_sum(words) - words;
    const int km = a.force_km > 0 ? a.force_km : 8;
    const int npc = staged ? (N + km - 1) / km : 0;  // merge pieces of the job
    const int p_first = warp_incl_sum(npc) - npc;
    if (staged) {
      S.jout[ord] = slot;
      S.na[ord] = na;
      S.nb[ord] = nb;
      S.pc[ord] = p_first;
      S.jcnt[ord] = 0;
      S.jlow[ord] = -1;
    }
    __syncwarp();
    unsigned rest = stmask;
    while (rest) {
      // batch: the staged jobs from lane c on whose spans fit together
      const int c = __ffs(rest) - 1;
      const int w0 = __shfl_sync(0xffffffffu, w_ex, c);
      const bool mine = staged && lane >= c && w_ex + words - w0 <= kStage;
      const unsigned bmask = __ballot_sync(0xffffffffu, mine);
      rest &= ~bmask;
      const int o0 = __popc(stmask & ((1u << c) - 1u));
      const int base = w_ex - w0;  // this job's spans in `in`
      if (mine) {
        S.ia[ord] = base + ra;
        S.ib[ord] = base + span_a + rb;
      }
      // stage: 16-byte chunks from the lists' aligned starts (the column stores carry slack
      // after their last column for the rounding); jobs of 16+ chunks by the whole warp,
      // shorter ones by their lane; all copies of the batch are in flight together
      const int ch_a = span_a >> 2;
      const int ch_n = ch_a + (B ? span_b >> 2 : 0);
      const int32_t* ga = A - ra;
      const int32_t* gb = B ? B - rb : nullptr;
      unsigned lmask = __ballot_sync(0xffffffffu, mine && ch_n >= 16);
      while (lmask) {
        const int src = __ffs(lmask) - 1;
        lmask &= lmask - 1;
        const int32_t* wa = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)ga, src);
        const int32_t* wb = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)gb, src);
        const int wca = __shfl_sync(0xffffffffu, ch_a, src);
        const int wcn = __shfl_sync(0xffffffffu, ch_n, src);
        int32_t* d = S.in + __shfl_sync(0xffffffffu, base, src);
        for (int q = lane; q < wcn; q += 32)
          cp_async16(d + 4 * q, q < wca ? wa + 4 * q : wb + 4 * (q - wca));
      }
      if (mine && ch_n < 16) {
        int32_t* d = S.in + base;
        for (int q = 0; q < ch_n; q++) cp_async16(d + 4 * q, q < ch_a ? ga + 4 * q : gb + 4 * (q - ch_a));
      }
      cp_async_wait_all();
      __syncwarp();
      if (mine) {  // the sentinels go after the copies, which may have covered their words
        S.in[base + ra + na] = INT32_MAX;
        S.in[base + span_a + rb + nb] = INT32_MAX;
      }
      __syncwarp();
      if constexpr (kLane) {  // each job by its own lane
        if (mine) {
          int32_t lastv;
          const int len = lane_merge_job(S.in, base + ra, base + span_a + rb, N, slot, &lastv);
          S.jcnt[ord] = len;
          S.jlow[ord] = lastv;
        }
      } else {  // pieces of every job spread over the lanes
        const int P0 = __shfl_sync(0xffffffffu, p_first, c);
        const int P1 = P0 + (int)__reduce_add_sync(0xffffffffu, mine ? (unsigned)npc : 0u);
        switch (km) {
          case 8: staged_rounds<8>(S, P0, P1, o0, mine, p_first, km); break;
          default: staged_rounds<0>(S, P0, P1, o0, mine, p_first, km); break;
        }
      }
      __syncwarp();
    }
    if (staged) {
      o_ptr = slot;
      o_len = S.jcnt[ord];
      low = S.jlow[ord];
    }
    // merges too long to stage: straight from global memory into their slot
    unsigned bmask = __ballot_sync(0xffffffffu, big);
    while (bmask) {
      const int src = __ffs(bmask) - 1;
      bmask &= bmask - 1;
      const int32_t* wA = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)A, src);
      const int32_t* wB = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)B, src);
      const int wna = __shfl_sync(0xffffffffu, na, src);
      const int wnb = __shfl_sync(0xffffffffu, nb, src);
      int32_t* wd = (int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)slot, src);
      int len;
      int32_t last = -1;
      if (wB) {
        len = warp_symdiff(wA, wna, wB, wnb, wd, last);
      } else {
        for (int q = lane; q < wna; q += 32) wd[q] = wA[q];
        len = wna;
      }
      if (lane == src) {
        low = last;
        o_ptr = wd;
        o_len = len;
      }
    }
  }
  // ---- bit-packed columns, one job at a time by the whole warp
  unsigned dnmask = kDense ? __ballot_sync(0xffffffffu, cls == 4) : 0u;
  while (dnmask) {
    const int src = __ffs(dnmask) - 1;
    dnmask &= dnmask - 1;
    const int32_t* wA = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)A, src);
    const int32_t* wB = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)B, src);
    const int wna = __shfl_sync(0xffffffffu, na, src);
    int32_t* wd = (int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)slot, src);
    const bool wdense_a = __shfl_sync(0xffffffffu, (int)dense_a, src) != 0;
    if (wB == nullptr) {  // a bit-packed column with nothing to add moves as it is
      for (int q = lane; q < wna; q += 32) wd[q] = wA[q];
      if (lane == src) {
        o_ptr = wd;
        o_len = dense_len(wna);
      }
      continue;
    }
    int32_t dlow, words;
    const int32_t rows = dense_job_warp(a, __shfl_sync(0xffffffffu, j, src), wA, wna, wdense_a,
                                        wB, __shfl_sync(0xffffffffu, nb, src),
                                        __shfl_sync(0xffffffffu, (int)dense_b, src) != 0, wd,
                                        wna + __shfl_sync(0xffffffffu, nb, src), dlow, words);
    if (lane == src) {
      o_ptr = wd;
      o_len = rows ? dense_len(words) : 0;  // a zero column stores nothing
      low = dlow;
    }
  }
  return cls;
}

// by thread 0, after the block's rounds: its counters into the pass's
__device__ __forceinline__ void flush_counters(const RArgs& a, const PV& v,
                                               const unsigned long long* s_cnt) {
  if (s_cnt[kCntTargets]) atomicAdd(&a.ds->targets, s_cnt[kCntTargets]);
  if (v.stats) {
    const int idx[kNumCnt] = {PH_PS_TARGETS, PH_PS_ACTIVE, PH_PS_CLEARED,
                              PH_PS_ADDS,    PH_PS_XORS,   PH_PS_COPIED, PH_PS_PACKED};
    for (int i = 0; i < kNumCnt; i++)
      if (s_cnt[i]) atomicAdd((unsigned long long*)&v.stats[idx[i]], s_cnt[i]);
  }
}

// Phase II for one chunk of the active list (128 slots of a block, or 32 of a warp). Survivors
// get their place in the next active list from a block (or warp) scan plus the look-back, and
// their rows a slot of the next arena from one atomic per chunk. New pivots are copied to the
// pivot store, one run per warp; survivors (with or without an addition) are merged in
// registers (short columns, one thread per job) or staged in shared memory and merged, each job
// by its own lane (short jobs) or by a merge path over the batch's jobs cut into pieces of km
// positions (8 unless ph_opts.merge_items says otherwise); merges longer than the staging
// bound run from global memory; bit-packed jobs run one at a time by the whole warp. Targets
// and zeroed columns are updated in place (no other job reads them this pass); new pivots and
// left-most survivors, which other jobs may be reading as sources, are updated by k_commit.
// kSlots > 0: the chunk is kSlots (32 or 8) slots of one warp, lanes kSlots.. without a job
// (warp scan, no block barrier); kSlots = 0: kBT slots of the whole block of kBT threads
template <bool kDense, int kSlots, bool kLane, int kBT>
__device__ __forceinline__ void add_chunk(const RArgs& a, const PV& v, int64_t chunk,
                                          WarpStage& S, int64_t* sh, int64_t* s_prefix,
                                          unsigned long long* s_cnt) {
  constexpr bool kWarp = kSlots > 0;
  const int lane = lane_id();
  const int64_t e = !kWarp         ? chunk * kBT + threadIdx.x
                    : kSlots == 32 ? chunk * 32 + lane
                                   : (lane < kSlots ? chunk * kSlots + lane : v.n_act);
  Job jb = job_of<kDense>(a, v, e);
  const int32_t pass = a.ds->pass;
  int64_t off, n_surv;
  int rank;
  if constexpr (kWarp) {
    // survivor ranks by ballot, arena words by a warp scan
    const unsigned survm = __ballot_sync(0xffffffffu, jb.surv);
    n_surv = __popc(survm);
    rank = __popc(survm & ((1u << lane) - 1));
    const int64_t w = jb.surv ? jb.words : 0;
    const int64_t wincl = warp_incl_sum(w);
    const int64_t wtot = __shfl_sync(0xffffffffu, wincl, 31);
    unsigned long long wbase = 0;
    if (lane == 0) {
      look_publish(a, pass, chunk, n_surv);
      // the chunk's survivors take one contiguous run of the next arena
      if (wtot) wbase = atomicAdd(&a.ds->arena_used, (unsigned long long)wtot);
    }
    off = (int64_t)__shfl_sync(0xffffffffu, wbase, 0) + wincl - w;
  } else {
    // one block scan gives both the survivor rank (high 16 bits) and the arena words (low 48)
    constexpr int kRankShift = 48;
    constexpr int64_t kWordMask = (int64_t(1) << kRankShift) - 1;
    const int64_t packed = jb.surv ? ((int64_t(1) << kRankShift) | jb.words) : 0;
    int64_t tot;
    const int64_t excl = block_excl_sum<int64_t, kBT / 32>(packed, sh, tot);
    n_surv = tot >> kRankShift;
    if (threadIdx.x == 0) {
      look_publish(a, pass, chunk, n_surv);
      // the chunk's survivors take one contiguous run of the next arena
      s_prefix[1] = (tot & kWordMask) ? (int64_t)atomicAdd(&a.ds->arena_used,
                                                           (unsigned long long)(tot & kWordMask))
                                      : 0;
    }
    __syncthreads();
    off = s_prefix[1] + (excl & kWordMask);
    rank = (int)(excl >> kRankShift);
  }

#ifdef PH_DEBUG
  // the job's slot lies in the arena this pass writes (else the job is dropped and reported)
  if (jb.surv && !PH_DCHECK(&a.ds->debug_fault, off >= 0 && off + jb.words <= v.arena_next_cap, 3)) {
    jb.surv = false;
    jb.newpiv = false;
  }
#endif
  const int32_t* A = jb.A;
  const int32_t* B = jb.B;
  const int na = jb.na, nb = jb.nb;
  int32_t* o_ptr = nullptr;  // the column's new place and length
  int o_len = 0;

  // ---- new pivots: their columns never change again; move them to the pivot store (a
  // bit-packed column moves as its stored words)
  unsigned pmask = __ballot_sync(0xffffffffu, jb.newpiv);
  if (pmask) {  // the warp's new pivots take one run of the pivot store
    const int mine = jb.newpiv ? na : 0;
    const int incl = warp_incl_sum(mine);
    const int ptot = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long w0 = 0;
    if (lane == 0) w0 = atomicAdd(&a.ds->piv_used, (unsigned long long)ptot);
    w0 = __shfl_sync(0xffffffffu, w0, 0) + (unsigned long long)(incl - mine);
#ifdef PH_DEBUG
    // the warp's run lies in the pivot store's chunk (else the warp's copies are dropped)
    const bool in_store = PH_DCHECK(&a.ds->debug_fault, (int64_t)(w0 + mine) <= v.piv_cap, 4);
    if (!__all_sync(0xffffffffu, in_store)) pmask = 0;
#endif
    if (jb.newpiv) o_ptr = v.piv_base + w0;
  }
  while (pmask) {
    const int src = __ffs(pmask) - 1;
    pmask &= pmask - 1;
    const int32_t* wA = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)A, src);
    const int wna = __shfl_sync(0xffffffffu, na, src);
    int32_t* dst = (int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)o_ptr, src);
    for (int q = lane; q < wna; q += 32) dst[q] = wA[q];
    if (lane == src) {
      o_ptr = dst;
      o_len = kDense && jb.dense_a ? dense_len(wna) : wna;
    }
  }

  // ---- survivors: every job writes into its own reserved slot of the next arena
  int cls = 0;
  {
    int32_t* m_ptr;
    int m_len;
    int32_t low;
    cls = merge_rows<kDense, kWarp ? kSlots : 32, kLane>(
        a, v, S, jb.j, jb.surv ? v.arena_next + off : nullptr, A, na, jb.dense_a, B, nb, jb.dense_b,
        m_ptr, m_len, low);
    if (jb.surv) {
      o_ptr = m_ptr;
      o_len = m_len;
      if (B) {
        a.low[jb.j] = low;
        next_tab<true>(a, v, low, jb.j);
      }
    }
  }
  // ---- the survivors' places in the next active list
  if constexpr (kWarp) {
    const int64_t pre = look_back(a, pass, chunk, n_surv);
    if (jb.surv && PH_DCHECK(&a.ds->debug_fault, pre + rank < v.n_act, 5)) {
      v.act2[pre + rank] = jb.j;
      v.alen2[pre + rank] = o_len;
    }
  } else {
    if (threadIdx.x < 32) {
      const int64_t pre = look_back(a, pass, chunk, n_surv);
      if (threadIdx.x == 0) s_prefix[0] = pre;
    }
    __syncthreads();
    if (jb.surv && PH_DCHECK(&a.ds->debug_fault, s_prefix[0] + rank < v.n_act, 5)) {
      v.act2[s_prefix[0] + rank] = jb.j;
      v.alen2[s_prefix[0] + rank] = o_len;
    }
  }
  // ---- publish: in place for targets and zeroed columns, through k_commit for the others
  if (jb.surv && B == nullptr) next_tab<false>(a, v, a.low[jb.j], jb.j);  // its low stays
  if (jb.j >= 0) {
    if (jb.surv && jb.target) {
      a.meta[jb.j].ptr = o_ptr;
      a.meta[jb.j].len = o_len;
    } else if (!jb.surv && !jb.newpiv) {
      a.meta[jb.j].flags |= F_FINAL;
      a.low[jb.j] = -1;
      a.meta[jb.j].len = 0;
    }
  }
  const bool defer = jb.newpiv || (jb.surv && !jb.target);
  const unsigned dmask = __ballot_sync(0xffffffffu, defer);
  if (dmask) {
    int d0 = 0;
    if (lane == __ffs(dmask) - 1) d0 = atomicAdd(&a.ds->n_deferred, __popc(dmask));
    d0 = __shfl_sync(0xffffffffu, d0, __ffs(dmask) - 1);
    if (defer) {
      d0 += __popc(dmask & ((1u << lane) - 1));
      a.dlist[d0] = jb.j;
      a.nxt_ptr[d0] = o_ptr;
      a.nxt_len[d0] = o_len;
    }
  }
  // ---- counters, per warp into the block's shared totals
  const int n_tgt = __popc(__ballot_sync(0xffffffffu, jb.target));
  if (lane == 0 && n_tgt) atomicAdd(&s_cnt[kCntTargets], (unsigned long long)n_tgt);
  if (v.stats) {
    const bool add = jb.surv && B != nullptr;
    const bool copy = jb.newpiv || (jb.surv && B == nullptr);
    const int n_act = __popc(__ballot_sync(0xffffffffu, jb.j >= 0));
    const int n_clr = __popc(__ballot_sync(0xffffffffu, jb.j >= 0 && a.meta[jb.j].cleared));
    const int n_add = __popc(__ballot_sync(0xffffffffu, add));
    const int n_pk = kDense ? __popc(__ballot_sync(0xffffffffu, add && cls == 4)) : 0;
    // row counts: a bit-packed column keeps its own in its header
    const int ra = kDense && jb.dense_a ? A[0] : na;
    const int64_t xr = warp_sum64(
        add ? (ra + (kDense && jb.dense_b ? B[0] : nb) + (kDense && o_len < 0 ? o_ptr[0] : o_len)) / 2
            : 0);
    const int64_t cp = warp_sum64(copy ? ra : 0);
    if (lane == 0) {
      atomicAdd(&s_cnt[kCntActive], (unsigned long long)n_act);
      atomicAdd(&s_cnt[kCntCleared], (unsigned long long)n_clr);
      atomicAdd(&s_cnt[kCntAdds], (unsigned long long)n_add);
      atomicAdd(&s_cnt[kCntXors], (unsigned long long)xr);
      atomicAdd(&s_cnt[kCntCopied], (unsigned long long)cp);
      if (n_pk) atomicAdd(&s_cnt[kCntPacked], (unsigned long long)n_pk);
    }
  }
}

// one pass's additions, by every block of the grid. kLoop: in the loop kernel (every block resident),
// where chunks are dealt out in order; otherwise they are claimed in order from a work queue
template <bool kDense, int kSlots, bool kLane, int kBT, bool kLoop>
__device__ __forceinline__ void add_pass(const RArgs& a, WarpStage& S, unsigned blocks) {
  constexpr bool kWarp = kSlots > 0;
  __shared__ int64_t sh[kBT / 32 + 1];
  __shared__ int64_t s_chunk;
  __shared__ int64_t s_prefix[2];
  __shared__ unsigned long long s_cnt[kNumCnt];
  __shared__ PV s_v;  // per-pass values from shared memory rather than held in registers
  if (threadIdx.x == 0) s_v = pass_view(a.ds);
  if (blockIdx.x == 0 && threadIdx.x == 0) a.ds->chunk_slots = kWarp ? kSlots : kBT;
  const PV& v = s_v;
  if (threadIdx.x < kNumCnt) s_cnt[threadIdx.x] = 0;
  if constexpr (kWarp) {
    __syncthreads();  // publishes s_v and the zeroed counters
    const int64_t nchunks = (v.n_act + kSlots - 1) / kSlots;
    unsigned int next = (threadIdx.x >> 5) * blocks + blockIdx.x;
    for (;;) {  // chunks of kSlots slots for whole warps
      unsigned int chunk = next;
      if (kLoop) {
        next += blocks * (kBT / 32);
      } else {
        if (lane_id() == 0) chunk = atomicAdd(&a.ds->queue, 1u);
        chunk = __shfl_sync(0xffffffffu, chunk, 0);
      }
      if ((int64_t)chunk >= nchunks) break;
      add_chunk<kDense, kSlots, kLane, kBT>(a, v, chunk, S, sh, s_prefix, s_cnt);
    }
    __syncthreads();
  } else {
    for (;;) {  // chunks of kBT slots for the whole block
      if (threadIdx.x == 0) s_chunk = atomicAdd(&a.ds->queue, 1u);
      __syncthreads();  // also publishes s_v, written by thread 0 before the loop
      const int64_t chunk = s_chunk;
      const int64_t nchunks = (v.n_act + kBT - 1) / kBT;
      __syncthreads();
      if (chunk >= nchunks) break;
      add_chunk<kDense, 0, kLane, kBT>(a, v, chunk, S, sh, s_prefix, s_cnt);
    }
  }
  if (threadIdx.x == 0) flush_counters(a, v, s_cnt);
}

// kDense: the pass may meet bit-packed columns or convert some; the row-list variant carries none
// of it. kSlots: chunks of kSlots (32 or 8) slots claimed by single warps, 0: chunks of 128 slots
// claimed by blocks. kLane: each staged job merged by its own lane (short columns), else merge
// pieces spread over the lanes. The host picks the variant from DevState::dense_on, warp_on,
// narrow_on and lane_on (a separate graph for each).
template <bool kDense, int kSlots, bool kLane, int kBT = kAddThreads>
__global__ void __launch_bounds__(kBT, 1024 / kBT) k_add(RArgs a) {
  extern __shared__ __align__(16) unsigned char add_smem[];
  pdl_wait();
  pdl_trigger();
  if (a.ds->status != ST_RUN) return;
  add_pass<kDense, kSlots, kLane, kBT, false>(
      a, reinterpret_cast<WarpStage*>(add_smem)[threadIdx.x >> 5], gridDim.x);
}

// what k_merge does with a column
enum : uint8_t {
  kNothing = 0,
  kMerge,     // its delta goes into its list
  kAdd,       // the source whose id is in its delta's first place is added to its list
  kMove,      // its list moves to this pass's arena
  kMoveLate,  // ... but others may be reading it in this pass: published by k_commit
};

// Phase II with look-ahead, first half: every column that is due gets its source for this pass. A
// source of few rows starts a visit (look_ahead), which leaves the column's list as it is, only
// shortened, and its delta beside it; the columns whose list has to be rewritten, or whose source is
// too long for a visit, are left to k_merge. In a pass that compacts that is every survivor: its
// place in the next active list comes from Phase I (newpos). New pivots are
// copied to the pivot store. Targets and zeroed columns are updated in place (no other job reads
// them this pass); new pivots and left-most survivors, which other jobs may be reading as
// sources, are updated by k_commit.
struct VisitStage {
  int32_t pend[32 + kScan];  // slots gathered for the next rounds
};

// by one warp. e, j: this lane's slot and its column (-1: none), which is due
__device__ __forceinline__ void visit_round(const RArgs& a, const PV& v, int32_t e, int32_t j,
                                            unsigned long long* s_cnt) {
  constexpr int R = kSourceRows, kNew = R * kAheadMax;
  const int lane = lane_id();
  const int32_t pass = a.ds->pass;
  // every load is issued up front: the column, its low and its source candidate are known from
  // the active list, the stored lows and k_phase1's per-slot source, so no load waits on
  // another's result
  Visit w;
  bool surv = false, newpiv = false, target = false, add = false, eager = false, dense_a = false;
  int32_t s = -1;
  w.low = -1;
  w.na = w.nb = w.k = 0;
  w.A = w.B = nullptr;
  w.rec = make_int4(0, 0, 0, 0);
  w.gone = w.settle = false;
  // its place in the next active list: compacted, or where it is (a due column's low is its own)
  int64_t pos = e;
  if (j >= 0) {
    w.low = a.low[j];
    if (v.compact) pos = a.newpos[e];
    const int32_t se = a.src_e[e];  // -1: no collision; <= -2: a target whose set waits
    const ColMeta mj = load_meta(a.meta + j);
    if (se >= 0) w.rec = a.prec[w.low];
    newpiv = (mj.flags & F_NEWPIV) != 0;
    surv = !(mj.flags & (F_PROVEN | F_FINAL)) && !mj.cleared;
    target = surv && se != -1;
    dense_a = mj.len < 0;
    w.A = mj.ptr;
    w.na = stored_words(mj.len);
    w.k = mj.spare;
    if (target && se >= 0 && v.do_adds) {
      s = se;
      if (w.rec.x > 0 && w.rec.x <= R + 1) {  // a proven pivot's record says it all
        add = true;
        eager = dense_a;
      } else {
        const ColMeta ms = load_meta(a.meta + s);
        add = !(ms.flags & F_FINAL) && !ms.cleared && (!a.strict || (ms.flags & F_PROVEN));
        w.B = ms.ptr;
        w.nb = ms.len;
        eager = add && (dense_a || ms.len < 0 || ms.len > kNew + 1);
      }
    }
  }
  w.due = pass + 1;
  const int na0 = w.na;
  const bool visit = add && !eager;
  bool no_beta = false;  // Corollary 10 may zero it
  if (__any_sync(0xffffffffu, visit)) {
    int32_t* block = a.delta + (int64_t)max(j, 0) * kDeltaRows;
#pragma unroll
    for (int i = 0; i < kOld; i += 4) {
      int4 x = make_int4(INT32_MAX, INT32_MAX, INT32_MAX, INT32_MAX);
      if (visit && i < w.k) x = *reinterpret_cast<const int4*>(block + i);
      w.d.c[i] = -x.x;
      w.d.c[i + 1] = i + 1 < w.k ? -x.y : kEmpty;
      w.d.c[i + 2] = i + 2 < w.k ? -x.z : kEmpty;
      w.d.c[i + 3] = i + 3 < w.k ? -x.w : kEmpty;
    }
#pragma unroll
    for (int i = kOld; i < kDeltaRows; i++) w.d.c[i] = kEmpty;
    const bool c10 = visit && a.cor10 && a.beta[j] < 0;
    no_beta = c10;
    // (at the time bound the loop may stop before the pass that zeroes the column: it keeps its rows)
    const int32_t fu = c10 && !a.ds->drain ? a.first_unp[seg_of(a, j) - a.nc] : INT32_MIN;
    if (look_ahead(a, v, pass, visit, fu, pos, w)) tidy<0>(w, visit && !w.gone);
    else tidy<kOld>(w, visit && !w.gone);
    if (visit) {
#pragma unroll
      for (int i = 0; i < kDeltaRows; i += 4)
        if (i < w.k)
          *reinterpret_cast<int4*>(block + i) =
              make_int4(w.d.c[i], w.d.c[i + 1], w.d.c[i + 2], w.d.c[i + 3]);
    }
  }

  // what is left to k_merge: a compacting pass rewrites every list, another one those whose delta
  // is full or that have to be whole; at the cap the lists are what the caller can read
  int kind = kNothing;
  if (eager) {
    kind = kAdd;
    a.delta[(int64_t)j * kDeltaRows] = s;
  } else if (visit) {
    if (!w.gone && (v.compact || w.k > kOld ||
                    (w.k > 0 && (w.settle || v.whole))))
      kind = kMerge;
  } else if (surv && v.compact) {
    kind = target ? kMove : kMoveLate;
  }
  if (v.compact) {
    if (j >= 0 && pos >= 0 && PH_DCHECK(&a.ds->debug_fault, pos < v.n_act, 5)) {
      v.act2[pos] = surv ? j : dead_slot(j);
      if (!surv) a.due[pos] = kDeadDue;
      v.alen2[pos] = w.na;
      a.kind[pos] = (uint8_t)kind;
    }
  } else {
    if (j >= 0 && !surv) {
      v.act[e] = dead_slot(j);
      a.due[e] = kDeadDue;
    }
    if (visit) v.alen[e] = w.na;
    const unsigned km = __ballot_sync(0xffffffffu, kind != kNothing);
    if (km) {
      unsigned int base = 0;
      if (lane == 0) base = atomicAdd(&a.ds->n_work, (unsigned int)__popc(km));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (kind) {
        a.work[base + __popc(km & ((1u << lane) - 1))] = e;
        a.kind[e] = (uint8_t)kind;
      }
    }
  }

  // ---- new pivots: their columns never change again; move them to the pivot store (a
  // bit-packed column moves as its stored words)
  int32_t* p_ptr = nullptr;
  unsigned pmask = __ballot_sync(0xffffffffu, newpiv);
  if (pmask) {  // the warp's new pivots take one run of the pivot store
    const unsigned all = pmask;
    const int mine = newpiv ? na0 : 0;
    const int incl = warp_incl_sum(mine);
    const int ptot = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long w0 = 0;
    int d0 = 0;
    if (lane == 0) {
      w0 = atomicAdd(&a.ds->piv_used, (unsigned long long)ptot);
      d0 = atomicAdd(&a.ds->n_deferred, __popc(all));
    }
    w0 = __shfl_sync(0xffffffffu, w0, 0) + (unsigned long long)(incl - mine);
    d0 = __shfl_sync(0xffffffffu, d0, 0) + __popc(all & ((1u << lane) - 1));
#ifdef PH_DEBUG
    // the warp's run lies in the pivot store's chunk (else the warp's copies are dropped)
    const bool in_store = PH_DCHECK(&a.ds->debug_fault, (int64_t)(w0 + mine) <= v.piv_cap, 4);
    if (!__all_sync(0xffffffffu, in_store)) pmask = 0;
#endif
    if (newpiv) {
      p_ptr = v.piv_base + w0;
      a.dlist[d0] = j;
      a.nxt_ptr[d0] = p_ptr;
      a.nxt_len[d0] = dense_a ? dense_len(na0) : na0;
    }
  }
  while (pmask) {
    const int src = __ffs(pmask) - 1;
    pmask &= pmask - 1;
    const int32_t* wA = (const int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)w.A, src);
    const int wna = __shfl_sync(0xffffffffu, na0, src);
    int32_t* dst = (int32_t*)__shfl_sync(0xffffffffu, (unsigned long long)p_ptr, src);
    for (int q = lane; q < wna; q += 32) dst[q] = wA[q];
  }

  // ---- publish: the lows of the coming passes (k_merge knows those of its additions), a visited
  // column's shortened list and its delta, a zeroed column
  if (surv && PH_DCHECK(&a.ds->debug_fault, pos >= 0 && pos < v.n_act, 5)) {
    a.due[pos] = no_beta ? ~w.due : w.due;
    if (visit) {
      if (w.due == pass + 1) next_tab<true>(a, v, w.low, j);
    } else if (!eager) {  // its low stays
      a.lows[(int64_t)((pass + 1) & a.ring) * a.lows_stride + pos] = w.low;
      next_tab<false>(a, v, w.low, j);
    }
  }
  if (visit) {
    a.low[j] = w.low;
    a.meta[j].len = w.na;
    a.meta[j].spare = (uint8_t)w.k;
  } else if (j >= 0 && !surv && !newpiv) {
    a.meta[j].flags |= F_FINAL;
    a.low[j] = -1;
    a.meta[j].len = 0;
  }
  // ---- counters, per warp into the block's shared totals
  const int n_tgt = __popc(__ballot_sync(0xffffffffu, target));
  if (lane == 0 && n_tgt) atomicAdd(&s_cnt[kCntTargets], (unsigned long long)n_tgt);
}

// one pass's visits, by every block of the grid
__device__ __forceinline__ void visit_pass(const RArgs& a, VisitStage& S, unsigned blocks) {
  __shared__ unsigned long long s_cnt[kNumCnt];
  __shared__ PV s_v;  // per-pass values from shared memory rather than held in registers
  if (threadIdx.x == 0) s_v = pass_view(a.ds);
  const PV& v = s_v;
  const int lane = lane_id();
  const int warps = blockDim.x >> 5;
  if (threadIdx.x < kNumCnt) s_cnt[threadIdx.x] = 0;
  __syncthreads();  // publishes s_v and the zeroed counters
  // A pass that compacts: every column is due, 32 slots per round. Otherwise few columns are due: those
  // that Phase I listed, and those among the first scan_end slots, where every warp looks through its
  // share and gathers the due ones for full rounds. A column ahead of the pass stays a target, unless
  // clearing zeroes it (only below the top dimension); its last stored low enters the next pass's
  // table when it is due then. (With every slot looked through, a pass of 10.67 M columns took 41 us.)
  const int32_t pass = a.ds->pass;
  const int32_t* lows_next = a.lows + (int64_t)((pass + 1) & a.ring) * a.lows_stride;
  const int64_t warp = (int64_t)blockIdx.x * warps + (threadIdx.x >> 5);
  int64_t i0 = warp * (v.compact ? 32 : kScan), k0 = warp * 32;
  const int64_t n_due = a.ds->n_due, scan_end = a.ds->scan_end;
  int np = 0, n_tgt = 0;
  if (!v.compact) {
    const int64_t n_enter = a.ds->n_enter;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n_enter;
         k += (int64_t)blocks * blockDim.x) {
      const int32_t x = v.act2[k];
      next_tab<true>(a, v, lows_next[x], v.act[x]);
    }
  }
  for (;;) {
    int32_t e = 0, jv = -1;
    if (v.compact) {
      if (i0 >= v.n_act) break;
      const int64_t x = i0 + lane;
      i0 += (int64_t)blocks * warps * 32;
      if (x < v.n_act) {
        e = (int32_t)x;
        jv = max(v.act[e], -1);
      }
    } else {
      for (; np < 32 && i0 < scan_end; i0 += (int64_t)blocks * warps * kScan) {
        // only columns below the top dimension can be cleared: those of the others are not read
        const bool below = slot_id(v.act[i0]) < a.rows_end;
        int32_t ds[kScan / 32];
#pragma unroll
        for (int u = 0; u < kScan / 32; u++) {
          const int64_t x = i0 + 32 * u + lane;
          ds[u] = x < scan_end ? a.due[x] : kDeadDue;
        }
#pragma unroll
        for (int u = 0; u < kScan / 32; u++) {
          const int32_t x = (int32_t)(i0 + 32 * u + lane);
          const int32_t d = due_pass(ds[u]);
          if (d > pass && d != kDeadDue) {
            const bool enters = d == pass + 1;
            const int32_t j = below || enters ? v.act[x] : INT32_MAX;
            if (below && j < a.rows_end && a.meta[j].cleared) {
              a.meta[j].flags |= F_FINAL;
              a.meta[j].len = 0;
              a.low[j] = -1;
              v.act[x] = dead_slot(j);
              a.due[x] = kDeadDue;
            } else {
              n_tgt++;
              if (enters) next_tab<true>(a, v, lows_next[x], j);
            }
          }
          const unsigned m = __ballot_sync(0xffffffffu, d <= pass);
          if (d <= pass) S.pend[np + __popc(m & ((1u << lane) - 1u))] = x;
          np += __popc(m);
        }
        __syncwarp();
      }
      if (np > 0) {
        const int n = min(np, 32);
        np -= n;
        if (lane < n) {
          e = S.pend[np + lane];
          jv = v.act[e];
        }
        __syncwarp();
      } else {  // then the columns that Phase I listed
        if (k0 >= n_due) break;
        if (k0 + lane < n_due) {
          e = a.newpos[k0 + lane];
          jv = v.act[e];
        }
        k0 += (int64_t)blocks * warps * 32;
      }
    }
    visit_round(a, v, e, jv, s_cnt);
  }
  if (!v.compact) {
    const unsigned t = __reduce_add_sync(0xffffffffu, (unsigned)n_tgt);
    if (lane == 0 && t) atomicAdd(&s_cnt[kCntTargets], (unsigned long long)t);
  }
  __syncthreads();
  if (threadIdx.x == 0) flush_counters(a, v, s_cnt);
}

__global__ void __launch_bounds__(kAddThreads, 1024 / kAddThreads) k_visit(RArgs a) {
  __shared__ VisitStage s_stage[kAddWarps];
  pdl_wait();
  pdl_trigger();
  if (a.ds->status != ST_RUN) return;
  visit_pass(a, s_stage[threadIdx.x >> 5], gridDim.x);
}

// the places of the next active list in a pass that compacts: the inclusive prefix that the last
// chunk of k_add, or with look-ahead Phase I's last tile, published in its look-back (false: there
// is none, an internal error)
__device__ __forceinline__ bool survivors(const RArgs& a, const DevState* ds, int64_t n_act,
                                          int32_t ahead, int32_t pass, int64_t& n) {
  const int64_t per = ahead > 1 ? kFTile : ds->chunk_slots;
  const int64_t nch = (n_act + per - 1) / per;
  n = 0;
  if (nch == 0) return true;
  const unsigned long long w = *(const volatile unsigned long long*)(a.look + nch - 1);
  if ((w >> 40) != (look_tag(pass) >> 40) || (w & kLookFlags) != kLookIncl) return false;
  n = (int64_t)(w & kLookVal);
  return true;
}

// Phase II with look-ahead, second half, by one warp: the lists of columns that k_visit left to it.
// pos: this lane's slot, kind: what to do with its column. The warp's jobs take one contiguous run
// of the arena, from one atomic.
template <bool kDense, bool kLane>
__device__ __forceinline__ void merge_round(const RArgs& a, const PV& v, int32_t pos, int kind,
                                            WarpStage& S) {
  const int lane = lane_id();
  int32_t j = -1;
  const int32_t* A = nullptr;
  const int32_t* B = nullptr;
  int na = 0, nb = 0;
  bool dense_a = false, dense_b = false;
  if (kind) {
    j = (v.compact ? v.act2 : v.act)[pos];
    const ColMeta mj = load_meta(a.meta + j);
    A = mj.ptr;
    na = kDense ? stored_words(mj.len) : mj.len;
    dense_a = kDense && mj.len < 0;
    if (kind == kMerge) {
      B = a.delta + (int64_t)j * kDeltaRows;
      nb = mj.spare;
    } else if (kind == kAdd) {
      const ColMeta ms = load_meta(a.meta + a.delta[(int64_t)j * kDeltaRows]);
      B = ms.ptr;
      nb = kDense ? stored_words(ms.len) : ms.len;
      dense_b = kDense && ms.len < 0;
    }
  }
  const int64_t words = kind ? na + nb : 0;
  const int64_t wincl = warp_incl_sum(words);
  const int64_t wtot = __shfl_sync(0xffffffffu, wincl, 31);
  unsigned long long wbase = 0;
  if (lane == 0 && wtot) wbase = atomicAdd(&a.ds->arena_used, (unsigned long long)wtot);
  const int64_t off = (int64_t)__shfl_sync(0xffffffffu, wbase, 0) + wincl - words;
#ifdef PH_DEBUG
  // the job's slot lies in the arena this pass writes (else the job is dropped and reported)
  if (kind && !PH_DCHECK(&a.ds->debug_fault, off >= 0 && off + words <= v.arena_next_cap, 3)) {
    kind = kNothing;
    j = -1;
  }
#endif
  int32_t* o_ptr;  // the column's new place, length and low
  int o_len;
  int32_t low;
  merge_rows<kDense, 32, kLane>(a, v, S, j, kind ? v.arena_next + off : nullptr, A, na,
                                                dense_a, B, nb, dense_b, o_ptr, o_len, low);
  // ---- publish
  if (kind) {
    (v.compact ? v.alen2 : v.alen)[pos] = o_len;
    if (kind != kMoveLate) {
      a.meta[j].ptr = o_ptr;
      a.meta[j].len = o_len;
    }
    if (kind == kMerge) a.meta[j].spare = 0;
    if (kind == kAdd) {
      a.low[j] = low;
      a.lows[(int64_t)((a.ds->pass + 1) & a.ring) * a.lows_stride + pos] = low;
      next_tab<true>(a, v, low, j);
    }
  }
  const unsigned dmask = __ballot_sync(0xffffffffu, kind == kMoveLate);
  if (dmask) {
    int d0 = 0;
    if (lane == 0) d0 = atomicAdd(&a.ds->n_deferred, __popc(dmask));
    d0 = __shfl_sync(0xffffffffu, d0, 0) + __popc(dmask & ((1u << lane) - 1));
    if (kind == kMoveLate) {
      a.dlist[d0] = j;
      a.nxt_ptr[d0] = o_ptr;
      a.nxt_len[d0] = o_len;
    }
  }
}

// kDense: the pass may meet bit-packed columns or convert some; the row-list variant carries none
// of it. kLane: each staged job merged by its own lane (short columns), else merge pieces spread over the
// lanes. The host picks the variant from DevState::dense_on and lane_on (a separate graph for each).
template <bool kDense, bool kLane>
__device__ __forceinline__ void merge_pass(const RArgs& a, WarpStage& S, unsigned blocks) {
  __shared__ PV s_v;  // per-pass values from shared memory rather than held in registers
  if (threadIdx.x == 0) s_v = pass_view(a.ds);
  const PV& v = s_v;
  const int lane = lane_id();
  __syncthreads();  // publishes s_v
  int64_t n = 0;
  if (!v.compact) n = a.ds->n_work;
  else if (!survivors(a, a.ds, v.n_act, v.ahead, a.ds->pass, n)) a.ds->fault = 1;
  // full rounds, or the few columns spread over all warps
  const int64_t warps = (int64_t)blocks * (blockDim.x >> 5);
  const int per = (int)std::min<int64_t>(32, (n + warps - 1) / warps);
  for (int64_t i = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per; i < n;
       i += warps * per) {
    const bool mine = lane < per && i + lane < n;
    const int32_t pos = !mine ? 0 : v.compact ? (int32_t)(i + lane) : a.work[i + lane];
    merge_round<kDense, kLane>(a, v, pos, mine ? a.kind[pos] : kNothing, S);
    __syncwarp();
  }
}

template <bool kDense, bool kLane>
__global__ void __launch_bounds__(kAddThreads, 1024 / kAddThreads) k_merge(RArgs a) {
  extern __shared__ __align__(16) unsigned char add_smem[];
  pdl_wait();
  pdl_trigger();
  if (a.ds->status != ST_RUN) return;
  merge_pass<kDense, kLane>(a, reinterpret_cast<WarpStage*>(add_smem)[threadIdx.x >> 5],
                                    gridDim.x);
}

// |E^l| after this pass's marks (per-pass counter; only with collect_stats)
__device__ __forceinline__ void ess_count(const RArgs& a, int64_t m, unsigned blocks) {
  __shared__ int64_t sh[kWarps + 1];
  int64_t n = 0;
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < m;
       x += (int64_t)blocks * blockDim.x)
    n += in_essential_estimate(load_meta(a.meta + x), a.beta[x], a.owner[x]);
  int64_t tot;
  block_excl_sum<int64_t>(n, sh, tot);
  if (threadIdx.x == 0 && tot)
    atomicAdd((unsigned long long*)&a.ds->stats[(int64_t)a.ds->pass * PH_PS_N + PH_PS_ESS_EST],
              (unsigned long long)tot);
}

__global__ void k_ess_count(RArgs a, int64_t m) {
  pdl_wait();
  pdl_trigger();
  if (a.ds->status != ST_RUN) return;
  ess_count(a, m, gridDim.x);
}

CloudIds cloud_ids(const ph_ctx* ctx, int32_t cloud) {
  CloudIds c;
  c.nd = ctx->max_dim + 1;
  for (int d = 0; d < c.nd; d++) {
    const int64_t* s = &ctx->seg_start[(int64_t)d * ctx->n_clouds + cloud];
    c.first[d] = c.n;
    c.lo[d] = s[0];
    c.n += s[1] - s[0];
  }
  c.first[c.nd] = c.n;
  return c;
}

// E^l of a cloud's ids, as bytes at their filtration index
__global__ void k_ess_flags(CloudIds ids, const ColMeta* __restrict__ meta,
                            const int32_t* __restrict__ beta, const int32_t* __restrict__ owner,
                            const int64_t* __restrict__ gidx, int64_t n, uint8_t* out,
                            int32_t* bad) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ids.n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = ids.id(t);
    const int64_t g = gidx[x];
    if (g < 0 || g >= n) {
      *bad = 1;
      continue;
    }
    out[g] = in_essential_estimate(load_meta(meta + x), beta[x], owner[x]) ? 1 : 0;
  }
}

// where a pass runs: host-driven, in the graph's loop (which stops when another variant of the
// additions, or the loop kernel, suits the next passes better), in the loop kernel
enum : int { kHostLoop = 0, kInGraph = 1, kInLoop = 2 };
__device__ void end_of_pass(const RArgs& a, cudaGraphConditionalHandle cond, int mode);

// the counters a pass accumulates, cleared for the next one
__host__ __device__ inline void reset_counters(DevState* ds) {
  ds->bound_words = 0;
  ds->bound_piv = 0;
  ds->queue = 0;
  ds->tile_queue = 0;
  ds->n_deferred = 0;
  ds->n_work = 0;
  ds->n_dirty = 0;
  ds->n_due = ds->n_enter = ds->scan_end = 0;
  ds->targets = 0;
}

// the deferred column updates and the next pass's row state, then (last block) the end of the
// pass and the reset of the per-pass counters. A pass stopped for space (ST_HOST) continues at
// Phase II on the row state it had, so neither is touched then (the host resets the counters).
__device__ __forceinline__ void commit_pass(const RArgs& a, unsigned blocks) {
  DevState* ds = a.ds;
  const int64_t n = (int64_t)ds->n_deferred;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)blocks * blockDim.x) {
    const int32_t j = a.dlist[i];
    const ColMeta mj = load_meta(a.meta + j);
    a.meta[j].ptr = a.nxt_ptr[i];
    a.meta[j].len = a.nxt_len[i];
    if (mj.flags & F_NEWPIV) {  // a long pivot's record points to its rows
      if (ds->ahead > 1 && mj.len > kRecRows) a.prec[a.low[j]] = rec_of(a.nxt_ptr[i], mj.len);
      a.meta[j].flags = (uint8_t)(mj.flags & ~F_NEWPIV);
    }
  }
  next_unpaired(a, blocks);
  if (a.predict) rows_of_pass<false>(a, blocks);
}
// by the last block
__device__ __forceinline__ void commit_last(const RArgs& a, cudaGraphConditionalHandle cond,
                                            int mode, unsigned blocks) {
  const bool run = a.ds->status == ST_RUN;
  if (run) {
    rows_of_pass_last(a);
    next_unpaired_last(a, blocks);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    end_of_pass(a, cond, mode);
    if (run) reset_counters(a.ds);
  }
}

__global__ void k_commit(RArgs a, cudaGraphConditionalHandle cond, int mode) {
  pdl_wait();
  DevState* ds = a.ds;
  if (ds->status == ST_RUN) commit_pass(a, gridDim.x);
  if (last_block(&ds->blocks_done, gridDim.x)) {
    if (threadIdx.x == 0) ds->blocks_done = 0;
    commit_last(a, cond, mode, gridDim.x);
  }
}

// ------------------------------------------------------------------------------------------
// the pass loop in one kernel
// ------------------------------------------------------------------------------------------
// On a short active list a pass's kernels take some microseconds each, whatever they do: launch,
// first loads, last-block handshakes, drain. k_loop runs all passes in one cooperative grid
// (every block resident, so they may wait for each other), the parts of a pass separated by
// grid barriers. Bound by latency: a pass is a chain of some forty loads and atomics that wait for
// L2, and three barriers (10,700 columns: 3.5 us Phase I, 7 us additions, 2 us commit, 8 us barriers
// and the end of the pass). As kernels of a graph 18 passes of 10,700 columns took 739 us, here 490;
// 237 passes of a 96 x 80 image grid 6.6 ms, here 2.6 to 3.1.
//
// A grid barrier is one counter: every block adds one and waits until all of the pass's blocks have,
// that many times the barriers so far (`target`). What was written before it is visible after it.
// The last barrier of a pass (grid_last) runs `tail` in the block that arrives last, which then
// clears the counter and lets the others go by a second word. The waits are bounded: a block that
// gives up records a fault, and both return false.
__device__ __forceinline__ bool poll_until(DevState* ds, const unsigned int* p, unsigned int value,
                                           bool at_least) {
  for (int it = 0; it < kBarrierLimit; it++) {
    const unsigned int x = *(const volatile unsigned int*)p;
    if (at_least ? x >= value : x != value) return true;
  }
  ds->fault = 1;
  return false;
}
__device__ __forceinline__ bool grid_sync(DevState* ds, unsigned blocks, unsigned int& target) {
  if (blocks == 1) {
    __syncthreads();
    return true;
  }
  target += blocks;
  bool ok = true;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&ds->bar_count, 1u);
    ok = poll_until(ds, &ds->bar_count, target, true);
    __threadfence();
  }
  return __syncthreads_and(ok);
}
template <typename F>
__device__ __forceinline__ bool grid_last(DevState* ds, unsigned blocks, unsigned int target,
                                          unsigned int& gen, F tail) {
  __shared__ int s_last;
  __syncthreads();
  if (blocks == 1) {
    tail();
    __syncthreads();
    return true;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&ds->bar_count, 1u) == target + blocks - 1;
  }
  __syncthreads();
  bool ok = true;
  if (s_last) {
    __threadfence();
    tail();
    __syncthreads();
    if (threadIdx.x == 0) {
      ds->bar_count = 0;
      __threadfence();
      atomicExch(&ds->bar_gen, gen + 1);
    }
  } else if (threadIdx.x == 0) {
    ok = poll_until(ds, &ds->bar_gen, gen, false);
    __threadfence();
  }
  gen++;
  return __syncthreads_and(ok);
}

// A call that begins with up to kLoopStart columns runs in k_loop alone: it saves the graph's launch
// and the return to the host, while its passes over long lists are slower than the graph's. Graph ->
// k_loop: 85,400 columns 881 -> 853 and 733 -> 715 us, 65,856 of a batch 402 -> 361; 102,425 columns
// 875 -> 799, but 495 -> 527 where lists stay long; 121,575 columns 1078 -> 1052, but 366 -> 443; 166,750
// columns, 8 passes, 336 -> 431. A call that begins in the graph goes over to it at kLoopBelow columns
// (16,384 to 65,536 measure alike, 131,072 costs 50 to 90 us).
constexpr int64_t kLoopBelow = (int64_t)1 << 14;
constexpr int64_t kLoopStart = 110000;
// Long columns, or bitmaps, want the whole machine: after a pass of more than kLoopWords arena words k_loop
// hands back to the graph, which hands over again below half of that. Random columns of three rows,
// k_loop alone -> with this rule: 14,000 on 8000 rows 98.4 -> 71.2 ms, 40,000 on 20,000 rows 565 -> 314
// ms; 24,600 random triangles on 80 points 31.7 -> 28.4 ms. With half as many words 6000 columns on 4000
// rows, whose passes k_loop does faster, take 22.9 ms instead of 19.0; with twice as many the triangles
// take 29.3, with four times the 14,000 columns stay at 98.5.
constexpr int64_t kLoopWords = (int64_t)1 << 20;
// columns left to one block, whose barriers are __syncthreads (64 and 256 measure alike)
constexpr int64_t kLoopSingle = 64;
constexpr int kLoopBlocks = 2;  // per SM: registers for every part of a pass without spills
__global__ void __launch_bounds__(kThreads, kLoopBlocks) k_loop(RArgs a, int64_t m) {
  extern __shared__ __align__(16) unsigned char add_smem[];
  WarpStage& S = reinterpret_cast<WarpStage*>(add_smem)[threadIdx.x >> 5];
  DevState* ds = a.ds;
  // (no block can let the others go before this one has arrived)
  unsigned int gen = *(volatile unsigned int*)&ds->bar_gen;
  // a shrinking list is left to fewer blocks, at last to one, whose barriers cost next to nothing
  for (;;) {
    const unsigned blocks = *(volatile unsigned int*)&ds->loop_blocks;
    if (blockIdx.x >= blocks || *(volatile int32_t*)&ds->status != ST_RUN) return;
    unsigned int target = 0;
    const int64_t n = *(volatile int64_t*)&ds->n_act;
    // what every block needs to see for itself whether the pass's space suffices, as it stands
    // before the additions take any
    const Space space = space_of(ds);
    phase1_pass<false, true>(a, blocks);
    if (!grid_sync(ds, blocks, target)) return;
    if (const int reason = lacks_space(ds, space)) {
      if (blockIdx.x == 0 && threadIdx.x == 0) stop_for_space(ds, reason);
      return;
    }
    if (ds->stats) {
      ess_count(a, m, blocks);
      if (!grid_sync(ds, blocks, target)) return;
    }
    // few columns: narrow chunks, so that every warp has some (a merge round of a warp takes 1.1 us
    // whatever its share: 25 columns of some hundred rows 13.5 us by one warp, 6.5 us by seven)
    if (n <= kWarps) add_pass<true, 1, false, kThreads, true>(a, S, blocks);
    else if (n <= 4 * kWarps) add_pass<true, 4, false, kThreads, true>(a, S, blocks);
    else if (n <= 8 * kWarps * (int64_t)blocks) add_pass<true, 8, false, kThreads, true>(a, S, blocks);
    else add_pass<true, 32, false, kThreads, true>(a, S, blocks);
    if (!grid_sync(ds, blocks, target)) return;
    commit_pass(a, blocks);
    if (!grid_last(ds, blocks, target, gen, [&] { commit_last(a, 0, kInLoop, blocks); })) return;
  }
}

// the device's global timer, in ns
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__global__ void k_clock_start(DevState* ds) { ds->t_start = global_ns(); }

// blocks of the loop kernel for an active list of n columns: a warp for 8 columns, up to kLoopMost
// blocks (a barrier of 64 blocks takes 1.4 us), then a thread for each
constexpr int kLoopMost = 64;
__host__ __device__ inline unsigned int loop_blocks_for(int64_t n) {
  const int64_t per8 = (n + 8 * kWarps - 1) / (8 * kWarps), per32 = (n + kThreads - 1) / kThreads;
  const int64_t many = per32 > kLoopMost ? per32 : kLoopMost;
  return n <= kLoopSingle ? 1u : (unsigned int)(per8 < kLoopMost ? per8 : many);
}

// end of a pass: the next active list, convergence (no target left), the pass cap, the time
// bound, and the graph's loop condition
__device__ void end_of_pass(const RArgs& a, cudaGraphConditionalHandle cond, int mode) {
  const bool in_graph = mode == kInGraph;
  DevState* ds = a.ds;
  // one thread's work, on the path of every pass: its loads are issued together
  const int32_t fault = ds->fault, debug_fault = ds->debug_fault, p = ds->pass;
  const int32_t dense_want = ds->dense_want, dense_on = ds->dense_on, compact = ds->compact;
  const int32_t was_ahead = ds->ahead, was_leave = ds->leave, horizon = ds->horizon;
  const int32_t arena_cur = ds->arena_cur, max_passes = ds->max_passes, warp_on = ds->warp_on;
  const int32_t lane_on = ds->lane_on, narrow_on = ds->narrow_on, drain = ds->drain;
  const int32_t stats_rows = ds->stats_rows;
  const int64_t n_act = ds->n_act, warp_below = ds->warp_below, warp_words = ds->warp_words;
  const int64_t lane_words = ds->lane_words, narrow_below = ds->narrow_below;
  const int64_t ahead_above = ds->ahead_above, loop_below = ds->loop_below;
  const unsigned long long used = ds->arena_used, targets = ds->targets;
  const unsigned long long t_start = ds->t_start, t_limit = ds->t_limit;
  int32_t* const act = ds->act;
  int32_t* const act2 = ds->act2;
  int32_t* const alen = ds->alen;
  int32_t* const alen2 = ds->alen2;
  const bool stats = ds->stats != nullptr;
  int32_t status = ds->status;
  int64_t n_surv = n_act;
  if (status == ST_RUN &&
      (fault || debug_fault || (compact && !survivors(a, ds, n_act, was_ahead, p, n_surv))))
    status = ST_FAULT;
  const bool to_dense = dense_want && !dense_on;
  if (to_dense) ds->dense_on = 1;
  if (status == ST_RUN) {
    ds->n_act = n_surv;
    if (compact) {
      ds->act = act2;
      ds->act2 = act;
      ds->alen = alen2;
      ds->alen2 = alen;
    }
    if (mode == kInLoop) ds->loop_blocks = min(ds->loop_blocks, loop_blocks_for(n_surv));
    // the next pass: at the horizon it compacts into the other arena; before it, visited columns
    // take new slots after the ones in use. Look-ahead ends with a compacting pass that runs no
    // column ahead and makes every list whole
    const bool next_compact = p + 1 >= horizon;
    const bool to_add = was_leave != 0;
    const int32_t ahead = to_add ? 1 : was_ahead;
    const bool leave = next_compact && ahead > 1 && n_surv < ahead_above;
    ds->compact = next_compact ? 1 : 0;
    ds->ahead = ahead;
    ds->leave = leave ? 1 : 0;
    if (next_compact) {
      ds->horizon = p + 1 + (leave ? 1 : ahead);
      ds->arena_cur = arena_cur ^ 1;
      ds->arena_used = 0;
    }
    if (targets == 0) {
      status = ST_DONE;
      ds->passes = p;
    } else if (p >= max_passes) {
      status = ST_CAPPED;
      ds->passes = p;
    } else {
      ds->pass = p + 1;
      // ... and only once the jobs are long (mean arena words per survivor), where warps of one
      // block would otherwise wait on each other's merges
      const bool to_warp = compact && !warp_on && n_surv < warp_below &&
                           used >= (unsigned long long)warp_words * n_surv;
      if (to_warp) ds->warp_on = 1;
      // merge pieces over the lanes once the jobs are long enough to share them out
      const bool to_pieces =
          compact && lane_on && used >= (unsigned long long)lane_words * n_surv;
      if (to_pieces) ds->lane_on = 0;
      // 8 columns per warp once the active list is short
      const bool to_narrow = compact && (warp_on || to_warp) && ahead == 1 &&
                             (!lane_on || to_pieces) && !narrow_on && n_surv < narrow_below;
      if (to_narrow) ds->narrow_on = 1;
      // past the time bound a later call resumes from the next pass, and what the caller reads until
      // then is this pass's result: with columns ahead of the pass it first runs on without look-ahead
      // to the horizon, whose pass visits every column, makes its list whole and runs it no further
      const bool late = drain || global_ns() - t_start > t_limit;
      const bool whole = was_ahead == 1 || (compact && drain);
      if (late) ds->drain = 1;
      if (late && whole) status = ST_TIMEOUT;
      else if (mode != kInLoop && (to_dense || to_warp || to_pieces || to_narrow || to_add))
        status = ST_SWITCH;
      else if (mode == kInLoop ? (int64_t)used > kLoopWords
                               : in_graph && ahead == 1 && n_surv <= loop_below &&
                                     2 * (int64_t)used <= kLoopWords)
        status = ST_SWITCH;
      // counter rows for the next pass: its first kernel writes them before any capacity check
      if (status != ST_TIMEOUT && stats && p + 1 >= stats_rows) {
        ds->host_reason = 4;
        status = ST_HOST;
      }
    }
  }
  if (status == ST_SWITCH) ds->pass_words = (int64_t)used;
  ds->status = status;
  if (in_graph) cudaGraphSetConditional(cond, status == ST_RUN ? 1u : 0u);
}

// ------------------------------------------------------------------------------------------
// set-up and host orchestration
// ------------------------------------------------------------------------------------------
struct InitLayout {
  int64_t dimoff[kMaxDim + 2];
  int64_t rowbase[kMaxDim + 2];
  int maxd;
};

// the boundary matrix of a simplicial complex: a column of dimension d > 0 has d + 1 rows,
// stored in id order from rowbase[d]
// col_off: the columns of a loaded matrix (any length); null: d + 1 rows at a fixed stride
__global__ void k_reduce_init(int64_t m, InitLayout L, int32_t* rows0,
                              const int64_t* __restrict__ col_off, ColMeta* meta, int32_t* low,
                              int32_t* act, int32_t* alen, int32_t* owner, unsigned long long* tab,
                              int32_t* lows0, int32_t* due, int4* prec) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < m;
       x += (int64_t)gridDim.x * blockDim.x) {
    int d = 0;
    while (d < L.maxd && x >= L.dimoff[d + 1]) d++;
    int32_t* c = col_off ? rows0 + col_off[x]
                         : rows0 + L.rowbase[d] + (int64_t)(d > 0 ? d + 1 : 0) * (x - L.dimoff[d]);
    const int32_t n = col_off ? (int32_t)(col_off[x + 1] - col_off[x]) : (d > 0 ? d + 1 : 0);
    ColMeta mx;
    mx.ptr = c;
    mx.len = n;
    mx.flags = 0;
    mx.cleared = 0;
    mx.low_seen = 0;
    mx.spare = 0;
    meta[x] = mx;
    const int32_t l = n > 0 ? c[n - 1] : -1;  // largest row of the unreduced column
    low[x] = l;
    if (due) {
      lows0[x] = l;
      due[x] = 0;
    }
    if (x < L.dimoff[L.maxd]) {  // rows: no pivot yet
      if (due) prec[x] = make_int4(0, INT32_MAX, INT32_MAX, INT32_MAX);
      tab[x] = ~0ull;
    }
    act[x] = (int32_t)x;
    alen[x] = n;
    owner[x] = -1;
  }
}

// look-back states: chunks of any shape (8 slots or more; 1 or 4 for a few columns), or tiles
static int64_t look_words(int64_t m) { return (m + 7) / 8 + 1 + kWarps; }

static RArgs make_args(ph_ctx* ctx) {
  ReduceState& rs = ctx->rs;
  RArgs a;
  std::memset(&a, 0, sizeof(a));  // (whole: pass_graph compares the bytes)
  a.ds = static_cast<DevState*>(rs.dstate);
  a.low = ctx->low;
  a.beta = ctx->beta;
  a.meta = static_cast<ColMeta*>(rs.meta);
  a.nxt_ptr = rs.nxt_ptr;
  a.nxt_len = rs.nxt_len;
  a.owner = rs.owner;
  a.first_unp = rs.first_unp;
  a.tab = rs.tab;
  a.seg = ctx->seg;
  a.rows_end = ctx->dimoff[ctx->max_dim];
  a.nseg = (int)ctx->seg_start.size() - 1;
  a.next_unp = rs.dirty;
  a.dirty_on = rs.dirty + a.nseg;
  a.dirty = rs.dirty + 2 * a.nseg;
  a.nc = ctx->n_clouds;
  a.strict = ctx->opts.strict_phase2;
  a.cor10 = ctx->opts.use_cor10;
  a.tile_st = static_cast<unsigned long long*>(rs.tiles);
  a.loop_tile_st = a.tile_st + (ctx->m + kFTile - 1) / kFTile + 1;
  a.look = static_cast<unsigned long long*>(rs.look);
  a.dlist = static_cast<int32_t*>(rs.dlist);
  a.src_e = static_cast<int32_t*>(rs.src_e);
  a.lows = rs.lows;
  a.due = rs.due;
  a.lows_stride = lows_stride_of(ctx->m);
  a.ring = kAheadMax - 1;
  a.prec = static_cast<int4*>(rs.prec);
  a.delta = rs.delta;
  a.kind = rs.kind;
  a.newpos = rs.newpos;
  a.work = rs.work;
  a.predict = ctx->opts.predict_pairs ? 1 : 0;
  a.unp_bits = rs.unp_bits;
  a.unp_words = rs.unp_words;
  a.pred = rs.pred;
  a.staged_max = ctx->opts.staged_merge_max > 0 ? std::min(ctx->opts.staged_merge_max, kStage)
                                                 : kStage;
  a.force_km = std::max(0, std::min(ctx->opts.merge_items, 64));
  a.set_n = rs.set_n;
  a.set_neg = rs.set_neg;
  a.set_on = rs.set_on;
  // bit-packed columns: per column dimension the smallest threshold over its row segments
  a.dense_mode = ctx->opts.dense_threshold;
  a.seg_start = ctx->d_seg_start;
  for (int d = 0; d <= kMaxDim; d++)
    a.dim_start[d] = (int32_t)(d <= ctx->max_dim ? ctx->dimoff[d] : ctx->m);
  const int64_t t0 = a.dense_mode > 0 ? a.dense_mode : 32;
  a.dense_floor = INT32_MAX;
  for (int d = 0; d <= kMaxDim; d++) {
    int64_t mn = INT32_MAX;
    for (int c = 0; a.dense_mode >= 0 && d >= 1 && d <= ctx->max_dim && c < ctx->n_clouds; c++) {
      const int rs = (d - 1) * ctx->n_clouds + c;
      const int64_t n = ctx->seg_start[rs + 1] - ctx->seg_start[rs];
      if (n > 0) mn = std::min<int64_t>(mn, std::max<int64_t>((n + 31) / 32 + kDenseHead, t0));
    }
    a.dense_min[d] = (int32_t)std::min<int64_t>(mn, INT32_MAX);
    a.dense_floor = std::min(a.dense_floor, a.dense_min[d]);
  }
  return a;
}

// the kernels of a pass's additions: k_add as 1 = handles bit-packed columns (DevState::dense_on) + 2
// = one chunk per warp (DevState::warp_on) + 4 = each job merged by its own lane
// (DevState::lane_on), 8 + 1 = bit-packed: 8-slot warp chunks with merge pieces
// (DevState::narrow_on); or k_visit and k_merge (DevState::ahead > 1), 10 + 1 = bit-packed + 2 = each
// job merged by its own lane
static int add_variant(const DevState& h) {
  if (h.ahead > 1) return 10 + (h.dense_on ? 1 : 0) + (h.lane_on ? 2 : 0);
  if (h.narrow_on) return 8 + (h.dense_on ? 1 : 0);
  return (h.dense_on ? 1 : 0) + (h.warp_on ? 2 : 0) + (h.lane_on ? 4 : 0);
}
static void (*const add_kernels[10])(RArgs) = {
    k_add<false, 0, false, kPieceBlockThreads>, k_add<true, 0, false, kPieceBlockThreads>,
    k_add<false, 32, false>, k_add<true, 32, false>, k_add<false, 0, true>, k_add<true, 0, true>,
    k_add<false, 32, true>, k_add<true, 32, true>, k_add<false, 8, false>, k_add<true, 8, false>};
static void (*const merge_kernels[4])(RArgs) = {k_merge<false, false>, k_merge<true, false>,
                                                k_merge<false, true>, k_merge<true, true>};

// grid of the persistent additions kernel: add_blocks_per_sm units of two 128-thread blocks per
// SM, no more blocks than the largest active list (all m columns) can use
static unsigned add_grid_of(const ph_ctx* ctx) {
  const int64_t m = std::max<int64_t>(ctx->m, 1);
  const int bps = ctx->opts.add_blocks_per_sm > 0 ? std::min(ctx->opts.add_blocks_per_sm, 4) : 4;
  const int64_t full = (int64_t)ctx->num_sms * bps * (kThreads / kAddThreads);
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(full, (m + kAddThreads - 1) / kAddThreads));
}

// launches one pass kernel; pdl: the kernel may start while the kernel before it in the stream
// drains (programmatic dependent launch; the kernel waits in pdl_wait)
constexpr bool kUsePdl = true;
template <typename... KArgs, typename... Args>
static void launch_k(ph_ctx* ctx, bool pdl, void (*kern)(KArgs...), unsigned grid, unsigned block,
                     size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl && kUsePdl ? 1 : 0;
  ctx->launches++;
  PH_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
}

// the kernels of one pass, in order; grids are fixed (persistent blocks loop over the work).
// The pass's first kernel (Phase I and the marks), then the rest: a pass stopped for more space
// after its marks continues with the rest alone (launch_pass_rest)
// variant: the additions kernel (add_variant)
static unsigned pass_blocks(ph_ctx* ctx, int64_t full, int64_t per_block) {
  // the full machine for large complexes, no more blocks than the largest active list (all m
  // columns) can use for small ones, so a small complex's pass costs little
  const int64_t m = std::max<int64_t>(ctx->m, 1);
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(full, (m + per_block - 1) / per_block));
}

static void launch_pass_rest(ph_ctx* ctx, const RArgs& a, cudaGraphConditionalHandle cond,
                             bool in_graph, int variant, bool time_add, cudaStream_t st) {
  ReduceState& rs = ctx->rs;
  const int sms = ctx->num_sms;
  auto blocks = [&](int64_t full, int64_t per_block) { return pass_blocks(ctx, full, per_block); };
  if (ctx->opts.collect_stats)
    launch_k(ctx, true, k_ess_count, (unsigned)sms * 4, kThreads, 0, st, a, ctx->m);
  if (ctx->opts.phase2_sets > 0 && a.rows_end > 0) {  // host-driven loop only
    const int64_t rows = a.rows_end;
    int bits = 1;
    while (bits < 31 && (int64_t(1) << bits) <= ctx->m) bits++;
    PH_CUDA(cudaMemsetAsync(rs.set_n, 0, (size_t)rows * sizeof(int32_t), st));
    PH_CUDA(cudaMemsetAsync(rs.set_neg, 0, (size_t)rows * sizeof(int32_t), st));
    k_set_count<<<blocks(sms * 8, kThreads), kThreads, 0, st>>>(a);
    PH_CHECK_LAUNCH();
    uint64_t* key = rs.set_key;
    uint64_t* row = rs.set_key + rows;
    k_set_tiekeys<<<grid_for(ctx, rows, kThreads), kThreads, 0, st>>>(a, ctx->gidx, key, row);
    PH_CHECK_LAUNCH();
    int32_t* fault = &static_cast<DevState*>(rs.dstate)->fault;
    radix_sort_u64(ctx, key, row, rows, 0, bits, rs.set_key + 2 * rows, rs.set_key + 3 * rows,
                   fault);
    k_set_keys<<<grid_for(ctx, rows, kThreads), kThreads, 0, st>>>(
        a, ctx->opts.phase2_priority, bits, key, row);
    PH_CHECK_LAUNCH();
    radix_sort_u64(ctx, key, row, rows, 0, ctx->opts.phase2_priority == 1 ? 2 * bits : bits,
                   rs.set_key + 2 * rows, rs.set_key + 3 * rows, fault);
    const int64_t p = std::min<int64_t>(ctx->opts.phase2_sets, rows);
    k_set_select<<<grid_for(ctx, p, kThreads), kThreads, 0, st>>>(a, p, row);
    PH_CHECK_LAUNCH();
    k_set_apply<<<blocks(sms * 8, kThreads), kThreads, 0, st>>>(a);
    PH_CHECK_LAUNCH();
  }
  if (time_add) {
    cudaEvent_t e0, e1;
    PH_CUDA(cudaEventCreate(&e0));
    PH_CUDA(cudaEventCreate(&e1));
    rs.ev.push_back(e0);
    rs.ev.push_back(e1);
    PH_CUDA(cudaEventRecord(e0, st));
  }
  // (an event recorded between two kernels needs the first one complete: no early start then)
  if (variant >= 10) {
    launch_k(ctx, !time_add, k_visit, add_grid_of(ctx), kAddThreads, 0, st, a);
    launch_k(ctx, true, merge_kernels[variant - 10], add_grid_of(ctx), kAddThreads, kAddSmem, st, a);
  } else {
    // block chunks with merge pieces (variants 0, 1) in smaller blocks, as many warps per SM
    const int bt = variant <= 1 ? kPieceBlockThreads : kAddThreads;
    launch_k(ctx, !time_add, add_kernels[variant], add_grid_of(ctx) * (kAddThreads / bt), bt,
             sizeof(WarpStage) * (bt / 32), st, a);
  }
  if (time_add) PH_CUDA(cudaEventRecord(rs.ev.back(), st));
  launch_k(ctx, !time_add, k_commit, blocks(sms * 2, kThreads), kThreads, 0, st, a, cond,
           in_graph ? kInGraph : kHostLoop);
}

static void launch_pass(ph_ctx* ctx, const RArgs& a, cudaGraphConditionalHandle cond,
                        bool in_graph, int variant, bool time_add, cudaStream_t st) {
  launch_k(ctx, true, variant >= 10 ? k_phase1<true> : k_phase1<false>,
           pass_blocks(ctx, ctx->num_sms * 8, kFTile), kThreads, 0, st, a);
  launch_pass_rest(ctx, a, cond, in_graph, variant, time_add, st);
}

// the new buffer is taken before the old one goes, so a failed allocation (PH_ERR_ALLOC)
// leaves the store, and the device state that points into it, as it was: a later call resumes
static void grow_store(ph_ctx* ctx, ColStore& s, int64_t need_words) {
  if (need_words <= s.cap) return;
  const int64_t cap = std::max<int64_t>(2 * need_words, 1 << 20);  // doubling: few regrowth stops
  int32_t* p = alloc_n<int32_t>(ctx, cap + kColSlack);
  if (s.p) ctx->dfree(s.p);
  s.p = p;
  s.cap = cap;
}

static int64_t first_arena(const ph_ctx* ctx, bool look_ahead) {
  return ctx->opts.arena_words > 0 ? ctx->opts.arena_words
         : look_ahead              ? ctx->nnz + kDeltaRows * (ctx->m - ctx->dimoff[1]) + 1
                                   : 2 * ctx->nnz + 1;
}

// the first arenas and the pivot store's first chunk: pass 0 needs at most the boundary matrix twice
// over, or once and a visit's rows per column; later passes need less (they grow on demand otherwise)
static void take_stores(ph_ctx* ctx, bool look_ahead) {
  ReduceState& rs = ctx->rs;
  for (ColStore& s : rs.arena) grow_store(ctx, s, first_arena(ctx, look_ahead));
  ColStore c{};
  grow_store(ctx, c, ctx->nnz / 4 + 1);
  rs.pivots.push_back(c);
}

static void free_ahead(ph_ctx* ctx) {
  ReduceState& rs = ctx->rs;
  for (void* p : {(void*)rs.prec, (void*)rs.lows, (void*)rs.due, (void*)rs.delta, (void*)rs.kind,
                  (void*)rs.newpos, (void*)rs.work})
    ctx->dfree(p);
  rs.prec = nullptr;
  rs.lows = rs.due = rs.delta = rs.newpos = rs.work = nullptr;
  rs.kind = nullptr;
}

// Look-ahead's arrays and stores: some 580 bytes per column, where pass by pass the stores take 100.
// They come last at set-up: without room for them, or when they would take more than two fifths of the
// device's memory, the reduction runs pass by pass. When a later allocation fails it starts again pass
// by pass (restart_pass_by_pass), and one that waits between two calls gives them back
// (give_up_ahead). So what fits without look-ahead fits.
// h: the state of a reduction that begins to look ahead now (null: at set-up). The arena that its
// next pass writes into holds nothing yet
static bool take_ahead(ph_ctx* ctx, DevState* h) {
  ReduceState& rs = ctx->rs;
  const int64_t m = ctx->m, rows = ctx->dimoff[ctx->max_dim];
  if (ctx->device_bytes == 0) {  // (how much of it is free tells little: allocators hold blocks back)
    size_t free_bytes = 0;
    PH_CUDA(cudaMemGetInfo(&free_bytes, &ctx->device_bytes));
  }
  const double bytes = 16.0 * rows + (4.0 * (kAheadMax + 1 + kDeltaRows + 2) + 1.0) * m +
                       16.0 * first_arena(ctx, true);  // (two arenas of twice that many words)
  if (bytes > 0.4 * ctx->device_bytes) return false;
  try {
    rs.prec = alloc_n<int4>(ctx, rows);
    rs.lows = alloc_n<int32_t>(ctx, kAheadMax * lows_stride_of(m));
    rs.due = alloc_n<int32_t>(ctx, lows_stride_of(m));
    rs.delta = alloc_n<int32_t>(ctx, kDeltaRows * m + kColSlack);
    rs.kind = alloc_n<uint8_t>(ctx, m);
    rs.newpos = alloc_n<int32_t>(ctx, m);
    rs.work = alloc_n<int32_t>(ctx, m);
    if (h) grow_store(ctx, rs.arena[h->arena_cur], first_arena(ctx, true));
    else take_stores(ctx, true);
    return true;
  } catch (const Fail&) {
    ctx->err.clear();
    free_ahead(ctx);
    for (ColStore& s : rs.arena) {
      if (h) break;
      ctx->dfree(s.p);
      s = ColStore{};
    }
    return false;
  }
}

// the unreduced columns of a reduction whose arrays are there, with or without look-ahead's; then, with
// its stores, the pass loop's state
static void set_up_columns(ph_ctx* ctx) {
  ReduceState& rs = ctx->rs;
  cudaStream_t st = ctx->stream;
  const int64_t m = ctx->m;
  const int nseg = (int)ctx->seg_start.size() - 1;
  PH_CUDA(cudaMemsetAsync(rs.first_unp, 0x7f, nseg * sizeof(int32_t), st));  // above every id
  PH_CUDA(cudaMemsetAsync(rs.dirty, 0x7f, nseg * sizeof(int32_t), st));
  PH_CUDA(cudaMemsetAsync(rs.dirty + nseg, 0, nseg * sizeof(int32_t), st));
  PH_CUDA(cudaMemsetAsync(rs.tiles, 0, rs.tiles_bytes, st));  // no state published yet
  PH_CUDA(cudaMemsetAsync(rs.look, 0, look_words(m) * sizeof(unsigned long long), st));
  if (rs.pred) PH_CUDA(cudaMemsetAsync(rs.pred, 0xff, (size_t)m * sizeof(int32_t), st));
  if (rs.pass_stats)
    PH_CUDA(cudaMemsetAsync(rs.pass_stats, 0, (size_t)rs.stats_rows * PH_PS_N * 8, st));
  InitLayout L{};
  L.maxd = ctx->max_dim;
  for (int d = 0; d <= ctx->max_dim + 1; d++) L.dimoff[d] = ctx->dimoff[d];
  int64_t rb = 0;
  for (int d = 0; d <= ctx->max_dim; d++) {
    L.rowbase[d] = rb;
    rb += (d > 0 ? d + 1 : 0) * (ctx->dimoff[d + 1] - ctx->dimoff[d]);
  }
  k_reduce_init<<<grid_for(ctx, m, kThreads), kThreads, 0, st>>>(
      m, L, ctx->rows0, ctx->col_off, static_cast<ColMeta*>(rs.meta), ctx->low, rs.act,
      rs.alen, rs.owner, rs.tab, rs.lows, rs.due, static_cast<int4*>(rs.prec));
  PH_CHECK_LAUNCH();
}

static void set_up_passes(ph_ctx* ctx) {
  ReduceState& rs = ctx->rs;
  cudaStream_t st = ctx->stream;
  const int64_t m = ctx->m;
  const int32_t ahead = rs.lows ? kAheadMax : 1;
  DevState& h = *static_cast<DevState*>(rs.hstate);
  h = DevState{};
  h.act = rs.act;
  h.act2 = rs.act2;
  h.alen = rs.alen;
  h.alen2 = rs.alen2;
  h.n_act = m;
  for (int i = 0; i < 2; i++) {
    h.arena[i] = rs.arena[i].p;
    h.arena_cap[i] = rs.arena[i].cap;
  }
  h.piv_base = rs.pivots.back().p;
  h.piv_cap = rs.pivots.back().cap;
  h.piv_used = 0;
  h.stats = rs.pass_stats;
  h.stats_rows = rs.stats_rows;
  h.pass = 0;
  h.status = ST_RUN;
  h.ahead = ahead;
  h.ahead_above = kAheadAbove;
  h.horizon = ahead;
  h.compact = 1;
  h.arena_cur = 0;
  h.warp_below = ctx->opts.warp_chunks_below < 0   ? 0
                 : ctx->opts.warp_chunks_below == 0 ? (int64_t)1 << 22
                                                    : ctx->opts.warp_chunks_below;
  h.warp_words = ctx->opts.warp_chunk_words < 0    ? 0
                 : ctx->opts.warp_chunk_words == 0 ? 40
                                                   : ctx->opts.warp_chunk_words;
  // the first passes' jobs are short: block chunks, unless any job length will do
  h.warp_on = h.warp_words == 0 && m < h.warp_below ? 1 : 0;
  h.lane_words = ctx->opts.lane_merge_words == 0 ? 20 : ctx->opts.lane_merge_words;
  h.lane_on = ctx->opts.lane_merge_words < 0 ? 0 : 1;
  h.narrow_below = ctx->opts.narrow_chunks_below < 0 ? 0
                   : ctx->opts.narrow_chunks_below == 0
                       ? (int64_t)add_grid_of(ctx) * kAddWarps * kNarrowColsPerWarp
                       : ctx->opts.narrow_chunks_below;
  h.narrow_on = 0;
  PH_CUDA(cudaMemcpyAsync(rs.dstate, &h, sizeof(DevState), cudaMemcpyHostToDevice, st));
  // the first pass's row state and table (the later ones come from the pass before)
  {
    const RArgs a0 = make_args(ctx);
    launch_k(ctx, false, k_first, (unsigned)grid_for(ctx, std::max(m, a0.rows_end), kThreads), kThreads,
             0, st, a0);
  }
  rs.fresh = true;
  rs.loop_ran = false;
}

// the stored lows of the active columns, which are all up to date, and the records of the pivots
__global__ void k_enter_ahead(RArgs a, const int32_t* __restrict__ act, int64_t n_act, int32_t pass) {
  int32_t* lows = a.lows + (int64_t)(pass & a.ring) * a.lows_stride;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (int64_t e = first; e < n_act; e += stride) {
    const int32_t j = act[e];
    lows[e] = j >= 0 ? a.low[j] : -1;
    a.due[e] = j >= 0 ? pass : kDeadDue;
  }
  for (int64_t x = first; x < a.rows_end; x += stride) {
    const int32_t o = a.owner[x];
    int4 r = make_int4(0, INT32_MAX, INT32_MAX, INT32_MAX);
    if (o >= 0) {
      const ColMeta mo = load_meta(a.meta + o);
      r = rec_of(mo.ptr, mo.len);
    }
    a.prec[x] = r;
  }
}

// Look-ahead pays from the third pass of a call on: of 10.67 M columns a call of no pass took 1.11 ms with
// it and 0.81 without, of one 2.00 and 1.37, of two 2.30 and 1.96, of three 2.46 and 2.59, of four 2.69
// and 3.17 (47.3 M in 512 clouds: 5.8 and 3.7, 10.3 and 6.1, 11.0 and 8.5, 11.4 and 11.2, 12.3 and 13.5).
// So a first and a second call capped below that run pass by pass; the next one begins to look ahead, as
// many such calls cost less with it than without (23 of one pass each and the rest: 53 and 76 ms).
constexpr int32_t kFewPasses = 2;
static void enter_ahead(ph_ctx* ctx, DevState& h) {
  ReduceState& rs = ctx->rs;
  if (h.ahead > 1 || h.n_act < kAheadFrom / 2 || !take_ahead(ctx, &h)) return;
  const ColStore& s = rs.arena[h.arena_cur];
  h.arena[h.arena_cur] = s.p;
  h.arena_cap[h.arena_cur] = s.cap;
  const RArgs a = make_args(ctx);
  k_enter_ahead<<<grid_for(ctx, std::max(h.n_act, a.rows_end), kThreads), kThreads, 0, ctx->stream>>>(
      a, h.act, h.n_act, h.pass);
  PH_CHECK_LAUNCH();
  h.ahead = kAheadMax;
  h.horizon = h.pass + kAheadMax;
}

void reduce_init(ph_ctx* ctx, int32_t max_passes) {
  free_reduce_state(ctx);  // whatever an earlier, failed initialisation left
  // Phase I's tile states carry a (cloud, dimension) segment in 23 bits
  PH_REQUIRE((int64_t)ctx->seg_start.size() - 1 < (1 << 23), PH_ERR_CAPACITY,
             "at most 8,388,607 (cloud, dimension) segments per reduction");
  ReduceState& rs = ctx->rs;
  const int64_t m = ctx->m;
  rs.act = alloc_n<int32_t>(ctx, m);
  rs.act2 = alloc_n<int32_t>(ctx, m);
  rs.alen = alloc_n<int32_t>(ctx, m);
  rs.alen2 = alloc_n<int32_t>(ctx, m);
  rs.meta = alloc_n<ColMeta>(ctx, m);
  rs.nxt_ptr = alloc_n<int32_t*>(ctx, m);
  rs.nxt_len = alloc_n<int32_t>(ctx, m);
  rs.owner = alloc_n<int32_t>(ctx, m);
  rs.tab = alloc_n<unsigned long long>(ctx, ctx->dimoff[ctx->max_dim]);
  int nseg = (int)ctx->seg_start.size() - 1;
  rs.first_unp = alloc_n<int32_t>(ctx, nseg);
  rs.dirty = alloc_n<int32_t>(ctx, 3 * nseg);  // next_unp, dirty_on, dirty
  // Phase I's tile states; the loop kernel's tiles are of another size and have their own
  const int64_t ntiles = (m + kFTile - 1) / kFTile;
  const int64_t loop_tiles = (std::min<int64_t>(m, kLoopStart) + kThreads - 1) / kThreads;
  rs.tiles_bytes = (ntiles + 1 + loop_tiles) * sizeof(unsigned long long);
  rs.tiles = ctx->dalloc(rs.tiles_bytes);
  rs.look = alloc_n<unsigned long long>(ctx, look_words(m));
  rs.dlist = alloc_n<int32_t>(ctx, m);
  // look-ahead for long lists (per-pass counters, and sets chosen pass by pass, need every pass to
  // take every column)
  const bool may = !ctx->opts.collect_stats && ctx->opts.phase2_sets <= 0 &&
                   ctx->three_row_columns() >= kAheadFrom;
  // (a block all the same: without it the others lie such that 0.57 M columns take 1650 us, not 1625)
  if (!may) rs.prec = alloc_n<int4>(ctx, 1);
  rs.src_e = alloc_n<int32_t>(ctx, m);
  if (ctx->opts.predict_pairs) {
    const int64_t rows = ctx->dimoff[ctx->max_dim];
    const int64_t nwords = (rows + 31) / 32;
    rs.unp_bits = alloc_n<uint32_t>(ctx, nwords + 1);
    rs.unp_words = alloc_n<int32_t>(ctx, nwords + 1);
    rs.pred = alloc_n<int32_t>(ctx, m);
  }
  if (ctx->opts.phase2_sets > 0) {
    const int64_t rows = std::max<int64_t>(ctx->dimoff[ctx->max_dim], 1);
    rs.set_n = alloc_n<int32_t>(ctx, rows);
    rs.set_neg = alloc_n<int32_t>(ctx, rows);
    rs.set_on = alloc_n<uint8_t>(ctx, rows);
    rs.set_key = alloc_n<uint64_t>(ctx, 4 * rows);
  }
  if (ctx->opts.collect_stats) {
    rs.stats_rows = 256;
    rs.pass_stats = alloc_n<int64_t>(ctx, (int64_t)rs.stats_rows * PH_PS_N);
  }
  rs.dstate = ctx->dalloc(sizeof(DevState));
  if (!rs.hstate) PH_CUDA(cudaMallocHost(&rs.hstate, sizeof(DevState)));  // kept by the context
  rs.h_stats.clear();
  rs.ahead_later = may && max_passes >= 0 && max_passes <= kFewPasses ? 2 : 0;
  const bool ahead = may && !rs.ahead_later && take_ahead(ctx, nullptr);
  set_up_columns(ctx);  // (the device is at work while the stores are taken)
  if (!ahead) take_stores(ctx, false);
  set_up_passes(ctx);
  rs.passes = 0;
  rs.init = true;
  rs.done = false;
  rs.status = PH_OK;
}

// A reduction with look-ahead that found no memory starts again pass by pass. Between two horizons
// columns are ahead of the pass, which is no state to leave behind; a pass-by-pass run decides the
// same (reduce_run takes the caps of earlier calls again on the way) and stops for want of memory
// before the pass that needs it, with all columns up to date. It keeps all memory it has, so that it
// comes as far as the run before if the allocator gives nothing more; look-ahead's larger arenas are
// exchanged for its own if it gives these.
static void restart_pass_by_pass(ph_ctx* ctx) {
  ReduceState& rs = ctx->rs;
  ColStore block{rs.delta, kDeltaRows * ctx->m};
  rs.delta = nullptr;
  free_ahead(ctx);
  for (auto& r : rs.retired) ctx->dfree(r.p);
  rs.retired.clear();
  const int64_t first = first_arena(ctx, false);
  for (ColStore& s : rs.arena) {
    ColStore c{};
    if (s.cap < block.cap / 2) {  // one that look-ahead had no use for yet: the deltas' block will do
      std::swap(c, block);
    } else if (ctx->opts.arena_words <= 0 && s.cap > 2 * first) {
      try {
        grow_store(ctx, c, first);
      } catch (const Fail&) {
        ctx->err.clear();
      }
    }
    if (!c.p) continue;
    ctx->dfree(s.p);
    s = c;
  }
  ctx->dfree(block.p);
  // the chunks of the pivot store: the largest one first
  std::sort(rs.pivots.begin(), rs.pivots.end(),
            [](const ColStore& x, const ColStore& y) { return x.cap < y.cap; });
  rs.spare.insert(rs.spare.end(), rs.pivots.begin(), rs.pivots.end() - 1);
  rs.pivots.erase(rs.pivots.begin(), rs.pivots.end() - 1);
  for (auto e : rs.ev) cudaEventDestroy(e);
  rs.ev.clear();
  rs.add_launches = 0;
  rs.ms_add = 0;
  rs.add_ms.clear();
  rs.caps_met = 0;
  set_up_columns(ctx);
  set_up_passes(ctx);
}

// A reduction with look-ahead that rests between two calls (capped, or stopped at the time bound: all
// columns up to date, all lists whole) goes on pass by pass, and gives look-ahead's arrays back. Its
// next pass compacts into the other arena.
bool give_up_ahead(ph_ctx* ctx) {
  ReduceState& rs = ctx->rs;
  if (!rs.resting || !rs.lows) return false;
  DevState& h = *static_cast<DevState*>(rs.hstate);
  if (h.ahead > 1) {
    if (!h.compact) {
      h.compact = 1;
      h.arena_cur ^= 1;
      h.arena_used = 0;
    }
    h.ahead = 1;
    h.leave = 0;
    h.horizon = (h.status == ST_CAPPED ? h.passes + 1 : h.pass) + 1;
    PH_CUDA(cudaMemcpyAsync(rs.dstate, &h, sizeof(DevState), cudaMemcpyHostToDevice, ctx->stream));
  }
  free_ahead(ctx);
  return true;
}

// grows whatever the stopped pass asked for, in the host mirror h
static void serve_host_request(ph_ctx* ctx, DevState& h) {
  ReduceState& rs = ctx->rs;
  cudaStream_t st = ctx->stream;
  // buffers retired between two compacting passes hold no column any more after the next one
  if (h.compact) {
    for (auto it = rs.retired.begin(); it != rs.retired.end();) {
      if (it->until < h.pass) {
        ctx->dfree(it->p);
        it = rs.retired.erase(it);
      } else {
        ++it;
      }
    }
  }
  if (h.host_reason & 1) {  // the arena this pass writes into
    ColStore& s = rs.arena[h.arena_cur];
    if (h.compact) {  // its contents are dead
      grow_store(ctx, s, (int64_t)h.bound_words);
    } else {  // it holds columns until the next compacting pass: a further buffer beside it
      ColStore c{};
      grow_store(ctx, c, (int64_t)h.bound_words);
      rs.retired.push_back({s.p, h.horizon});
      s = c;
      h.arena_used = 0;
    }
    h.arena[h.arena_cur] = s.p;
    h.arena_cap[h.arena_cur] = s.cap;
  }
  if (h.host_reason & 2) {  // a new pivot chunk; the old ones stay (their columns live there)
    ColStore c{};
    if (!rs.spare.empty() && rs.spare.back().cap >= (int64_t)h.bound_piv) {  // a restart left it
      c = rs.spare.back();
      rs.spare.pop_back();
    } else {
      grow_store(ctx, c, std::max<int64_t>(2 * (int64_t)h.bound_piv, ctx->nnz / 4 + 1));
    }
    rs.pivots.push_back(c);
    h.piv_base = c.p;
    h.piv_cap = c.cap;
    h.piv_used = 0;
  }
  if (h.host_reason & 4) {
    int32_t rows = std::max(256, rs.stats_rows * 2);
    while (rows <= h.pass) rows *= 2;
    int64_t* ns = alloc_n<int64_t>(ctx, (int64_t)rows * PH_PS_N);
    PH_CUDA(cudaMemsetAsync(ns, 0, (size_t)rows * PH_PS_N * 8, st));
    PH_CUDA(cudaMemcpyAsync(ns, rs.pass_stats, (size_t)rs.stats_rows * PH_PS_N * 8,
                            cudaMemcpyDeviceToDevice, st));
    ctx->dfree(rs.pass_stats);
    rs.pass_stats = ns;
    rs.stats_rows = rows;
    h.stats = ns;
    h.stats_rows = rows;
  }
  h.host_reason = 0;
  h.status = ST_RUN;
}

// grid of the loop kernel: no more blocks than can be resident at once, or than the columns
// can use (0: the device cannot run it)
constexpr size_t kLoopSmem = sizeof(WarpStage) * kWarps;
static_assert(kAddSmem <= 48 * 1024 && kLoopSmem <= 48 * 1024, "above, kernels must opt in");
static unsigned loop_grid(ph_ctx* ctx) {
  if (ctx->loop_blocks_per_sm < 0)  // asked once per context
    PH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctx->loop_blocks_per_sm, k_loop, kThreads,
                                                          kLoopSmem));
  const int64_t most = (int64_t)ctx->num_sms * ctx->loop_blocks_per_sm;
  return (unsigned)most;
}

// the pass loop as one graph: a conditional while node around one pass, with one of the
// additions kernel variants (see launch_pass)
static void free_loop(ReduceState::Loop& l) {
  if (l.exec) cudaGraphExecDestroy(l.exec);
  if (l.graph) cudaGraphDestroy(l.graph);
  l = ReduceState::Loop{};
}
static void free_retired(ph_ctx* ctx) {
  for (auto& l : ctx->retired) free_loop(l);
  ctx->retired.clear();
}
void free_graphs(ph_ctx* ctx) {
  for (auto& l : ctx->loops) free_loop(l);
  free_retired(ctx);
  if (ctx->capture_stream) cudaStreamDestroy(ctx->capture_stream);
  ctx->capture_stream = nullptr;
}

// Passes per round of the while node: a round's end costs 4.3 us against 1.5 us between two kernels
// of the body. The passes after the last one find their work done and leave at once (some 5 us each).
// 574,000 columns, 34 passes: 1740 us with one, 1665 us with four
constexpr int kGraphPasses = 4;
static cudaGraphExec_t pass_graph(ph_ctx* ctx, const RArgs& a, int variant) {
  // everything the graph's kernels and grids depend on besides the context's options
  ReduceState::Loop& loop = ctx->loops[variant];
  std::vector<unsigned char> args(sizeof(RArgs) + sizeof(int64_t));
  std::memcpy(args.data(), &a, sizeof(RArgs));
  std::memcpy(args.data() + sizeof(RArgs), &ctx->m, sizeof(int64_t));
  if (loop.exec && loop.args == args) return loop.exec;
  // (given back once the new graph runs: it takes as long as making one)
  if (loop.graph) ctx->retired.push_back(std::move(loop));
  loop = ReduceState::Loop{};
  cudaGraph_t g;
  cudaError_t ce;
  PH_CUDA(cudaGraphCreate(&g, 0));
  cudaGraphConditionalHandle cond;
  PH_CUDA(cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault));
  cudaGraphNodeParams p{};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = cond;
  p.conditional.type = cudaGraphCondTypeWhile;
  p.conditional.size = 1;
  cudaGraphNode_t node;
  PH_CUDA(cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &p));
  cudaGraph_t body = p.conditional.phGraph_out[0];
  // capture on a private stream (the legacy default stream cannot capture); the graph is
  // then launched on the context's stream
  if (!ctx->capture_stream) {
    ce = cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking);
    if (ce != cudaSuccess) {
      ctx->capture_stream = nullptr;
      cudaGraphDestroy(g);
    }
    PH_CUDA(ce);
  }
  const cudaStream_t cs = ctx->capture_stream;
  ce = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
  if (ce != cudaSuccess) {
    cudaGraphDestroy(g);
    PH_CUDA(ce);
  }
  const int64_t counted = ctx->launches;  // captured launches run later, counted per pass
  try {
    for (int i = 0; i < kGraphPasses; i++) launch_pass(ctx, a, cond, true, variant, false, cs);
    ctx->launches = counted;
  } catch (...) {
    cudaStreamEndCapture(cs, &body);
    cudaGraphDestroy(g);
    throw;
  }
  ce = cudaStreamEndCapture(cs, &body);
  if (ce != cudaSuccess) cudaGraphDestroy(g);
  PH_CUDA(ce);
  loop.graph = g;  // (freed with the loop, also when the next call fails)
  PH_CUDA(cudaGraphInstantiate(&loop.exec, g, 0));
  loop.args = std::move(args);
  return loop.exec;
}

int reduce_run(ph_ctx* ctx, int32_t max_passes) {
  ReduceState& rs = ctx->rs;
  cudaStream_t st = ctx->stream;
  // the budgeted Phase II ranks its sets with host-sized sort launches: host-driven loop
  const bool use_graph = ctx->opts.use_graph != 0 && ctx->opts.phase2_sets <= 0;
  const bool time_add = ctx->opts.time_kernels != 0 && !use_graph;
  DevState& h = *static_cast<DevState*>(rs.hstate);
  const bool rested = rs.resting;
  rs.resting = false;
  // a resumed reduction continues after the pass that hit the previous cap
  bool loop_states_clear = rs.fresh;  // k_loop's tile states: nothing of an earlier pass in them
  if (!rs.fresh) {  // (what set-up wrote is still in the host's copy)
    PH_CUDA(cudaMemcpyAsync(&h, rs.dstate, sizeof(DevState), cudaMemcpyDeviceToHost, st));
    PH_CUDA(cudaStreamSynchronize(st));
  }
  rs.fresh = false;
  if (h.status == ST_CAPPED) {  // every column is up to date there
    h.pass = h.passes + 1;
    h.status = ST_RUN;
  } else if (h.status == ST_TIMEOUT) {  // stopped between two passes
    h.status = ST_RUN;
  }
  if (rs.ahead_later && rested) {
    rs.ahead_later--;
    if (max_passes < 0 || max_passes - h.pass > kFewPasses || rs.ahead_later == 0) {
      rs.ahead_later = 0;
      enter_ahead(ctx, h);
    }
  }
  if (h.stats && h.pass >= h.stats_rows) {  // counter rows for the first pass of this call
    h.host_reason = 4;
    serve_host_request(ctx, h);
  }
  // every pass proves or zeroes at least one column, so m + 1 passes always suffice
  int32_t cap = max_passes < 0 ? (int32_t)std::min<int64_t>(ctx->m + 1, INT32_MAX) : max_passes;
  unsigned loop_blocks = use_graph ? loop_grid(ctx) : 0;
  const int64_t limit_ms = ctx->opts.timeout_ms > 0 ? ctx->opts.timeout_ms : 60000;
  auto next_cap = [&] { return rs.caps_met < rs.caps.size() ? rs.caps[rs.caps_met] : cap; };
  auto begin = [&] {
    h.max_passes = next_cap();
    h.blocks_done = 0;
    h.bar_count = h.bar_gen = 0;
    h.loop_below = loop_blocks ? kLoopBelow : -1;
    h.pass_words = 0;
    h.drain = 0;
    h.t_limit = (unsigned long long)limit_ms * 1000000ull;
    PH_CUDA(cudaMemcpyAsync(rs.dstate, &h, sizeof(DevState), cudaMemcpyHostToDevice, st));
    k_clock_start<<<1, 1, 0, st>>>(static_cast<DevState*>(rs.dstate));
    PH_CHECK_LAUNCH();
  };
  begin();
  RArgs a = make_args(ctx);

  bool started = false;    // this call has launched passes
  bool in_loop = false;    // the last of them by k_loop
  bool rest_only = false;  // a pass stopped for space after its marks continues at Phase II
  for (;;) {
    const int32_t first_pass = h.pass;
    NvtxRange nvtx_range_(use_graph ? "pass loop (graph)" : "pass");
    bool ran_graph = false;
    const int variant = add_variant(h);
    if (rest_only) {
      rest_only = false;
      launch_pass_rest(ctx, a, 0, false, variant, time_add, st);
      if (time_add) rs.add_launches++;
    } else if (use_graph && loop_blocks && h.ahead == 1 && h.pass_words <= kLoopWords &&
               h.n_act <= (started && !in_loop ? h.loop_below : kLoopStart)) {
      // a state's tag has eight bits: one left by an earlier stay in k_loop could pass for this one's
      if (!in_loop && !loop_states_clear) {
        const int64_t tiles = (std::min<int64_t>(ctx->m, kLoopStart) + kThreads - 1) / kThreads;
        PH_CUDA(cudaMemsetAsync(a.loop_tile_st, 0, tiles * sizeof(unsigned long long), st));
      }
      loop_states_clear = false;
      in_loop = true;
      h.loop_blocks = std::min(loop_blocks, loop_blocks_for(h.n_act));
      PH_CUDA(cudaMemcpyAsync(&static_cast<DevState*>(rs.dstate)->loop_blocks, &h.loop_blocks,
                              sizeof(h.loop_blocks), cudaMemcpyHostToDevice, st));
      RArgs args = a;
      int64_t m = ctx->m;
      void* params[] = {&args, &m};
      const cudaError_t ce = cudaLaunchCooperativeKernel(
          (const void*)k_loop, dim3(h.loop_blocks), dim3(kThreads), params, kLoopSmem, st);
      if (ce == cudaErrorCooperativeLaunchTooLarge || ce == cudaErrorNotSupported) {
        cudaGetLastError();  // a share of the device without room for it: the graph throughout
        loop_blocks = 0;
        in_loop = false;
        h.loop_below = -1;
        PH_CUDA(cudaMemcpyAsync(rs.dstate, &h, sizeof(DevState), cudaMemcpyHostToDevice, st));
        PH_CUDA(cudaStreamSynchronize(st));
        continue;
      }
      PH_CUDA(ce);
      PH_CHECK_LAUNCH();
      rs.loop_ran = true;
    } else {
      if (rs.loop_ran) {  // (a later call on a share of the device without room for k_loop)
        PH_CUDA(cudaMemsetAsync(a.tile_st, 0, (a.loop_tile_st - a.tile_st) * sizeof(unsigned long long),
                                st));
        rs.loop_ran = false;
      }
      in_loop = false;
      if (use_graph) {
        ran_graph = true;
        PH_CUDA(cudaGraphLaunch(pass_graph(ctx, a, variant), st));
      } else {
        launch_pass(ctx, a, 0, false, variant, time_add, st);
        if (time_add) rs.add_launches++;
      }
    }
    started = true;
    PH_CUDA(cudaMemcpyAsync(&h, rs.dstate, sizeof(DevState), cudaMemcpyDeviceToHost, st));
    free_retired(ctx);
    PH_CUDA(cudaStreamSynchronize(st));
    h.bar_count = 0;  // k_loop leaves a pass without space half-way
    if (ran_graph) {  // kernels per executed pass of the graph's loop
      const int32_t last = (h.status == ST_DONE || h.status == ST_CAPPED) ? h.passes : h.pass;
      const int per_pass = (variant >= 10 ? 4 : 3) + (ctx->opts.collect_stats ? 1 : 0);
      ctx->launches += per_pass * (int64_t)(last - first_pass + 1);
    }
    if (h.status == ST_RUN) continue;
    if (h.status == ST_SWITCH) {  // the next pass on, with the bit-packing additions kernel
      h.status = ST_RUN;
      PH_CUDA(cudaMemcpyAsync(rs.dstate, &h, sizeof(DevState), cudaMemcpyHostToDevice, st));
      continue;
    }
    if (h.status == ST_CAPPED && rs.caps_met < rs.caps.size()) {  // after a restart
      rs.caps_met++;
      h.max_passes = next_cap();
      h.pass = h.passes + 1;
      h.status = ST_RUN;
      PH_CUDA(cudaMemcpyAsync(rs.dstate, &h, sizeof(DevState), cudaMemcpyHostToDevice, st));
      continue;
    }
    if (h.status == ST_HOST) {
      if (time_add && rs.ev.size() >= 2) {  // the stopped pass's k_add did no work
        cudaEventDestroy(rs.ev.back());
        rs.ev.pop_back();
        cudaEventDestroy(rs.ev.back());
        rs.ev.pop_back();
        rs.add_launches--;
      }
      // space for Phase II (reasons 1, 2): the pass continues there, its marks made; counter
      // rows (reason 4): asked for between two passes, the next pass runs whole
      rest_only = (h.host_reason & 3) != 0;
      try {
        serve_host_request(ctx, h);
      } catch (const Fail& f) {
        if (f.code != PH_ERR_ALLOC || !rs.lows) throw;
        ctx->err.clear();
        if (h.ahead > 1) {  // (as far as it had come, if the call's cap lies below)
          cap = std::max(cap, h.pass);
          restart_pass_by_pass(ctx);
          rs.fresh = false;
          rest_only = started = in_loop = false;
          loop_states_clear = true;
          begin();
          a = make_args(ctx);
          continue;
        }
        free_ahead(ctx);  // (look-ahead is over)
        a = make_args(ctx);
        serve_host_request(ctx, h);
      }
      if (rest_only) {
        const DevState marked = h;  // what the marks left for the rest of the pass stays
        reset_counters(&h);
        h.n_dirty = marked.n_dirty;
        h.n_due = marked.n_due;
        h.n_enter = marked.n_enter;
        h.scan_end = marked.scan_end;
        h.targets = marked.targets;
      }
      PH_CUDA(cudaMemcpyAsync(rs.dstate, &h, sizeof(DevState), cudaMemcpyHostToDevice, st));
      continue;
    }
    break;
  }
  PH_REQUIRE(h.status != ST_FAULT || h.debug_fault == 0, PH_ERR_CUDA,
             "device bounds check " + std::to_string(h.debug_fault) + " failed (debug build)");
  PH_REQUIRE(h.status != ST_FAULT, PH_ERR_CUDA,
             "a bounded wait in the addition kernel ran out (look-back did not complete)");
  rs.resting = true;
  PH_REQUIRE(h.status != ST_TIMEOUT, PH_ERR_TIMEOUT,
             "the pass loop ran past the time bound (ph_opts.timeout_ms)");
  rs.passes = h.passes;
  if (h.status == ST_CAPPED) rs.caps.push_back(h.passes);
  rs.caps_met = rs.caps.size();
  rs.status = h.status == ST_DONE ? PH_OK : PH_NOT_CONVERGED;
  if (ctx->opts.collect_stats) {
    rs.h_stats.assign((size_t)(rs.passes + 1) * PH_PS_N, 0);
    PH_CUDA(cudaMemcpyAsync(rs.h_stats.data(), rs.pass_stats,
                            rs.h_stats.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  }
  PH_CUDA(cudaStreamSynchronize(st));
  for (size_t i = 0; i + 1 < rs.ev.size(); i += 2) {
    float ms = 0;
    PH_CUDA(cudaEventElapsedTime(&ms, rs.ev[i], rs.ev[i + 1]));
    rs.ms_add += ms;
    rs.add_ms.push_back(ms);
    cudaEventDestroy(rs.ev[i]);
    cudaEventDestroy(rs.ev[i + 1]);
  }
  rs.ev.clear();
  rs.done = true;
  if (rs.status == PH_OK) free_ahead(ctx);
  return rs.status;
}

void essential_estimate(ph_ctx* ctx, int32_t cloud, uint8_t* host_out, int64_t n) {
  ReduceState& rs = ctx->rs;
  uint8_t* d_out = alloc_n<uint8_t>(ctx, n);
  int32_t* d_bad = alloc_n<int32_t>(ctx, 1);
  PH_CUDA(cudaMemsetAsync(d_bad, 0, sizeof(int32_t), ctx->stream));
  const CloudIds ids = cloud_ids(ctx, cloud);
  k_ess_flags<<<grid_for(ctx, ids.n, kThreads), kThreads, 0, ctx->stream>>>(
      ids, static_cast<const ColMeta*>(rs.meta), ctx->beta, rs.owner, ctx->gidx, n, d_out, d_bad);
  PH_CHECK_LAUNCH();
  int32_t* bad = static_cast<int32_t*>(ctx->pinned(sizeof(int32_t)));
  PH_CUDA(cudaMemcpyAsync(bad, d_bad, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
  PH_CUDA(cudaMemcpyAsync(host_out, d_out, (size_t)n, cudaMemcpyDeviceToHost, ctx->stream));
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  ctx->dfree(d_out);
  ctx->dfree(d_bad);
  PH_REQUIRE(*bad == 0, PH_ERR_INVALID, "internal error: filtration index out of range");
}

__global__ void k_pred_out(CloudIds ids, const int32_t* __restrict__ pred,
                           const int64_t* __restrict__ gidx, int64_t n, int32_t* out,
                           int32_t* bad) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ids.n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = ids.id(t);
    const int64_t g = gidx[x];
    if (g < 0 || g >= n) {
      *bad = 1;
      continue;
    }
    const int32_t p = pred[x];
    out[g] = p >= 0 ? (int32_t)gidx[p] : -1;
  }
}

void predicted_lows(ph_ctx* ctx, int32_t cloud, int32_t* host_out, int64_t n) {
  ReduceState& rs = ctx->rs;
  int32_t* d_out = alloc_n<int32_t>(ctx, std::max<int64_t>(n, 1));
  int32_t* d_bad = alloc_n<int32_t>(ctx, 1);
  PH_CUDA(cudaMemsetAsync(d_bad, 0, sizeof(int32_t), ctx->stream));
  const CloudIds ids = cloud_ids(ctx, cloud);
  k_pred_out<<<grid_for(ctx, ids.n, kThreads), kThreads, 0, ctx->stream>>>(ids, rs.pred, ctx->gidx, n,
                                                                         d_out, d_bad);
  PH_CHECK_LAUNCH();
  int32_t* bad = static_cast<int32_t*>(ctx->pinned(sizeof(int32_t)));
  PH_CUDA(cudaMemcpyAsync(bad, d_bad, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
  PH_CUDA(cudaMemcpyAsync(host_out, d_out, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost,
                          ctx->stream));
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  ctx->dfree(d_out);
  ctx->dfree(d_bad);
  PH_REQUIRE(*bad == 0, PH_ERR_INVALID, "internal error: filtration index out of range");
}

// ------------------------------------------------------------------------------------------
// the reduced matrix R of one cloud, CSC over its filtration indices
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int32_t col_rows(const ColMeta& mx) {
  return mx.len >= 0 ? mx.len : mx.ptr[0];  // a bit-packed column's header holds its rows
}

__global__ void k_col_counts(CloudIds ids, const ColMeta* __restrict__ meta,
                             const int64_t* __restrict__ gidx, int64_t n, int32_t* cnt,
                             int32_t* bad) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ids.n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = ids.id(t);
    const int64_t f = gidx[x];
    if (f < 0 || f >= n) {
      *bad = 1;
      continue;
    }
    cnt[f] = col_rows(load_meta(meta + x));
  }
}

// rows as filtration indices of the same cloud, ascending (ids of one dimension and cloud are in
// filtration order); a bitmap is read word by word, bit by bit
// A warp takes 32 columns: each lane its own if it is short, as nearly all are (most are empty), the warp
// together every longer one. With a thread per column the longest column of a 96 x 80 image grid took 64
// us of the kernel's; with a warp per column the read-out of 10.67 M columns took 7.0 ms, now 4.5 (0.56 M,
// most of three rows: 541 -> 456 us; the grid: 110 us either way).
constexpr int32_t kLaneRows = 8;
__global__ void k_col_rows(CloudIds ids, const ColMeta* __restrict__ meta,
                           const int64_t* __restrict__ gidx, const int32_t* __restrict__ seg,
                           const int64_t* __restrict__ seg_start, int nc,
                           const int64_t* __restrict__ off, int64_t n, int64_t nnz, int32_t* out,
                           int32_t* bad) {
  const int lane = lane_id();
  for (int64_t t0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) & ~31; t0 < ids.n;
       t0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = t0 + lane;
    int64_t x = 0, at = 0;
    int32_t len = 0;  // of a bit-packed column: negative
    const int32_t* rows = nullptr;
    if (t < ids.n) {
      x = ids.id(t);
      const int64_t f = gidx[x];
      if (f < 0 || f >= n) {
        *bad = 1;
      } else {
        const ColMeta mx = load_meta(meta + x);
        at = off[f];
        rows = mx.ptr;
        len = mx.len;
        if (at + col_rows(mx) > nnz) {
          *bad = 1;
          len = 0;
        }
      }
    }
    if (len > 0 && len <= kLaneRows)
      for (int q = 0; q < len; q++) out[at + q] = (int32_t)gidx[rows[q]];
    unsigned longer = __ballot_sync(0xffffffffu, len < 0 || len > kLaneRows);
    for (; longer; longer &= longer - 1) {
      const int src = __ffs(longer) - 1;
      const int32_t wlen = __shfl_sync(0xffffffffu, len, src);
      const auto* wrows = reinterpret_cast<const int32_t*>(
          __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(rows), src));
      int32_t* o = out + __shfl_sync(0xffffffffu, at, src);
      if (wlen > 0) {
        for (int64_t q = lane; q < wlen; q += 32) o[q] = (int32_t)gidx[wrows[q]];
        continue;
      }
      const int rs = seg[__shfl_sync(0xffffffffu, x, src)] - nc;
      const int64_t base = seg_start[rs];
      const int64_t words = (seg_start[rs + 1] - base + 31) / 32;
      const uint32_t* bits = reinterpret_cast<const uint32_t*>(wrows + kDenseHead);
      const int64_t room = wrows[0];
      int64_t k = 0;
      for (int64_t w0 = 0; w0 < words; w0 += 32) {
        const uint32_t word = w0 + lane < words ? bits[w0 + lane] : 0;
        const int incl = warp_incl_sum(__popc(word));
        int64_t p = k + incl - __popc(word);
        for (uint32_t b = word; b && p < room; b &= b - 1)
          o[p++] = (int32_t)gidx[base + 32 * (w0 + lane) + (__ffs(b) - 1)];
        k += __shfl_sync(0xffffffffu, incl, 31);
      }
      if (k != room) *bad = 1;
    }
  }
}
void reduced_columns(ph_ctx* ctx, int32_t cloud, int64_t n, int64_t* colptr, int32_t* rows,
                     int64_t capacity, int64_t* nnz_out) {
  ReduceState& rs = ctx->rs;
  const ColMeta* meta = static_cast<const ColMeta*>(rs.meta);
  const CloudIds ids = cloud_ids(ctx, cloud);
  int64_t* d_off = alloc_n<int64_t>(ctx, n + 1);
  int32_t* d_cnt = alloc_n<int32_t>(ctx, n + 2);
  int32_t* d_bad = d_cnt + n;  // bad index, a bounded wait that ran out
  PH_CUDA(cudaMemsetAsync(d_bad, 0, 2 * sizeof(int32_t), ctx->stream));
  k_col_counts<<<grid_for(ctx, n, kThreads), kThreads, 0, ctx->stream>>>(ids, meta, ctx->gidx, n, d_cnt,
                                                                       d_bad);
  PH_CHECK_LAUNCH();
  scan_counts(ctx, d_cnt, nullptr, n, d_off, nullptr, d_bad + 1);
  int32_t* bad = static_cast<int32_t*>(ctx->pinned(2 * sizeof(int32_t)));
  PH_CUDA(cudaMemcpyAsync(bad, d_bad, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
  PH_CUDA(cudaMemcpyAsync(colptr, d_off, (size_t)(n + 1) * sizeof(int64_t),
                          cudaMemcpyDeviceToHost, ctx->stream));
  PH_CUDA(cudaStreamSynchronize(ctx->stream));
  PH_REQUIRE(bad[1] == 0, PH_ERR_CUDA, "a bounded wait of the column scan ran out");
  const int64_t nnz = colptr[n];
  if (nnz_out) *nnz_out = nnz;
  if (bad[0] == 0 && rows && nnz <= capacity && nnz > 0) {
    int32_t* d_rows = alloc_n<int32_t>(ctx, nnz);
    k_col_rows<<<grid_for(ctx, n, kThreads), kThreads, 0, ctx->stream>>>(
        ids, meta, ctx->gidx, ctx->seg, ctx->d_seg_start, ctx->n_clouds, d_off, n, nnz, d_rows, d_bad);
    PH_CHECK_LAUNCH();
    PH_CUDA(cudaMemcpyAsync(bad, d_bad, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    PH_CUDA(cudaMemcpyAsync(rows, d_rows, (size_t)nnz * sizeof(int32_t), cudaMemcpyDeviceToHost,
                            ctx->stream));
    PH_CUDA(cudaStreamSynchronize(ctx->stream));
    ctx->dfree(d_rows);
  }
  ctx->dfree(d_off);
  ctx->dfree(d_cnt);
  PH_REQUIRE(bad[0] == 0, PH_ERR_INVALID, "internal error: column index out of range");
  PH_REQUIRE(!rows || nnz <= capacity, PH_ERR_CAPACITY,
             "rows holds " + std::to_string(capacity) + " entries, the columns need " +
                 std::to_string(nnz));
}

void free_reduce_state(ph_ctx* ctx) {
  ReduceState& rs = ctx->rs;
  for (void* p : {(void*)rs.act, (void*)rs.act2, (void*)rs.alen, (void*)rs.alen2, rs.meta,
                  (void*)rs.nxt_ptr, (void*)rs.nxt_len, (void*)rs.owner, (void*)rs.tab,
                  (void*)rs.first_unp, (void*)rs.dirty, rs.tiles, rs.dstate,
                  rs.look, rs.dlist, rs.src_e, (void*)rs.lows, (void*)rs.due, rs.prec,
                  (void*)rs.delta, (void*)rs.kind, (void*)rs.newpos, (void*)rs.work,
                  (void*)rs.unp_bits, (void*)rs.unp_words,
                  (void*)rs.pred, (void*)rs.set_n, (void*)rs.set_neg, (void*)rs.set_on,
                  (void*)rs.set_key,
                  (void*)rs.pass_stats})
    ctx->dfree(p);
  for (auto& a : rs.arena) ctx->dfree(a.p);
  for (auto& r : rs.retired) ctx->dfree(r.p);
  for (auto& c : rs.pivots) ctx->dfree(c.p);
  for (auto& c : rs.spare) ctx->dfree(c.p);
  for (auto e : rs.ev) cudaEventDestroy(e);
  void* hstate = rs.hstate;  // (page-locked: kept by the context)
  rs = ReduceState{};
  rs.hstate = hstate;
}

}  // namespace ph
