// Local-moving phase (Alg. 5) with Dynamic Frontier expansion.
//
// One iteration visits the frontier in `substeps` hash classes.  For each
// class, the decide kernels (one per degree bin) evaluate every frontier
// vertex i against the membership C', totals Sigma' and sizes left by the
// previous class:
//   scanCommunities: H[c] = sum of w_ij over neighbours j != i with C'[j] = c
//   best c != d = C'[i] by score(c) = 2m*H[c] - K_i*Sigma_c (ties: smaller c)
//   move iff score(c*) > stay = 2m*H[d] - K_i*(Sigma_d - K_i)   (Eq. 2 > 0)
//   except a singleton moving into a singleton community with a larger id.
// A mover is recorded, its numerator score - stay is added to S, and its
// neighbours (in the affected range) are marked for the next iteration
// (Section 4.1: a mover makes its neighbours affected).  The commit kernel then
// applies the class's moves to C', Sigma' and the sizes.
#include <chrono>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "common.cuh"

namespace dfl {

namespace {

struct DecideArgs {
  GraphView g;
  const uint32_t* C;
  const long long* K;
  const long long* Sigma;
  const int* size;
  const long long* m2p;   // 2m, read from device memory so captured graphs stay valid
  const uint32_t* list;
  const unsigned int* count;
  uint32_t* fbits_next;
  uint32_t* next_lists;
  Segs seg;
  int next_buf;
  const uint32_t* rbits;  // affected range, nullptr = every vertex
  uint32_t* ever;         // first-pass processed set, nullptr = not tracked
  uint32_t* mv_i;
  uint32_t* mv_c;
  uint32_t* mv_d;
  Ctrl* ctrl;
  uint32_t k;
  uint2* gtable;          // block bins: per-block global overflow tables
  uint32_t gslots;        // slots per block (power of two)
  uint2* bigmv;           // queue of the movers of degree > kMarkInline (push_row)
  unsigned int* movers;   // movers of the sub-step (slot counter into mv_i/mv_c/mv_d)
  unsigned long long* nbig;  // ... its counter
  unsigned int* clear_movers;  // the next sub-step's three counters, zeroed by this sub-step's
  unsigned long long* clear_nbig;  // commit (null: nothing to zero)
  unsigned int* clear_bignd;
  // group of graphs (ngraphs > 0): the vertex's graph gives its 2m, whether
  // it is still processed, and where its movers' dQ sum goes
  uint32_t ngraphs;
  const uint32_t* goff;   // first vertex of each graph at this level
  const long long* gm2;
  const uint8_t* gdone;
  unsigned long long* gS;
};

// Group lookup for vertex i: false if its graph is no longer processed;
// otherwise its graph and 2m.
__device__ __forceinline__ bool group_active(const DecideArgs& a, uint32_t i, long long* m2,
                                             uint32_t* gi) {
  if (!a.ngraphs) return true;
  const uint32_t g = graph_of(a.goff, a.ngraphs, i);
  if (a.gdone[g]) return false;
  *gi = g;
  *m2 = a.gm2[g];
  return true;
}

// m2 * h - k * sig, the numerator of a modularity gain (Eq. 2 scaled by
// 2m^2; a candidate's score or the stay term).  Every factor is below 2^32:
// 2m < 2^32 holds on every graph (dfl_create and dfl_apply_batch refuse
// more), and h, k and sig are sums of parts of 2m.  So each product is one
// 32 x 32 -> 64-bit multiply, and the difference is exact in 128 bits.
__device__ __forceinline__ i128 gain_num(long long m2, unsigned long long h, long long k, long long sig) {
  const unsigned long long p = (unsigned long long)(uint32_t)m2 * (uint32_t)h;
  const unsigned long long q = (unsigned long long)(uint32_t)k * (uint32_t)sig;
  return (i128)p - (i128)q;
}

// Sigma_c as a 32-bit word (the low half of the int64: Sigma_c is in [0, 2m)).
__device__ __forceinline__ uint32_t sigma32(const long long* Sigma, uint32_t c) {
  return reinterpret_cast<const uint32_t*>(Sigma)[2ull * c];
}

// Outcome of one vertex's decision, identical on every lane / thread.
__device__ __forceinline__ bool decide_move(const DecideArgs& a, long long m2, uint32_t i, uint32_t d,
                                            long long Ki, bool have, i128 best, uint32_t bc,
                                            unsigned long long Hd, i128* gain) {
  if (!have) return false;
  const i128 stay = gain_num(m2, Hd, Ki, a.Sigma[d] - Ki);
  if (!(best > stay)) return false;
  if (a.size[d] == 1 && a.size[bc] == 1 && bc > d) return false;  // singleton-swap guard
  *gain = best - stay;
  return true;
}

// A decide kernel's counters: summed in registers by the thread that owns a
// vertex's outcome, then once per block (flush_sums).
struct MoveSums {
  unsigned long long bytes = 0, processed = 0, ever = 0, s_lo = 0, s_hi = 0;
};

__device__ __forceinline__ void record_move(const DecideArgs& a, uint32_t i, uint32_t c, uint32_t d,
                                            i128 gain, uint32_t gi, MoveSums& sums) {
  uint32_t slot = atomicAdd(a.movers, 1u);
  a.mv_i[slot] = i;
  a.mv_c[slot] = c;
  a.mv_d[slot] = d;
  sums.s_lo += (unsigned long long)((u128)gain & 0xFFFFFFFFull);
  sums.s_hi += (unsigned long long)((u128)gain >> 32);
  if (a.ngraphs) {
    const u128 v = (u128)gain;
    const unsigned long long lo = (unsigned long long)(v & 0xFFFFFFFFull);
    const unsigned long long hi = (unsigned long long)(v >> 32);
    if (lo) atomicAdd(a.gS + 2 * gi, lo);
    if (hi) atomicAdd(a.gS + 2 * gi + 1, hi);
  }
}

// Block-wide sums of the counters held by `holder` threads, one global
// atomic each per block.  Every thread of the block must call it.
__device__ __forceinline__ void flush_sums(const DecideArgs& a, const MoveSums& v, bool holder) {
  __shared__ unsigned long long sh[5];
  if (threadIdx.x < 5) sh[threadIdx.x] = 0;
  __syncthreads();
  if (holder) {
    if (v.bytes) atomicAdd(&sh[0], v.bytes);
    if (v.processed) atomicAdd(&sh[1], v.processed);
    if (v.ever) atomicAdd(&sh[2], v.ever);
    if (v.s_lo) atomicAdd(&sh[3], v.s_lo);
    if (v.s_hi) atomicAdd(&sh[4], v.s_hi);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (sh[0]) atomicAdd(&a.ctrl->move_bytes, sh[0]);
    if (sh[1]) atomicAdd(&a.ctrl->processed, sh[1]);
    if (sh[2]) atomicAdd(&a.ctrl->ever_count, sh[2]);
    if (sh[3]) atomicAdd(&a.ctrl->s_lo, sh[3]);
    if (sh[4]) atomicAdd(&a.ctrl->s_hi, sh[4]);
  }
}

// flush_sums for kernels where every thread holds counts: the warp sums
// them first, so the block's shared counters take one update per warp.
__device__ __forceinline__ void flush_sums_all(const DecideArgs& a, MoveSums v) {
#pragma unroll
  for (int x = 16; x; x >>= 1) {
    v.bytes += __shfl_xor_sync(0xFFFFFFFFu, v.bytes, x);
    v.s_lo += __shfl_xor_sync(0xFFFFFFFFu, v.s_lo, x);
    v.s_hi += __shfl_xor_sync(0xFFFFFFFFu, v.s_hi, x);
  }
  v.processed = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.processed));
  v.ever = __reduce_add_sync(0xFFFFFFFFu, uint32_t(v.ever));
  flush_sums(a, v, (threadIdx.x & 31u) == 0);
}

// The commit marks the movers' neighbours for the next iteration (the decide
// kernels only record the moves): of a mover of at most kMarkInline arcs from
// the mover list, of a larger one from a queue cut into pieces of kMarkChunk
// arcs, so that every mover's arcs are read coalesced and spread over the GPU.
constexpr uint32_t kMarkInline = 512;
constexpr uint32_t kMarkChunk = 512;

__device__ __forceinline__ void queue_marks(const DecideArgs& a, unsigned long long* counter, uint32_t i,
                                            uint32_t dg) {
  push_row(a.bigmv, counter, i, (dg + kMarkChunk - 1) / kMarkChunk);
}

// Mark arcs [k0, k1) of mover i's row at o, this lane's from k0 + first on in
// steps of `step`, four arcs' bitmap words in flight: the neighbours' bits in
// the next frontier's bitmap (the lists are built from it once, at the end of
// the iteration).  The bits are read first, so a vertex marked by many movers
// takes one atomic.  kAppend: a vertex newly marked also goes straight onto its
// list of the next frontier (the small-frontier kernel; the others build the
// lists from the bitmap).
__device__ __forceinline__ void append_next(const DecideArgs& a, uint32_t v) {
  const uint32_t key = vertex_class(v, a.k, a.seg) * kBins + degree_bin(a.g.deg[v], a.seg);
  const uint32_t r = atomicAdd(&a.ctrl->count[a.next_buf][key / kBins][key % kBins], 1u);
  if (r < a.seg.cap[key]) a.next_lists[a.seg.off[key] + r] = v;
  else atomicOr(&a.ctrl->err, kErrInternal);
}

template <bool kAppend>
__device__ __forceinline__ void mark_arcs(const DecideArgs& a, uint32_t i, unsigned long long o, uint32_t k0,
                                          uint32_t k1, uint32_t first, uint32_t step) {
  for (uint32_t b = k0 + first; b < k1; b += 4 * step) {
    uint2 e[4];
    bool on[4];
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) e[u] = b + u * step < k1 ? a.g.arcs[o + b + u * step] : make_uint2(i, 0u);
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      on[u] = e[u].x != i && e[u].y != 0;  // not a self-loop, not a deleted arc
      if (on[u]) on[u] = !bit_test(a.fbits_next, e[u].x);
    }
    if (a.rbits) {
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u) on[u] = on[u] && bit_test(a.rbits, e[u].x);
    }
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u)
      if (on[u] && bit_set(a.fbits_next, e[u].x) && kAppend) append_next(a, e[u].x);
  }
}

// ---------------------------------------------------------------------------
// The tiny bin (at most W <= 32 arcs), W lanes per vertex, so one
// warp decides 32 / W vertices at once, one arc per lane; aggregation by
// community in registers inside each W-lane segment (W shuffles and
// compares).  A long list instead takes a vertex per lane (k_decide_lanes,
// below).
// ---------------------------------------------------------------------------

// Argmax of (score, -c) over the aligned W-lane segment of each lane.
template <int W>
__device__ __forceinline__ void segment_argmax(bool& have, i128& score, uint32_t& c) {
#pragma unroll
  for (int s = W / 2; s >= 1; s >>= 1) {
    unsigned long long lo = (unsigned long long)(u128)score;
    unsigned long long hi = (unsigned long long)((u128)score >> 64);
    unsigned long long olo = __shfl_xor_sync(0xFFFFFFFFu, lo, s);
    unsigned long long ohi = __shfl_xor_sync(0xFFFFFFFFu, hi, s);
    uint32_t oc = __shfl_xor_sync(0xFFFFFFFFu, c, s);
    bool oh = __shfl_xor_sync(0xFFFFFFFFu, have ? 1 : 0, s) != 0;
    i128 os = (i128)(((u128)ohi << 64) | (u128)olo);
    if (oh && (!have || os > score || (os == score && oc < c))) {
      have = true;
      score = os;
      c = oc;
    }
  }
}

// A move: vertex i (row at o, dg arcs, weight K) from community d to c, whose
// numerator 2m^2 * dQ is gain.
struct Move {
  unsigned long long o;
  uint32_t i, d, c, dg, Ki;
  i128 gain;
};

// Decision of one vertex per W-lane segment (`active` false: the segment
// idles).  Every lane of the warp must call it; the move is returned on every
// lane of the segment.  The chain list entry -> row header -> arcs (with
// Sigma and size of the own community) -> communities -> their Sigma bounds it.
template <int W>
__device__ __forceinline__ bool decide_segment(const DecideArgs& a, bool active, uint32_t i, long long m2, Move* mvo,
                                               MoveSums& sums) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t seg = lane / W, sl = lane % W;
  const unsigned segmask = W == 32 ? 0xFFFFFFFFu : (((1u << W) - 1u) << (seg * W));
  const uint32_t d = active ? a.C[i] : 0u;
  const long long Ki = active ? a.K[i] : 0;
  const unsigned long long o = active ? a.g.off[i] : 0ull;
  const uint32_t dg = active ? a.g.deg[i] : 0u;
  const long long Sd = active ? a.Sigma[d] : 0;
  const int szd = active ? a.size[d] : 0;
  uint2 arc = sl < dg ? a.g.arcs[o + sl] : make_uint2(i, 0u);
  const bool valid = sl < dg && arc.x != i && arc.y != 0;  // weight 0 = deleted arc
  const uint32_t c = valid ? a.C[arc.x] : kEmpty;
  // weight of this lane's community within the segment, and whether this is
  // the community's first lane: W shuffles and compares (cheaper here than
  // match/reduce over many groups)
  uint32_t hsum = 0;
  bool leader = valid;
  const uint32_t wv = valid ? arc.y : 0u;
  const uint32_t sg = (valid && c != d) ? sigma32(a.Sigma, c) : 0u;  // (in flight during the rounds)
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const uint32_t src = seg * W + k;
    const uint32_t ck = __shfl_sync(0xFFFFFFFFu, c, src);
    const uint32_t wk = __shfl_sync(0xFFFFFFFFu, wv, src);
    if (valid && ck == c) {
      hsum += wk;
      if (uint32_t(k) < sl) leader = false;
    }
  }
  const unsigned dm = __ballot_sync(0xFFFFFFFFu, leader && c == d) & segmask;
  // every lane shuffles (from its segment's holder of d, or from itself)
  const uint32_t hd_src = dm ? uint32_t(__ffs(dm) - 1) : lane;
  const uint32_t hd_val = __shfl_sync(0xFFFFFFFFu, hsum, hd_src);
  const unsigned long long Hd = dm ? hd_val : 0u;
  const bool cand = leader && c != d;
  const unsigned cm = __ballot_sync(0xFFFFFFFFu, cand) & segmask;
  i128 score = 0;
  if (cand) score = gain_num(m2, hsum, Ki, sg);
  bool have = cand;
  uint32_t bc = c;
  segment_argmax<W>(have, score, bc);
  const i128 stay = gain_num(m2, Hd, Ki, Sd - Ki);
  bool mv = active && have && score > stay;
  if (mv && szd == 1 && bc > d && a.size[bc] == 1) mv = false;  // singleton-swap guard
  if (active && sl == 0) sums.bytes += 24 + 12ull * dg + 12ull * __popc(cm) + (mv ? 16 + 4ull * dg : 0ull);
  *mvo = Move{o, i, d, bc, dg, uint32_t(Ki), score - stay};
  return mv;
}

// The same for list positions [first, first + 32 / W) below cnt; counted as
// processed.  The ever-bit's old value is only looked at after the decision.
template <int W>
__device__ __forceinline__ bool decide_position(const DecideArgs& a, const uint32_t* list, uint64_t first, uint32_t cnt, long long m2_one,
                                                uint32_t* gi, Move* mvo, MoveSums& sums) {
  const uint32_t lane = threadIdx.x & 31u, seg = lane / W, sl = lane % W;
  const uint64_t t = first + seg;
  bool active = t < cnt;
  const uint32_t i = active ? list[t] : 0u;
  long long m2 = m2_one;
  *gi = 0;
  if (active && !group_active(a, i, &m2, gi)) active = false;
  const bool head = active && sl == 0;
  const uint32_t em = 1u << (i & 31u);
  const uint32_t old = (head && a.ever) ? atomicOr(a.ever + (i >> 5), em) : em;
  if (active && a.rbits && !bit_test(a.rbits, i)) active = false;  // processed, not in range
  const bool mv = decide_segment<W>(a, active, i, m2, mvo, sums);
  if (head) {
    ++sums.processed;
    if (!(old & em)) ++sums.ever;
  }
  return mv;
}

template <int W>
__device__ __forceinline__ void decide_segments(const DecideArgs& a, uint64_t first, uint32_t cnt, long long m2_one,
                                                MoveSums& sums) {
  uint32_t gi;
  Move m;
  const bool mv = decide_position<W>(a, a.list, first, cnt, m2_one, &gi, &m, sums);
  if (mv && (threadIdx.x & 31u) % W == 0) record_move(a, m.i, m.c, m.d, m.gain, gi, sums);
}

// Short lists of small vertices: W lanes per vertex of the first list, then
// (list2, if given) a warp per vertex of a second one, whose vertices are
// dealt to the warps from the last one down.  One launch for both: each would
// leave most of the GPU idle.
template <int W>
__global__ void __launch_bounds__(256, 5) k_decide_warp(DecideArgs a, const uint32_t* list2,
                                                        const unsigned int* count2) {
  constexpr uint32_t kSegs = 32 / W;
  const long long m2_one = *a.m2p;
  const uint32_t cnt = *a.count, cnt2 = count2 ? *count2 : 0u;
  // a block without a vertex leaves at once (a replayed graph's grids are fixed)
  const uint64_t bw = blockDim.x >> 5;
  if (blockIdx.x * bw * kSegs >= cnt && (gridDim.x - 1 - blockIdx.x) * bw >= cnt2) return;
  const uint64_t warp = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) >> 5;
  const uint64_t nwarps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
  MoveSums sums;
  for (uint64_t t0 = warp * kSegs; t0 < cnt; t0 += nwarps * kSegs) decide_segments<W>(a, t0, cnt, m2_one, sums);
  a.list = list2;
  for (uint64_t t = nwarps - 1 - warp; t < cnt2; t += nwarps) decide_segments<32>(a, t, cnt2, m2_one, sums);
  flush_sums(a, sums, (threadIdx.x & 31u) % W == 0);
}

// Open-addressing insert (linear probing) of weight w under key c; gives up
// after `limit` probes (the caller then falls back to a larger table).
__device__ __forceinline__ bool table_add(uint32_t* keys, uint32_t* vals, uint32_t mask, uint32_t c,
                                          uint32_t w, uint32_t limit) {
  uint32_t s = hash_move(c) & mask;
  for (uint32_t probe = 0; probe < limit; ++probe) {
    uint32_t prev = keys[s];
    if (prev == kEmpty) prev = atomicCAS(&keys[s], kEmpty, c);
    if (prev == kEmpty || prev == c) {
      atomicAdd(&vals[s], w);
      return true;
    }
    s = (s + 1) & mask;
  }
  return false;
}

// scanCommunities over arcs [k0, dg) of row o, lanes striding by `step`:
// every lane adds its arc's weight under its neighbour's community (shared
// memory atomics).  Grouping equal communities inside the warp first was
// measured slower on this GPU both ways tried: match/reduce when a warp
// holds many communities, and ballot/shuffle rounds that sum the lanes of
// the first pending lane's community (even for hubs whose thousands of arcs
// lead to a few dozen communities, the DF decide phase on R-MAT 2^22 went
// from 0.219 to 0.246-0.296 ms with 2-8 such rounds).  Loads of kUnroll
// chunks are issued before use.
template <int kUnroll>
__device__ __forceinline__ bool scan_row(const DecideArgs& a, uint32_t i, unsigned long long o,
                                         uint32_t dg, uint32_t k0, uint32_t step, uint32_t* keys,
                                         uint32_t* vals, uint32_t mask, uint32_t limit) {
  const uint32_t lane = threadIdx.x & 31u;
  bool ok = true;
  for (uint32_t base = k0; base < dg; base += step * kUnroll) {
    uint2 arc[kUnroll];
    uint32_t c[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      uint32_t k = base + u * step + lane;
      arc[u] = k < dg ? a.g.arcs[o + k] : make_uint2(i, 0u);
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      bool valid = arc[u].x != i && arc[u].y != 0;  // skip self-loops and deleted arcs
      c[u] = valid ? a.C[arc[u].x] : kEmpty;
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      if (c[u] != kEmpty) ok &= table_add(keys, vals, mask, c[u], arc[u].y, limit);
  }
  return ok;
}

// Best candidate of table slots start, start + step, ... below `slots`: U
// slots' keys and values, then their Sigma gathers, are issued before any is
// used, so a thread waits once per U occupied slots.  Returns (per thread)
// the weight to d if this thread met d's slot, and counts candidates.
template <int U>
__device__ __forceinline__ unsigned long long table_argmax(const DecideArgs& a, const uint32_t* keys,
                                                           const uint32_t* vals, uint32_t slots,
                                                           uint32_t start, uint32_t step, uint32_t d,
                                                           long long m2, long long Ki, bool& have,
                                                           i128& best, uint32_t& bc, uint32_t& ncand) {
  unsigned long long hd = 0;
  for (uint32_t s0 = start; s0 < slots; s0 += step * U) {
    uint32_t c[U], w[U];
    long long sg[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t sl = s0 + u * step;
      c[u] = sl < slots ? keys[sl] : kEmpty;
      w[u] = sl < slots ? vals[sl] : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) sg[u] = (c[u] != kEmpty && c[u] != d) ? a.Sigma[c[u]] : 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (c[u] == kEmpty) continue;
      if (c[u] == d) {
        hd = w[u];
        continue;
      }
      ++ncand;
      const i128 sc = gain_num(m2, w[u], Ki, sg[u]);
      if (!have || sc > best || (sc == best && c[u] < bc)) {
        have = true;
        best = sc;
        bc = c[u];
      }
    }
  }
  return hd;
}

// Reduce (have, score, c) of every thread of the block to thread 0 (larger
// score wins, ties to the smaller c); every thread calls it.
constexpr uint32_t kMaxBlockWarps = 32;  // blocks of up to 1024 threads

__device__ __forceinline__ void block_argmax(bool& have, i128& best, uint32_t& bc) {
  __shared__ unsigned long long s_lo[kMaxBlockWarps], s_hi[kMaxBlockWarps];
  __shared__ uint32_t s_c[kMaxBlockWarps];
  __shared__ int s_have[kMaxBlockWarps];
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5, nw = blockDim.x / 32;
  warp_argmax(have, best, bc);
  __syncthreads();
  if (lane == 0) {
    s_lo[wib] = (unsigned long long)(u128)best;
    s_hi[wib] = (unsigned long long)((u128)best >> 64);
    s_c[wib] = bc;
    s_have[wib] = have;
  }
  __syncthreads();
  if (wib == 0) {
    have = lane < nw && s_have[lane];
    best = lane < nw ? (i128)(((u128)s_hi[lane] << 64) | (u128)s_lo[lane]) : 0;
    bc = lane < nw ? s_c[lane] : 0;
    warp_argmax(have, best, bc);
  }
}

// ---------------------------------------------------------------------------
// One warp per vertex with a shared table, a vertex at a time (the persistent
// and small-frontier kernels, and scores of 128 bits).
// ---------------------------------------------------------------------------
constexpr uint32_t kWarpSlots = 512;
constexpr int kWarpHashWarps = 8;
static_assert(kBinWarpHash <= 8 * 32 && 2 * kBinWarpHash <= kWarpSlots, "a table-bin vertex fits 8 arcs a lane and its table");

// One vertex of the table bin by one warp (its degree up to kWarpSlots / 2): up to
// 32 arcs by the register path, else a shared table of the warp.  Every lane
// of the warp calls it.
__device__ __forceinline__ bool warp_table_vertex(const DecideArgs& a, uint32_t i, long long m2, uint32_t* keys,
                                                  uint32_t* vals, Move* mvo, MoveSums& sums) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t dg = a.g.deg[i];
  if (dg <= 32) return decide_segment<32>(a, true, i, m2, mvo, sums);  // (the lane bin's) registers, not a table
  const uint32_t d = a.C[i];
  const long long Ki = a.K[i];
  const unsigned long long o = a.g.off[i];
  uint32_t slots = 64;
  while (slots < 2 * dg && slots < kWarpSlots) slots <<= 1;
  const uint32_t mask = slots - 1;
  for (uint32_t s = lane; s < slots; s += 32) {
    keys[s] = kEmpty;
    vals[s] = 0;
  }
  __syncwarp();
  bool ok = scan_row<8>(a, i, o, dg, 0, 32, keys, vals, mask, slots);
  if (!__all_sync(0xFFFFFFFFu, ok) && lane == 0) atomicOr(&a.ctrl->err, kErrInternal);
  __syncwarp();
  bool have = false;
  i128 best = 0;
  uint32_t bc = 0;
  uint32_t ncand = 0;
  unsigned long long Hd = table_argmax<4>(a, keys, vals, slots, lane, 32, d, m2, Ki, have, best, bc, ncand);
  for (int x = 16; x; x >>= 1) {
    Hd += __shfl_xor_sync(0xFFFFFFFFu, Hd, x);
    ncand += __shfl_xor_sync(0xFFFFFFFFu, ncand, x);
  }
  warp_argmax(have, best, bc);
  i128 gain = 0;
  const bool mv = decide_move(a, m2, i, d, Ki, have, best, bc, Hd, &gain);
  if (lane == 0) sums.bytes += 24 + 12ull * dg + 12ull * ncand + (mv ? 16 + 4ull * dg : 0ull);
  *mvo = Move{o, i, d, bc, dg, uint32_t(Ki), gain};
  __syncwarp();
  return mv;
}

// A move decided by one thread (or the leader of a warp): recorded, and its
// row queued for marking if it is long.
__device__ __forceinline__ void record(const DecideArgs& a, const Move& m, uint32_t gi, MoveSums& sums) {
  record_move(a, m.i, m.c, m.d, m.gain, gi, sums);
  if (m.dg > kMarkInline) queue_marks(a, a.nbig, m.i, m.dg);
}

// ---------------------------------------------------------------------------
// Vertex headers a warp at a time.  A vertex's decision is a chain of
// dependent loads: list entry -> its row offset, degree, community and K ->
// the Sigma and size of its community -> its arcs -> the neighbours'
// communities -> the candidates' Sigma.  The kernels below take the first
// links of that chain for up to 32 list positions at once (one lane each),
// so they wait for them once per batch of vertices instead of once per
// vertex.
// ---------------------------------------------------------------------------

// K_i, Sigma_d and 2m are below 2^32 (2m < 2^32 on every graph, and K_i and
// Sigma_d are parts of 2m), so they travel as 32-bit words.
struct VHdr {
  unsigned long long o;  // row offset
  uint32_t Ki, Sd, m2;   // K_i, Sigma of its community d, 2m of its graph
  uint32_t i, d, dg, gi;
  int szd;               // size of d
  bool act;              // processed and in the affected range: decide it
};

// Exact 64-bit form of Eq. 2's comparisons.  Adding K_i * 2m to every score
// of vertex i shifts them all by the same amount:
//   score'(c) = 2m * H[c] + K_i * (2m - Sigma_c)           (a candidate c)
//   stay'     = 2m * H[d] + K_i * (2m - (Sigma_d - K_i))
// so the best candidate, the move test score > stay and the gain score - stay
// are unchanged.  Each is at most 2 * 2m * K_i (H[c] <= K_i and Sigma_c <= 2m),
// so it fits 64 bits whenever 2m * K_i < 2^63, which holds unless 2m and K_i
// both approach 2^32; those vertices take the 128-bit path.  A candidate's
// score' is at least 1 (H[c] >= 1).
__device__ __forceinline__ bool fits64(uint32_t m2, uint32_t Ki) {
  return (unsigned long long)m2 * Ki < (1ull << 63);
}
__device__ __forceinline__ unsigned long long score64(uint32_t m2, uint32_t h, uint32_t Ki, uint32_t sig) {
  return (unsigned long long)m2 * h + (unsigned long long)Ki * (m2 - sig);
}

// Warp-wide best (largest score', then smallest c) of the lanes with `have`,
// by three warp reductions; the result on every lane.
__device__ __forceinline__ void warp_best64(bool& have, unsigned long long& s, uint32_t& c) {
  const uint32_t hi = have ? uint32_t(s >> 32) : 0u, lo = have ? uint32_t(s) : 0u;
  const uint32_t mh = __reduce_max_sync(0xFFFFFFFFu, hi);
  const uint32_t ml = __reduce_max_sync(0xFFFFFFFFu, (have && hi == mh) ? lo : 0u);
  c = __reduce_min_sync(0xFFFFFFFFu, (have && hi == mh && lo == ml) ? c : kEmpty);
  s = ((unsigned long long)mh << 32) | ml;
  have = c != kEmpty;
}

// This lane's header of list position t (`valid`: t is in the list).  The
// vertex is counted as processed (and newly ever-processed) as in the
// per-vertex kernels.
__device__ __forceinline__ void load_header(const DecideArgs& a, uint64_t t, bool valid, long long m2_one,
                                            MoveSums& sums, VHdr& h) {
  h.i = valid ? a.list[t] : 0u;
  long long m2 = m2_one;
  h.gi = 0;
  if (valid && !group_active(a, h.i, &m2, &h.gi)) valid = false;
  h.m2 = uint32_t(m2);
  // the row and state loads are issued before the bookkeeping atomics
  h.d = valid ? a.C[h.i] : 0u;
  h.Ki = valid ? uint32_t(a.K[h.i]) : 0u;
  h.o = valid ? a.g.off[h.i] : 0ull;
  h.dg = valid ? a.g.deg[h.i] : 0u;
  bool inr = valid;
  if (valid) {
    if (a.ever && bit_set(a.ever, h.i)) ++sums.ever;
    ++sums.processed;
    if (a.rbits) inr = bit_test(a.rbits, h.i);
  }
  h.act = inr;
  h.Sd = inr ? sigma32(a.Sigma, h.d) : 0u;
  h.szd = inr ? a.size[h.d] : 0;
}

__device__ __forceinline__ VHdr shfl_header(const VHdr& h, int k) {
  VHdr v;
  v.o = __shfl_sync(0xFFFFFFFFu, h.o, k);
  v.Ki = __shfl_sync(0xFFFFFFFFu, h.Ki, k);
  v.Sd = __shfl_sync(0xFFFFFFFFu, h.Sd, k);
  v.m2 = __shfl_sync(0xFFFFFFFFu, h.m2, k);
  v.i = __shfl_sync(0xFFFFFFFFu, h.i, k);
  v.d = __shfl_sync(0xFFFFFFFFu, h.d, k);
  v.dg = __shfl_sync(0xFFFFFFFFu, h.dg, k);
  v.gi = __shfl_sync(0xFFFFFFFFu, h.gi, k);
  v.szd = __shfl_sync(0xFFFFFFFFu, h.szd, k);
  v.act = true;
  return v;
}

// The move decision of Eq. 2 from the best candidate (score' form), with the
// community's Sigma and size already loaded: the best candidate's size is
// read only when the singleton-swap guard needs it.
__device__ __forceinline__ bool decide64(const DecideArgs& a, const VHdr& v, bool have, unsigned long long best,
                                         uint32_t bc, uint32_t Hd, i128* gain) {
  if (!have) return false;
  const unsigned long long stay = score64(v.m2, Hd, v.Ki, v.Sd - v.Ki);
  if (!(best > stay)) return false;
  if (v.szd == 1 && bc > v.d && a.size[bc] == 1) return false;  // singleton-swap guard
  *gain = (i128)(best - stay);
  return true;
}

// record_move for every mover lane of the warp with one slot reservation.
// Every lane of the warp calls it.
__device__ __forceinline__ void record_moves_warp(const DecideArgs& a, bool mv, uint32_t i, uint32_t c,
                                                  uint32_t d, i128 gain, uint32_t gi, MoveSums& sums) {
  const unsigned m = __ballot_sync(0xFFFFFFFFu, mv);
  if (!m) return;
  const uint32_t lane = threadIdx.x & 31u;
  const int first = __ffs(m) - 1;
  uint32_t base = 0;
  if (int(lane) == first) base = atomicAdd(a.movers, uint32_t(__popc(m)));
  base = __shfl_sync(0xFFFFFFFFu, base, first);
  if (!mv) return;
  const uint32_t slot = base + __popc(m & ((1u << lane) - 1u));
  a.mv_i[slot] = i;
  a.mv_c[slot] = c;
  a.mv_d[slot] = d;
  const u128 v = (u128)gain;
  const unsigned long long lo = (unsigned long long)(v & 0xFFFFFFFFull);
  const unsigned long long hi = (unsigned long long)(v >> 32);
  sums.s_lo += lo;
  sums.s_hi += hi;
  if (a.ngraphs) {
    if (lo) atomicAdd(a.gS + 2 * gi, lo);
    if (hi) atomicAdd(a.gS + 2 * gi + 1, hi);
  }
}

// ---------------------------------------------------------------------------
// Long lists of small vertices (bins 0 and 1: at most 32 arcs): a lane per
// vertex.  Issue slots bound these kernels (the gathers of 32 vertices are in
// flight together), so the communities are grouped by a sorting network over
// registers instead of comparing every pair: a key is (community << 5 | arc),
// one 32-bit word, so a comparator is a min and a max, and the arcs' weights
// wait in shared memory until their order is known.  A run of equal
// communities is scored at its last key; runs come in ascending order, so the
// first best wins the tie.
// On 100,000 vertices of mean degree 16 (one sub-step of a 400,000-vertex
// graph) a warp per vertex, with a shuffle and compare round per arc, issued
// 354 instructions a vertex and took 65 us; a lane or two per vertex comparing
// all pairs 165 and 60 us; this 91 and 40 us (492,000 vertices: 414 -> 226 us).
// ---------------------------------------------------------------------------
constexpr uint32_t kLaneLabels = (1u << 27) - 1;  // labels below this fit a key (and ~0 is none of theirs)
constexpr int kLaneThreads = 128;

// Batcher's odd-even merge sort of N keys, ascending: the comparators of stage
// (P, K) join i and i + K within blocks of 2P.
template <int N, int P = 1, int K = 1>
__device__ __forceinline__ void sort_keys(uint32_t (&x)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i >= K % P && (i - K % P) % (2 * K) < K && i + K < N && i / (2 * P) == (i + K) / (2 * P)) {
      const uint32_t lo = min(x[i], x[i + K]), hi = max(x[i], x[i + K]);
      x[i] = lo;
      x[i + K] = hi;
    }
  if constexpr (K > 1) sort_keys<N, P, K / 2>(x);
  else if constexpr (2 * P < N) sort_keys<N, 2 * P, 2 * P>(x);
}

// Decision of this lane's vertex v (if v.act; at most D arcs, scores in 64
// bits).  `w`: this lane's column of the warp's weights, 32 words apart.  Rows
// start 16-byte aligned and have an even capacity, so the pair of an odd last
// arc is readable.
template <int D>
__device__ __forceinline__ bool lane_vertex(const DecideArgs& a, const VHdr& v, uint32_t* w, uint32_t* bco,
                                            unsigned long long* gain, uint32_t* ncand) {
  const uint4* row = reinterpret_cast<const uint4*>(a.g.arcs + v.o);
  const uint32_t dg = v.act ? v.dg : 0u;
  uint32_t key[D];
#pragma unroll
  for (int q = 0; q < D / 2; ++q) {
    const uint4 x = 2 * q < dg ? row[q] : make_uint4(v.i, 0u, v.i, 0u);
    // self-loops and deleted arcs (weight 0) are no arcs
    key[2 * q] = x.y ? x.x : v.i;
    key[2 * q + 1] = (x.w && 2 * q + 1 < dg) ? x.z : v.i;
    w[(2 * q) * 32] = x.y;
    w[(2 * q + 1) * 32] = x.w;
  }
#pragma unroll
  for (int k = 0; k < D; ++k) key[k] = key[k] != v.i ? (a.C[key[k]] << 5) | uint32_t(k) : kEmpty;
  sort_keys<D>(key);
  uint32_t Hd = 0, nc = 0, run = 0, bc = kEmpty;
  unsigned long long best = 0;  // (a candidate's score' is at least 1)
#pragma unroll
  for (int k0 = 0; k0 < D; k0 += 8) {  // eight runs' Sigma in flight
    uint32_t sg[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + u;
      const uint32_t c = key[k] >> 5;
      const bool last = key[k] != kEmpty && (k + 1 == D || (key[k + 1 < D ? k + 1 : k] >> 5) != c);
      sg[u] = (last && c != v.d) ? sigma32(a.Sigma, c) : 0u;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + u;
      const uint32_t c = key[k] >> 5;
      const bool last = key[k] != kEmpty && (k + 1 == D || (key[k + 1 < D ? k + 1 : k] >> 5) != c);
      run += key[k] != kEmpty ? w[(key[k] & 31u) * 32] : 0u;
      if (last) {
        if (c == v.d) {
          Hd = run;
        } else {
          ++nc;
          const unsigned long long sc = score64(v.m2, run, v.Ki, sg[u]);
          if (sc > best) {
            best = sc;
            bc = c;
          }
        }
        run = 0;
      }
    }
  }
  *bco = bc;
  *ncand = nc;
  i128 g = 0;
  const bool mv = v.act && decide64(a, v, bc != kEmpty, best, bc, Hd, &g);
  *gain = (unsigned long long)g;  // a gain is positive and below 2^64
  return mv;
}

// The rare vertices whose scores need 128 bits, a warp each, out of line.
__device__ __noinline__ void lane_vertices_128(const DecideArgs& a, const VHdr& h, unsigned m, MoveSums& sums) {
  for (; m; m &= m - 1) {
    const VHdr v = shfl_header(h, __ffs(m) - 1);
    Move mv;
    if (decide_segment<32>(a, true, v.i, v.m2, &mv, sums) && (threadIdx.x & 31u) == 0)
      record_move(a, v.i, mv.c, mv.d, mv.gain, v.gi, sums);
  }
}

// Vertices of at most D arcs (D = 8, or 32: a warp with no vertex over 16 arcs
// sorts 16 keys).  Labels must be below kLaneLabels.
template <int D>
__global__ void __launch_bounds__(kLaneThreads, D == 8 ? 8 : 5) k_decide_lanes(DecideArgs a) {
  __shared__ uint32_t s_w[kLaneThreads / 32][D][32];
  const long long m2_one = *a.m2p;
  const uint32_t cnt = *a.count;
  if (blockIdx.x * uint64_t(blockDim.x) >= cnt) return;  // no vertex for this block
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t* w = &s_w[threadIdx.x >> 5][0][lane];
  const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
  MoveSums sums;
  for (uint64_t t0 = blockIdx.x * uint64_t(blockDim.x) + (threadIdx.x & ~31u); t0 < cnt; t0 += stride) {
    const uint64_t t = t0 + lane;  // warp-uniform loop: the movers are recorded per warp
    VHdr h;
    load_header(a, t, t < cnt, m2_one, sums, h);
    const unsigned wide = __ballot_sync(0xFFFFFFFFu, h.act && !fits64(h.m2, h.Ki));
    if (wide) {
      lane_vertices_128(a, h, wide, sums);
      if ((wide >> lane) & 1u) h.act = false;
    }
    uint32_t bc = 0, ncand = 0;
    unsigned long long gain = 0;
    bool mv;
    if (D == 8) mv = lane_vertex<8>(a, h, w, &bc, &gain, &ncand);
    else if (__any_sync(0xFFFFFFFFu, h.act && h.dg > 16)) mv = lane_vertex<D>(a, h, w, &bc, &gain, &ncand);
    else mv = lane_vertex<16>(a, h, w, &bc, &gain, &ncand);
    if (h.act) sums.bytes += 24 + 12ull * h.dg + 12ull * ncand + (mv ? 16 + 4ull * h.dg : 0ull);
    record_moves_warp(a, mv, h.i, bc, h.d, (i128)gain, h.gi, sums);
  }
  flush_sums_all(a, sums);
}

// ---------------------------------------------------------------------------
// The table bin: one warp per vertex (more than 32 arcs), vertices taken in
// batches of up to 32 headers, each decided in the warp's shared table.  The
// table is empty at rest: the lane that creates a community's slot loads that community's Sigma at once,
// and after the last arc is in, scores the slot and clears it, so the table
// is neither cleared nor scanned as a whole.  Vertices whose scores need
// 128 bits take the per-vertex path of the persistent kernel.
// ---------------------------------------------------------------------------

// Decision of vertex v (32 < degree <= 32 U) in the warp's table (keys kEmpty
// and values 0 at rest, and left so).  `a0` is this lane's first arc,
// loaded ahead.  Returns the decision on every lane.
template <int U>
__device__ __forceinline__ bool table_vertex(const DecideArgs& a, const VHdr& v, uint2 a0, uint32_t* keys,
                                             uint32_t* vals, uint32_t* bco, i128* gain, uint32_t* ncand) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t slots = 64;
  while (slots < 2 * v.dg) slots <<= 1;  // at most 64 U: never full
  const uint32_t mask = slots - 1;
  uint2 arc[U];
  arc[0] = a0;
#pragma unroll
  for (int u = 1; u < U; ++u) {
    const uint32_t k = u * 32 + lane;
    arc[u] = k < v.dg ? a.g.arcs[v.o + k] : make_uint2(v.i, 0u);
  }
  uint32_t c[U];
#pragma unroll
  for (int u = 0; u < U; ++u) c[u] = (arc[u].x != v.i && arc[u].y != 0) ? a.C[arc[u].x] : kEmpty;
  uint32_t cs[U], sg[U];
  bool ok = true;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    cs[u] = kEmpty;
    sg[u] = 0;
    if (c[u] == kEmpty) continue;
    uint32_t s = hash_move(c[u]) & mask;
    bool placed = false;
    for (uint32_t probe = 0; probe < slots; ++probe) {
      uint32_t prev = keys[s];
      if (prev == kEmpty) prev = atomicCAS(&keys[s], kEmpty, c[u]);
      if (prev == kEmpty) {  // created: this lane scores the slot
        cs[u] = s;
        if (c[u] != v.d) sg[u] = sigma32(a.Sigma, c[u]);
      }
      if (prev == kEmpty || prev == c[u]) {
        atomicAdd(&vals[s], arc[u].y);
        placed = true;
        break;
      }
      s = (s + 1) & mask;
    }
    ok &= placed;
  }
  if (!__all_sync(0xFFFFFFFFu, ok) && lane == 0) atomicOr(&a.ctrl->err, kErrInternal);
  __syncwarp();  // every arc is in
  bool have = false;
  unsigned long long best = 0;
  uint32_t bc = 0, nc = 0, Hd = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (cs[u] == kEmpty) continue;
    const uint32_t hw = vals[cs[u]];
    keys[cs[u]] = kEmpty;  // only this lane reads the slot it created
    vals[cs[u]] = 0;
    if (c[u] == v.d) {
      Hd = hw;
      continue;
    }
    ++nc;
    const unsigned long long sc = score64(v.m2, hw, v.Ki, sg[u]);
    if (!have || sc > best || (sc == best && c[u] < bc)) {
      have = true;
      best = sc;
      bc = c[u];
    }
  }
  __syncwarp();  // the table is empty again before the next vertex
  Hd = __reduce_add_sync(0xFFFFFFFFu, Hd);
  *ncand = __reduce_add_sync(0xFFFFFFFFu, nc);
  warp_best64(have, best, bc);
  *bco = bc;
  return decide64(a, v, have, best, bc, Hd, gain);
}

// The rare 128-bit vertices, out of line so that they do not cost the common
// path registers.
__device__ __noinline__ void warp_vertex_128(const DecideArgs& a, const VHdr& v, uint32_t* keys, uint32_t* vals,
                                             MoveSums& sums) {
  Move m;
  if (warp_table_vertex(a, v.i, v.m2, keys, vals, &m, sums) && (threadIdx.x & 31u) == 0) record(a, m, v.gi, sums);
}

__global__ void __launch_bounds__(256, 3) k_decide_warp_hash(DecideArgs a) {
  __shared__ uint32_t skeys[kWarpHashWarps][kWarpSlots];
  __shared__ uint32_t svals[kWarpHashWarps][kWarpSlots];
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  const long long m2_one = *a.m2p;
  const uint32_t cnt = *a.count;
  const uint64_t warp = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) >> 5;
  const uint64_t nwarps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
  // vertices per warp and round: up to 32, fewer when the list is short
  uint64_t B = (uint64_t(cnt) + nwarps - 1) / nwarps;
  B = B < 1 ? 1 : B > 32 ? 32 : B;
  if (blockIdx.x * uint64_t(kWarpHashWarps) * B >= cnt) return;  // no vertex for this block
  uint32_t* keys = skeys[wib];
  uint32_t* vals = svals[wib];
  for (uint32_t s = lane; s < kWarpSlots; s += 32) {
    keys[s] = kEmpty;
    vals[s] = 0;
  }
  __syncwarp();
  MoveSums sums;
  for (uint64_t t0 = warp * B; t0 < cnt; t0 += nwarps * B) {
    VHdr h;
    load_header(a, t0 + lane, lane < B && t0 + lane < cnt, m2_one, sums, h);
    bool my_mv = false;
    uint32_t my_c = 0;
    i128 my_gain = 0;
    unsigned m = __ballot_sync(0xFFFFFFFFu, h.act);
    // each vertex's first 32 arcs are loaded while the one before is decided
    uint2 pre = make_uint2(0u, 0u);
    if (m) {
      const int k = __ffs(m) - 1;
      const unsigned long long o = __shfl_sync(0xFFFFFFFFu, h.o, k);
      const uint32_t dg = __shfl_sync(0xFFFFFFFFu, h.dg, k), i = __shfl_sync(0xFFFFFFFFu, h.i, k);
      pre = lane < dg ? a.g.arcs[o + lane] : make_uint2(i, 0u);
    }
    while (m) {
      const int k = __ffs(m) - 1;
      m &= m - 1;
      const VHdr v = shfl_header(h, k);
      const uint2 a0 = pre;
      if (m) {
        const int k1 = __ffs(m) - 1;
        const unsigned long long o = __shfl_sync(0xFFFFFFFFu, h.o, k1);
        const uint32_t dg = __shfl_sync(0xFFFFFFFFu, h.dg, k1), i = __shfl_sync(0xFFFFFFFFu, h.i, k1);
        pre = lane < dg ? a.g.arcs[o + lane] : make_uint2(i, 0u);
      }
      if (!fits64(v.m2, v.Ki)) {  // 128-bit scores: the per-vertex path, then the table emptied again
        warp_vertex_128(a, v, keys, vals, sums);
        for (uint32_t s = lane; s < kWarpSlots; s += 32) {
          keys[s] = kEmpty;
          vals[s] = 0;
        }
        __syncwarp();
        continue;
      }
      uint32_t bc = 0, ncand = 0;
      i128 gain = 0;
      bool mv;
      if (v.dg <= 64) {
        mv = table_vertex<2>(a, v, a0, keys, vals, &bc, &gain, &ncand);
      } else if (v.dg <= 128) {
        mv = table_vertex<4>(a, v, a0, keys, vals, &bc, &gain, &ncand);
      } else {
        mv = table_vertex<8>(a, v, a0, keys, vals, &bc, &gain, &ncand);
      }
      if (int(lane) == k) {
        sums.bytes += 24 + 12ull * v.dg + 12ull * ncand + (mv ? 16 + 4ull * v.dg : 0ull);
        my_mv = mv;
        my_c = bc;
        my_gain = gain;
      }
    }
    record_moves_warp(a, my_mv, h.i, my_c, h.d, my_gain, h.gi, sums);
  }
  flush_sums_all(a, sums);
}

// ---------------------------------------------------------------------------
// One block per vertex with a shared table of kBlockSlots (a degree above
// kBinBlock, which only a tuning sends here, may overflow it: the vertex is then
// redone with a table in a per-block slice of global memory sized from the
// maximum degree).
// ---------------------------------------------------------------------------
constexpr uint32_t kBlockSlots = 2 * kBinBlock;  // 8192 keys + 8192 values = 64 KB

// Shared scalars of the block-level bodies.
struct BlockScratch {
  unsigned long long hd;
  uint32_t ncand;
  int ok, last;
};

// One vertex by the whole block (up to 512 threads): a shared table of
// 2 x degree slots at `dyn` (at most kSlots keys + values); a vertex of
// larger degree whose distinct communities overflow it is redone in the
// block's slice of the global table.  Every thread of the block calls it.
// The decision and its move are thread 0's.
template <int kThreads, uint32_t kSlots>
__device__ __forceinline__ bool block_vertex(const DecideArgs& a, uint32_t i, long long m2, uint32_t* dyn,
                                             BlockScratch& sc, Move* mvo, MoveSums& sums) {
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  constexpr uint32_t nthr = kThreads;  // compile-time strides
  const uint32_t d = a.C[i];
  const long long Ki = a.K[i];
  const unsigned long long o = a.g.off[i];
  const uint32_t dg = a.g.deg[i];
  uint32_t slots = 1024;
  while (slots < 2 * dg && slots < kSlots) slots <<= 1;
  uint32_t* keys = dyn;
  uint32_t* vals = dyn + slots;
  bool global = false;
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (attempt == 1) {  // shared table overflowed: global slice of gslots
      global = true;
      slots = a.gslots;
      keys = reinterpret_cast<uint32_t*>(a.gtable + uint64_t(blockIdx.x) * a.gslots);
      vals = keys + a.gslots;
    }
    const uint32_t mask = slots - 1;
    for (uint32_t s = threadIdx.x; s < slots; s += nthr) {
      keys[s] = kEmpty;
      vals[s] = 0;
    }
    if (threadIdx.x == 0) {
      sc.hd = 0;
      sc.ncand = 0;
      sc.ok = 1;
    }
    __syncthreads();
    // a table of >= 2 * deg slots cannot overflow: probe it to the end;
    // a smaller shared table gives up early and falls back
    const uint32_t limit = (global || slots >= 2 * dg) ? slots : 64;
    bool ok = scan_row<8>(a, i, o, dg, wib * 32, nthr, keys, vals, mask, limit);
    if (!ok) sc.ok = 0;
    __syncthreads();
    const bool done = sc.ok;
    __syncthreads();  // everyone has read sc.ok before the retry resets it
    if (done) break;
    if (global || !a.gtable) {
      if (threadIdx.x == 0) atomicOr(&a.ctrl->err, kErrInternal);
      break;
    }
  }
  bool have = false;
  i128 best = 0;
  uint32_t bc = 0;
  uint32_t ncand = 0;
  {
    const unsigned long long hd = table_argmax<4>(a, keys, vals, slots, threadIdx.x, nthr, d, m2, Ki,
                                                   have, best, bc, ncand);
    if (hd) sc.hd = hd;  // exactly one slot holds d
  }
  for (int x = 16; x; x >>= 1) ncand += __shfl_xor_sync(0xFFFFFFFFu, ncand, x);
  if (lane == 0 && ncand) atomicAdd(&sc.ncand, ncand);
  block_argmax(have, best, bc);
  bool mv = false;
  if (threadIdx.x == 0) {
    i128 gain = 0;
    mv = decide_move(a, m2, i, d, Ki, have, best, bc, sc.hd, &gain);
    sums.bytes += 24 + 12ull * dg + 12ull * sc.ncand + (mv ? 16 + 4ull * dg : 0ull);
    *mvo = Move{o, i, d, bc, dg, uint32_t(Ki), gain};
  }
  __syncthreads();
  return mv;
}

// The block bins: one block per vertex, of 128 threads with a table of 2,048
// slots up to kMidDeg arcs, else of block_threads with kBlockSlots slots.  The
// barriers between a vertex's phases bound it, so the smaller bin's gain is
// eight vertices in progress per SM instead of three (ND on the 2^22-vertex
// R-MAT graph: 452 us of block kernels an iteration in one bin, 185 + 158 in two).
// Headers are loaded by warp 0 for up to 32 of the block's vertices at once.
// The shared table (kSlots keys + values) is empty at rest: a vertex uses the first power of two >= 2 x degree slots, and the scan that
// scores the occupied slots also clears them.  Two block barriers per
// vertex: after the inserts, and after the per-warp bests; warp 0 then
// decides while the other warps start the next vertex (the per-vertex
// scratch is double-buffered), the batch's movers are recorded together at
// its end, and their neighbours are marked by the commit kernel (the mover
// list it spreads over all blocks).  Vertices of degree above kBinBlock, or
// whose scores need 128 bits, take block_vertex (which may fall back to a
// global table) and the table is emptied after it.
template <int kThreads, uint32_t kSlots>
__device__ __noinline__ void block_vertex_slow(const DecideArgs& a, const VHdr& v, uint32_t* dyn, BlockScratch& sc,
                                               MoveSums& sums) {
  Move m;
  if (block_vertex<kThreads, kSlots>(a, v.i, v.m2, dyn, sc, &m, sums)) record(a, m, v.gi, sums);
}

template <int kThreads, uint32_t kSlots>
__global__ void __launch_bounds__(kThreads) k_decide_block(DecideArgs a) {
  extern __shared__ __align__(16) uint32_t dyn[];
  uint32_t* keys = dyn;
  uint32_t* vals = dyn + kSlots;
  __shared__ BlockScratch sc;  // the 128-bit path's
  __shared__ VHdr s_hdr[32];
  __shared__ unsigned long long s_best[2][kMaxBlockWarps];
  __shared__ uint32_t s_bc[2][kMaxBlockWarps];
  __shared__ uint32_t s_hd[2], s_nc[2];
  __shared__ unsigned long long s_gain[32];
  __shared__ uint32_t s_mvc[32];
  __shared__ int s_mv[32];
  constexpr uint32_t nthr = kThreads;
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  const long long m2_one = *a.m2p;
  const uint32_t cnt = *a.count;
  if (blockIdx.x >= cnt) return;  // no vertex for this block
  const uint64_t G = gridDim.x;
  for (uint32_t s = threadIdx.x; s < kSlots; s += nthr) {
    keys[s] = kEmpty;
    vals[s] = 0;
  }
  if (threadIdx.x < 2) {
    s_hd[threadIdx.x] = 0;
    s_nc[threadIdx.x] = 0;
  }
  MoveSums sums;
  __syncthreads();
  for (uint64_t t0 = blockIdx.x; t0 < cnt; t0 += 32 * G) {
    if (wib == 0) {
      const uint64_t t = t0 + lane * G;
      VHdr h;
      load_header(a, t, t < cnt, m2_one, sums, h);
      s_hdr[lane] = h;
      s_mv[lane] = 0;
    }
    __syncthreads();
    const uint64_t left = (uint64_t(cnt) - t0 + G - 1) / G;
    const uint32_t nv = uint32_t(left < 32 ? left : 32);
    uint32_t p = 0;  // scratch buffer of the current vertex
    for (uint32_t k = 0; k < nv; ++k) {
      const VHdr v = s_hdr[k];
      if (!v.act) continue;  // block-uniform
      if (v.dg > kSlots / 2 || !fits64(v.m2, v.Ki)) {
        __syncthreads();  // warp 0 has finished the decisions before (it uses sc)
        block_vertex_slow<kThreads, kSlots>(a, v, dyn, sc, sums);
        for (uint32_t s = threadIdx.x; s < kSlots; s += nthr) {
          keys[s] = kEmpty;
          vals[s] = 0;
        }
        __syncthreads();
        continue;
      }
      uint32_t slots = 64;
      while (slots < 2 * v.dg) slots <<= 1;
      const uint32_t mask = slots - 1;
      // every arc's weight under its neighbour's community (a table of
      // >= 2 x degree slots cannot overflow)
      const bool ok = scan_row<8>(a, v.i, v.o, v.dg, wib * 32, nthr, keys, vals, mask, slots);
      if (!ok) atomicOr(&a.ctrl->err, kErrInternal);
      __syncthreads();
      // score the occupied slots and clear them; four slots' Sigma loads in flight
      bool have = false;
      unsigned long long best = 0;
      uint32_t bc = 0, nc = 0;
      for (uint32_t s0 = threadIdx.x; s0 < slots; s0 += nthr * 4) {
        uint32_t c[4], w[4], sg[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t sl = s0 + u * nthr;
          c[u] = sl < slots ? keys[sl] : kEmpty;
          w[u] = c[u] != kEmpty ? vals[sl] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) sg[u] = (c[u] != kEmpty && c[u] != v.d) ? sigma32(a.Sigma, c[u]) : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (c[u] == kEmpty) continue;
          const uint32_t sl = s0 + u * nthr;
          keys[sl] = kEmpty;
          vals[sl] = 0;
          if (c[u] == v.d) {
            s_hd[p] = w[u];  // exactly one slot holds d
            continue;
          }
          ++nc;
          const unsigned long long s = score64(v.m2, w[u], v.Ki, sg[u]);
          if (!have || s > best || (s == best && c[u] < bc)) {
            have = true;
            best = s;
            bc = c[u];
          }
        }
      }
      nc = __reduce_add_sync(0xFFFFFFFFu, nc);
      if (lane == 0 && nc) atomicAdd(&s_nc[p], nc);
      warp_best64(have, best, bc);
      if (lane == 0) {
        s_best[p][wib] = have ? best : 0ull;
        s_bc[p][wib] = bc;
      }
      __syncthreads();
      if (wib == 0) {  // the other warps go on to the next vertex
        have = lane < nthr / 32 && s_bc[p][lane] != kEmpty;
        best = have ? s_best[p][lane] : 0ull;
        bc = have ? s_bc[p][lane] : kEmpty;
        warp_best64(have, best, bc);
        if (lane == 0) {
          i128 gain = 0;
          const bool mv = decide64(a, v, have, best, bc, s_hd[p], &gain);
          sums.bytes += 24 + 12ull * v.dg + 12ull * s_nc[p] + (mv ? 16 + 4ull * v.dg : 0ull);
          s_mv[k] = mv;
          s_mvc[k] = bc;
          s_gain[k] = (unsigned long long)gain;  // a gain is positive and below 2^64
          s_hd[p] = 0;  // ready for the vertex after next
          s_nc[p] = 0;
        }
      }
      p ^= 1;
    }
    __syncthreads();  // every decision of the batch is made
    if (wib == 0) {  // the batch's movers: one slot reservation
      const bool mv = lane < nv && s_mv[lane];
      const VHdr& v = s_hdr[lane];
      record_moves_warp(a, mv, v.i, s_mvc[lane], v.d, (i128)s_gain[lane], v.gi, sums);
      if (mv && v.dg > kMarkInline) queue_marks(a, a.nbig, v.i, v.dg);
    }
    __syncthreads();  // s_hdr and s_mv are rewritten by the next round
  }
  flush_sums_all(a, sums);
}

// ---------------------------------------------------------------------------
// The largest degrees: three kernels, every step parallel and
// proportional to the vertex's arcs or its distinct neighbour communities.
//   k_giant_prefix  at the start of an iteration, for every sub-step class
//                   (one block each), lays out per listed vertex its chunks
//                   (kGiantSingle, kGiantChunk), a global open-addressing table of a
//                   power of two >= 2 x degree slots (empty at rest) and a
//                   list of the table's occupied slots (capacity = degree);
//   k_giant_accum   one block per chunk: the chunk's arcs are aggregated by
//                   community in shared memory, then every distinct (community,
//                   weight) is added into the vertex's table; a new key's slot
//                   is appended to the vertex's occupied list;
//   k_giant_decide  one block per kGiantPart occupied slots of a vertex: those
//                   entries are read and cleared, the part's best candidate is
//                   kept (and the weight to the own community, when met); the
//                   vertex's last part block reduces the parts and decides.
// ---------------------------------------------------------------------------
// Chunk sizes: a chunk's fixed chain (headers, flush, fence, last-block decision)
// takes longer than a few more rounds of arcs, so chunks of 1,024 arcs lost
// (R-MAT 2^22 vertices: DF at 1e-3|E| 425 us a step, ND 1.64 ms, static 22.0
// ms) against these (374 us, 1.48 ms, 20.6 ms); larger ones (8,192 or a single
// chunk up to 16,384) lose where hubs are few (temporal stream 254 -> 263 us).
constexpr uint32_t kGiantSingle = 8192;  // a vertex of at most this degree is one chunk ...
constexpr uint32_t kGiantChunk = 4096;   // ... a larger one has chunks of this many arcs
// From singletons a hub's arcs meet as many communities as there are arcs, so a
// chunk's time is its flushes into the vertex's table, and a class with few
// chunks needs more of them to fill the GPU: chunks of kGiantFine arcs where there
// would be fewer than kGiantFew of the others.  Static Louvain on R-MAT graphs
// of 2^16, 2^18 and 2^19 vertices 2.68, 4.39 and 4.61 ms with chunks of 4,096,
// now 2.32, 3.20 and 4.37; on 2^20 to 2^22 the same.  The line is flat from 24
// to 76 chunks; at 12 the run on 2^18 vertices loses 11%, at 152 the one on 2^20
// 1.4%.  Updates start from communities, where a hub's arcs meet few, and lose
// with finer chunks (DF of 4,000 edges on 2^20 vertices 262 -> 275 us).  Labels
// that the caller has set count as singletons, since nothing is known of them
// (an iteration from communities of seven vertices, 2^18 in all, 950 us with the
// larger chunks, now 692; 718 when every chunk was small).
constexpr uint32_t kGiantFine = 1024;
constexpr uint32_t kGiantFew = 76;
constexpr int kAccumThreads = 256;
constexpr uint32_t kGiantRound = 8 * kAccumThreads;  // arcs in flight
constexpr uint32_t kGiantSlots = 4096;               // shared chunk table: keys + values = 32 KB
constexpr uint32_t kGiantFlush = 512;                // entries before a round (see ChunkTable)
constexpr uint32_t kGiantPart = 2048;               // occupied slots per decide block
constexpr int kGiantThreads = 256;
constexpr uint32_t kGiantListSmem = 2048;          // chunk prefix cached in shared memory

struct GiantRes {
  unsigned long long lo, hi;  // best score of the part
  uint32_t c;
  uint32_t have;
};

struct GiantDecide {
  unsigned long long* toff;   // per list position: first slot of its table
  unsigned long long* loff;   // ... first entry of its occupied-slot list
  uint32_t* cpre;             // exclusive prefix of chunk counts (+ total)
  uint32_t* ndist;            // occupied slots of its table (zeroed by k_giant_prefix)
  uint32_t* done;             // part blocks finished (zero at rest)
  unsigned long long* hd;     // weight to the own community (zero at rest)
  GiantRes* res;              // per part
  uint32_t* tkeys;            // tables (kEmpty at rest)
  uint32_t* tvals;            // (0 at rest)
  uint2* tlist;               // occupied-slot lists: (slot, community) per entry
  unsigned int* nitems;       // chunk total
  unsigned int* nbignd;       // vertices left to the part blocks (counted)
};

__device__ __forceinline__ uint32_t giant_deg(const DecideArgs& a, const uint32_t* list, uint32_t t) {
  const uint32_t v = list[t];
  uint32_t d = a.g.deg[v];
  if (d && a.ngraphs && a.gdone[graph_of(a.goff, a.ngraphs, v)]) d = 0;  // finished graph: skipped
  return d;
}

// Arcs per chunk of a vertex of degree d in a class of coarse or fine chunks.
__device__ __forceinline__ uint32_t giant_chunk_arcs(uint32_t d, bool fine) {
  return fine ? kGiantFine : d <= kGiantSingle ? kGiantSingle : kGiantChunk;
}
// The same from the vertex's number of chunks (of several chunks, 1,024 arcs
// each and 4,096 each are never the same number).
__device__ __forceinline__ uint32_t giant_chunk_arcs_of(uint32_t d, uint32_t nch) {
  return nch == 1 ? kGiantSingle : nch == (d + kGiantChunk - 1) / kGiantChunk ? kGiantChunk : kGiantFine;
}

// Table of a vertex of degree d: a power of two >= 2d (at least 64 slots).
__device__ __forceinline__ uint64_t giant_table_slots(uint32_t d) {
  if (!d) return 0;
  uint64_t p = 64;
  while (p < 2 * uint64_t(d)) p <<= 1;
  return p;
}

// One block: exclusive prefixes over the huge bin's list of chunks, table slots
// and list capacities.
__device__ __forceinline__ void giant_prefix_body(const DecideArgs& a, const uint32_t* list, uint32_t cnt,
                                                  const GiantDecide& gd) {
  __shared__ unsigned long long s_t[32], s_l[32];
  __shared__ uint32_t s_c[32];
  __shared__ unsigned long long s_tbase, s_lbase;
  __shared__ uint32_t s_cbase;
  __shared__ unsigned long long s_arcs;
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_tbase = s_lbase = s_arcs = 0;
    s_cbase = 0;
  }
  __syncthreads();
  const uint32_t d0 = threadIdx.x < cnt ? giant_deg(a, list, threadIdx.x) : 0u;
  bool fine = a.ctrl->from_singletons != 0;
  if (fine) {  // (the same in every thread) and if the class has few arcs
    unsigned long long x = d0;
    for (uint32_t t = threadIdx.x + blockDim.x; t < cnt; t += blockDim.x) x += giant_deg(a, list, t);
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    if (lane == 0 && x) atomicAdd(&s_arcs, x);
    __syncthreads();
    fine = s_arcs < uint64_t(kGiantFew) * kGiantChunk;
  }
  for (uint32_t t0 = 0; t0 < cnt; t0 += blockDim.x) {
    const uint32_t t = t0 + threadIdx.x;
    const uint32_t d = t0 == 0 ? d0 : t < cnt ? giant_deg(a, list, t) : 0u;
    const uint32_t size = giant_chunk_arcs(d, fine), ch = (d + size - 1) / size;
    const unsigned long long ts = giant_table_slots(d);
    unsigned long long xt = ts, xl = d;
    uint32_t xc = ch;
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long yt = __shfl_up_sync(0xFFFFFFFFu, xt, o);
      unsigned long long yl = __shfl_up_sync(0xFFFFFFFFu, xl, o);
      uint32_t yc = __shfl_up_sync(0xFFFFFFFFu, xc, o);
      if (lane >= (uint32_t)o) {
        xt += yt;
        xl += yl;
        xc += yc;
      }
    }
    if (lane == 31) {
      s_t[w] = xt;
      s_l[w] = xl;
      s_c[w] = xc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long rt = s_tbase, rl = s_lbase;
      uint32_t rc = s_cbase;
      for (uint32_t k = 0; k < blockDim.x / 32; ++k) {
        const unsigned long long tt = s_t[k], tl = s_l[k];
        const uint32_t tc = s_c[k];
        s_t[k] = rt;
        s_l[k] = rl;
        s_c[k] = rc;
        rt += tt;
        rl += tl;
        rc += tc;
      }
      s_tbase = rt;
      s_lbase = rl;
      s_cbase = rc;
    }
    __syncthreads();
    if (t < cnt) {
      gd.toff[t] = s_t[w] + xt - ts;
      gd.loff[t] = s_l[w] + xl - d;
      gd.cpre[t] = s_c[w] + xc - ch;
      gd.ndist[t] = 0;  // counted by k_giant_accum, read by every k_giant_decide block
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    gd.cpre[cnt] = s_cbase;
    *gd.nitems = s_cbase;
  }
}

// Class s's region of the huge bin's arrays: every sub-step class has its own
// layout (at s * gstride), so all of an iteration's layouts are made at once.
__host__ __device__ __forceinline__ GiantDecide giant_class(GiantDecide gd, uint32_t s, uint64_t gstride,
                                                          Ctrl* ctrl) {
  const uint64_t o = uint64_t(s) * gstride;
  gd.toff += o;
  gd.loff += o;
  gd.cpre += o;
  gd.ndist += o;
  gd.done += o;
  gd.hd += o;
  gd.nitems = &ctrl->it_items[s];
  return gd;
}

// The huge bin's layouts of every sub-step class (block s: class s), at the start
// of an iteration, when all classes' lists are final; each sub-step's chain
// of largest-degree kernels then starts with its chunks.
__global__ void __launch_bounds__(1024) k_giant_prefix(DecideArgs a, GiantDecide gd, uint64_t gstride,
                                                       const uint32_t* lists, int cur) {
  pdl_wait_only();
  const uint32_t s = blockIdx.x;
  giant_prefix_body(a, lists + a.seg.off[s * kBins + kBinHuge], a.ctrl->count[cur][s][kBinHuge],
                    giant_class(gd, s, gstride, a.ctrl));
}

// Entries [e0, e1) of vertex t's occupied list: read and clear them, keep the
// best candidate of this thread (and the weight to d, in hd[t]); returns the
// number of candidates this thread saw.  Four entries' loads are in flight
// at a time (slot, then key and weight, then Sigma).
template <int U>
__device__ __forceinline__ uint32_t giant_scan_entries(const DecideArgs& a, const GiantDecide& gd, uint32_t t,
                                                       uint32_t e0, uint32_t e1, uint32_t d, long long m2,
                                                       long long Ki, bool& have, i128& best, uint32_t& bc) {
  uint32_t* gk = gd.tkeys + gd.toff[t];
  uint32_t* gv = gd.tvals + gd.toff[t];
  const uint2* gl = gd.tlist + gd.loff[t];
  uint32_t ncand = 0;
  for (uint32_t b = e0 + threadIdx.x; b < e1; b += blockDim.x * U) {
    uint2 en[U];  // (slot, community): the weight and Sigma loads go out together
    uint32_t h[U], sg[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t e = b + u * blockDim.x;
      en[u] = e < e1 ? __ldcg(gl + e) : make_uint2(kEmpty, kEmpty);  // written by other blocks of this kernel
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      h[u] = en[u].x != kEmpty ? __ldcg(gv + en[u].x) : 0u;
      sg[u] = (en[u].x != kEmpty && en[u].y != d) ? sigma32(a.Sigma, en[u].y) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (en[u].x == kEmpty) continue;
      gk[en[u].x] = kEmpty;
      gv[en[u].x] = 0;
      if (en[u].y == d) {
        gd.hd[t] = h[u];  // exactly one entry of the table holds d
        continue;
      }
      ++ncand;
      const i128 sc = gain_num(m2, h[u], Ki, sg[u]);
      if (!have || sc > best || (sc == best && en[u].y < bc)) {
        have = true;
        best = sc;
        bc = en[u].y;
      }
    }
  }
  return ncand;
}

constexpr uint32_t kSmallDecide = 4096;  // occupied slots the last chunk block decides alone

// Shared table of a chunk's block, empty at rest.  Its entries move to the
// vertex's global table at the end of the chunk, or when a further round of
// arcs could overfill it: the arcs of a converged hub meet a few dozen
// communities, so a chunk of 4,096 arcs costs one flush, while a singleton
// start flushes every round (the table is then 5/8 full at the worst).
struct ChunkTable {
  uint32_t keys[kGiantSlots], vals[kGiantSlots];
  uint16_t list[kGiantFlush + kGiantRound];  // occupied slots, compacted for the flush
  uint32_t claimed, n;
};

__device__ __forceinline__ void chunk_table_init(ChunkTable& t) {
  for (uint32_t s = threadIdx.x; s < kGiantSlots; s += kAccumThreads) {
    t.keys[s] = kEmpty;
    t.vals[s] = 0;
  }
  if (threadIdx.x == 0) t.claimed = t.n = 0;
  __syncthreads();
}

// Every entry of the chunk table into list position t's global table, four per
// thread in flight; new keys' slots go onto its occupied list (one counter
// update per warp).  The chunk table is empty again.
__device__ __forceinline__ void chunk_flush(const DecideArgs& a, const GiantDecide& gd, uint32_t t, uint32_t tmask,
                                            ChunkTable& ct) {
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  for (uint32_t s0 = wib * 32; s0 < kGiantSlots; s0 += kAccumThreads) {
    const bool has = ct.keys[s0 + lane] != kEmpty;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, has);
    if (!m) continue;
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&ct.n, uint32_t(__popc(m)));
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (has) ct.list[at + __popc(m & ((1u << lane) - 1u))] = uint16_t(s0 + lane);
  }
  __syncthreads();
  const uint32_t ne = ct.n;
  uint32_t* gk = gd.tkeys + gd.toff[t];
  uint32_t* gv = gd.tvals + gd.toff[t];
  uint2* gl = gd.tlist + gd.loff[t];
  constexpr int U = 4;
  for (uint32_t b0 = wib * 32 * U; b0 < ne; b0 += kAccumThreads * U) {  // warp-uniform
    uint32_t c[U], w[U], slot[U], prev[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t e = b0 + u * 32 + lane;
      c[u] = kEmpty;
      w[u] = 0;
      if (e < ne) {
        const uint32_t q = ct.list[e];
        c[u] = ct.keys[q];
        w[u] = ct.vals[q];
        ct.keys[q] = kEmpty;
        ct.vals[q] = 0;
      }
      slot[u] = hash_move(c[u]) & tmask;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) prev[u] = c[u] != kEmpty ? atomicCAS(&gk[slot[u]], kEmpty, c[u]) : kEmpty;
    unsigned cm[U];  // lanes that created a slot, per group
#pragma unroll
    for (int u = 0; u < U; ++u) {
      bool created = false;
      if (c[u] != kEmpty) {
        // load <= 1/2: the probe ends within the table
        for (uint32_t probe = 0; prev[u] != kEmpty && prev[u] != c[u] && probe < tmask; ++probe) {
          slot[u] = (slot[u] + 1) & tmask;
          prev[u] = atomicCAS(&gk[slot[u]], kEmpty, c[u]);
        }
        if (prev[u] != kEmpty && prev[u] != c[u]) {
          atomicOr(&a.ctrl->err, kErrInternal);  // (cannot happen: the table is never full)
        } else {
          created = prev[u] == kEmpty;
          atomicAdd(&gv[slot[u]], w[u]);
        }
      }
      cm[u] = __ballot_sync(0xFFFFFFFFu, created);
    }
    // the new keys' slots onto the vertex's occupied list: one reservation for
    // all groups of the warp
    uint32_t total = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) total += __popc(cm[u]);
    if (total) {
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(&gd.ndist[t], total);
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if ((cm[u] >> lane) & 1u) gl[base + __popc(cm[u] & ((1u << lane) - 1u))] = make_uint2(slot[u], c[u]);
        base += __popc(cm[u]);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) ct.claimed = ct.n = 0;
}

// One chunk of list position t by the whole block (kAccumThreads threads):
// aggregated in the chunk table and added into the vertex's global table; the
// vertex's last chunk block decides it when the table holds at most
// kSmallDecide communities.  A vertex of one chunk whose table was never
// flushed is decided from the chunk table itself.  `nch` is the vertex's chunk
// count.  Every thread of the block calls it.
__device__ __forceinline__ void giant_chunk(const DecideArgs& a, const GiantDecide& gd, uint32_t t,
                                            uint32_t chunk, uint32_t nch, long long m2_one, ChunkTable& ct,
                                            BlockScratch& sc, MoveSums& sums) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t i = a.list[t];
  if (chunk == 0 && threadIdx.x == 0) {
    if (a.ever && bit_set(a.ever, i)) ++sums.ever;
    ++sums.processed;
  }
  if (a.rbits && !bit_test(a.rbits, i)) return;  // processed, not in the affected range
  const unsigned long long o = a.g.off[i];
  const uint32_t dg = a.g.deg[i];
  const uint32_t size = giant_chunk_arcs_of(dg, nch);
  const uint32_t k0 = chunk * size;
  const uint32_t k1 = min(dg, k0 + size);
  const uint32_t tmask = uint32_t(giant_table_slots(dg) - 1);
  long long m2 = m2_one;
  uint32_t gi = 0;
  group_active(a, i, &m2, &gi);  // (a finished graph's vertices have no chunk)
  const uint32_t d = a.C[i];
  const long long Ki = a.K[i];
  bool flushed = false, decided = false;
  for (uint32_t b = k0; b < k1; b += kGiantRound) {  // block-uniform
    constexpr int U = kGiantRound / kAccumThreads;
    uint2 e[U];
    uint32_t c[U], made = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t k = b + u * kAccumThreads + threadIdx.x;
      e[u] = k < k1 ? a.g.arcs[o + k] : make_uint2(i, 0u);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = (e[u].x != i && e[u].y != 0) ? a.C[e[u].x] : kEmpty;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (c[u] == kEmpty) continue;
      uint32_t q = hash_move(c[u]) & (kGiantSlots - 1);
      for (;;) {  // (the table is never full: the probe ends)
        uint32_t prev = ct.keys[q];
        if (prev == kEmpty) {
          prev = atomicCAS(&ct.keys[q], kEmpty, c[u]);
          if (prev == kEmpty) ++made;
        }
        if (prev == kEmpty || prev == c[u]) break;
        q = (q + 1) & (kGiantSlots - 1);
      }
      atomicAdd(&ct.vals[q], e[u].y);
    }
    const bool last = b + kGiantRound >= k1;
    if (!last) {
      made = __reduce_add_sync(0xFFFFFFFFu, made);
      if (lane == 0 && made) atomicAdd(&ct.claimed, made);
    }
    __syncthreads();
    const bool full = !last && ct.claimed > kGiantFlush;
    decided = last && nch == 1 && !flushed;
    if (full || (last && !decided)) chunk_flush(a, gd, t, tmask, ct);
    flushed |= full;
    if (!last) __syncthreads();  // the count has been read, or reset
  }
  if (decided) {
    if (threadIdx.x == 0) sc.ncand = 0;
    bool have = false;
    i128 best = 0;
    uint32_t bc = 0, ncand = 0;
    const unsigned long long hd = table_argmax<4>(a, ct.keys, ct.vals, kGiantSlots, threadIdx.x, kAccumThreads, d, m2,
                                                  Ki, have, best, bc, ncand);
    if (threadIdx.x == 0) sc.hd = 0;
    ncand = __reduce_add_sync(0xFFFFFFFFu, ncand);
    __syncthreads();  // the table has been read
    if (hd) sc.hd = hd;  // exactly one slot holds d
    if (lane == 0 && ncand) atomicAdd(&sc.ncand, ncand);
    for (uint32_t s = threadIdx.x; s < kGiantSlots; s += kAccumThreads) {
      ct.keys[s] = kEmpty;
      ct.vals[s] = 0;
    }
    if (threadIdx.x == 0) ct.claimed = 0;
    block_argmax(have, best, bc);
    if (threadIdx.x == 0) {
      i128 gain = 0;
      const bool mv = decide_move(a, m2, i, d, Ki, have, best, bc, sc.hd, &gain);
      sums.bytes += 24 + 12ull * dg + 12ull * sc.ncand + (mv ? 16 + 4ull * dg : 0ull);
      if (mv) record(a, Move{o, i, d, bc, dg, uint32_t(Ki), gain}, gi, sums);
    }
    __syncthreads();
    return;
  }
  // the vertex's last chunk block decides it when its table holds few
  // communities; the part blocks take the rest
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) sc.last = atomicAdd(&gd.done[t], 1u) == nch - 1;
  __syncthreads();
  if (sc.last) {
    __threadfence();
    const uint32_t nd = __ldcg(gd.ndist + t);
    if (threadIdx.x == 0) {
      gd.done[t] = 0;  // the part blocks count from 0
      sc.ncand = 0;
    }
    if (nd > kSmallDecide && threadIdx.x == 0) atomicAdd(gd.nbignd, 1u);
    if (nd <= kSmallDecide) {
      bool have = false;
      i128 best = 0;
      uint32_t bc = 0;
      uint32_t ncand = giant_scan_entries<4>(a, gd, t, 0, nd, d, m2, Ki, have, best, bc);
      for (int x = 16; x; x >>= 1) ncand += __shfl_xor_sync(0xFFFFFFFFu, ncand, x);
      __threadfence();
      __syncthreads();
      if (lane == 0 && ncand) atomicAdd(&sc.ncand, ncand);
      block_argmax(have, best, bc);
      if (threadIdx.x == 0) {
        const unsigned long long Hd = __ldcg(gd.hd + t);
        gd.hd[t] = 0;
        i128 gain = 0;
        const bool mv = decide_move(a, m2, i, d, Ki, have, best, bc, Hd, &gain);
        sums.bytes += 24 + 12ull * dg + 12ull * sc.ncand;
        if (mv) {
          record_move(a, i, bc, d, gain, gi, sums);
          queue_marks(a, a.nbig, i, dg);
          sums.bytes += 16 + 4ull * dg;
        }
      }
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kAccumThreads, 4) k_giant_accum(DecideArgs a, GiantDecide gd) {
  pdl_wait_only();
  __shared__ ChunkTable ct;
  __shared__ uint32_t s_pre[kGiantListSmem];
  __shared__ BlockScratch sc;
  const long long m2_one = *a.m2p;
  const uint32_t cnt = *a.count;
  const uint32_t nitems = *gd.nitems;
  if (blockIdx.x >= nitems) return;  // no chunk for this block
  chunk_table_init(ct);
  // the chunk prefix, cached in shared memory when it fits
  const uint32_t* cp = gd.cpre;
  if (cnt + 1 <= kGiantListSmem) {
    for (uint32_t k = threadIdx.x; k <= cnt; k += blockDim.x) s_pre[k] = gd.cpre[k];
    __syncthreads();
    cp = s_pre;
  }
  MoveSums sums;
  for (uint32_t item = blockIdx.x; item < nitems; item += gridDim.x) {
    uint32_t lo = 0, hi = cnt;  // list position owning this chunk
    while (hi - lo > 1) {
      uint32_t mid = (lo + hi) >> 1;
      if (cp[mid] <= item) lo = mid;
      else hi = mid;
    }
    giant_chunk(a, gd, lo, item - cp[lo], cp[lo + 1] - cp[lo], m2_one, ct, sc, sums);
  }
  flush_sums(a, sums, threadIdx.x == 0);
}

// Vertices whose tables hold more than kSmallDecide communities: kGiantPart
// occupied slots per block (blocks of kGiantThreads threads), the vertex's
// last part block reduces.  The block sweeps the list in tiles to number
// the parts.  Every thread of the block calls it.
__device__ __forceinline__ void giant_parts(const DecideArgs& a, const GiantDecide& gd, long long m2_one,
                                            MoveSums& sums) {
  __shared__ uint32_t s_ipre[kGiantThreads + 1];  // part prefix of one tile of the list
  __shared__ uint32_t s_ncand;
  __shared__ int s_last;
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  const uint32_t cnt = *a.count;
  // sweep the list in tiles of blockDim.x positions; part items of a tile
  // are numbered from `ibase` and dealt round-robin over the blocks
  uint32_t ibase = 0;
  for (uint32_t t0 = 0; t0 < cnt; t0 += kGiantThreads) {
    {
      const uint32_t t = t0 + threadIdx.x;
      const uint32_t nd = t < cnt ? gd.ndist[t] : 0u;
      const uint32_t np = nd > kSmallDecide ? (nd + kGiantPart - 1) / kGiantPart : 0u;  // else decided
      uint32_t x = np;
      for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      __shared__ uint32_t s_w[kGiantThreads / 32];
      if (lane == 31) s_w[wib] = x;
      __syncthreads();
      uint32_t wbase = 0;
      for (uint32_t k = 0; k < wib; ++k) wbase += s_w[k];
      s_ipre[threadIdx.x + 1] = wbase + x;
      if (threadIdx.x == 0) s_ipre[0] = 0;
      __syncthreads();
    }
    const uint32_t tile_items = s_ipre[kGiantThreads];
    const uint32_t first = (blockIdx.x + gridDim.x - ibase % gridDim.x) % gridDim.x;
    for (uint32_t it = first; it < tile_items; it += gridDim.x) {
      uint32_t lo = 0, hi = kGiantThreads;  // tile position owning part item `it`
      while (hi - lo > 1) {
        uint32_t mid = (lo + hi) >> 1;
        if (s_ipre[mid] <= it) lo = mid;
        else hi = mid;
      }
      const uint32_t t = t0 + lo;
      const uint32_t part = it - s_ipre[lo];
      const uint32_t nparts = s_ipre[lo + 1] - s_ipre[lo];
      const uint32_t ridx = ibase + s_ipre[lo];  // results of this vertex start here
      const uint32_t nd = gd.ndist[t];
      const uint32_t i = a.list[t];
      long long m2 = m2_one;
      uint32_t gi = 0;
      group_active(a, i, &m2, &gi);  // its graph is active: it has entries
      const uint32_t d = a.C[i];
      const long long Ki = a.K[i];
      if (threadIdx.x == 0) s_ncand = 0;
      // 1. this part's entries: best candidate, weight to d; then clear them
      bool have = false;
      i128 best = 0;
      uint32_t bc = 0;
      uint32_t ncand = giant_scan_entries<4>(a, gd, t, part * kGiantPart, min(nd, (part + 1) * kGiantPart), d, m2,
                                          Ki, have, best, bc);
      for (int x = 16; x; x >>= 1) ncand += __shfl_xor_sync(0xFFFFFFFFu, ncand, x);
      __syncthreads();  // s_ncand reset seen
      if (lane == 0 && ncand) atomicAdd(&s_ncand, ncand);
      block_argmax(have, best, bc);
      __threadfence();  // hd[t] (from whichever thread met d) ...
      __syncthreads();  // ... before thread 0's done count
      if (threadIdx.x == 0) {
        GiantRes r;
        r.lo = (unsigned long long)(u128)best;
        r.hi = (unsigned long long)((u128)best >> 64);
        r.c = bc;
        r.have = have ? 1u : 0u;
        gd.res[ridx + part] = r;
        sums.bytes += 12ull * s_ncand;
        __threadfence();
        s_last = atomicAdd(&gd.done[t], 1u) == nparts - 1;
      }
      __syncthreads();
      if (s_last) {
        // 2. last part block of the vertex: reduce the parts and decide
        __threadfence();
        have = false;
        best = 0;
        bc = 0;
        for (uint32_t k = threadIdx.x; k < nparts; k += kGiantThreads) {
          const GiantRes* src = gd.res + ridx + k;
          const unsigned long long rlo = __ldcg(&src->lo), rhi = __ldcg(&src->hi);
          const uint32_t rc = __ldcg(&src->c), rh = __ldcg(&src->have);
          const i128 sc = (i128)(((u128)rhi << 64) | (u128)rlo);
          if (rh && (!have || sc > best || (sc == best && rc < bc))) {
            have = true;
            best = sc;
            bc = rc;
          }
        }
        block_argmax(have, best, bc);
        if (threadIdx.x == 0) {
          const unsigned long long Hd = __ldcg(gd.hd + t);
          gd.hd[t] = 0;  // zero at rest for the next use of this list position
          gd.done[t] = 0;
          const uint32_t dg = a.g.deg[i];
          i128 gain = 0;
          const bool mv = decide_move(a, m2, i, d, Ki, have, best, bc, Hd, &gain);
          sums.bytes += 24 + 12ull * dg;
          if (mv) {
            record_move(a, i, bc, d, gain, gi, sums);
            queue_marks(a, a.nbig, i, dg);
            sums.bytes += 16 + 4ull * dg;
          }
        }
      }
      __syncthreads();
    }
    ibase += tile_items;
    __syncthreads();  // s_ipre is rewritten for the next tile
  }
}

__global__ void __launch_bounds__(kGiantThreads) k_giant_decide(DecideArgs a, GiantDecide gd) {
  pdl_wait_only();
  if (*gd.nbignd == 0) return;  // every vertex was decided by its last chunk block
  MoveSums sums;
  giant_parts(a, gd, *a.m2p, sums);
  flush_sums(a, sums, threadIdx.x == 0);
}

// Warp `warp` of `nwarps`' pieces of the queued movers' rows (`big`: the queue's counter).
template <bool kAppend>
__device__ __forceinline__ void mark_queued(const DecideArgs& a, unsigned long long big, uint32_t warp,
                                            uint32_t nwarps) {
  const uint32_t rows = uint32_t(big >> 32), pieces = uint32_t(big);
  for (uint64_t p = warp; p < pieces; p += nwarps) {
    const uint2 e = a.bigmv[find_row(a.bigmv, rows, uint32_t(p))];
    const uint32_t k0 = (uint32_t(p) - e.y) * kMarkChunk, dg = a.g.deg[e.x];
    mark_arcs<kAppend>(a, e.x, a.g.off[e.x], k0, dg - k0 < kMarkChunk ? dg : k0 + kMarkChunk, threadIdx.x & 31u, 32);
  }
}

constexpr int kCommitThreads = 256;

// Apply the moves of one sub-step and mark the movers' neighbours for the
// next iteration.  Latency bounds it, so the two jobs go to different warps
// where there are enough: the moves to the first warps, 32 a warp (movers of a
// warp joining or leaving one community are summed first, so a popular
// community takes one update per warp), the marks to the last, one mover a
// warp while they last and up to 32 beyond, eight lanes a mover then.  The
// decide kernels marked their own movers' rows before, at the end of each
// vertex's chain: without it the lane kernel takes 27 us instead of 40 on
// 100,000 vertices of mean degree 16 and the warp tables 45 instead of 55, the
// commit 25 instead of 9; a small commit takes 4 us as before.
// Warp `warp` of `nwarps`; every lane of it calls this.
__device__ __forceinline__ void commit_body(const DecideArgs& a, uint32_t m, unsigned long long big, uint32_t warp,
                                            uint32_t nwarps) {
  uint32_t* C = const_cast<uint32_t*>(a.C);
  long long* Sigma = const_cast<long long*>(a.Sigma);
  int* size = const_cast<int*>(a.size);
  const uint32_t lane = threadIdx.x & 31u;
  if (warp == 0 && lane == 0 && m) atomicAdd(&a.ctrl->moved, (unsigned long long)m);
  for (uint64_t t0 = uint64_t(warp) * 32; t0 < m; t0 += uint64_t(nwarps) * 32) {
    const uint64_t t = t0 + lane;
    const bool ok = t < m;
    const uint32_t i = ok ? a.mv_i[t] : 0u;
    const uint32_t c = ok ? a.mv_c[t] : kEmpty, d = ok ? a.mv_d[t] : kEmpty;
    const long long ki = ok ? a.K[i] : 0;
    if (ok) C[i] = c;
    for (int side = 0; side < 2; ++side) {
      const uint32_t key = side ? d : c;
      long long sk = 0;
      int cnt = 0;
      bool first = ok;
      // sum over the lanes with the same community (32 shuffles)
      for (int k = 0; k < 32; ++k) {
        const uint32_t kk = __shfl_sync(0xFFFFFFFFu, key, k);
        const long long kv = __shfl_sync(0xFFFFFFFFu, ki, k);
        if (ok && kk == key) {
          sk += kv;
          ++cnt;
          if (uint32_t(k) < lane) first = false;
        }
      }
      if (first) {
        atomicAdd((unsigned long long*)&Sigma[key], (unsigned long long)(side ? -sk : sk));
        atomicAdd(&size[key], side ? -cnt : cnt);
      }
    }
  }
  // marks, the warps counted from the last one down
  const uint32_t rev = nwarps - 1 - warp;
  uint32_t per = (m + nwarps - 1) / nwarps;
  per = per < 32 ? per : 32;
  for (uint64_t t0 = uint64_t(rev) * per; t0 < m; t0 += uint64_t(nwarps) * per) {
    const bool ok = lane < per && t0 + lane < m;
    const uint32_t i = ok ? a.mv_i[t0 + lane] : 0u;
    const unsigned long long o = ok ? a.g.off[i] : 0ull;
    uint32_t dg = ok ? a.g.deg[i] : 0u;
    if (dg > kMarkInline) dg = 0;  // queued
    // whole-warp rows: all of them while a warp has few movers, else the long ones
    const uint32_t narrow = per > 4 ? 64u : 0u;
    for (unsigned mk = __ballot_sync(0xFFFFFFFFu, dg > narrow); mk; mk &= mk - 1) {
      const int src = __ffs(mk) - 1;
      mark_arcs<false>(a, __shfl_sync(0xFFFFFFFFu, i, src), __shfl_sync(0xFFFFFFFFu, o, src), 0,
                __shfl_sync(0xFFFFFFFFu, dg, src), lane, 32);
    }
    if (!narrow) continue;
    if (dg > narrow) dg = 0;
    for (uint32_t s = 0; s * 4 < per; ++s) {
      const int src = int(s * 4 + (lane >> 3));
      mark_arcs<false>(a, __shfl_sync(0xFFFFFFFFu, i, src), __shfl_sync(0xFFFFFFFFu, o, src), 0,
                __shfl_sync(0xFFFFFFFFu, dg, src), lane & 7u, 8);
    }
  }
  mark_queued<false>(a, big, rev, nwarps);
}

__global__ void __launch_bounds__(kCommitThreads) k_commit(DecideArgs a) {
  pdl_wait_only();
  // the next sub-step counts into the other pair of counters, last used two
  // sub-steps ago: zeroed here, so no memset separates the sub-steps
  if (blockIdx.x == 0 && threadIdx.x == 0 && a.clear_movers) {
    *a.clear_movers = 0;
    *a.clear_nbig = 0;
    *a.clear_bignd = 0;
  }
  commit_body(a, *a.movers, *a.nbig, blockIdx.x * (kCommitThreads / 32) + (threadIdx.x >> 5),
                     gridDim.x * (kCommitThreads / 32));
}

int read_ctrl(Handle* h) {
  DFL_CUDA(h, cudaMemcpyAsync(h->hctrl, h->ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, h->stream));
  DFL_CUDA(h, cudaStreamSynchronize(h->stream));
  return DFL_OK;
}

// A control read of local-moving.  The first one after a batch apply that
// was enqueued without a host wait also settles that apply, in the same
// wait; if the batch was not written (an invalid batch, or buffers to grow
// first) the code is returned and local-moving stops -- its iteration ran on
// an empty frontier, since nothing was marked.
int read_move_ctrl(Handle* h, bool* settled) {
  const bool pend = h->papply.active;
  // (the apply's control blocks follow this one: one copy takes both)
  const size_t blocks = pend ? size_t(2 + h->papply.par) : 1;
  DFL_CUDA(h, cudaMemcpyAsync(h->hctrl, h->ctrl, blocks * sizeof(Ctrl), cudaMemcpyDeviceToHost, h->stream));
  DFL_CUDA(h, cudaStreamSynchronize(h->stream));
  *settled = pend;
  return pend ? settle_apply(h) : DFL_OK;
}

// floor(tau_num * m2^2 / (2 * tau_den * drop^pass)), the exact form of
// "sum of dQ <= tau" (Alg. 5) with S = sum of the movers' 2m^2 * dQ.
__host__ __device__ inline u128 tolerance_threshold(uint64_t tau_num, uint64_t tau_den, uint64_t drop, long long m2,
                                                    uint32_t pass) {
  u128 num = (u128)tau_num * (u128)(uint64_t)m2 * (u128)(uint64_t)m2;
  u128 den = (u128)2 * (u128)tau_den;
  for (uint32_t p = 0; p < pass; ++p) {
    if (den > num) return 0;
    den *= (u128)drop;
  }
  if (den == 0) return ~(u128)0;
  return num / den;
}

u128 tolerance_threshold(const dfl_options& o, long long m2, uint32_t pass) {
  return tolerance_threshold(o.tau_num, o.tau_den, o.tolerance_drop, m2, pass);
}

uint32_t next_pow2(uint64_t x) {
  uint64_t p = 1;
  while (p < x) p <<= 1;
  return uint32_t(p);
}




// ---------------------------------------------------------------------------
// Persistent iteration kernel: one cooperative launch runs a whole
// local-moving iteration.  Its blocks take work units of a sub-step from a
// shared counter (largest-degree chunks first, then block, warp and
// segment units), meet at grid barriers between deciding and committing,
// and build the next frontier's lists at the end.  It replaces the per
// sub-step launches, stream forks and joins of issue_iteration.
// ---------------------------------------------------------------------------
constexpr int kIterThreads = 256;
constexpr uint32_t kIterPreCache = kGiantListSmem;                   // chunk prefix cached in shared memory
constexpr uint32_t kIterDynWords = 2 * kBlockSlots + kIterPreCache;  // tables + chunk prefix cache
constexpr unsigned long long kBarrierPolls = 1ull << 22;             // x 256 ns: about a second
constexpr unsigned long long kTestBarrierPolls = 1ull << 14;         // a few ms (the timeout test hook)
// vertices per warp in one work unit of bins 1 and 0 (rounds of 1 and of
// 32 / W vertices); larger units save counter updates on big frontiers but
// measured slower on small DF frontiers, where they leave blocks idle
constexpr uint32_t kIterRounds1 = 1;
constexpr uint32_t kIterRounds0 = 1;

struct IterArgs {
  DecideArgs a;            // list/count/movers/nbig are set per bin and sub-step
  GiantDecide gd;          // class 0's arrays; class s at + s * gstride
  uint32_t gstride;
  uint32_t k;
  int cur;
  uint32_t seg_lanes;      // W: lanes per tiny-bin vertex
  const uint32_t* lists_cur;
  uint32_t* fbits_cur;     // cleared at the end (the processed frontier)
  uint32_t words;
  // grid barriers: arrivals beyond the grid that complete one (0; 1 makes
  // every barrier unreachable, DFL_FLAG_TEST_UNREACHABLE_BARRIER) and polls
  // before a wait gives up
  uint32_t bar_extra;
  unsigned long long bar_polls;
};

// Grid-wide barrier with a bounded wait: false if it gave up (the error bit
// kErrTimeout is then set and the kernel must return).  Every thread calls it.
__device__ __forceinline__ bool grid_barrier(Ctrl* ctrl, uint32_t extra, unsigned long long max_polls) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned int* genp = &ctrl->bar_gen;
    const unsigned int gen = *genp;
    __threadfence();
    int ok = 1;
    if (atomicAdd(&ctrl->bar_count, 1u) == gridDim.x - 1 + extra) {
      ctrl->bar_count = 0;
      __threadfence();
      atomicAdd(&ctrl->bar_gen, 1u);
    } else {
      unsigned long long polls = 0;
      while (*genp == gen) {
        if (++polls > max_polls || (*((volatile unsigned int*)&ctrl->err) & kErrTimeout)) {
          ok = 0;
          atomicOr(&ctrl->err, kErrTimeout);
          break;
        }
        __nanosleep(256);
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  __threadfence();  // every thread: later reads see what other blocks wrote before the barrier
  return s_ok;
}

// (The list's offset is looked up in the parameters: looked up in the copy, it
// would put the layout of every bin's copy on the stack, 1,368 bytes a thread
// and sub-step: a DF step on 50,000 vertices 393 us in this form, now 220.)
__device__ __forceinline__ DecideArgs bin_args(const IterArgs& ia, uint32_t s, int b) {
  DecideArgs a = ia.a;
  a.list = ia.lists_cur + ia.a.seg.off[s * kBins + b];
  a.count = &a.ctrl->count[ia.cur][s][b];
  a.movers = &a.ctrl->it_movers[s & 1];
  a.nbig = &a.ctrl->it_nbig[s & 1];
  return a;
}

__device__ __forceinline__ GiantDecide class_giant(const IterArgs& ia, uint32_t s) {
  GiantDecide gd = giant_class(ia.gd, s, ia.gstride, ia.a.ctrl);
  gd.nbignd = &ia.a.ctrl->it_bignd[s & 1];
  return gd;
}

static_assert(kIterThreads == kGiantThreads && kIterThreads == kCommitThreads,
              "the part blocks and the commit sweep their lists in tiles of one block");
static_assert(kIterThreads == kListThreads, "the list builder's tiles are one block's");
static_assert(kIterDynWords >= 2 * kBlockSlots && 8 * 2 * kWarpSlots <= 2 * kBlockSlots &&
                  sizeof(ChunkTable) <= sizeof(uint32_t) * 2 * kBlockSlots && kIterThreads == kAccumThreads,
              "the dynamic tables hold every unit kind");

// two blocks per SM: 128 registers a thread (three blocks, at 80 registers,
// spilled and measured slower)
__global__ void __launch_bounds__(kIterThreads, 2) k_iterate(IterArgs ia) {
  extern __shared__ __align__(16) uint32_t dyn[];
  __shared__ BlockScratch sc;
  __shared__ uint32_t s_unit;
  Ctrl* ctrl = ia.a.ctrl;
  const long long m2_one = *ia.a.m2p;
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  uint32_t* pre_cache = dyn + 2 * kBlockSlots;
  MoveSums sums;
  // 1. the largest-degree lists of every class: chunk, table and list layouts
  if (blockIdx.x < ia.k) {
    giant_prefix_body(ia.a, ia.lists_cur + ia.a.seg.off[blockIdx.x * kBins + kBinHuge],
                      ctrl->count[ia.cur][blockIdx.x][kBinHuge], class_giant(ia, blockIdx.x));
  }
  if (!grid_barrier(ctrl, ia.bar_extra, ia.bar_polls)) return;
  for (uint32_t s = 0; s < ia.k; ++s) {
    const uint32_t par = s & 1;
    if (blockIdx.x == 0 && threadIdx.x == 0 && s >= 1) {  // the other parity's counters are idle now
      ctrl->it_movers[par ^ 1] = 0;
      ctrl->it_nbig[par ^ 1] = 0;
      ctrl->it_work[par ^ 1] = 0;
      ctrl->it_bignd[par ^ 1] = 0;
    }
    // (the lane bin's vertices are warp units here too, in units of their own)
    const DecideArgs a0 = bin_args(ia, s, kBinTiny), al = bin_args(ia, s, kBinLanes), a1 = bin_args(ia, s, kBinTable),
                     am = bin_args(ia, s, kBinMid), a2 = bin_args(ia, s, kBinWhole), a3 = bin_args(ia, s, kBinHuge);
    const GiantDecide gd = class_giant(ia, s);
    const uint32_t n0 = *a0.count, nl = *al.count, n1 = *a1.count, nm = *am.count, n2 = nm + *a2.count, n3 = *a3.count;
    const uint32_t G = *gd.nitems;
    // chunk prefix of the class, cached when it fits
    const uint32_t* cp = gd.cpre;
    if (n3 + 1 <= kIterPreCache) {
      for (uint32_t q = threadIdx.x; q <= n3; q += blockDim.x) pre_cache[q] = gd.cpre[q];
      __syncthreads();
      cp = pre_cache;
    }
    const uint32_t per_warp0 = 32 / ia.seg_lanes;
    const uint64_t U0 = (uint64_t(n0) + per_warp0 * 8 * kIterRounds0 - 1) / (per_warp0 * 8 * kIterRounds0);
    const uint64_t U1 = (uint64_t(n1) + 8 * kIterRounds1 - 1) / (8 * kIterRounds1);
    const uint64_t UL = (uint64_t(nl) + 8 * kIterRounds1 - 1) / (8 * kIterRounds1);
    const uint64_t total = uint64_t(G) + n2 + U1 + UL + U0;
    // 2. decide: work units from the shared counter
    for (;;) {
      if (threadIdx.x == 0) s_unit = atomicAdd(&ctrl->it_work[par], 1u);
      __syncthreads();
      const uint64_t u = s_unit;
      __syncthreads();
      if (u >= total) break;
      if (u < G) {
        uint32_t lo = 0, hi = n3;  // list position owning chunk u
        while (hi - lo > 1) {
          uint32_t mid = (lo + hi) >> 1;
          if (cp[mid] <= u) lo = mid;
          else hi = mid;
        }
        ChunkTable& ct = *reinterpret_cast<ChunkTable*>(dyn);
        chunk_table_init(ct);  // (other units used the memory)
        giant_chunk(a3, gd, lo, uint32_t(u) - cp[lo], cp[lo + 1] - cp[lo], m2_one, ct, sc, sums);
      } else if (u < uint64_t(G) + n2) {
        const uint32_t i = u - G < nm ? am.list[u - G] : a2.list[u - G - nm];
        long long m2 = m2_one;
        uint32_t gi = 0;
        if (!group_active(a2, i, &m2, &gi)) continue;
        if (threadIdx.x == 0) {
          if (a2.ever && bit_set(a2.ever, i)) ++sums.ever;
          ++sums.processed;
        }
        if (a2.rbits && !bit_test(a2.rbits, i)) continue;
        Move m;
        if (block_vertex<kIterThreads, kBlockSlots>(a2, i, m2, dyn, sc, &m, sums)) record(a2, m, gi, sums);
      } else if (u < uint64_t(G) + n2 + U1 + UL) {
        // one table-bin or lane-bin vertex per warp and round, in the warp's own table
        const bool table = u < uint64_t(G) + n2 + U1;
        const uint64_t unit = table ? u - G - n2 : u - G - n2 - U1;
        const DecideArgs& aw = table ? a1 : al;
        for (uint32_t r = 0; r < kIterRounds1; ++r) {
          const uint64_t t = (unit * kIterRounds1 + r) * 8 + wib;
          if (t >= (table ? n1 : nl)) break;
          const uint32_t i = aw.list[t];
          long long m2 = m2_one;
          uint32_t gi = 0;
          if (!group_active(aw, i, &m2, &gi)) continue;
          if (lane == 0) {
            if (aw.ever && bit_set(aw.ever, i)) ++sums.ever;
            ++sums.processed;
          }
          Move m;
          if (!aw.rbits || bit_test(aw.rbits, i))
            if (warp_table_vertex(aw, i, m2, dyn + wib * 2 * kWarpSlots, dyn + wib * 2 * kWarpSlots + kWarpSlots, &m,
                                  sums) &&
                lane == 0)
              record(aw, m, gi, sums);
        }
      } else {
        for (uint32_t r = 0; r < kIterRounds0; ++r) {
          const uint64_t first =
              ((u - G - n2 - U1 - UL) * kIterRounds0 + r) * (per_warp0 * 8) + uint64_t(wib) * per_warp0;
          if (first >= n0) break;  // warp-uniform
          switch (ia.seg_lanes) {
            case 4: decide_segments<4>(a0, first, n0, m2_one, sums); break;
            case 8: decide_segments<8>(a0, first, n0, m2_one, sums); break;
            case 16: decide_segments<16>(a0, first, n0, m2_one, sums); break;
            default: decide_segments<32>(a0, first, n0, m2_one, sums); break;
          }
        }
      }
    }
    if (!grid_barrier(ctrl, ia.bar_extra, ia.bar_polls)) return;
    // 3. vertices with many distinct communities: spread over part blocks
    if (*((volatile unsigned int*)&ctrl->it_bignd[par])) {
      giant_parts(a3, gd, m2_one, sums);
      if (!grid_barrier(ctrl, ia.bar_extra, ia.bar_polls)) return;
    }
    // 4. commit the sub-step's moves (and mark around high-degree movers)
    commit_body(a0, *((volatile unsigned int*)a0.movers), *((volatile unsigned long long*)a0.nbig),
                       blockIdx.x * (kCommitThreads / 32) + wib, gridDim.x * (kCommitThreads / 32));
    if (!grid_barrier(ctrl, ia.bar_extra, ia.bar_polls)) return;
  }
  // 5. the next frontier's lists; clear the processed frontier's bitmap
  lists_body<true>(ia.a.fbits_next, ia.a.g.nv, ia.a.g.deg, ia.a.next_lists, ia.a.seg, ctrl, ia.a.next_buf, ia.k);
  for (uint64_t w = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; w < ia.words;
       w += uint64_t(gridDim.x) * blockDim.x)
    ia.fbits_cur[w] = 0;
  flush_sums_all(ia.a, sums);  // every thread holds counts (segment and warp leaders, block leaders)
}

// ---------------------------------------------------------------------------
// Small frontiers: one thread-block cluster runs whole local-moving
// iterations, one after another, in one launch.  A frontier of a few thousand
// vertices leaves most of the GPU idle, and its iteration is a chain of about
// a dozen kernels of 2-8 us each (launches, stream forks and joins, a control
// read), so the chain itself bounds it.  Here the sub-steps' phases are
// separated by hardware cluster barriers (no polling), newly marked vertices go
// straight onto the next frontier's lists, and the tolerance test is made on
// the device.  Vertices are dealt statically: a vertex of the last bin to the
// whole cluster, over one table spread over the CTAs' shared memory; of the
// block bins to a CTA, of the table and lane bins to a warp, of the tiny bin to a few
// lanes.  The kernel stops before an iteration whose estimated time is above
// what the per-bin kernels need (small_cost), leaving its frontier to them.
// A DF step's four sub-steps of 100 edges on 10,000 vertices take 34 us here
// (30 + 15 us of decide and commit kernels, 4 us of lists, and the launches and
// the control read between them before: 195 -> 130 us the whole step); an
// iteration of the same graph's static run takes 49 us, 75 before.
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 512;
constexpr uint32_t kSmallCtas = 16;
constexpr uint32_t kSmallWarps = kSmallThreads / 32 * kSmallCtas;
constexpr uint32_t kSmallSlots = 16384;                  // slots per CTA of the cluster's table
constexpr uint32_t kSmallHuge = kSmallSlots * kSmallCtas / 2;  // largest degree it always holds
constexpr size_t kSmallSmem = sizeof(uint32_t) * 2 * kSmallSlots;
static_assert(2 * kSmallSlots >= 2 * kBlockSlots + kSmallThreads / 32 * 2 * kWarpSlots,
              "the cluster table's memory also holds a block table and the warps' tables");

// Estimated ns of one iteration's decisions over lists of the given lengths
// (measured: a warp decides a vertex, or four tiny ones, in about 2.5 us, a CTA
// one of the block bins in 3 or 6 us, the cluster one of the last bin in 10 us).
__host__ __device__ inline uint64_t small_cost(const uint32_t* n) {
  return (uint64_t(n[kBinTiny] / 4) + n[kBinLanes] + 2ull * n[kBinTable]) * 2500 / kSmallWarps +
         (3000ull * n[kBinMid] + 6000ull * n[kBinWhole]) / kSmallCtas + uint64_t(n[kBinHuge]) * 10000;
}
// Flat down to 45 us.  At 30 us static Louvain on 10,000 vertices loses the
// iterations that gain most (2.59 -> 2.75 ms); at 120 us the cluster keeps
// iterations that the per-bin kernels do faster with the whole GPU (static on
// 400,000 vertices 4.24 -> 4.90 ms, on 32 graphs 15.4 -> 16.2 ms).
constexpr uint64_t kSmallCostMax = 60000;

struct SmallArgs {
  DecideArgs a[2];         // by the processed frontier's buffer
  int cur;                 // ... of the first iteration
  uint32_t seg_lanes;      // W: lanes per tiny-bin vertex
  uint32_t* lists[2];
  uint32_t* fbits[2];
  uint32_t max_iters;      // iterations left to the pass
  uint32_t single;         // stop after one iteration (a group: the host tests each graph's tolerance)
  uint32_t pass;           // tolerance test
  uint64_t tau_num, tau_den, drop;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Barrier of the whole cluster: what any thread wrote before it is visible to
// every thread after it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Address of shared variable p in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(uint32_t(__cvta_generic_to_shared(p))), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t cluster_cas(uint32_t addr, uint32_t cmp, uint32_t val) {
  uint32_t r;
  asm volatile("atom.shared::cluster.cas.b32 %0, [%1], %2, %3;" : "=r"(r) : "r"(addr), "r"(cmp), "r"(val) : "memory");
  return r;
}
__device__ __forceinline__ void cluster_add(uint32_t addr, uint32_t val) {
  asm volatile("red.shared::cluster.add.u32 [%0], %1;" ::"r"(addr), "r"(val) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t addr, uint32_t val) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(val) : "memory");
}

// The cluster's parts of one vertex, gathered in CTA 0.
struct SmallParts {
  uint32_t lo[4][kSmallCtas];  // the best score's words
  uint32_t c[kSmallCtas], have[kSmallCtas], ncand[kSmallCtas];
  uint32_t hd;                 // weight to the own community
};

// One vertex by the whole cluster: its arcs' weights summed by community in an
// open-addressing table of kSmallCtas x kSmallSlots slots (linear probing runs
// on into the next CTA's slots), then each CTA scores its own slots.  Every
// thread of the cluster calls it; the move is thread 0's of CTA 0.
__device__ __forceinline__ bool cluster_vertex(const DecideArgs& a, uint32_t i, long long m2, uint32_t* dyn,
                                               SmallParts& sp, BlockScratch& sc, Move* mvo, MoveSums& sums) {
  constexpr uint32_t kMask = kSmallCtas * kSmallSlots - 1;
  const uint32_t rank = cluster_rank();
  uint32_t* keys = dyn;
  uint32_t* vals = dyn + kSmallSlots;
  const uint32_t d = a.C[i];
  const long long Ki = a.K[i];
  const unsigned long long o = a.g.off[i];
  const uint32_t dg = a.g.deg[i];
  for (uint32_t s = threadIdx.x; s < kSmallSlots; s += kSmallThreads) {
    keys[s] = kEmpty;
    vals[s] = 0;
  }
  if (threadIdx.x == 0) {
    sp.hd = 0;
    sc.ncand = 0;
  }
  cluster_sync();
  constexpr uint32_t U = 4, kStep = kSmallCtas * kSmallThreads;
  for (uint32_t b = rank * kSmallThreads + threadIdx.x; b < dg; b += U * kStep) {
    uint2 e[U];
    uint32_t c[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) e[u] = b + u * kStep < dg ? a.g.arcs[o + b + u * kStep] : make_uint2(i, 0u);
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) c[u] = (e[u].x != i && e[u].y != 0) ? a.C[e[u].x] : kEmpty;
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      if (c[u] == kEmpty) continue;
      uint32_t at = hash_move(c[u]) & kMask;
      bool placed = false;
      for (uint32_t probe = 0; probe <= kMask && !placed; ++probe) {  // load <= 1/2: the probe ends
        const uint32_t owner = at / kSmallSlots, slot = at % kSmallSlots;
        const uint32_t prev = cluster_cas(cluster_addr(keys + slot, owner), kEmpty, c[u]);
        if (prev == kEmpty || prev == c[u]) {
          cluster_add(cluster_addr(vals + slot, owner), e[u].y);
          placed = true;
        }
        at = (at + 1) & kMask;
      }
      if (!placed) atomicOr(&a.ctrl->err, kErrInternal);
    }
  }
  cluster_sync();
  bool have = false;
  i128 best = 0;
  uint32_t bc = 0, ncand = 0;
  const unsigned long long hd =
      table_argmax<4>(a, keys, vals, kSmallSlots, threadIdx.x, kSmallThreads, d, m2, Ki, have, best, bc, ncand);
  if (hd) cluster_store(cluster_addr(&sp.hd, 0), uint32_t(hd));  // exactly one slot of the table holds d
  ncand = __reduce_add_sync(0xFFFFFFFFu, ncand);
  if ((threadIdx.x & 31u) == 0 && ncand) atomicAdd(&sc.ncand, ncand);
  block_argmax(have, best, bc);
  if (threadIdx.x == 0) {
    for (int q = 0; q < 4; ++q) cluster_store(cluster_addr(&sp.lo[q][rank], 0), uint32_t((u128)best >> (32 * q)));
    cluster_store(cluster_addr(&sp.c[rank], 0), bc);
    cluster_store(cluster_addr(&sp.have[rank], 0), have ? 1u : 0u);
    cluster_store(cluster_addr(&sp.ncand[rank], 0), sc.ncand);
  }
  cluster_sync();
  bool mv = false;
  if (rank == 0 && threadIdx.x == 0) {
    have = false;
    ncand = 0;
    for (uint32_t r = 0; r < kSmallCtas; ++r) {
      ncand += sp.ncand[r];
      if (!sp.have[r]) continue;
      u128 x = 0;
      for (int q = 3; q >= 0; --q) x = (x << 32) | sp.lo[q][r];
      if (!have || (i128)x > best || ((i128)x == best && sp.c[r] < bc)) {
        have = true;
        best = (i128)x;
        bc = sp.c[r];
      }
    }
    i128 gain = 0;
    mv = decide_move(a, m2, i, d, Ki, have, best, bc, sp.hd, &gain);
    sums.bytes += 24 + 12ull * dg + 12ull * ncand + (mv ? 16 + 4ull * dg : 0ull);
    *mvo = Move{o, i, d, bc, dg, uint32_t(Ki), gain};
  }
  __syncthreads();  // (the parts are rewritten only after the next cluster barrier)
  return mv;
}

// The moves a CTA decided in a sub-step, in its shared memory until they are
// committed.
struct SmallMove {
  unsigned long long o;
  uint32_t i, c, d, dg, Ki, pad;
};
constexpr uint32_t kSmallMoves = 1024;
// Vertices of a sub-step class at most: a CTA then decides at most
// kSmallClass / kSmallCtas + 8 a warp + 8 of them.
constexpr uint32_t kSmallClass = 12000;
static_assert(kSmallClass / kSmallCtas + 8 * kSmallThreads / 32 + kSmallThreads / 32 + 8 <= kSmallMoves,
              "a CTA's moves fit");
constexpr size_t kSmallSmemAll = kSmallSmem + sizeof(SmallMove) * kSmallMoves;
static_assert(alignof(SmallMove) <= 16 && kSmallSmem % alignof(SmallMove) == 0, "the moves are aligned behind the tables");

__device__ __forceinline__ void small_record(const DecideArgs& a, const Move& m, uint32_t gi, SmallMove* moves,
                                             uint32_t* count, unsigned long long* nbig, MoveSums& sums) {
  const uint32_t at = atomicAdd(count, 1u);
  moves[at] = SmallMove{m.o, m.i, m.c, m.d, m.dg, m.Ki, 0u};
  const unsigned long long lo = (unsigned long long)((u128)m.gain & 0xFFFFFFFFull);
  const unsigned long long hi = (unsigned long long)((u128)m.gain >> 32);
  sums.s_lo += lo;
  sums.s_hi += hi;
  if (a.ngraphs) {
    if (lo) atomicAdd(a.gS + 2 * gi, lo);
    if (hi) atomicAdd(a.gS + 2 * gi + 1, hi);
  }
  if (m.dg > kMarkInline) queue_marks(a, nbig, m.i, m.dg);
}

__global__ void __launch_bounds__(kSmallThreads, 1) k_small_move(const __grid_constant__ SmallArgs q) {
  pdl_wait_only();
  // the warps' tables (empty at rest) and a block table, or the cluster's table; then the moves
  extern __shared__ __align__(16) uint32_t dyn[];
  __shared__ SmallParts sp;
  __shared__ BlockScratch sc;
  __shared__ uint32_t s_n[kMaxSubsteps][kBins];
  __shared__ unsigned long long s_cost;
  __shared__ uint32_t s_refuse, s_huge, s_nmv[2];
  __shared__ int s_stop;
  Ctrl* ctrl = q.a[0].ctrl;
  const Segs& seg = q.a[0].seg;
  const uint32_t k = q.a[0].k, rank = cluster_rank();
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  const uint32_t warp = rank * (kSmallThreads / 32) + wib, rev = kSmallWarps - 1 - warp;
  uint32_t* keys = dyn + wib * 2 * kWarpSlots;
  uint32_t* vals = keys + kWarpSlots;
  uint32_t* block_table = dyn + kSmallThreads / 32 * 2 * kWarpSlots;
  SmallMove* moves = reinterpret_cast<SmallMove*>(dyn + 2 * kSmallSlots);
  const long long m2_one = *q.a[0].m2p;
  u128 threshold = 0;
  if (threadIdx.x == 0 && !q.single) threshold = tolerance_threshold(q.tau_num, q.tau_den, q.drop, m2_one, q.pass);
  if (threadIdx.x < 2) s_nmv[threadIdx.x] = 0;
  auto empty_table = [&] {
    for (uint32_t x = lane; x < kWarpSlots; x += 32) {
      keys[x] = kEmpty;
      vals[x] = 0;
    }
    __syncwarp();
  };
  empty_table();
  int cur = q.cur;
  uint32_t it = 0, step = 0;
  MoveSums sums;
  for (;;) {
    // the frontier's lengths (every CTA reads them and decides alike)
    if (threadIdx.x == 0) {
      s_cost = 0;
      s_refuse = s_huge = 0;
    }
    __syncthreads();
    if (threadIdx.x < k) {
      uint32_t n[kBins], total = 0;
      for (int b = 0; b < kBins; ++b) total += s_n[threadIdx.x][b] = n[b] = __ldcg(&ctrl->count[cur][threadIdx.x][b]);
      atomicAdd(&s_cost, (unsigned long long)small_cost(n));
      if (total > kSmallClass) s_refuse = 1;
    }
    __syncthreads();
    if (s_cost > kSmallCostMax || s_refuse) break;  // left to the per-bin kernels
    for (uint32_t s = 0; s < k; ++s)
      for (uint32_t t = threadIdx.x; t < s_n[s][kBinHuge]; t += kSmallThreads)
        if (q.a[0].g.deg[q.lists[cur][seg.off[s * kBins + kBinHuge] + t]] > kSmallHuge) s_huge = 1;
    const int nxt = cur ^ 1;
    const DecideArgs& a = q.a[cur];  // (marks and appends into the other buffer)
    const uint32_t* base = q.lists[cur];
    cluster_sync();  // every CTA has read what is reset here
    if (s_huge) break;
    if (rank == 0) {
      if (threadIdx.x == 0) {
        if (it == 0) {
          unsigned long long first = 0;
          for (uint32_t s = 0; s < k; ++s)
            for (int b = 0; b < kBins; ++b) first += s_n[s][b];
          ctrl->sm_first = first;
        }
        ctrl->s_lo = ctrl->s_hi = 0;
        ctrl->processed = ctrl->moved = 0;
      }
      if (threadIdx.x < 2) ctrl->it_nbig[threadIdx.x] = 0;
      for (uint32_t x = threadIdx.x; x < kMaxSubsteps * kBins; x += kSmallThreads) (&ctrl->count[nxt][0][0])[x] = 0;
    }
    cluster_sync();
    for (uint32_t s = 0; s < k; ++s) {
      const uint32_t n0 = s_n[s][kBinTiny], nl = s_n[s][kBinLanes], n1 = s_n[s][kBinTable], nm = s_n[s][kBinMid],
                     n2 = nm + s_n[s][kBinWhole], n3 = s_n[s][kBinHuge];
      if (!(n0 + nl + n1 + n2 + n3)) continue;
      const uint32_t par = step++ & 1;  // the counters of this sub-step that is run
      unsigned long long* nbig = &ctrl->it_nbig[par];
      uint32_t gi;
      Move m;
      // 1. decide
      for (uint32_t t = 0; t < n3; ++t) {
        const uint32_t i = base[seg.off[s * kBins + kBinHuge] + t];
        long long m2 = m2_one;
        gi = 0;
        if (!group_active(a, i, &m2, &gi)) continue;
        if (rank == 0 && threadIdx.x == 0) {
          if (a.ever && bit_set(a.ever, i)) ++sums.ever;
          ++sums.processed;
        }
        if (a.rbits && !bit_test(a.rbits, i)) continue;
        if (cluster_vertex(a, i, m2, dyn, sp, sc, &m, sums)) small_record(a, m, gi, moves, &s_nmv[par], nbig, sums);
      }
      if (n3) {
        cluster_sync();  // the table's last reader is done: its memory is the warps' again
        empty_table();
      }
      for (uint32_t t = rank; t < n2; t += kSmallCtas) {
        const uint32_t i = t < nm ? base[seg.off[s * kBins + kBinMid] + t] : base[seg.off[s * kBins + kBinWhole] + t - nm];
        long long m2 = m2_one;
        gi = 0;
        if (!group_active(a, i, &m2, &gi)) continue;
        if (threadIdx.x == 0) {
          if (a.ever && bit_set(a.ever, i)) ++sums.ever;
          ++sums.processed;
        }
        if (a.rbits && !bit_test(a.rbits, i)) continue;
        if (block_vertex<kSmallThreads, kBlockSlots>(a, i, m2, block_table, sc, &m, sums))
          small_record(a, m, gi, moves, &s_nmv[par], nbig, sums);
      }
      for (uint32_t u = warp; u < n1; u += kSmallWarps) {
        // (every lane loads the one header: broadcasts)
        VHdr v;
        v.i = base[seg.off[s * kBins + kBinTable] + u];
        long long m2 = m2_one;
        v.gi = 0;
        if (!group_active(a, v.i, &m2, &v.gi)) continue;
        v.m2 = uint32_t(m2);
        v.d = a.C[v.i];
        v.Ki = uint32_t(a.K[v.i]);
        v.o = a.g.off[v.i];
        v.dg = a.g.deg[v.i];
        const uint32_t em = 1u << (v.i & 31u);
        const uint32_t old = (lane == 0 && a.ever) ? atomicOr(a.ever + (v.i >> 5), em) : em;
        if (!a.rbits || bit_test(a.rbits, v.i)) {
          v.Sd = sigma32(a.Sigma, v.d);
          v.szd = a.size[v.d];
          v.act = true;
          bool mv;
          if (!fits64(v.m2, v.Ki)) {
            mv = warp_table_vertex(a, v.i, m2, keys, vals, &m, sums);
            empty_table();
          } else {
            const uint2 a0 = lane < v.dg ? a.g.arcs[v.o + lane] : make_uint2(v.i, 0u);
            uint32_t bc = 0, ncand = 0;
            i128 gain = 0;
            mv = v.dg <= 64    ? table_vertex<2>(a, v, a0, keys, vals, &bc, &gain, &ncand)
                 : v.dg <= 128 ? table_vertex<4>(a, v, a0, keys, vals, &bc, &gain, &ncand)
                               : table_vertex<8>(a, v, a0, keys, vals, &bc, &gain, &ncand);
            if (lane == 0) sums.bytes += 24 + 12ull * v.dg + 12ull * ncand + (mv ? 16 + 4ull * v.dg : 0ull);
            m = Move{v.o, v.i, v.d, bc, v.dg, v.Ki, gain};
          }
          if (mv && lane == 0) small_record(a, m, v.gi, moves, &s_nmv[par], nbig, sums);
        }
        if (lane == 0) {
          ++sums.processed;
          if (!(old & em)) ++sums.ever;
        }
      }
      for (uint32_t t = warp; t < nl; t += kSmallWarps)
        if (decide_position<32>(a, base + seg.off[s * kBins + kBinLanes], t, nl, m2_one, &gi, &m, sums) && lane == 0)
          small_record(a, m, gi, moves, &s_nmv[par], nbig, sums);
      const uint32_t* tiny = base + seg.off[s * kBins + kBinTiny];
      const uint32_t per = 32 / q.seg_lanes;
      for (uint32_t first = rev * per; first < n0; first += kSmallWarps * per) {
        bool mv;
        switch (q.seg_lanes) {
          case 4: mv = decide_position<4>(a, tiny, first, n0, m2_one, &gi, &m, sums); break;
          case 8: mv = decide_position<8>(a, tiny, first, n0, m2_one, &gi, &m, sums); break;
          case 16: mv = decide_position<16>(a, tiny, first, n0, m2_one, &gi, &m, sums); break;
          default: mv = decide_position<32>(a, tiny, first, n0, m2_one, &gi, &m, sums); break;
        }
        if (mv && lane % q.seg_lanes == 0) small_record(a, m, gi, moves, &s_nmv[par], nbig, sums);
      }
      cluster_sync();
      // 2. commit the CTA's own moves and mark around them; the other pair of counters is idle
      const uint32_t done = s_nmv[par];
      if (threadIdx.x == 0) {
        s_nmv[par ^ 1] = 0;
        if (rank == 0) ctrl->it_nbig[par ^ 1] = 0;
        if (done) atomicAdd(&ctrl->moved, (unsigned long long)done);
      }
      // a warp per move, or eight lanes when there are many
      const uint32_t L = done > 2 * kSmallThreads / 32 ? 8u : 32u, sl = lane & (L - 1);
      for (uint32_t e0 = wib * (32 / L); e0 < done; e0 += kSmallThreads / L) {
        const uint32_t e = e0 + lane / L;
        if (e >= done) continue;
        const SmallMove v = moves[e];
        if (sl == 0) const_cast<uint32_t*>(a.C)[v.i] = v.c;
        if (sl == 1 || sl == 2) {
          const unsigned long long ki = v.Ki;
          atomicAdd((unsigned long long*)const_cast<long long*>(a.Sigma) + (sl == 1 ? v.c : v.d), sl == 1 ? ki : 0ull - ki);
        }
        if (sl == 3 || sl == 4) atomicAdd(const_cast<int*>(a.size) + (sl == 3 ? v.c : v.d), sl == 3 ? 1 : -1);
        if (v.dg <= kMarkInline) mark_arcs<true>(a, v.i, v.o, 0, v.dg, sl, L);
      }
      const unsigned long long big = __ldcg(nbig);
      mark_queued<true>(a, big, rev, kSmallWarps);
      cluster_sync();
    }
    // 3. the processed frontier's bits, the sums, the tolerance test
    for (uint32_t s = 0; s < k; ++s)
      for (int b = 0; b < kBins; ++b)
        for (uint32_t t = rank * kSmallThreads + threadIdx.x; t < s_n[s][b]; t += kSmallCtas * kSmallThreads)
          q.fbits[cur][base[seg.off[s * kBins + b] + t] >> 5] = 0u;
    flush_sums_all(a, sums);
    sums = MoveSums();
    cluster_sync();
    cur = nxt;
    if (threadIdx.x == 0) {
      const unsigned long long lo = __ldcg(&ctrl->s_lo), hi = __ldcg(&ctrl->s_hi);
      const u128 S = ((u128)hi << 32) + (u128)lo;
      if (rank == 0) {
        unsigned long long* tr = ctrl->sm_trace[it];
        tr[0] = __ldcg(&ctrl->processed);
        tr[1] = __ldcg(&ctrl->moved);
        tr[2] = (unsigned long long)(S >> 64);
        tr[3] = (unsigned long long)S;
      }
      s_stop = (!q.single && S <= threshold) || it + 1 == q.max_iters ? 2 : (q.single || it + 1 == kSmallIters) ? 1 : 0;
    }
    __syncthreads();
    ++it;
    if (s_stop) break;
  }
  if (rank == 0 && threadIdx.x == 0) {
    ctrl->sm_iters = it;
    ctrl->sm_done = it && s_stop == 2;  // converged, or the pass is out of iterations
  }
}

// The start of an iteration: its sums (s_lo .. moved), both pairs of mover
// counters (sub-step s counts into pair s & 1) and the next list buffer's
// lengths are zeroed.
__global__ void k_iter_start(Ctrl* ctrl, int nxt) {
  pdl_wait();
  if (threadIdx.x == 0) {
    ctrl->s_lo = ctrl->s_hi = 0;
    ctrl->processed = ctrl->moved = 0;
  }
  if (threadIdx.x < 2) {
    ctrl->it_movers[threadIdx.x] = 0;
    ctrl->it_nbig[threadIdx.x] = 0;
    ctrl->it_bignd[threadIdx.x] = 0;
  }
  unsigned int* c = &ctrl->count[nxt][0][0];
  for (uint32_t q = threadIdx.x; q < sizeof(ctrl->count[0]) / sizeof(unsigned int); q += blockDim.x) c[q] = 0u;
}

// What a local-moving call sets in its control block: whether it starts from
// singletons, its counters, and its 2m; with a batch apply enqueued just before (ap),
// the batch's change of 2m if its gate opened
__global__ void k_set_m2(Ctrl* ctrl, long long m2, const Ctrl* ap, uint32_t from_singletons) {
  pdl_wait();
  ctrl->from_singletons = from_singletons;
  ctrl->m2v = m2 + (ap && ap->apply_go ? ap->m2_delta : 0ll);
  ctrl->move_bytes = 0;  // this call's counters
  ctrl->ever_count = 0;
}

// largest grid of the block-per-vertex kernel; each of its blocks owns one
// slice of the global overflow table
constexpr uint32_t kBlockGridMax = 3 * 152;

// Profile class of each bin (the lane and table bins are one class, as are the block bins).
constexpr int kBinClass[kBins] = {DFL_PROF_BIN0, DFL_PROF_BIN1, DFL_PROF_BIN1, DFL_PROF_BIN2, DFL_PROF_BIN2, DFL_PROF_BIN3};

// k_decide_lanes for a list of c vertices (~0: its length is on the device) of
// at most lim arcs.
void launch_lanes(const DecideArgs& a, uint32_t lim, uint32_t c, cudaStream_t st) {
  if (lim <= 8)
    k_decide_lanes<8><<<c == ~0u ? 152 * 8 : grid_for(c, kLaneThreads, 152 * 64), kLaneThreads, 0, st>>>(a);
  else
    k_decide_lanes<32><<<c == ~0u ? 152 * 5 : grid_for(c, kLaneThreads, 152 * 64), kLaneThreads, 0, st>>>(a);
}

// Issue one local-moving iteration (all sub-steps) on h->stream.  With
// `counts` (host-known list lengths) empty bins are skipped and grids are
// sized to the work; without (graph capture) every bin is launched with a
// fixed grid and reads its length on the device.
int issue_iteration(Handle* h, DecideArgs a, int cur, const unsigned int (*counts)[kBins],
                    const GiantDecide& gd_base, bool decide_only = false, bool small_hint = false) {
  const uint32_t k = a.k;
  const int nxt = cur ^ 1;
  // reset the iteration's sums, both pairs of mover counters and the next
  // buffer's list lengths (one launch)
  {
    LaunchScope ls(h, DFL_PROF_OTHER);
    launch_pdl(k_iter_start, 1, 64, 0, h->stream, h->ctrl, nxt);
    DFL_TRY(check_launch(h, "iteration start"));
  }
  if (a.ngraphs)
    DFL_CUDA(h, cudaMemsetAsync(a.gS, 0, sizeof(unsigned long long) * 2 * a.ngraphs, h->stream));
  a.fbits_next = h->fbits[nxt];
  a.next_lists = h->lists[nxt];
  a.next_buf = nxt;
  const uint64_t gstride = h->g_items_cap / kMaxSubsteps;
  // The degree bins of a sub-step are independent and run concurrently.  The
  // chain that bounds a sub-step -- the largest-degree chunks, their
  // decisions, the commit -- runs on one stream (the spine, the highest-
  // priority auxiliary stream), so that each of its kernels is a dependent
  // launch of the one before; the spine forks the other bins (the tiny one on
  // the handle's stream, the rest on auxiliary streams) at the start of a
  // sub-step and joins them before the commit.  With DFL_FLAG_SERIAL_BINS
  // everything runs on the handle's stream.
  const bool par = !(h->opt.flags & DFL_FLAG_SERIAL_BINS);
  cudaStream_t spine = par ? h->aux[kBins - 2] : h->stream;
  cudaStream_t bst[kBins] = {h->stream, par ? h->aux[0] : h->stream, par ? h->aux[1] : h->stream,
                             par ? h->aux[2] : h->stream, par ? h->aux[3] : h->stream, spine};
  if (par) {
    DFL_CUDA(h, cudaEventRecord(h->ev_fork, h->stream));
    DFL_CUDA(h, cudaStreamWaitEvent(spine, h->ev_fork, 0));
  }
  const bool wide_labels = a.g.nv >= kLaneLabels;  // labels that do not fit k_decide_lanes' keys
  bool any_huge = !counts;
  for (uint32_t s = 0; counts && s < k; ++s) any_huge |= counts[s][kBinHuge] != 0;
  if (any_huge) {  // the largest-degree layouts of all classes, once
    LaunchScope ls(h, DFL_PROF_BIN3, spine);
    launch_pdl(k_giant_prefix, k, 1024, 0, spine, a, gd_base, gstride, h->lists[cur], cur);
    DFL_TRY(check_launch(h, "giant prefix"));
  }
  for (uint32_t s = 0; s < k; ++s) {
    a.movers = &h->ctrl->it_movers[s & 1];
    a.nbig = &h->ctrl->it_nbig[s & 1];
    a.clear_movers = s + 1 < k ? &h->ctrl->it_movers[(s + 1) & 1] : nullptr;
    a.clear_nbig = s + 1 < k ? &h->ctrl->it_nbig[(s + 1) & 1] : nullptr;
    a.clear_bignd = s + 1 < k ? &h->ctrl->it_bignd[(s + 1) & 1] : nullptr;
    bool has[kBins], any = false;
    for (int b = 0; b < kBins; ++b) {
      has[b] = !counts || counts[s][b];
      any |= has[b];
    }
    // short lists of the two register bins share a launch
    const uint64_t n0 = counts ? counts[s][kBinTiny] : 0, n1 = counts ? counts[s][kBinLanes] : 0;
    const bool short0 = wide_labels || (counts ? n0 < kSmallList : small_hint);
    const bool short1 = wide_labels || (counts ? n1 < kSmallLanes : small_hint);
    const bool merged = short0 && short1 && has[kBinLanes];
    if (merged) {
      has[kBinTiny] = true;
      has[kBinLanes] = false;
    }
    cudaEvent_t pa = nullptr, pb = nullptr;  // wall time of the decide phase (profiling)
    if (any && (h->opt.flags & (DFL_FLAG_PROFILE | DFL_FLAG_PROFILE_MOVE))) {
      pa = take_event(h);
      pb = take_event(h);
      if (pa) record_timing_event(pa, spine);
    }
    // the fork point is this sub-step's start on the spine, before its own kernels
    bool fork = false;
    for (int b = 0; b < kBins; ++b) fork |= bst[b] != spine && has[b];
    if (fork) DFL_CUDA(h, cudaEventRecord(h->ev_fork, spine));
    bool joined[kBins - 1] = {};
    for (int b = kBins - 1; b >= 0; --b) {
      const uint32_t c = counts ? counts[s][b] : 0u;
      if (!has[b]) continue;
      cudaStream_t st = bst[b];
      if (st != spine) {
        DFL_CUDA(h, cudaStreamWaitEvent(st, h->ev_fork, 0));
        joined[b] = true;
      }
      a.list = h->lists[cur] + h->segs.off[s * kBins + b];
      a.count = &h->ctrl->count[cur][s][b];
      LaunchScope ls(h, kBinClass[b], st);
      if (b == kBinTiny) {
        const uint32_t lim = h->tune.bin_warp;
        const uint32_t segs = lim <= 4 ? 8 : lim <= 8 ? 4 : lim <= 16 ? 2 : 1;
        const uint32_t grid = counts ? grid_for(((n0 + segs - 1) / segs + (merged ? n1 : 0)) * 32, 256, 152 * 64) : 152 * 8;
        const uint32_t* l2 = merged ? h->lists[cur] + h->segs.off[s * kBins + kBinLanes] : nullptr;
        const unsigned int* c2 = merged ? &h->ctrl->count[cur][s][kBinLanes] : nullptr;
        if (!short0) launch_lanes(a, lim, counts ? c : ~0u, st);
        else if (segs == 8) k_decide_warp<4><<<grid, 256, 0, st>>>(a, l2, c2);
        else if (segs == 4) k_decide_warp<8><<<grid, 256, 0, st>>>(a, l2, c2);
        else if (segs == 2) k_decide_warp<16><<<grid, 256, 0, st>>>(a, l2, c2);
        else k_decide_warp<32><<<grid, 256, 0, st>>>(a, l2, c2);
      } else if (b == kBinLanes) {
        if (short1)  // a warp per vertex: the shorter chain
          k_decide_warp<32><<<counts ? grid_for(uint64_t(c) * 32, 256, 152 * 64) : 152 * 8, 256, 0, st>>>(a, nullptr,
                                                                                                       nullptr);
        else
          launch_lanes(a, h->segs.hi[kBinLanes], counts ? c : ~0u, st);
      } else if (b == kBinTable) {
        // a warp per vertex, headers in batches of up to 32 (fewer when the list is short)
        k_decide_warp_hash<<<counts ? grid_for(uint64_t(c) * 32, 256, 152 * 6) : 152 * 3, 256, 0, st>>>(a);
      } else if (b == kBinMid) {
        // (a replayed graph launches every bin at once: with all eight blocks an SM
        // this one keeps the lane bin's blocks, of the lowest priority too, waiting:
        // ND on 2^18, 2^20 and 2^22 vertices 315, 533 and 1,468 us so, 295, 514 and
        // 1,475 with five, 301, 522 and 1,490 with four)
        k_decide_block<128, 2 * kMidDeg>
            <<<counts ? grid_for(c, 1, 152 * 8) : 152 * 5, 128, sizeof(uint32_t) * 4 * kMidDeg, st>>>(a);
      } else if (b == kBinWhole) {
        const size_t smem = sizeof(uint32_t) * 2 * kBlockSlots;
        const uint32_t bt = h->tune.block_threads;
        const uint32_t per_sm = bt == 512 ? 2 : 3;  // 64 KB table each; grid <= kBlockGridMax
        const uint32_t grid = counts ? grid_for(c, 1, 152 * per_sm) : 152 * per_sm;
        if (bt == 128) k_decide_block<128, kBlockSlots><<<grid, 128, smem, st>>>(a);
        else if (bt == 512) k_decide_block<512, kBlockSlots><<<grid, 512, smem, st>>>(a);
        else k_decide_block<256, kBlockSlots><<<grid, 256, smem, st>>>(a);
      } else {
        GiantDecide gd = giant_class(gd_base, s, gstride, h->ctrl);  // laid out above
        gd.nbignd = &h->ctrl->it_bignd[s & 1];
        launch_pdl(k_giant_accum, 152 * 4, kAccumThreads, 0, st, a, gd);
        DFL_TRY(check_launch(h, "giant accumulate"));
        launch_pdl(k_giant_decide, 152 * 4, kGiantThreads, 0, st, a, gd);
      }
      DFL_TRY(check_launch(h, "decide"));
    }
    for (int b = 0; b < kBins - 1; ++b)
      if (joined[b]) {
        DFL_CUDA(h, cudaEventRecord(h->ev_join[b], bst[b]));
        DFL_CUDA(h, cudaStreamWaitEvent(spine, h->ev_join[b], 0));
      }
    if (pa && pb) {
      record_timing_event(pb, spine);
      h->ev_pending.push_back(Handle::Ev{pa, pb, DFL_PROF_MOVE});
      h->prof.launches[DFL_PROF_MOVE]++;
    } else {
      if (pa) h->ev_free.push_back(pa);
      if (pb) h->ev_free.push_back(pb);
    }
    if (any && decide_only) {
      // (it_nbig, it_movers and it_bignd are adjacent)
      DFL_CUDA(h, cudaMemsetAsync(&h->ctrl->it_nbig[0], 0, sizeof(h->ctrl->it_nbig) + 2 * sizeof(h->ctrl->it_movers), spine));
    } else if (any) {
      LaunchScope ls(h, DFL_PROF_COMMIT, spine);
      launch_pdl(k_commit, 152 * 4, kCommitThreads, 0, spine, a);
      DFL_TRY(check_launch(h, "commit"));
    } else if (a.clear_movers) {  // no commit ran: zero the next sub-step's counters here
      DFL_CUDA(h, cudaMemsetAsync(a.clear_movers, 0, sizeof(unsigned int), spine));
      DFL_CUDA(h, cudaMemsetAsync(a.clear_nbig, 0, sizeof(*a.clear_nbig), spine));
      DFL_CUDA(h, cudaMemsetAsync(a.clear_bignd, 0, sizeof(*a.clear_bignd), spine));
    }
  }
  // the next frontier's lists, from its bitmap
  {
    LaunchScope ls(h, DFL_PROF_MARK, spine);
    // (the processed frontier's bitmap, cleared alongside, becomes the next-next target)
    launch_pdl(k_lists_bits, lists_grid(a.g.nv), kListThreads, 0, spine, a.fbits_next, a.g.nv, a.g.deg, a.next_lists,
               a.seg, h->ctrl, nxt, k, h->fbits[cur], h->words);
    DFL_TRY(check_launch(h, "next frontier lists"));
  }
  if (par) {  // the handle's stream continues after the spine
    DFL_CUDA(h, cudaEventRecord(h->ev_fork, spine));
    DFL_CUDA(h, cudaStreamWaitEvent(h->stream, h->ev_fork, 0));
  }
  return DFL_OK;
}

// Launch configuration of the small-frontier kernel.
struct SmallLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  explicit SmallLaunch(cudaStream_t s) {
    cfg.gridDim = kSmallCtas;
    cfg.blockDim = kSmallThreads;
    cfg.dynamicSmemBytes = kSmallSmemAll;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kSmallCtas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
};

// Whether lists of these lengths are a small frontier (the kernel's own rule).
bool small_frontier(const unsigned int (*n)[kBins]) {
  uint64_t cost = 0, longest = 0;
  for (uint32_t s = 0; s < kMaxSubsteps; ++s) {
    uint64_t total = 0;
    for (int b = 0; b < kBins; ++b) total += n[s][b];
    longest = longest > total ? longest : total;
    cost += small_cost(n[s]);
  }
  return cost <= kSmallCostMax && longest <= kSmallClass;
}

// A frontier of at most this many vertices is tried without reading its
// lengths first: the kernel checks them itself, and a refusal costs its empty
// launch (the read it comes back with is needed either way; 12 us on a skewed
// graph of 2^14 vertices, whose DS updates know the lengths instead).
constexpr uint64_t kSmallTry = 16384;

// Whether the GPU can hold the small-frontier kernel's cluster; queried once per process.
bool small_available() {
  static std::once_flag once;
  static bool ok = false;
  std::call_once(once, [] {
    int n = 0;
    if (cudaFuncSetAttribute(k_small_move, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(k_small_move, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmallSmemAll)) ==
            cudaSuccess) {
      SmallLaunch l(nullptr);
      l.cfg.numAttrs = 1;
      ok = cudaOccupancyMaxActiveClusters(&n, k_small_move, &l.cfg) == cudaSuccess && n >= 1;
    }
    if (!ok) cudaGetLastError();
  });
  return ok;
}

// Blocks of the cooperative iteration kernel that are resident at once
// (0: it cannot run); queried once per process.
uint32_t persistent_grid() {
  static std::once_flag once;
  static uint32_t grid = 0;
  std::call_once(once, [] {
    int dev = 0, sms = 0, per_sm = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return;
    if (cudaFuncSetAttribute(k_iterate, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(sizeof(uint32_t) * kIterDynWords)) != cudaSuccess)
      return;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_iterate, kIterThreads,
                                                      sizeof(uint32_t) * kIterDynWords) != cudaSuccess)
      return;
    uint64_t g = uint64_t(sms) * uint64_t(per_sm);
    // each block may own a slice of the block kernel's overflow table
    grid = uint32_t(g < kBlockGridMax ? g : kBlockGridMax);
  });
  return grid;
}

// One local-moving iteration as a single cooperative launch of k_iterate.
int issue_persistent(Handle* h, const DecideArgs& a_base, int cur, const GiantDecide& gd, uint32_t grid) {
  const int nxt = cur ^ 1;
  DFL_CUDA(h, cudaMemsetAsync(h->ctrl, 0, offsetof(Ctrl, move_bytes), h->stream));
  DFL_CUDA(h, cudaMemsetAsync(&h->ctrl->it_nbig[0], 0,
                              offsetof(Ctrl, bar_gen) + sizeof(unsigned int) - offsetof(Ctrl, it_nbig),
                              h->stream));
  DFL_CUDA(h, cudaMemsetAsync(&h->ctrl->count[nxt][0][0], 0, sizeof(h->ctrl->count[0]), h->stream));
  if (a_base.ngraphs)
    DFL_CUDA(h, cudaMemsetAsync(a_base.gS, 0, sizeof(unsigned long long) * 2 * a_base.ngraphs, h->stream));
  IterArgs ia;
  std::memset(&ia, 0, sizeof(ia));
  ia.a = a_base;
  ia.a.fbits_next = h->fbits[nxt];
  ia.a.next_lists = h->lists[nxt];
  ia.a.next_buf = nxt;
  ia.gd = gd;
  ia.gstride = uint32_t(h->g_items_cap / kMaxSubsteps);
  ia.k = a_base.k;
  ia.cur = cur;
  const uint32_t lim = h->tune.bin_warp;
  ia.seg_lanes = lim <= 4 ? 4 : lim <= 8 ? 8 : lim <= 16 ? 16 : 32;
  ia.lists_cur = h->lists[cur];
  ia.fbits_cur = h->fbits[cur];
  ia.words = h->words;
  const bool test_timeout = (h->opt.flags & DFL_FLAG_TEST_UNREACHABLE_BARRIER) != 0;
  ia.bar_extra = test_timeout ? 1u : 0u;
  ia.bar_polls = test_timeout ? kTestBarrierPolls : kBarrierPolls;
  void* args[] = {&ia};
  {
    LaunchScope ls(h, DFL_PROF_MOVE);
    DFL_CUDA(h, cudaLaunchCooperativeKernel((const void*)k_iterate, dim3(grid), dim3(kIterThreads), args,
                                            sizeof(uint32_t) * kIterDynWords, h->stream));
  }
  return DFL_OK;
}

// Local-moving iterations of a small frontier (list buffer `cur`) in one
// launch; how many ran, and whether the pass is done, is in the control block.
int issue_small(Handle* h, const DecideArgs& a, int cur, uint32_t pass, uint32_t iters_left) {
  if (a.ngraphs)
    DFL_CUDA(h, cudaMemsetAsync(a.gS, 0, sizeof(unsigned long long) * 2 * a.ngraphs, h->stream));
  SmallArgs q;
  std::memset(&q, 0, sizeof(q));
  for (int b = 0; b < 2; ++b) {
    q.a[b] = a;
    q.a[b].fbits_next = h->fbits[b ^ 1];
    q.a[b].next_lists = h->lists[b ^ 1];
    q.a[b].next_buf = b ^ 1;
  }
  q.cur = cur;
  const uint32_t lim = h->tune.bin_warp;
  q.seg_lanes = lim <= 4 ? 4 : lim <= 8 ? 8 : lim <= 16 ? 16 : 32;
  for (int b = 0; b < 2; ++b) {
    q.lists[b] = h->lists[b];
    q.fbits[b] = h->fbits[b];
  }
  q.max_iters = iters_left;
  q.single = a.ngraphs ? 1u : 0u;
  q.pass = pass;
  q.tau_num = h->opt.tau_num;
  q.tau_den = h->opt.tau_den;
  q.drop = h->opt.tolerance_drop;
  LaunchScope ls(h, DFL_PROF_MOVE);
  SmallLaunch l(h->stream);
  cudaLaunchKernelEx(&l.cfg, k_small_move, q);
  return check_launch(h, "small frontier");
}

// Everything an iteration graph bakes in; a different key means re-capture.
struct GraphKey {
  DecideArgs a;
  GiantDecide gd;
  int cur;
  int small;
  uint32_t flags;
  void* stream;
  uint32_t block_threads;
};

// The cached graph for this iteration's key (captured on a miss, evicting
// the least recently used entry of this parity).
int ensure_iteration_graph(Handle* h, const DecideArgs& a, const GiantDecide& gd, int cur, bool small,
                           Handle::IterGraph** out) {
  GraphKey key;
  std::memset(&key, 0, sizeof(key));
  key.a = a;
  key.gd = gd;
  key.cur = cur;
  key.small = small;
  key.flags = h->opt.flags;
  key.stream = h->stream;
  key.block_threads = h->tune.block_threads;
  Handle::IterGraph* slot = nullptr;
  for (auto& e : h->igraph[cur])
    if (e.exec && e.key.size() == sizeof(key) && std::memcmp(e.key.data(), &key, sizeof(key)) == 0) {
      e.last_use = ++h->graph_use;
      *out = &e;
      return DFL_OK;
    }
  for (auto& e : h->igraph[cur])
    if (!slot || !e.exec || (slot->exec && e.last_use < slot->last_use)) slot = &e;
  Handle::IterGraph& g = *slot;
  destroy_iteration_graph(g);
  const auto t0 = std::chrono::steady_clock::now();
  const size_t ev0 = h->ev_pending.size();
  const uint64_t l0 = h->launches;
  uint64_t cl0[DFL_PROF_CLASSES];
  for (int q = 0; q < DFL_PROF_CLASSES; ++q) cl0[q] = h->prof.launches[q];
  DFL_CUDA(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
  int rc = issue_iteration(h, a, cur, nullptr, gd, false, small);
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(h->stream, &graph);
  if (rc) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return set_error(h, DFL_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(e));
  e = cudaGraphInstantiate(&g.exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) {
    g.exec = nullptr;
    return set_error(h, DFL_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
  }
  // events recorded inside the graph are harvested after every replay
  g.evs.assign(h->ev_pending.begin() + ev0, h->ev_pending.end());
  h->ev_pending.resize(ev0);
  g.kernels = h->launches - l0;
  h->launches = l0;
  for (int q = 0; q < DFL_PROF_CLASSES; ++q) {  // counted per replay instead
    g.class_launches[q] = h->prof.launches[q] - cl0[q];
    h->prof.launches[q] = cl0[q];
  }
  g.key.assign(reinterpret_cast<const char*>(&key), reinterpret_cast<const char*>(&key) + sizeof(key));
  g.last_use = ++h->graph_use;
  h->graph_captures++;
  h->graph_capture_ms +=
      std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  *out = &g;
  return DFL_OK;
}

}  // namespace

void destroy_iteration_graph(Handle::IterGraph& g) {
  if (g.exec) cudaGraphExecDestroy(g.exec);
  for (auto& ev : g.evs) {
    cudaEventDestroy(ev.a);
    cudaEventDestroy(ev.b);
  }
  g.evs.clear();
  g.key.clear();
  g.exec = nullptr;
  g.kernels = 0;
}

namespace {

// Buffers, streams and kernel attributes one local-moving run needs, and its
// decide arguments.
int prepare_move(Handle* h, const MoveArgs& ma, DecideArgs* out, GiantDecide* gdo) {
  const uint32_t k = h->opt.substeps;
  make_segs(h, k);
  // overflow tables of the block-per-vertex kernel, needed only when its bin
  // takes degrees beyond what its shared table always holds: one slice of
  // gslots keys + gslots values per block, gslots >= 2 * (largest degree it takes)
  const uint32_t blk_max = ma.max_deg < h->tune.bin_block ? ma.max_deg : h->tune.bin_block;
  const bool need_gtable = blk_max > kBinBlock;
  const uint32_t gslots = next_pow2(2ull * (need_gtable ? blk_max : kBinBlock));
  if (need_gtable && uint64_t(kBlockGridMax) * gslots > h->gtable_cap) {
    if (h->gtable) {
      cudaStreamSynchronize(h->stream);
      cudaFree(h->gtable);
      h->gtable = nullptr;
      h->gtable_cap = 0;
    }
    DFL_CUDA(h, dev_malloc(&h->gtable, sizeof(uint2) * uint64_t(kBlockGridMax) * gslots));
    h->gtable_cap = uint64_t(kBlockGridMax) * gslots;
  }
  // once per process (handles may be driven from several host threads)
  static std::once_flag smem_once;
  static cudaError_t smem_rc = cudaSuccess;
  std::call_once(smem_once, [] {
    const int tb = int(sizeof(uint32_t) * 2 * kBlockSlots);
    smem_rc = cudaFuncSetAttribute(k_decide_block<128, kBlockSlots>, cudaFuncAttributeMaxDynamicSharedMemorySize, tb);
    if (smem_rc == cudaSuccess)
      smem_rc = cudaFuncSetAttribute(k_decide_block<256, kBlockSlots>, cudaFuncAttributeMaxDynamicSharedMemorySize, tb);
    if (smem_rc == cudaSuccess)
      smem_rc = cudaFuncSetAttribute(k_decide_block<512, kBlockSlots>, cudaFuncAttributeMaxDynamicSharedMemorySize, tb);
    if (smem_rc == cudaSuccess)
      smem_rc = cudaFuncSetAttribute(k_iterate, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     int(sizeof(uint32_t) * kIterDynWords));

  });
  DFL_CUDA(h, smem_rc);
  // the huge bin's buffers, sized by bounds (arcs: of the listed vertices'
  // degrees): at most arcs / (bin_block + 1) listed vertices; tables of at most
  // 4 x degree (>= 64) slots each; occupied lists of at most degree entries; at
  // most arcs / kGiantPart + items parts
  {
    uint64_t arcs = slots_bound(live_arcs_bound(h), tombs_bound(h), h->tune.bin_block);
    for (int q = 0; q < 2; ++q) arcs = arcs > h->sg[q].arc_cap ? arcs : h->sg[q].arc_cap;
    // (one region per sub-step class: the persistent kernel lays out all
    // classes at the start of an iteration)
    const uint64_t items = (arcs / (uint64_t(h->tune.bin_block) + 1) + 64 + 1) * kMaxSubsteps;
    const bool any = ma.max_deg > h->tune.bin_block;
    const uint64_t tab = any ? 4 * arcs + 64 * items : 0;
    const uint64_t lst = any ? arcs + 64 : 0;
    const uint64_t res = any ? arcs / kGiantPart + items : 0;
    auto regrow = [&](auto** p, uint64_t& cap, uint64_t need, size_t elem, int fill) -> int {
      if (need <= cap) return DFL_OK;
      cudaStreamSynchronize(h->stream);
      cudaFree(*p);
      *p = nullptr;
      cap = 0;
      const uint64_t want = need + need / 4;
      DFL_CUDA(h, dev_malloc(p, elem * want));
      if (fill >= 0) DFL_CUDA(h, cudaMemsetAsync(*p, fill, elem * want, h->stream));
      cap = want;
      return DFL_OK;
    };
    if (items > h->g_items_cap) {
      uint64_t c0 = h->g_items_cap, c1 = c0, c2 = c0, c3 = c0, c4 = c0, c5 = c0;
      DFL_TRY(regrow(&h->g_toff, c0, items, sizeof(unsigned long long), -1));
      DFL_TRY(regrow(&h->g_loff, c1, items, sizeof(unsigned long long), -1));
      DFL_TRY(regrow(&h->g_cpre, c2, items + 1, sizeof(uint32_t), -1));
      DFL_TRY(regrow(&h->g_ndist, c3, items, sizeof(uint32_t), 0));
      DFL_TRY(regrow(&h->g_done, c4, items, sizeof(uint32_t), 0));
      DFL_TRY(regrow(&h->g_hd, c5, items, sizeof(unsigned long long), 0));
      h->g_items_cap = c0 < c2 ? c0 : c2 - 1;
    }
    {
      uint64_t c = h->g_res_cap;
      GiantRes* r = static_cast<GiantRes*>(h->g_res);
      const int rc = regrow(&r, c, res, sizeof(GiantRes), -1);
      h->g_res = r;  // also when the allocation failed: the old buffer is gone
      h->g_res_cap = c;
      DFL_TRY(rc);
    }
    if (tab > h->g_tab_cap) {
      uint64_t c0 = h->g_tab_cap, c1 = c0;
      DFL_TRY(regrow(&h->g_tkeys, c0, tab, sizeof(uint32_t), 0xFF));  // kEmpty
      DFL_TRY(regrow(&h->g_tvals, c1, tab, sizeof(uint32_t), 0));
      h->g_tab_cap = c0;
    }
    DFL_TRY(regrow(&h->g_tlist, h->g_lst_cap, lst, sizeof(uint2), -1));
  }
  {  // the queue of movers whose rows k_commit marks in pieces: at most one per
     // vertex of degree > kMarkInline
    uint64_t arcs = pool_top_bound(h);
    for (int q = 0; q < 2; ++q) arcs = arcs > h->sg[q].arc_cap ? arcs : h->sg[q].arc_cap;
    uint64_t need = arcs / (kMarkInline + 1) + 64;
    if (need > uint64_t(h->n) + 64) need = uint64_t(h->n) + 64;
    if (need > h->bigmv_cap) {
      cudaStreamSynchronize(h->stream);
      cudaFree(h->bigmv);
      h->bigmv = nullptr;
      h->bigmv_cap = 0;
      DFL_CUDA(h, dev_malloc(&h->bigmv, sizeof(uint2) * (need + need / 2)));
      h->bigmv_cap = need + need / 2;
    }
  }
  if (!h->ev_fork) {  // (created last: a failure part-way is completed by the next call)
    // the largest degrees make the longest chains of a sub-step: their
    // stream gets the highest priority, the block-per-vertex bin the next
    int least = 0, greatest = 0;
    DFL_CUDA(h, cudaDeviceGetStreamPriorityRange(&least, &greatest));
    for (int b = 0; b < kBins - 1; ++b) {
      int prio = b == kBins - 2 ? greatest : b == kBins - 3 ? (greatest < least ? greatest + 1 : least) : least;
      if (!h->aux[b]) DFL_CUDA(h, cudaStreamCreateWithPriority(&h->aux[b], cudaStreamNonBlocking, prio));
      if (!h->ev_join[b]) DFL_CUDA(h, cudaEventCreateWithFlags(&h->ev_join[b], cudaEventDisableTiming));
    }
    DFL_CUDA(h, cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
  }
  {
    LaunchScope ls(h, DFL_PROF_OTHER);
    launch_pdl(k_set_m2, 1, 1, 0, h->stream, h->ctrl, ma.m2,
               h->papply.active ? h->actrl + h->papply.par : nullptr, ma.from_singletons ? 1u : 0u);
    DFL_TRY(check_launch(h, "set m2"));
  }
  DecideArgs& a = *out;
  std::memset(&a, 0, sizeof(a));
  a.g = ma.g;
  a.C = ma.C;
  a.K = ma.K;
  a.Sigma = ma.Sigma;
  a.size = ma.size;
  a.m2p = &h->ctrl->m2v;
  a.seg = h->segs;
  a.rbits = ma.use_range ? h->rbits : nullptr;
  a.ever = ma.track_ever ? h->ever : nullptr;
  a.mv_i = h->mv_i;
  a.mv_c = h->mv_c;
  a.mv_d = h->mv_d;
  a.ctrl = h->ctrl;
  a.k = k;
  a.gtable = need_gtable ? h->gtable : nullptr;
  a.gslots = gslots;
  a.bigmv = h->bigmv;
  a.movers = &h->ctrl->it_movers[0];
  a.nbig = &h->ctrl->it_nbig[0];
  if (h->ngraphs) {
    a.ngraphs = h->ngraphs;
    a.goff = h->d_goff;
    a.gm2 = h->d_gm2;
    a.gdone = h->d_gdone;
    a.gS = h->d_gS;
  }
  *gdo = GiantDecide{h->g_toff, h->g_loff, h->g_cpre, h->g_ndist, h->g_done, h->g_hd,
                     static_cast<GiantRes*>(h->g_res), h->g_tkeys, h->g_tvals, h->g_tlist, nullptr,
                     nullptr};
  return DFL_OK;
}

}  // namespace

int local_move(Handle* h, const MoveArgs& ma, uint32_t pass, uint32_t* iterations,
               bool record_trace, uint64_t* initial, uint64_t* ever) {
  const uint32_t G = h->ngraphs;
  u128 threshold = tolerance_threshold(h->opt, ma.m2, pass);
  MoveArgs mv = ma;
  bool settled = false;  // a pending batch apply settled by a control read (2m changed)
  // a group tests each graph against its own threshold; graphs that have
  // finished (h->gfin) or converge stop being processed
  std::vector<u128> gthr(G);
  std::vector<uint8_t> gactive(G);
  uint32_t nactive = 0;
  for (uint32_t g = 0; g < G; ++g) {
    gthr[g] = tolerance_threshold(h->opt, h->gm2[g], pass);
    gactive[g] = !h->gfin[g];
    nactive += gactive[g];
    h->h_gdone[g] = !gactive[g];
    if (ma.graph_iters) ma.graph_iters[g] = 0;
  }
  if (G) DFL_TRY(group_upload_flags(h, h->d_gdone, h->h_gdone));
  // the persistent kernel when asked for; else graph replay, which needs
  // stable buffers (the base graph) and a capturable (non-default) stream,
  // unless forbidden, or unless the caller prefers host launches (a small
  // update, a group) and replay was not asked for explicitly; else host
  // launches
  const uint32_t pgrid = (h->opt.flags & DFL_FLAG_PERSISTENT) ? persistent_grid() : 0u;
  const bool use_persistent = pgrid >= kMaxSubsteps;
  const uint32_t fl = h->opt.flags;
  const bool want_graph = !(fl & DFL_FLAG_NO_GRAPH) && ((fl & DFL_FLAG_GRAPH) || !ma.prefer_host);
  const bool use_graph = !use_persistent && want_graph && ma.g.off == h->off && h->stream != nullptr;
  // small frontiers: one launch for whole iterations, unless the launch form or
  // the phases' times were asked for
  bool can_small = !use_persistent && ma.g.nv && small_available() &&
                   !(fl & (DFL_FLAG_SERIAL_BINS | DFL_FLAG_PROFILE | DFL_FLAG_PROFILE_MOVE)) &&
                   !((fl & DFL_FLAG_GRAPH) && use_graph);
  unsigned int cur_count[kMaxSubsteps][kBins];
  unsigned long long skipped = 0;
  // a frontier that can only be small needs no read of its lengths first
  bool small_next = can_small && !use_graph && !ma.counted && ma.frontier_hint <= kSmallTry;
  if (!use_graph && !use_persistent && !small_next) {
    if (!ma.counted) DFL_TRY(read_move_ctrl(h, &settled));  // list lengths of the initial frontier (buffer 0)
    if (settled && !G) {
      threshold = tolerance_threshold(h->opt, h->m2, pass);
      mv.m2 = h->m2;  // the batch's 2m, for the decide kernels
    }
    if (h->hctrl->err) return set_error(h, DFL_ERR_CUDA, "internal error in frontier marking");
    for (uint32_t s = 0; s < kMaxSubsteps; ++s)
      for (int b = 0; b < kBins; ++b) cur_count[s][b] = h->hctrl->count[0][s][b];
    skipped = h->hctrl->skipped;
    small_next = can_small && small_frontier(cur_count);
  }
  DecideArgs a;
  GiantDecide gd;
  DFL_TRY(prepare_move(h, mv, &a, &gd));
  int cur = 0;
  uint32_t it = 0;
  uint64_t hint = ma.frontier_hint;  // upper bound of this iteration's frontier
  Handle::IterGraph* graph_used[2] = {nullptr, nullptr};
  // the graphs that meet their own tolerance after iteration `it` stop being processed
  auto group_converged = [&]() -> int {
    bool changed = false;
    for (uint32_t g = 0; g < G; ++g) {
      if (!gactive[g]) continue;
      if (ma.graph_iters) ma.graph_iters[g] = it;
      const u128 Sg = ((u128)h->h_gS[2 * g + 1] << 32) + (u128)h->h_gS[2 * g];
      if (Sg <= gthr[g]) {  // this graph converged: skip its vertices from now on
        gactive[g] = 0;
        h->h_gdone[g] = 1;
        --nactive;
        changed = true;
      }
    }
    if (changed && nactive) DFL_TRY(group_upload_flags(h, h->d_gdone, h->h_gdone));
    return DFL_OK;
  };
  auto take_counts = [&](int buf) {
    hint = 0;
    for (uint32_t s = 0; s < kMaxSubsteps; ++s)
      for (int b = 0; b < kBins; ++b) hint += cur_count[s][b] = h->hctrl->count[buf][s][b];
    small_next = can_small && small_frontier(cur_count);
  };
  while (it < h->opt.max_iterations && (!G || nactive)) {
    if (small_next) {
      DFL_TRY(issue_small(h, a, cur, pass, h->opt.max_iterations - it));
      if (G)
        DFL_CUDA(h, cudaMemcpyAsync(h->h_gS, h->d_gS, sizeof(unsigned long long) * 2 * G,
                                    cudaMemcpyDeviceToHost, h->stream));
      DFL_TRY(read_move_ctrl(h, &settled));
      if (settled && !G) threshold = tolerance_threshold(h->opt, h->m2, pass);
      const Ctrl& c = *h->hctrl;
      if (c.err) return set_error(h, DFL_ERR_CUDA, "internal error in local-moving (table overflow)");
      if (it == 0) {
        skipped = c.skipped;
        if (initial && c.sm_iters) *initial = skipped + c.sm_first;
      }
      for (uint32_t r = 0; r < c.sm_iters && record_trace; ++r)
        for (int q = 0; q < 4; ++q) h->trace.push_back(c.sm_trace[r][q] + (q == 0 && r == 0 ? skipped : 0));
      if (c.sm_iters) skipped = 0;
      it += c.sm_iters;
      cur ^= int(c.sm_iters & 1);
      const bool ran = c.sm_iters != 0, done = c.sm_done != 0;
      take_counts(cur);
      if (!ran) {  // it refused the frontier (above small_cost's limit, or a vertex too large)
        if (small_next) can_small = false;
        small_next = false;
      } else if (G) {
        DFL_TRY(group_converged());
      } else if (done) {
        break;
      }
      continue;
    }
    ++it;
    const int nxt = cur ^ 1;
    if (use_graph) {
      Handle::IterGraph* gp = nullptr;
      DFL_TRY(ensure_iteration_graph(h, a, gd, cur, hint / h->opt.substeps < kSmallList, &gp));
      const Handle::IterGraph& g = *gp;
      graph_used[cur] = gp;
      DFL_CUDA(h, cudaGraphLaunch(g.exec, h->stream));
      h->launches += g.kernels;
      for (int q = 0; q < DFL_PROF_CLASSES; ++q) h->prof.launches[q] += g.class_launches[q];
    } else if (use_persistent) {
      DFL_TRY(issue_persistent(h, a, cur, gd, pgrid));
    } else {
      DFL_TRY(issue_iteration(h, a, cur, cur_count, gd));
    }
    if (G)
      DFL_CUDA(h, cudaMemcpyAsync(h->h_gS, h->d_gS, sizeof(unsigned long long) * 2 * G,
                                  cudaMemcpyDeviceToHost, h->stream));
    DFL_TRY(read_move_ctrl(h, &settled));
    if (settled && !G) threshold = tolerance_threshold(h->opt, h->m2, pass);
    const Ctrl& c = *h->hctrl;
    if (c.err & kErrTimeout) return set_error(h, DFL_ERR_TIMEOUT, "grid barrier of the iteration kernel gave up");
    if (c.err) return set_error(h, DFL_ERR_CUDA, "internal error in local-moving (table overflow)");
    if (use_persistent) {
      if (it == 1) {
        skipped = c.skipped;
        if (initial) {
          *initial = skipped;
          for (uint32_t s = 0; s < kMaxSubsteps; ++s)
            for (int b = 0; b < kBins; ++b) *initial += c.count[0][s][b];
        }
      }
    } else if (use_graph) {
      for (const auto& ev : graph_used[cur]->evs) {  // harvest this replay's timings
        float ms = 0;
        if (cudaEventElapsedTime(&ms, ev.a, ev.b) == cudaSuccess) h->prof.ms[ev.cls] += ms;
      }
      if (it == 1) {
        skipped = c.skipped;
        if (initial) {
          *initial = skipped;
          for (uint32_t s = 0; s < kMaxSubsteps; ++s)
            for (int b = 0; b < kBins; ++b) *initial += c.count[0][s][b];
        }
      }
    } else if (it == 1 && initial) {
      *initial = skipped;
      for (uint32_t s = 0; s < kMaxSubsteps; ++s)
        for (int b = 0; b < kBins; ++b) *initial += cur_count[s][b];
    }
    u128 S = ((u128)c.s_hi << 32) + (u128)c.s_lo;
    if (record_trace) {
      h->trace.push_back(c.processed + skipped);
      h->trace.push_back(c.moved);
      h->trace.push_back(uint64_t(S >> 64));
      h->trace.push_back(uint64_t(S));
    }
    cur = nxt;
    take_counts(cur);
    skipped = 0;
    if (!G) {
      if (S <= threshold) break;  // locally converged
      continue;
    }
    DFL_TRY(group_converged());
  }
  h->prof.bytes[DFL_PROF_MOVE] += h->hctrl->move_bytes;
  if (ever) *ever = h->hctrl->ever_count;
  // leave the unprocessed frontier behind: clear the other buffer's bitmap
  DFL_CUDA(h, cudaMemsetAsync(h->fbits[cur], 0, sizeof(uint32_t) * h->words, h->stream));
  *iterations = it;
  return DFL_OK;
}

// Decide phase of one local-moving iteration over the frontier in list
// buffer 0, without applying the moves: `reps` timed runs (the autotuner).
int time_decide(Handle* h, const MoveArgs& ma, uint32_t reps, std::vector<float>* ms) {
  DFL_TRY(read_ctrl(h));
  unsigned int counts[kMaxSubsteps][kBins];
  for (uint32_t s = 0; s < kMaxSubsteps; ++s)
    for (int b = 0; b < kBins; ++b) counts[s][b] = h->hctrl->count[0][s][b];
  if (h->ngraphs) {
    for (uint32_t g = 0; g < h->ngraphs; ++g) h->h_gdone[g] = 0;
    DFL_TRY(group_upload_flags(h, h->d_gdone, h->h_gdone));
  }
  DecideArgs a;
  GiantDecide gd;
  DFL_TRY(prepare_move(h, ma, &a, &gd));
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  DFL_CUDA(h, cudaEventCreate(&e0));
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return set_error(h, DFL_ERR_CUDA, "event");
  }
  int rc = DFL_OK;
  ms->clear();
  for (uint32_t r = 0; r < reps && !rc; ++r) {
    if (cudaMemsetAsync(h->fbits[1], 0, sizeof(uint32_t) * h->words, h->stream) != cudaSuccess)
      rc = set_error(h, DFL_ERR_CUDA, "memset");
    if (!rc) rc = cudaEventRecord(e0, h->stream) == cudaSuccess ? DFL_OK : DFL_ERR_CUDA;
    if (!rc) rc = issue_iteration(h, a, 0, counts, gd, true);
    if (!rc) rc = cudaEventRecord(e1, h->stream) == cudaSuccess ? DFL_OK : DFL_ERR_CUDA;
    if (!rc) rc = read_ctrl(h);
    if (!rc && h->hctrl->err) rc = set_error(h, DFL_ERR_CUDA, "internal error in local-moving");
    float t = 0;
    if (!rc && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) ms->push_back(t);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return rc;
}

}  // namespace dfl
