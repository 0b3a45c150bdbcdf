// Aggregation phase (Alg. 6): collapse each community of G' into one
// super-vertex of G''.
//   1. community vertex counts and total degrees (one pass over vertices),
//   2. exclusive scans: community-vertex CSR offsets, and super-vertex row
//      offsets from the total degree (an over-estimate, so rows have holes),
//   3. community-vertex CSR fill,
//   4. per community, a hash merge of its members' arcs keyed by the
//      neighbour's community, self-loops included (scanCommunities with
//      self = true); distinct keys are written as the super-vertex's row, and
//      its weight K'' = Sigma'' is the row sum (Alg. 4, weight reset).
// Communities are binned by total degree: one warp with a shared-memory
// table (<= 256), one block with a shared-memory table (<= 1024 and <= 4096); a
// larger community is split into chunks of members, each chunk aggregated by
// one block in shared memory and merged into the community's global table,
// which is then emitted slot-parallel.  Every arc goes straight into a table
// with a shared-memory (or, for a giant community's overflow, global) atomic.
//
// Latency bounds these kernels (member -> row -> arcs -> communities), and most
// members have a few arcs, so a tile of members is flattened first: a prefix
// sum over their degrees numbers the tile's arcs, which the lanes then take in
// order, four in flight each.  A warp per member row, one member after another,
// took 1.95 ms (block bin) and 1.79 ms (warp bin, which also took a warp per
// isolated vertex) for the two levels of the 2^22-vertex R-MAT graph's static
// run; this 0.61 and 0.57 ms.
#include <mutex>
#include <vector>

#include "common.cuh"

namespace dfl {

namespace {

// Lanes of the warp with this lane's community: its first lane, this lane's
// rank among them and their number.  Every lane calls it (kEmpty: none).
struct Peers {
  unsigned mask;
  bool first;
  uint32_t rank;
  __device__ __forceinline__ explicit Peers(uint32_t c) {
    mask = __match_any_sync(0xFFFFFFFFu, c);
    rank = __popc(mask & ((1u << (threadIdx.x & 31u)) - 1u));
    first = rank == 0;
  }
};

// (one update per warp and community: a giant community's counters are the
// contended ones)
__global__ void k_agg_count(GraphView g, const uint32_t* __restrict__ Cp, uint32_t* __restrict__ cnt,
                            unsigned long long* __restrict__ tdeg) {
  const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
  for (uint64_t v0 = blockIdx.x * uint64_t(blockDim.x); v0 < g.nv; v0 += stride) {
    const uint64_t v = v0 + threadIdx.x;
    const uint32_t c = v < g.nv ? Cp[v] : kEmpty;
    const uint32_t d = v < g.nv ? g.deg[v] : 0u;
    const Peers p(c);
    unsigned long long sum = d;
    if (p.mask & (p.mask - 1)) {  // (a lane alone needs no sum; the sums of 16-bit halves cannot wrap)
      const uint32_t lo = __reduce_add_sync(p.mask, d & 0xFFFFu), hi = __reduce_add_sync(p.mask, d >> 16);
      sum = ((unsigned long long)hi << 16) + lo;
    }
    if (c == kEmpty || !p.first) continue;
    atomicAdd(&cnt[c], uint32_t(__popc(p.mask)));
    if (sum) atomicAdd(&tdeg[c], sum);
  }
}

// Bins of communities by total degree.
enum : int { kAggByWarp = 0, kAggByBlock = 1, kAggByBigBlock = 2, kAggGiant = 3, kAggBins = 4 };
constexpr uint32_t kAggBlockDeg = 1024;

// Round every community's total degree up to an even count (rows then start
// 16-byte aligned) and bin the community; one without arcs (an isolated
// vertex) is a finished empty row.
__global__ void __launch_bounds__(256) k_agg_bins(uint32_t ncomm, unsigned long long* __restrict__ tdeg,
                                                  uint32_t* lists, uint64_t lstride, uint32_t* __restrict__ deg_out,
                                                  long long* __restrict__ Knew, Ctrl* ctrl) {
  __shared__ uint32_t s_cnt[kAggBins], s_base[kAggBins];
  constexpr uint32_t U = 4;
  const uint64_t stride = uint64_t(gridDim.x) * blockDim.x * U;
  for (uint64_t c0 = blockIdx.x * uint64_t(blockDim.x) * U; c0 < ncomm; c0 += stride) {
    uint32_t key[U], rank[U];
    if (threadIdx.x < kAggBins) s_cnt[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const uint64_t c = c0 + u * blockDim.x + threadIdx.x;
      key[u] = kAggBins;
      if (c < ncomm) {
        const unsigned long long t = tdeg[c];
        if (t == 0) {
          deg_out[c] = 0;
          Knew[c] = 0;
        } else {
          if (t & 1ull) tdeg[c] = t + 1;
          key[u] = t <= kBinWarpHash ? kAggByWarp : t <= kAggBlockDeg ? kAggByBlock : t <= kBinBlock ? kAggByBigBlock : kAggGiant;
        }
      }
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const Peers p(key[u]);
      rank[u] = 0;
      if (key[u] < kAggBins && p.first) rank[u] = atomicAdd(&s_cnt[key[u]], uint32_t(__popc(p.mask)));
      rank[u] = __shfl_sync(0xFFFFFFFFu, rank[u], __ffs(p.mask) - 1) + p.rank;
    }
    __syncthreads();
    if (threadIdx.x < kAggBins) {
      const uint32_t n = s_cnt[threadIdx.x];
      s_base[threadIdx.x] = n ? atomicAdd(&ctrl->count[1][0][threadIdx.x], n) : 0u;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t u = 0; u < U; ++u)
      if (key[u] < kAggBins) lists[key[u] * lstride + s_base[key[u]] + rank[u]] = uint32_t(c0 + u * blockDim.x + threadIdx.x);
    __syncthreads();
  }
}

__global__ void k_agg_fill(uint32_t nv, const uint32_t* __restrict__ Cp, const uint32_t* __restrict__ coff,
                           uint32_t* __restrict__ fillc, uint32_t* __restrict__ members) {
  const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
  for (uint64_t v0 = blockIdx.x * uint64_t(blockDim.x); v0 < nv; v0 += stride) {
    const uint64_t v = v0 + threadIdx.x;
    const uint32_t c = v < nv ? Cp[v] : kEmpty;
    const Peers p(c);
    uint32_t at = 0;
    if (c != kEmpty && p.first) at = coff[c] + atomicAdd(&fillc[c], uint32_t(__popc(p.mask)));
    at = __shfl_sync(0xFFFFFFFFu, at, __ffs(p.mask) - 1) + p.rank;
    if (c != kEmpty) members[at] = uint32_t(v);
  }
}

struct AggArgs {
  GraphView g;
  const uint32_t* Cp;
  const uint32_t* coff;
  const uint32_t* members;
  const unsigned long long* soff;
  uint32_t* deg_out;
  uint2* arcs_out;
  long long* Knew;
  const uint32_t* list;
  const unsigned int* count;
  Ctrl* ctrl;
};

// Open-addressing insert: 0 if no slot was found within `limit` probes, 2 if
// it created its slot, else 1.
__device__ __forceinline__ int agg_insert(uint32_t* keys, uint32_t* vals, uint32_t mask, uint32_t c, uint32_t w,
                                          uint32_t limit) {
  uint32_t s = hash32(c) & mask;
  for (uint32_t probe = 0; probe < limit; ++probe) {
    uint32_t prev = keys[s];
    if (prev == kEmpty) prev = atomicCAS(&keys[s], kEmpty, c);
    if (prev == kEmpty || prev == c) {
      atomicAdd(&vals[s], w);
      return prev == kEmpty ? 2 : 1;
    }
    s = (s + 1) & mask;
  }
  return 0;
}

__device__ __forceinline__ bool agg_add(uint32_t* keys, uint32_t* vals, uint32_t mask, uint32_t c, uint32_t w,
                                        uint32_t limit) {
  return agg_insert(keys, vals, mask, c, w, limit) != 0;
}

constexpr uint32_t kAggWarpSlots = 512;
constexpr int kAggWarps = 8;
constexpr int kAggThreads = 256;
constexpr uint32_t kChunkMembers = kAggThreads;     // members per block of a giant community
constexpr uint32_t kAggBigMember = 128;             // larger member rows go to k_agg_big ...
constexpr uint32_t kAggUnit = 64;                   // ... which deals their arcs in units of this many
constexpr uint32_t kGiantSlots = 4096;              // shared table of a giant-community block
constexpr uint32_t kGiantTile = 1024;               // global tables are multiples of this many slots

// Arc `k` of a flattened tile of `rows` rows (a power of two): the row's
// position by a binary search of the exclusive prefix `pre`, whose entry j is
// the first arc of row j; base[j] + k is then the arc's index.
template <int kRows>
__device__ __forceinline__ uint32_t flat_row(const uint32_t* pre, uint32_t k) {
  uint32_t j = 0;
#pragma unroll
  for (uint32_t s = kRows / 2; s; s >>= 1)
    if (pre[j + s] <= k) j += s;
  return j;
}

// A tile of up to kAggThreads rows, one per thread: d arcs from index o on.
// Returns the tile's number of arcs.  Every thread of the block calls it; the
// tile is rewritten by the next call, which a block barrier must separate.
struct FlatTile {
  unsigned long long base[kAggThreads];
  uint32_t pre[kAggThreads];
  uint32_t w[kAggThreads / 32];
  __device__ __forceinline__ unsigned long long arc(uint32_t k) const { return base[flat_row<kAggThreads>(pre, k)] + k; }
};
__device__ __forceinline__ uint32_t flat_rows(FlatTile& ft, unsigned long long o, uint32_t d) {
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  uint32_t x = d;
#pragma unroll
  for (int q = 1; q < 32; q <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, q);
    if (lane >= uint32_t(q)) x += y;
  }
  if (lane == 31) ft.w[wib] = x;
  __syncthreads();
  uint32_t before = 0, total = 0;
#pragma unroll
  for (uint32_t q = 0; q < kAggThreads / 32; ++q) {
    if (q == wib) before = total;
    total += ft.w[q];
  }
  ft.pre[threadIdx.x] = before + x - d;
  ft.base[threadIdx.x] = o - (before + x - d);
  __syncthreads();
  return total;
}

// This thread's member of [m0, m1): its row.
__device__ __forceinline__ uint32_t member_row(const AggArgs& a, uint32_t m0, uint32_t m1, unsigned long long* o,
                                               uint32_t* d) {
  const uint32_t m = m0 + threadIdx.x;
  const uint32_t v = m < m1 ? a.members[m] : 0u;
  *o = m < m1 ? a.g.off[v] : 0ull;
  *d = m < m1 ? a.g.deg[v] : 0u;
  return v;
}

// This thread's arcs k0, k0 + kAggThreads, ... (four of them, below total) and
// their neighbours' communities, all loads in flight; kEmpty where there is none.
__device__ __forceinline__ void load_arcs(const AggArgs& a, const FlatTile& ft, uint32_t k0, uint32_t total,
                                          uint32_t (&c)[4], uint32_t (&w)[4]) {
  uint2 e[4];
#pragma unroll
  for (uint32_t u = 0; u < 4; ++u) {
    const uint32_t k = k0 + u * kAggThreads;
    e[u] = k < total ? a.g.arcs[ft.arc(k)] : make_uint2(0u, 0u);
  }
#pragma unroll
  for (uint32_t u = 0; u < 4; ++u) {
    c[u] = e[u].y ? a.Cp[e[u].x] : kEmpty;  // deleted arcs (weight 0) skipped
    w[u] = e[u].y;
  }
}

// Write the table's entries as the row of super-vertex c (ballot order).
__device__ __forceinline__ void emit_warp(const AggArgs& a, uint32_t c, const uint32_t* keys,
                                          const uint32_t* vals, uint32_t slots, uint32_t* maxd) {
  const uint32_t lane = threadIdx.x & 31u;
  const unsigned long long base = a.soff[c];
  uint32_t pos = 0;
  unsigned long long ksum = 0;
  for (uint32_t s0 = 0; s0 < slots; s0 += 32) {
    uint32_t s = s0 + lane;
    uint32_t key = s < slots ? keys[s] : kEmpty;
    bool has = key != kEmpty;
    unsigned m = __ballot_sync(0xFFFFFFFFu, has);
    if (has) {
      uint32_t val = vals[s];
      a.arcs_out[base + pos + __popc(m & ((1u << lane) - 1u))] = make_uint2(key, val);
      ksum += val;
    }
    pos += __popc(m);
  }
  for (int x = 16; x; x >>= 1) ksum += __shfl_xor_sync(0xFFFFFFFFu, ksum, x);
  if (lane == 0) {
    a.deg_out[c] = pos;
    a.Knew[c] = (long long)ksum;
  }
  *maxd = max(*maxd, pos);
}

// Bin 0: one warp per community (total degree <= 256).
__global__ void __launch_bounds__(256) k_agg_warp(AggArgs a) {
  __shared__ uint32_t skeys[kAggWarps][kAggWarpSlots];
  __shared__ uint32_t svals[kAggWarps][kAggWarpSlots];
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  uint32_t* keys = skeys[wib];
  uint32_t* vals = svals[wib];
  const uint32_t cnt = *a.count;
  uint64_t warp = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) >> 5;
  uint64_t nwarps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
  uint32_t maxd = 0;
  for (uint64_t t = warp; t < cnt; t += nwarps) {
    const uint32_t c = a.list[t];
    const unsigned long long td = a.soff[c + 1] - a.soff[c];
    uint32_t slots = 32;
    while (slots < 2 * td && slots < kAggWarpSlots) slots <<= 1;
    for (uint32_t s = lane; s < slots; s += 32) {
      keys[s] = kEmpty;
      vals[s] = 0;
    }
    __syncwarp();
    bool ok = true;
    const uint32_t mend = a.coff[c + 1];
    for (uint32_t m0 = a.coff[c]; m0 < mend; m0 += 32) {  // tiles of 32 members, flattened
      uint32_t d = 0;
      unsigned long long o = 0;
      if (m0 + lane < mend) {
        const uint32_t v = a.members[m0 + lane];
        o = a.g.off[v];
        d = a.g.deg[v];
      }
      uint32_t x = d;
#pragma unroll
      for (int q = 1; q < 32; q <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, q);
        if (lane >= uint32_t(q)) x += y;
      }
      const uint32_t total = __shfl_sync(0xFFFFFFFFu, x, 31);
      const uint32_t pre = x - d;
      o -= pre;
      constexpr uint32_t U = 4;
      for (uint32_t k0 = 0; k0 < total; k0 += 32 * U) {
        uint2 e[U];
        uint32_t nc[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
          const uint32_t k = k0 + u * 32 + lane;
          uint32_t j = 0;  // the last row whose first arc is at or before k
#pragma unroll
          for (uint32_t s = 16; s; s >>= 1)
            if (__shfl_sync(0xFFFFFFFFu, pre, j + s) <= k) j += s;
          const unsigned long long ob = __shfl_sync(0xFFFFFFFFu, o, j);
          e[u] = k < total ? a.g.arcs[ob + k] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) nc[u] = e[u].y ? a.Cp[e[u].x] : kEmpty;
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
          if (nc[u] != kEmpty) ok &= agg_add(keys, vals, slots - 1, nc[u], e[u].y, slots);
      }
    }
    if (!__all_sync(0xFFFFFFFFu, ok) && lane == 0) atomicOr(&a.ctrl->err, kErrInternal);
    __syncwarp();
    emit_warp(a, c, keys, vals, slots, &maxd);
    __syncwarp();
  }
  if (lane == 0 && maxd) atomicMax(&a.ctrl->max_deg, maxd);
}

// Bins 1 and 2: one block per community, its table of kSlots keys + values in
// dynamic shared memory (kSlots >= 2 x total degree).
template <uint32_t kSlots>
__global__ void __launch_bounds__(kAggThreads) k_agg_block(AggArgs a) {
  extern __shared__ __align__(16) uint32_t dyn[];
  __shared__ FlatTile ft;
  __shared__ unsigned int s_pos;
  __shared__ unsigned long long s_sum;
  __shared__ int s_ok;
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  const uint32_t cnt = *a.count;
  unsigned int maxd = 0;
  for (uint64_t t = blockIdx.x; t < cnt; t += gridDim.x) {
    const uint32_t c = a.list[t];
    const unsigned long long td = a.soff[c + 1] - a.soff[c];
    uint32_t slots = 512;
    while (slots < 2 * td && slots < kSlots) slots <<= 1;
    uint32_t* keys = dyn;
    uint32_t* vals = dyn + slots;
    for (uint32_t s = threadIdx.x; s < slots; s += blockDim.x) {
      keys[s] = kEmpty;
      vals[s] = 0;
    }
    if (threadIdx.x == 0) {
      s_pos = 0;
      s_sum = 0;
      s_ok = 1;
    }
    __syncthreads();
    bool ok = true;
    const uint32_t mend = a.coff[c + 1];
    for (uint32_t m0 = a.coff[c]; m0 < mend; m0 += kAggThreads) {
      unsigned long long o;
      uint32_t d;
      member_row(a, m0, mend, &o, &d);
      const uint32_t total = flat_rows(ft, o, d);
      for (uint32_t k0 = threadIdx.x; k0 < total; k0 += 4 * kAggThreads) {
        uint32_t nc[4], w[4];
        load_arcs(a, ft, k0, total, nc, w);
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
          if (nc[u] != kEmpty) ok &= agg_add(keys, vals, slots - 1, nc[u], w[u], slots);
      }
      __syncthreads();  // the tile is rewritten
    }
    if (!ok) s_ok = 0;
    __syncthreads();
    if (!s_ok && threadIdx.x == 0) atomicOr(&a.ctrl->err, kErrInternal);
    const unsigned long long base = a.soff[c];
    unsigned long long ksum = 0;
    for (uint32_t s0 = wib * 32; s0 < slots; s0 += blockDim.x) {
      uint32_t s = s0 + lane;
      uint32_t key = s < slots ? keys[s] : kEmpty;
      bool has = key != kEmpty;
      unsigned m = __ballot_sync(0xFFFFFFFFu, has);
      uint32_t wbase = 0;
      if (lane == 0 && m) wbase = atomicAdd(&s_pos, __popc(m));
      wbase = __shfl_sync(0xFFFFFFFFu, wbase, 0);
      if (has) {
        uint32_t val = vals[s];
        a.arcs_out[base + wbase + __popc(m & ((1u << lane) - 1u))] = make_uint2(key, val);
        ksum += val;
      }
    }
    for (int x = 16; x; x >>= 1) ksum += __shfl_xor_sync(0xFFFFFFFFu, ksum, x);
    if (lane == 0 && ksum) atomicAdd(&s_sum, ksum);
    __syncthreads();
    if (threadIdx.x == 0) {
      a.deg_out[c] = s_pos;
      a.Knew[c] = (long long)s_sum;
      maxd = max(maxd, s_pos);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && maxd) atomicMax(&a.ctrl->max_deg, maxd);
}

// Giant communities (the last bin).  giant[g] = community, gtab[g] = offset of
// its global table of gsize[g] slots in the key and value arrays.
struct GiantArgs {
  const uint32_t* giant;
  unsigned long long* gtab;
  uint32_t* gsize;
  uint32_t* chunk0;        // first work item of each giant (exclusive scan of chunk counts)
  uint32_t ngiant;
  uint32_t nitems;         // total (giant, chunk) work items
  uint32_t* keys;          // empty before the first kernel
  uint32_t* vals;          // zero
  uint32_t* units;         // per (work item, thread): units of a high-degree member; then their exclusive scan
};

// Giant owning work item `item`.
__device__ __forceinline__ uint32_t giant_of(const GiantArgs& gi, uint32_t item) {
  uint32_t lo = 0, hi = gi.ngiant;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (gi.chunk0[mid] <= item) lo = mid;
    else hi = mid;
  }
  return lo;
}

// One block: the giants' tables and chunks laid out (a table holds twice the
// distinct communities a row can have: at most its arcs, and at most the
// communities that have arcs), their totals into red_a and red_b and the super
// graph's row slots into red_c, so that the host reads one control block.
__global__ void __launch_bounds__(1024) k_giant_layout(uint32_t ncomm, const unsigned long long* __restrict__ soff,
                                                       const uint32_t* __restrict__ coff, GiantArgs gi,
                                                       uint32_t* __restrict__ deg_out, long long* __restrict__ Knew,
                                                       Ctrl* ctrl) {
  __shared__ unsigned long long s_t[32], s_tbase;
  __shared__ uint32_t s_c[32], s_cbase;
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  const uint32_t ng = ctrl->count[1][0][kAggGiant];
  unsigned long long live = 0;
  for (int b = 0; b < kAggBins; ++b) live += ctrl->count[1][0][b];
  if (threadIdx.x == 0) {
    s_tbase = 0;
    s_cbase = 0;
  }
  __syncthreads();
  for (uint32_t t0 = 0; t0 < ng; t0 += blockDim.x) {
    const uint32_t t = t0 + threadIdx.x;
    unsigned long long size = 0;
    uint32_t chunks = 0;
    if (t < ng) {
      const uint32_t c = gi.giant[t];
      const unsigned long long td = soff[c + 1] - soff[c], distinct = td < live ? td : live;
      size = kGiantTile;
      while (size < 2 * distinct) size <<= 1;
      chunks = (coff[c + 1] - coff[c] + kChunkMembers - 1) / kChunkMembers;
      deg_out[c] = 0;
      Knew[c] = 0;
    }
    unsigned long long xt = size;
    uint32_t xc = chunks;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long yt = __shfl_up_sync(0xFFFFFFFFu, xt, o);
      const uint32_t yc = __shfl_up_sync(0xFFFFFFFFu, xc, o);
      if (lane >= uint32_t(o)) {
        xt += yt;
        xc += yc;
      }
    }
    if (lane == 31) {
      s_t[w] = xt;
      s_c[w] = xc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (uint32_t k = 0; k < blockDim.x / 32; ++k) {
        const unsigned long long tt = s_t[k];
        const uint32_t tc = s_c[k];
        s_t[k] = s_tbase;
        s_c[k] = s_cbase;
        s_tbase += tt;
        s_cbase += tc;
      }
    }
    __syncthreads();
    if (t < ng) {
      gi.gtab[t] = s_t[w] + xt - size;
      gi.gsize[t] = uint32_t(size);
      gi.chunk0[t] = s_c[w] + xc - chunks;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    ctrl->red_a = s_tbase;
    ctrl->red_b = s_cbase;
    ctrl->red_c = soff[ncomm];
  }
}

// Shared table of a giant's block (empty at rest): when a round of arcs could
// overfill it, its entries move to the giant's global table.  Rows of
// converged communities meet few distinct communities, so most chunks flush once.
struct GiantTable {
  uint32_t keys[kGiantSlots], vals[kGiantSlots];
  uint16_t list[kGiantSlots];  // occupied slots, compacted for the flush
  uint32_t claimed, n;
};
// Entries before a round of 4 x kAggThreads arcs: the table stays half empty
// at the worst (long probes cost more than flushes: 1,754 us for both kernels
// on the 2^22-vertex R-MAT graph's two levels, 1,787 with 2,048, 1,822 with
// 512, 2,150 with 3,072 of 8,192 slots; 2,355 for a warp per member row, with
// one merge per 256 members or per 2,048 arcs of a larger one).
constexpr uint32_t kGiantFlush = 1024;

__device__ __forceinline__ void giant_table_init(GiantTable& t) {
  for (uint32_t s = threadIdx.x; s < kGiantSlots; s += kAggThreads) {
    t.keys[s] = kEmpty;
    t.vals[s] = 0;
  }
  if (threadIdx.x == 0) t.claimed = t.n = 0;
  __syncthreads();
}

// Every entry into the global table, four per thread in flight; the shared
// table is empty again.  Returns false if one found no slot.
__device__ __forceinline__ bool giant_flush(GiantTable& t, uint32_t* gkeys, uint32_t* gvals, uint32_t gmask) {
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t s0 = threadIdx.x & ~31u; s0 < kGiantSlots; s0 += kAggThreads) {
    const bool has = t.keys[s0 + lane] != kEmpty;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, has);
    if (!m) continue;
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&t.n, uint32_t(__popc(m)));
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (has) t.list[at + __popc(m & ((1u << lane) - 1u))] = uint16_t(s0 + lane);
  }
  __syncthreads();
  const uint32_t n = t.n;
  bool ok = true;
  for (uint32_t e0 = threadIdx.x; e0 < n; e0 += 4 * kAggThreads) {
    uint32_t c[4], w[4], at[4], prev[4];
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      const uint32_t e = e0 + u * kAggThreads;
      c[u] = kEmpty;
      if (e >= n) continue;
      const uint32_t s = t.list[e];
      c[u] = t.keys[s];
      w[u] = t.vals[s];
      t.keys[s] = kEmpty;
      t.vals[s] = 0;
      at[u] = hash32(c[u]) & gmask;
    }
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) prev[u] = c[u] != kEmpty ? atomicCAS(&gkeys[at[u]], kEmpty, c[u]) : kEmpty;
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      if (c[u] == kEmpty) continue;
      for (uint32_t probe = 0; prev[u] != kEmpty && prev[u] != c[u] && probe < gmask; ++probe) {
        at[u] = (at[u] + 1) & gmask;
        prev[u] = atomicCAS(&gkeys[at[u]], kEmpty, c[u]);
      }
      if (prev[u] == kEmpty || prev[u] == c[u]) atomicAdd(&gvals[at[u]], w[u]);
      else ok = false;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) t.claimed = t.n = 0;
  __syncthreads();
  return ok;
}

// The tile's arcs into the shared table, flushed when a further round could
// overfill it.  Every thread of the block calls it.
__device__ __forceinline__ bool giant_arcs(const AggArgs& a, GiantTable& t, const FlatTile& ft, uint32_t total,
                                           uint32_t* gkeys, uint32_t* gvals, uint32_t gmask) {
  bool ok = true;
  for (uint32_t b = 0; b < total; b += 4 * kAggThreads) {  // block-uniform
    uint32_t c[4], w[4], made = 0;
    load_arcs(a, ft, b + threadIdx.x, total, c, w);
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      if (c[u] == kEmpty) continue;
      const int r = agg_insert(t.keys, t.vals, kGiantSlots - 1, c[u], w[u], kGiantSlots);
      ok &= r != 0;
      made += r == 2 ? 1u : 0u;
    }
    made = __reduce_add_sync(0xFFFFFFFFu, made);
    if ((threadIdx.x & 31u) == 0 && made) atomicAdd(&t.claimed, made);
    __syncthreads();
    if (t.claimed > kGiantFlush) ok &= giant_flush(t, gkeys, gvals, gmask);
    else __syncthreads();  // (everyone has read the count)
  }
  return ok;
}

// Work item (g, chunk): members [chunk*256, +256) of giant g.  A block takes a
// run of items and flushes its table when the giant changes.  The units of
// rows of more than kAggBigMember arcs are noted for k_agg_big.
__global__ void __launch_bounds__(kAggThreads) k_agg_giant_accum(AggArgs a, GiantArgs gi) {
  extern __shared__ __align__(16) uint32_t dyn[];
  GiantTable& t = *reinterpret_cast<GiantTable*>(dyn);
  __shared__ FlatTile ft;
  const uint32_t i0 = uint32_t(uint64_t(gi.nitems) * blockIdx.x / gridDim.x);
  const uint32_t i1 = uint32_t(uint64_t(gi.nitems) * (blockIdx.x + 1) / gridDim.x);
  if (i0 == i1) return;  // block-uniform
  bool ok = true;
  giant_table_init(t);
  uint32_t g = giant_of(gi, i0);
  for (uint32_t item = i0; item < i1; ++item) {
    const uint32_t c = gi.giant[g], gmask = gi.gsize[g] - 1;
    unsigned long long o;
    uint32_t d;
    member_row(a, a.coff[c] + (item - gi.chunk0[g]) * kChunkMembers, a.coff[c + 1], &o, &d);
    const bool big = d > kAggBigMember;
    gi.units[uint64_t(item) * kAggThreads + threadIdx.x] = big ? (d + kAggUnit - 1) / kAggUnit : 0u;
    const uint32_t total = flat_rows(ft, o, big ? 0u : d);
    uint32_t* gkeys = gi.keys + gi.gtab[g];
    uint32_t* gvals = gi.vals + gi.gtab[g];
    ok &= giant_arcs(a, t, ft, total, gkeys, gvals, gmask);
    const bool next = g + 1 < gi.ngiant && gi.chunk0[g + 1] == item + 1;  // the next item is another giant's
    if (next || item + 1 == i1) ok &= giant_flush(t, gkeys, gvals, gmask);
    else __syncthreads();  // the tile is rewritten
    g += next ? 1u : 0u;
  }
  if (!ok) atomicOr(&a.ctrl->err, kErrInternal);
}

// The giant communities' high-degree members: every block takes an equal share
// of their arcs (a run of units, which may begin and end inside a row), work
// item by work item.
__global__ void __launch_bounds__(kAggThreads) k_agg_big(AggArgs a, GiantArgs gi) {
  extern __shared__ __align__(16) uint32_t dyn[];
  GiantTable& t = *reinterpret_cast<GiantTable*>(dyn);
  __shared__ FlatTile ft;
  const uint32_t units = gi.units[uint64_t(gi.nitems) * kAggThreads];
  const uint32_t u0 = uint32_t(uint64_t(units) * blockIdx.x / gridDim.x);
  const uint32_t u1 = uint32_t(uint64_t(units) * (blockIdx.x + 1) / gridDim.x);
  if (u0 == u1) return;  // block-uniform
  bool ok = true, filled = false;
  giant_table_init(t);
  uint32_t lo = 0, hi = gi.nitems;  // the last item whose first unit is at or before u0
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (gi.units[uint64_t(mid) * kAggThreads] <= u0) lo = mid;
    else hi = mid;
  }
  uint32_t g = giant_of(gi, lo);
  for (uint32_t item = lo; item < gi.nitems; ++item) {
    const uint32_t* un = gi.units + uint64_t(item) * kAggThreads;
    const uint32_t first = un[0], end = un[kAggThreads];
    if (first >= u1) break;  // block-uniform, as the branches below
    uint32_t* gkeys = gi.keys + gi.gtab[g];
    uint32_t* gvals = gi.vals + gi.gtab[g];
    const uint32_t gmask = gi.gsize[g] - 1;
    if (end > first && end > u0) {
      // this thread's row, if it is a high-degree one with arcs in the share
      const uint32_t ue = un[threadIdx.x], ux = un[threadIdx.x + 1];
      unsigned long long o = 0;
      uint32_t d = 0;
      if (ux > ue && ux > u0 && ue < u1) {
        const uint32_t c = gi.giant[g];
        const uint32_t v = a.members[a.coff[c] + (item - gi.chunk0[g]) * kChunkMembers + threadIdx.x];
        const uint32_t dv = a.g.deg[v], k0 = ue < u0 ? (u0 - ue) * kAggUnit : 0u;
        const uint64_t k1 = uint64_t(u1 - ue) * kAggUnit;
        o = a.g.off[v] + k0;
        d = (k1 < dv ? uint32_t(k1) : dv) - k0;
      }
      const uint32_t total = flat_rows(ft, o, d);
      ok &= giant_arcs(a, t, ft, total, gkeys, gvals, gmask);
      __syncthreads();  // the tile is rewritten
      filled = true;
    }
    const bool next = g + 1 < gi.ngiant && gi.chunk0[g + 1] == item + 1;  // the next item is another giant's
    if (filled && (next || item + 1 == gi.nitems || end >= u1)) {
      ok &= giant_flush(t, gkeys, gvals, gmask);
      filled = false;
    }
    g += next ? 1u : 0u;
  }
  if (!ok) atomicOr(&a.ctrl->err, kErrInternal);
}

// The giants' tables as super arcs, a block per tile of kGiantTile slots (all
// of one giant): the tile's row positions are claimed with one atomic (one per
// entry took 1,053 us for the two levels above, this 135).
__global__ void __launch_bounds__(kAggThreads) k_agg_giant_emit(AggArgs a, GiantArgs gi, unsigned long long total) {
  pdl_wait_only();
  __shared__ uint32_t s_w[kAggThreads / 32], s_base;
  __shared__ unsigned long long s_k[kAggThreads / 32];
  constexpr uint32_t U = kGiantTile / kAggThreads;
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  uint32_t maxd = 0;
  for (unsigned long long t0 = blockIdx.x * (unsigned long long)kGiantTile; t0 < total;
       t0 += gridDim.x * (unsigned long long)kGiantTile) {
    uint32_t key[U], val[U], n = 0;
    unsigned long long ksum = 0;
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      key[u] = gi.keys[t0 + u * kAggThreads + threadIdx.x];
      val[u] = gi.vals[t0 + u * kAggThreads + threadIdx.x];
      n += key[u] != kEmpty ? 1u : 0u;
      ksum += val[u];  // (0 in an empty slot)
    }
    // giant owning the tile (tables are laid out in giant order)
    uint32_t lo = 0, hi = gi.ngiant;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (gi.gtab[mid] <= t0) lo = mid;
      else hi = mid;
    }
    const uint32_t c = gi.giant[lo];
    uint32_t x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= uint32_t(o)) x += y;
    }
    for (int o = 16; o; o >>= 1) ksum += __shfl_xor_sync(0xFFFFFFFFu, ksum, o);
    if (lane == 31) s_w[wib] = x;
    if (lane == 0) s_k[wib] = ksum;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t run = 0;
      unsigned long long kt = 0;
      for (uint32_t q = 0; q < kAggThreads / 32; ++q) {
        const uint32_t y = s_w[q];
        s_w[q] = run;
        run += y;
        kt += s_k[q];
      }
      if (run) {
        s_base = atomicAdd(&a.deg_out[c], run);
        maxd = max(maxd, s_base + run);
        atomicAdd((unsigned long long*)&a.Knew[c], kt);
      }
    }
    __syncthreads();
    unsigned long long at = a.soff[c] + s_base + s_w[wib] + x - n;
#pragma unroll
    for (uint32_t u = 0; u < U; ++u)
      if (key[u] != kEmpty) a.arcs_out[at++] = make_uint2(key[u], val[u]);
    __syncthreads();  // s_w, s_k and s_base are rewritten by the next tile
  }
  if (threadIdx.x == 0 && maxd) atomicMax(&a.ctrl->max_deg, maxd);
}

int read_ctrl(Handle* h) {
  DFL_CUDA(h, cudaMemcpyAsync(h->hctrl, h->ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, h->stream));
  DFL_CUDA(h, cudaStreamSynchronize(h->stream));
  return DFL_OK;
}

}  // namespace

// Aggregate g under the renumbered membership Cp (labels in [0, ncomm)) into
// super graph sg[dst]; Knew receives the super-vertex weights.  Returns the
// super graph's maximum degree in h->hctrl->max_deg.
int aggregate(Handle* h, const GraphView& g, const uint32_t* Cp, uint32_t ncomm, int dst,
              long long* Knew) {
  SuperGraph& sg = h->sg[dst];
  if (ncomm + 1 > sg.nv_cap) {
    cudaStreamSynchronize(h->stream);
    cudaFree(sg.off);
    cudaFree(sg.deg);
    sg.off = nullptr;
    sg.deg = nullptr;
    sg.nv_cap = 0;
    DFL_CUDA(h, dev_malloc(&sg.off, sizeof(unsigned long long) * (uint64_t(h->n) + 1)));
    DFL_CUDA(h, dev_malloc(&sg.deg, sizeof(uint32_t) * (uint64_t(h->n) + 1)));
    sg.nv_cap = h->n + 1;
  }
  DFL_CUDA(h, cudaMemsetAsync(h->ctrl, 0, sizeof(Ctrl), h->stream));
  DFL_CUDA(h, cudaMemsetAsync(h->cnt, 0, sizeof(uint32_t) * (uint64_t(ncomm) + 1), h->stream));
  DFL_CUDA(h, cudaMemsetAsync(h->fillc, 0, sizeof(uint32_t) * uint64_t(ncomm), h->stream));
  DFL_CUDA(h, cudaMemsetAsync(sg.off, 0, sizeof(unsigned long long) * (uint64_t(ncomm) + 1),
                              h->stream));
  {
    LaunchScope ls(h, DFL_PROF_AGG);
    k_agg_count<<<grid_for(g.nv, 256), 256, 0, h->stream>>>(g, Cp, h->cnt, sg.off);
    DFL_TRY(check_launch(h, "agg count"));
  }
  uint32_t* lists = h->lists[1];  // kAggBins lists of up to n communities
  {
    LaunchScope ls(h, DFL_PROF_AGG);
    k_agg_bins<<<grid_for(ncomm, 1024, 152 * 8), 256, 0, h->stream>>>(ncomm, sg.off, lists, h->n, sg.deg, Knew, h->ctrl);
    DFL_TRY(check_launch(h, "agg bins"));
  }
  DFL_TRY(scan_u32(h, h->cnt, h->cnt, ncomm));
  DFL_TRY(scan_u64(h, sg.off, sg.off, ncomm));
  {
    LaunchScope ls(h, DFL_PROF_AGG);
    k_agg_fill<<<grid_for(g.nv, 256), 256, 0, h->stream>>>(g.nv, Cp, h->cnt, h->fillc, h->members);
    DFL_TRY(check_launch(h, "agg fill"));
  }
  // the giants' layout (in the idle frontier lists), then one control read
  GiantArgs gi;
  gi.giant = lists + uint64_t(kAggGiant) * h->n;
  gi.gtab = reinterpret_cast<unsigned long long*>(h->lists[0]);
  gi.gsize = h->lists[0] + 2ull * h->n;
  gi.chunk0 = gi.gsize + h->n;
  {
    LaunchScope ls(h, DFL_PROF_AGG);
    k_giant_layout<<<1, 1024, 0, h->stream>>>(ncomm, sg.off, h->cnt, gi, sg.deg, Knew, h->ctrl);
    DFL_TRY(check_launch(h, "giant layout"));
  }
  DFL_TRY(read_ctrl(h));
  const Ctrl c = *h->hctrl;
  if (c.err) return set_error(h, DFL_ERR_CUDA, "internal error in aggregation lists");
  if (c.red_c > sg.arc_cap) {
    cudaFree(sg.arcs);
    sg.arcs = nullptr;
    sg.arc_cap = 0;
    uint64_t want = c.red_c + c.red_c / 8 + 1024;
    DFL_CUDA(h, dev_malloc(&sg.arcs, sizeof(uint2) * want));
    sg.arc_cap = want;
  }
  // once per process (handles may be driven from several host threads)
  static std::once_flag smem_once;
  static cudaError_t smem_rc = cudaSuccess;
  std::call_once(smem_once, [] {
    smem_rc = cudaFuncSetAttribute(k_agg_block<2 * kBinBlock>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   int(sizeof(uint32_t) * 4 * kBinBlock));
  });
  DFL_CUDA(h, smem_rc);
  AggArgs a;
  a.g = g;
  a.Cp = Cp;
  a.coff = h->cnt;
  a.members = h->members;
  a.soff = sg.off;
  a.deg_out = sg.deg;
  a.arcs_out = sg.arcs;
  a.Knew = Knew;
  a.ctrl = h->ctrl;
  for (int b = 0; b < kAggGiant; ++b) {
    const uint32_t nc = c.count[1][0][b];
    if (!nc) continue;
    a.list = lists + uint64_t(b) * h->n;
    a.count = &h->ctrl->count[1][0][b];
    LaunchScope ls(h, DFL_PROF_AGG);
    if (b == kAggByWarp)
      k_agg_warp<<<grid_for(uint64_t(nc) * 32, 256, 152 * 16), 256, 0, h->stream>>>(a);
    else if (b == kAggByBlock)
      k_agg_block<2 * kAggBlockDeg><<<grid_for(nc, 1, 152 * 8), kAggThreads, sizeof(uint32_t) * 4 * kAggBlockDeg,
                                      h->stream>>>(a);
    else
      k_agg_block<2 * kBinBlock><<<grid_for(nc, 1, 152 * 3), kAggThreads, sizeof(uint32_t) * 4 * kBinBlock,
                                   h->stream>>>(a);
    DFL_TRY(check_launch(h, "aggregate"));
  }
  gi.ngiant = c.count[1][0][kAggGiant];
  if (gi.ngiant) {
    const uint64_t total = c.red_a;
    gi.nitems = uint32_t(c.red_b);
    if (total > h->gtable_cap) {
      cudaFree(h->gtable);
      h->gtable = nullptr;
      h->gtable_cap = 0;
      DFL_CUDA(h, dev_malloc(&h->gtable, sizeof(uint2) * total));
      h->gtable_cap = total;
    }
    gi.keys = reinterpret_cast<uint32_t*>(h->gtable);
    gi.vals = gi.keys + total;
    const uint64_t entries = uint64_t(gi.nitems) * kAggThreads;
    if (entries + 1 > h->aggq_cap) {
      cudaStreamSynchronize(h->stream);
      cudaFree(h->aggq);
      h->aggq = nullptr;
      h->aggq_cap = 0;
      DFL_CUDA(h, dev_malloc(&h->aggq, sizeof(uint32_t) * (entries + 1)));
      h->aggq_cap = entries + 1;
    }
    gi.units = h->aggq;
    DFL_CUDA(h, cudaMemsetAsync(gi.keys, 0xFF, sizeof(uint32_t) * total, h->stream));
    DFL_CUDA(h, cudaMemsetAsync(gi.vals, 0, sizeof(uint32_t) * total, h->stream));
    {
      LaunchScope ls(h, DFL_PROF_AGG);
      k_agg_giant_accum<<<grid_for(gi.nitems, 1, 152 * 5), kAggThreads, sizeof(GiantTable), h->stream>>>(a, gi);
      DFL_TRY(check_launch(h, "giant accum"));
    }
    DFL_TRY(scan_u32(h, gi.units, gi.units, entries));
    {
      LaunchScope ls(h, DFL_PROF_AGG);
      k_agg_big<<<152 * 5, kAggThreads, sizeof(GiantTable), h->stream>>>(a, gi);
      DFL_TRY(check_launch(h, "giant members"));
    }
    {
      LaunchScope ls(h, DFL_PROF_AGG);
      launch_pdl(k_agg_giant_emit, grid_for(total, kGiantTile, 152 * 8), kAggThreads, 0, h->stream, a, gi,
                 (unsigned long long)total);
      DFL_TRY(check_launch(h, "giant emit"));
    }
  }
  DFL_TRY(read_ctrl(h));
  if (h->hctrl->err) return set_error(h, DFL_ERR_CUDA, "internal error in aggregation (table overflow)");
  return DFL_OK;
}

}  // namespace dfl
