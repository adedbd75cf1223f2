// Join-order enumeration over sketch estimates (Sec. 5, Algorithm 1): for every join graph,
// a depth-first search over left-deep orders that follow the graph's edges, from every
// source vertex in increasing f(v) = alpha card(v) / max card + beta deg(v) / max deg,
// extending a prefix by its neighbours in increasing estimate of the extended sub-plan,
// pruning a prefix whose cost exceeds the best complete plan's, and ending a source's
// search after max_plans complete plans.
//
// Cost of a plan: the sum of the estimates of its join prefixes of two or more tables (the
// first table adds nothing).  Ties: sources and candidates by table id.  A NaN estimate
// (beyond the exact range) counts as +inf, a negative one as 0.  Pruning and the update of
// the best plan are strict, so of equal-cost plans the first found is kept.
//
// One CTA per graph.  The search is sequential by definition: every completed plan may lower
// the best cost, which decides what is pruned from then on, and the counters count what the
// sequential search visits.  But between two completed plans the best cost does not change,
// and the subtrees still to be searched are independent.  So the first warp searches, and
// when it has extended kEnumSeqNodes prefixes without completing a plan, the CTA runs a
// round: the unvisited prefixes, in search order, are split (the shallowest first) into up to
// kEnumItems pieces, the warps search the pieces side by side under the current best cost,
// and the results are taken in search order up to and including the first piece that
// completed a plan (all of it: its warp lowered the best cost for itself).  What came after
// that piece is discarded and searched again under the new best cost.  The counters, the
// costs and the plan are those of the sequential search; a round that would exceed the
// search budget is discarded and the sequential search goes on alone, to the end, as it does
// when a paused search has more than kEnumItems unvisited prefixes.
//
// A batch of more graphs than there are SMs takes two launches.  A CTA of 16 warps of 118
// registers has an SM to itself, and most searches of a large batch are short: so the first launch
// gives every graph one warp (up to 32 CTAs per SM) and a number of extensions, and the
// second one goes on with the searches it left open in the workspace.  3000 graphs of five tables
// (88 extensions each): 892 us with a CTA of 16 warps for every graph, 89 us now; 3000 chains of
// 12 (622 on average, at most 7205): 5197 and 2074 us; 600 mixed graphs of 5 to 13 tables (2164 on
// average, at most 82,884): 3704 and 3716 us.
//
// Everything a prefix extension touches is kept close, for its latency is what a search
// costs:
//  - the search frames (one per prefix length and warp) live in shared memory;
//  - the graph's open-addressing table of (sub-plan mask, estimate) is staged in shared
//    memory when it has at most kEnumStageSlots slots (64 KB), else read through the
//    read-only cache (mask slot, then the estimate the slot points to);
//  - a prefix's candidates are looked up side by side, lane v taking table v (and v + 32),
//    and sorted by (estimate, id) by counting each one's predecessors;
//  - estimates and costs are never negative, so they are ordered as their bit patterns, in
//    integers (double comparisons run at 1/64 of their rate here); the one double addition
//    per candidate, its cost, is made for all candidates of a prefix side by side;
//  - candidates are in ascending estimate order and cost + estimate is monotone under
//    rounding, so the first pruned candidate prunes the rest of its frame at once.
// Ten chains and cycles of 4 to 17 tables (993 sub-plans, 100,000 extensions): 46.2 ms with one
// lane per graph and its frames in global memory, 33.7 ms with the above on one warp, 4.6 ms
// with the rounds.
// f(v) and the costs are computed with explicitly rounded double operations (no fused
// multiply-add), so every comparison sees the same values as a plain IEEE evaluation.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.cuh"

namespace cmpk {
namespace {

constexpr int kEnumMaxN = CMP_MAX_TABLES;  // 64

struct EnumGraph {
  int32_t n, h_log2;            // tables; log2 of its hash table's slots
  int64_t h_begin, n_masks;     // its hash table in the slot array; its sub-plans
  const int64_t* card;          // device [n]: exact selected counts
  uint64_t adj[kEnumMaxN];
  int32_t deg[kEnumMaxN];
};
// One slot of a graph's table: a sub-plan mask (0 = empty; masks are nonzero) and the
// index of its estimate.  Linear probing from enum_hash(mask); at most half the slots used.
struct EnumSlot {
  uint64_t mask;
  int64_t sub;
};
// (the high bits of the product are hashed: shift by 64 - log2 of the table's slots)
__host__ __device__ inline uint64_t enum_hash(uint64_t m, int log2_size) {
  return ((m ^ (m >> 29)) * 0x9E3779B97F4A7C15ull) >> (64 - log2_size);
}

struct EnumPlanHdr {
  uint64_t magic;
  int32_t version, n_graphs;
  int64_t n_sub, n_slots;
  int64_t off_graphs, off_slots, total_bytes, ws_bytes;
  int32_t n_max, stage_slots;  // most tables of a graph; slots of the largest staged table
};
constexpr int32_t kEnumPlanVersion = 4;
constexpr uint64_t kEnumPlanMagic = 0x434d50454e554d31ull;  // "CMPENUM1"

constexpr int kEnumMaxWarps = 16;
constexpr int kEnumStageSlots = 4096;    // 64 KB
constexpr int kEnumItems = 256;          // pieces of a round
constexpr int kEnumTasksWanted = 96;     // pieces to search that a round stops splitting at
constexpr int64_t kEnumSeqNodes = 192;   // prefixes extended alone before a round
constexpr int32_t kEnumBatch = 152;      // graphs (one CTA per SM) beyond which a plan takes two launches
// Extensions of a graph in the first launch: 48 for every graph per SM, at least 96.  What one
// warp ends costs no CTA of its own later, but the longest search waits for it (96 / 192 for
// every graph per SM: 3000 chains of 12 1850 / 2215 us, but the 600 mixed graphs 3801 / 3901 us).
constexpr int64_t kEnumFirstNodes = 48, kEnumFirstLeast = 96;
constexpr size_t kEnumFirstSmem = 6 << 10;  // shared memory of a first launch's CTA: 32 of them per SM

// Shared memory of one warp's search over n tables: per prefix length its candidates sorted
// by (estimate, id) with the costs of the prefixes they extend to, the prefix, its
// neighbours, its cost, the next candidate; the best plan.
struct EnumFrame {
  int e, cost, mask, nb, n_cand, next, path, best, cand, bytes;
};
__host__ __device__ inline EnumFrame enum_frame(int n) {
  EnumFrame L;
  int o = 0;
  L.e = o;      o += 8 * n * n;
  L.cost = o;   o += 8 * n;
  L.mask = o;   o += 8 * n;
  L.nb = o;     o += 8 * n;
  L.n_cand = o; o += 4 * n;
  L.next = o;   o += 4 * n;
  L.path = o;   o += 4 * n;
  L.best = o;   o += 4 * n;
  L.cand = o;   o += n * n;
  L.bytes = (o + 15) & ~15;
  return L;
}
// One piece of a round: nothing (kNone), an unsearched prefix (kTask, itself one extension),
// `count` pruned extensions (kPruned) or a complete plan (kPlan).  pre: extensions visited
// right before it (prefixes split into pieces); missing: one of them lacked an estimate.
enum { kNone = 0, kTask = 1, kPruned = 2, kPlan = 3 };
struct EnumPiece {
  uint64_t mask, cost;
  int32_t pre, count;
  uint8_t kind, len, missing, pad[5];  // len: tables of the prefix
};
struct EnumResult {  // of a searched piece: extensions (itself included), pruned ones, plans, best cost
  int64_t nodes, pruned;
  uint64_t cost;
  int32_t plans;
  uint8_t warp, missing, over, improved;
};
// The block's shared memory: warp frames, two lists of pieces with their paths (n bytes each),
// results (not in a first launch: one warp), the source order, the staged table.
struct EnumSmem {
  int frame, piece[2], path[2], result, src, table;
};
__host__ __device__ inline EnumSmem enum_smem(int n, int warps, bool first = false) {
  EnumSmem L;
  int o = 0;
  L.frame = o;  o += enum_frame(n).bytes * warps;
  const int items = first ? 0 : kEnumItems;
  for (int k = 0; k < 2; k++) {
    L.piece[k] = o;
    o += int(sizeof(EnumPiece)) * items;
    L.path[k] = o;
    o += (n * items + 15) & ~15;
  }
  L.result = o; o += int(sizeof(EnumResult)) * items;
  L.src = o;    o += 4 * n;
  L.table = (o + 15) & ~15;
  return L;
}
// A search as the first launch of a batch leaves it (open: at frame d of the frames after it),
// one per graph in the workspace.
struct EnumSaved {
  uint64_t min_cost;
  int64_t plans, nodes, pruned, p, quiet;
  int32_t si, d;
  uint8_t open, have, missing, pad[5];
};
__host__ __device__ inline size_t enum_saved_bytes(int n) { return align16(sizeof(EnumSaved)) + size_t(enum_frame(n).bytes); }
// workspace of a plan of one launch: it needs none beyond shared memory; the entry point still
// takes a buffer of this size
constexpr size_t kEnumWsBytes = 16;

struct EnumArgs {
  const EnumGraph* graphs;
  const EnumSlot* slots;
  const double* est;
  int32_t n_graphs;
  double alpha, beta;
  int64_t max_plans, max_nodes;
  int32_t n_max, stage_slots, warps;  // most tables of a graph; slots of the shared-memory table; warps per CTA
  unsigned char* saved;  // a batch's searches between its two launches, else null
  int64_t first_nodes;   // extensions of a graph in a first launch
  int32_t* order;
  double* cost;
  int64_t* stats;
  int32_t* status;
};

// The bits of an estimate as the search takes it: NaN (beyond the exact range) as +inf, a
// negative one (or -0) as 0.  Bits of non-negative doubles order as the values.
constexpr uint64_t kInfBits = 0x7ff0000000000000ull;
__device__ __forceinline__ uint64_t est_bits(double v) {
  const uint64_t b = uint64_t(__double_as_longlong(v));
  if ((b & ~(1ull << 63)) > kInfBits) return kInfBits;  // NaN
  return (b >> 63) ? 0ull : b;
}
__device__ __forceinline__ double bits_double(uint64_t b) { return __longlong_as_double((long long)b); }

// A slot's fields through the read-only cache.
__device__ __forceinline__ uint64_t load_mask(const EnumSlot* s) {
  return __ldg(reinterpret_cast<const unsigned long long*>(&s->mask));
}
__device__ __forceinline__ int64_t load_sub(const EnumSlot* s) {
  return __ldg(reinterpret_cast<const long long*>(&s->sub));
}

// The estimate of sub-plan m in the staged table (tmask, tval) or the plan's slots.
__device__ __forceinline__ uint64_t lookup(const EnumArgs& A, const EnumGraph& g, const uint64_t* tmask,
                                           const uint64_t* tval, bool staged, uint64_t m, bool* missing) {
  const uint64_t size = uint64_t(1) << g.h_log2;
  uint64_t i = enum_hash(m, g.h_log2);
  for (uint64_t probe = 0; probe < size; probe++) {  // the table has empty slots: ends early
    if (staged) {
      const uint64_t k = tmask[i];
      if (k == m) return tval[i];
      if (k == 0) break;
    } else {
      const EnumSlot* sl = A.slots + g.h_begin + int64_t(i);
      const uint64_t k = load_mask(sl);
      const int64_t sub = load_sub(sl);
      if (k == m) return est_bits(__ldg(A.est + sub));
      if (k == 0) break;
    }
    i = (i + 1) & (size - 1);
  }
  *missing = true;
  return kInfBits;
}

// A warp's search: its frames in shared memory, the current frame in registers (warp-uniform).
struct EnumWarp {
  const EnumArgs& A;
  const EnumGraph& g;
  const uint64_t *tmask, *tval;
  bool staged;
  int n, lane;
  uint64_t full;
  uint64_t *fe, *fcost, *fmask, *fnb;
  int32_t *fn, *fnext, *path, *best;
  uint8_t* fcand;
  int d, nx, nc;
  uint64_t m, nb, cost;
  bool missing;

  __device__ EnumWarp(const EnumArgs& A_, const EnumGraph& g_, unsigned char* base, const uint64_t* tm,
                      const uint64_t* tv, bool st)
      : A(A_), g(g_), tmask(tm), tval(tv), staged(st), n(g_.n), lane(threadIdx.x & 31) {
    const EnumFrame L = enum_frame(A_.n_max);
    full = n == 64 ? ~0ull : ((1ull << n) - 1);
    fe = reinterpret_cast<uint64_t*>(base + L.e);
    fcost = reinterpret_cast<uint64_t*>(base + L.cost);
    fmask = reinterpret_cast<uint64_t*>(base + L.mask);
    fnb = reinterpret_cast<uint64_t*>(base + L.nb);
    fn = reinterpret_cast<int32_t*>(base + L.n_cand);
    fnext = reinterpret_cast<int32_t*>(base + L.next);
    path = reinterpret_cast<int32_t*>(base + L.path);
    best = reinterpret_cast<int32_t*>(base + L.best);
    fcand = base + L.cand;
    missing = false;
  }
  // Neighbours of a set of tables.
  __device__ __forceinline__ uint64_t neighbours(uint64_t mask) const {
    uint64_t r = 0;
    for (; mask; mask &= mask - 1) r |= g.adj[__ffsll(static_cast<long long>(mask)) - 1];
    return r;
  }
  // Candidates of frame fd for the prefix pm with neighbours pnb and cost pc, sorted by
  // (estimate, id), with the costs of the extended prefixes.  Returns their number.
  __device__ int expand(int fd, uint64_t pm, uint64_t pnb, uint64_t pc) {
    const uint64_t c = pnb & ~pm;
    const int v0 = lane, v1 = lane + 32;
    const bool h0 = (c >> v0) & 1, h1 = (c >> v1) & 1;
    uint64_t e0 = kInfBits, e1 = kInfBits;
    bool miss = false;
    if (h0) e0 = lookup(A, g, tmask, tval, staged, pm | (1ull << v0), &miss);
    if (h1) e1 = lookup(A, g, tmask, tval, staged, pm | (1ull << v1), &miss);
    if (__any_sync(0xffffffffu, miss)) missing = true;
    int r0 = 0, r1 = 0;
    if (c & (c - 1)) {
      for (uint64_t rest = c; rest; rest &= rest - 1) {
        const int j = __ffsll(static_cast<long long>(rest)) - 1;
        const uint64_t ej = __shfl_sync(0xffffffffu, (unsigned long long)(j < 32 ? e0 : e1), j & 31);
        r0 += ej < e0 || (ej == e0 && j < v0);
        r1 += ej < e1 || (ej == e1 && j < v1);
      }
    }
    const double base = bits_double(pc);
    if (h0) {
      fe[fd * n + r0] = uint64_t(__double_as_longlong(__dadd_rn(base, bits_double(e0))));
      fcand[fd * n + r0] = uint8_t(v0);
    }
    if (h1) {
      fe[fd * n + r1] = uint64_t(__double_as_longlong(__dadd_rn(base, bits_double(e1))));
      fcand[fd * n + r1] = uint8_t(v1);
    }
    __syncwarp();
    return __popcll(c);
  }
  // The current frame to shared memory (read by the warp's later returns to it, and by rounds).
  __device__ __forceinline__ void save() {
    __syncwarp();  // every lane has read what is rewritten now
    if (lane == 0) {
      fmask[d] = m;
      fnb[d] = nb;
      fcost[d] = cost;
      fnext[d] = nx;
      fn[d] = nc;
    }
    __syncwarp();
  }
  __device__ __forceinline__ void load(int fd) {
    d = fd;
    m = fmask[d];
    nb = fnb[d];
    cost = fcost[d];
    nx = fnext[d];
    nc = fn[d];
  }
  enum { kDone, kLimit, kPause, kFull, kAbort };
  // Depth-first search of everything left at depths >= d0 (kDone), until `limit` extensions
  // have been made (kLimit: another one was due), `pause` of them without completing a plan
  // (kPause; quiet: those since the last plan), or `plans` has reached max_plans (kFull); `stop`: a piece with an index below
  // `self` completed a plan (kAbort).
  __device__ int run(int d0, int64_t limit, int64_t pause, int64_t max_plans, int64_t& nodes, int64_t& pruned,
                     int64_t& plans, uint64_t& min_cost, bool& improved, const volatile int* stop, int self,
                     int64_t& quiet) {
    while (true) {
      if (nx == nc) {  // back to the previous prefix
        if (d == d0) return kDone;
        load(d - 1);
        continue;
      }
      if (nodes == limit) return kLimit;
      if (quiet >= pause) return kPause;
      if (stop && (quiet & 15) == 0 && __shfl_sync(0xffffffffu, *stop, 0) < self) return kAbort;
      const uint64_t cc = fe[d * n + nx];
      if (cc > min_cost) {  // early pruning, of this candidate and the dearer ones after it
        const int64_t take = min(int64_t(nc - nx), limit - nodes);
        nodes += take;
        pruned += take;
        nx += int(take);
        quiet++;
        continue;
      }
      const int v = fcand[d * n + nx];
      nodes++;
      nx++;
      quiet++;
      const uint64_t cm = m | (1ull << v);
      if (cm == full) {  // complete plan
        plans++;
        quiet = 0;
        if (cc < min_cost) {
          min_cost = cc;
          improved = true;
          __syncwarp();
          for (int t = lane; t <= d; t += 32) best[t] = path[t];
          if (lane == 0) best[d + 1] = v;
          __syncwarp();
        }
        if (max_plans > 0 && plans >= max_plans) return kFull;  // (-1: never)
        continue;
      }
      save();
      if (lane == 0) path[d + 1] = v;
      d++;
      m = cm;
      nb |= g.adj[v];
      cost = cc;
      nx = 0;
      nc = expand(d, m, nb, cost);
    }
  }
};

// A round's shared state.
struct EnumRound {
  int cmd, n_items, next, first, cur;  // cur: the list in use
  uint64_t min_cost;
  int64_t limit, plans;
};
enum { kCmdExit = 0, kCmdRound = 1 };

}  // namespace

// FIRST: the first launch of a batch, one warp per CTA and no rounds.
template <bool FIRST>
__global__ void __launch_bounds__(FIRST ? 32 : 32 * kEnumMaxWarps) k_enumerate(const __grid_constant__ EnumArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  EnumSaved* const saved =
      A.saved ? reinterpret_cast<EnumSaved*>(A.saved + enum_saved_bytes(A.n_max) * blockIdx.x) : nullptr;
  if (!FIRST && saved && !saved->open) return;  // the first launch has ended it
  const EnumGraph& g = A.graphs[blockIdx.x];
  const int n = g.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = A.warps;
  const EnumSmem L = enum_smem(A.n_max, W, FIRST);
  uint64_t* tmask = reinterpret_cast<uint64_t*>(smem + L.table);
  uint64_t* tval = tmask + A.stage_slots;
  int32_t* src = reinterpret_cast<int32_t*>(smem + L.src);
  EnumPiece* piece[2] = {reinterpret_cast<EnumPiece*>(smem + L.piece[0]), reinterpret_cast<EnumPiece*>(smem + L.piece[1])};
  uint8_t* ppath[2] = {smem + L.path[0], smem + L.path[1]};  // [kEnumItems][n]
  EnumResult* result = reinterpret_cast<EnumResult*>(smem + L.result);
  const int64_t size = int64_t(1) << g.h_log2;
  const bool staged = size <= A.stage_slots;
  if (staged)
    for (int64_t i = threadIdx.x; i < size; i += blockDim.x) {
      const EnumSlot* sl = A.slots + g.h_begin + i;
      const uint64_t k = load_mask(sl);
      tmask[i] = k;
      tval[i] = k ? est_bits(__ldg(A.est + load_sub(sl))) : 0;
    }
  if (warp == 0) {  // source order: f(v) increasing, ties by id; lane v takes tables v and v + 32
    const int v0 = lane, v1 = lane + 32;
    const int64_t card0 = v0 < n ? g.card[v0] : 0, card1 = v1 < n ? g.card[v1] : 0;
    int64_t mc = max(int64_t(0), max(card0, card1));
    int32_t md = max(v0 < n ? g.deg[v0] : 0, v1 < n ? g.deg[v1] : 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mc = max(mc, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)mc, o));
      md = max(md, __shfl_xor_sync(0xffffffffu, md, o));
    }
    auto f_of = [&](int v, int64_t card) {
      if (v >= n) return double(INFINITY);
      const double a = mc > 0 ? __ddiv_rn(__ll2double_rn(card), __ll2double_rn(mc)) : 0.0;
      const double b = md > 0 ? __ddiv_rn(double(g.deg[v]), double(md)) : 0.0;
      return __dadd_rn(__dmul_rn(A.alpha, a), __dmul_rn(A.beta, b));
    };
    const double f0 = f_of(v0, card0), f1 = f_of(v1, card1);
    int r0 = 0, r1 = 0;
    for (int j = 0; j < n; j++) {
      const double fj = __shfl_sync(0xffffffffu, j < 32 ? f0 : f1, j & 31);
      r0 += fj < f0 || (fj == f0 && j < v0);
      r1 += fj < f1 || (fj == f1 && j < v1);
    }
    if (v0 < n) src[r0] = v0;
    if (v1 < n) src[r1] = v1;
  }
  const int frame_words = enum_frame(A.n_max).bytes / 16;
  uint4* const frame0 = reinterpret_cast<uint4*>(smem + L.frame);
  uint4* const saved_frame = saved ? reinterpret_cast<uint4*>(saved) + align16(sizeof(EnumSaved)) / 16 : nullptr;
  if (!FIRST && saved)  // warp 0 goes on from the frames of the first launch
    for (int i = threadIdx.x; i < frame_words; i += blockDim.x) frame0[i] = saved_frame[i];
  __syncthreads();
  EnumWarp S(A, g, smem + L.frame + size_t(enum_frame(A.n_max).bytes) * warp, tmask, tval, staged);

  // ---- the sequential search's state (warp 0; uniform over its lanes)
  uint64_t min_cost = kInfBits;
  bool have = false, missing = false, out_of_budget = false, alone = W < 2;
  int64_t plans = 0, nodes = 0, pruned = 0, p = 0;  // p: plans completed from this source
  int64_t quiet = 0;  // extensions since the search's last plan (or round, or source)
  int si = -1;
  bool open = false;  // a source's search is under way, at S's current frame
  // The next source (false: there is none left).
  auto next_source = [&]() {
    while (++si < n) {
      p = 0;
      quiet = 0;
      S.d = 0;
      S.m = 1ull << src[si];
      S.nb = g.adj[src[si]];
      S.cost = 0;  // 0.0
      S.nx = 0;
      __syncwarp();
      if (lane == 0) S.path[0] = src[si];
      if (S.m != S.full) {
        S.nc = S.expand(0, S.m, S.nb, S.cost);
        return open = true;
      }
      plans++;  // one table: the plan is complete and costs nothing
      if (min_cost != 0) {
        min_cost = 0;
        if (lane == 0) S.best[0] = src[si];
        have = true;
      }
    }
    return false;
  };
  // The open search from where it is, until its source, the budget, `limit` extensions or the
  // pause ends it.
  auto search = [&](int64_t limit, int64_t pause) {
    bool improved = false;
    const int64_t p0 = p;
    const int why = S.run(0, limit, pause, A.max_plans, nodes, pruned, p, min_cost, improved, nullptr, 0, quiet);
    plans += p - p0;
    have |= improved;
    if (why == EnumWarp::kDone || why == EnumWarp::kFull) open = false;
    if (why == EnumWarp::kLimit && nodes == A.max_nodes) out_of_budget = true;  // exactly max_nodes extensions
    return why;
  };
  // The graph's result (warp 0).
  auto finish = [&]() {
    for (int t = lane; t < kEnumMaxN; t += 32)
      A.order[int64_t(blockIdx.x) * kEnumMaxN + t] = (have && t < n) ? S.best[t] : -1;
    if (lane != 0) return;
    A.cost[blockIdx.x] = bits_double(have ? min_cost : kInfBits);
    A.stats[int64_t(blockIdx.x) * 3 + 0] = plans;
    A.stats[int64_t(blockIdx.x) * 3 + 1] = nodes;
    A.stats[int64_t(blockIdx.x) * 3 + 2] = pruned;
    if (missing) set_status(A.status, CMP_EUNSUPPORTED);
    if (out_of_budget) set_status(A.status, CMP_ETIMEOUT);
  };

  if constexpr (FIRST) {
    const int64_t limit = A.max_plans < 0 ? A.max_nodes : min(A.max_nodes, A.first_nodes);
    bool more = true;
    while (more && (open || next_source())) more = search(limit, INT64_MAX) != EnumWarp::kLimit;
    open &= !out_of_budget;
    if (open) {
      S.save();
      for (int i = lane; i < frame_words; i += 32) saved_frame[i] = frame0[i];
    }
    if (lane == 0) *saved = {min_cost, plans, nodes, pruned, p, quiet, si, S.d, open, have, S.missing};
    missing = S.missing;
    if (!open) finish();
    return;
  }
  __shared__ EnumRound R;
  __shared__ int scan[kEnumMaxWarps * 32 + 1];
  if (saved && warp == 0) {
    const EnumSaved v = *saved;
    min_cost = v.min_cost, plans = v.plans, nodes = v.nodes, pruned = v.pruned, p = v.p, quiet = v.quiet, si = v.si;
    have = v.have, missing = v.missing, open = true;
    S.load(v.d);
  }

  // Warp 0: the unvisited prefixes of the open search as the first list of pieces, in search
  // order (the deepest frame's remaining candidates first); false when they are too many.
  auto collect = [&]() {
    int at = 0;
    for (int fd = S.d; fd >= 0; fd--) {
      const int k0 = S.fnext[fd], k1 = S.fn[fd];
      int live = 0;  // candidates not yet pruned: a prefix of the frame's order
      for (int k = k0; k < k1; k++) live += S.fe[fd * n + k] <= min_cost;
      const int rest = k1 - k0 - live;
      if (at + live + (rest > 0) > kEnumItems) return false;
      for (int k = k0 + lane; k < k0 + live; k += 32) {
        EnumPiece q;
        const int v = S.fcand[fd * n + k];
        q.mask = S.fmask[fd] | (1ull << v);
        q.cost = S.fe[fd * n + k];
        q.pre = q.count = 0;
        q.kind = q.mask == S.full ? kPlan : kTask;
        q.len = uint8_t(fd + 2);
        q.missing = 0;
        uint8_t* pp = ppath[0] + size_t(at + k - k0) * n;
        for (int t = 0; t <= fd; t++) pp[t] = uint8_t(S.path[t]);
        pp[fd + 1] = uint8_t(v);
        piece[0][at + k - k0] = q;
      }
      at += live;
      if (rest > 0) {
        if (lane == 0) {
          EnumPiece q = {};
          q.kind = kPruned;
          q.count = rest;
          piece[0][at] = q;
        }
        at++;
      }
    }
    __syncwarp();
    if (lane == 0) {
      R.n_items = at;
      R.cur = 0;
    }
    return true;
  };

  for (;;) {
    if (warp == 0) {
      int cmd = kCmdExit;
      while (!out_of_budget && (open || next_source())) {
        // (a search without a limit on its plans completes them all the time: alone)
        const int why = search(A.max_nodes, alone || A.max_plans < 0 ? INT64_MAX : kEnumSeqNodes);
        if (why == EnumWarp::kPause) {
          S.save();
          quiet = 0;
          if (!collect()) {
            alone = true;
            continue;
          }
          cmd = kCmdRound;
          if (lane == 0) {
            R.min_cost = min_cost;
            R.limit = A.max_nodes - nodes;
            R.plans = p;
            R.next = 0;
          }
          break;
        }
      }
      if (lane == 0) R.cmd = cmd;
      missing |= S.missing;
      S.missing = false;
    }
    __syncthreads();
    if (R.cmd == kCmdExit) break;

    // ---- a round.  Split the shallowest unsearched prefixes while the list has room.
    for (int step = 0; step < 64; step++) {
      const int ni = R.n_items, cur = R.cur, i = threadIdx.x;
      int len = 1 << 20;
      bool task = false;
      if (i < ni && i < kEnumItems && piece[cur][i].kind == kTask) {
        task = true;
        len = piece[cur][i].len;
      }
      const int n_task = __syncthreads_count(task);
      // shallowest length (prefixes of n - 2 tables and more are searched whole)
      scan[threadIdx.x] = len;
      __syncthreads();
      for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (i < o) scan[i] = min(scan[i], scan[i + o]);
        __syncthreads();
      }
      const int shallow = scan[0];
      __syncthreads();
      if (n_task == 0 || n_task >= kEnumTasksWanted || shallow > n - 3) break;  // block-uniform
      // pieces each one becomes, in order, as long as the whole list fits
      const bool want = task && len == shallow;
      int more = 0;
      if (want) more = __popcll(S.neighbours(piece[cur][i].mask) & ~piece[cur][i].mask);  // its children + pruned rest
      int incl = more;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      if (lane == 31) scan[warp] = incl;
      __syncthreads();
      for (int k = 0; k < warp; k++) incl += scan[k];
      const bool fits = ni + incl <= kEnumItems;
      const int dst = i + (fits ? incl - more : 0);
      // (once one does not fit, none after it does: incl is monotone; they move by the last fitting sum)
      __syncthreads();
      if (i == 0) scan[0] = 0;
      __syncthreads();
      if (fits) atomicMax(&scan[0], incl);
      __syncthreads();
      const int grown = scan[0];
      const int to = fits ? dst : i + grown;
      const int any = __syncthreads_or(want && fits && more > 0);
      if (!any) break;
      if (i < ni && !(want && fits)) {  // moves
        piece[cur ^ 1][to] = piece[cur][i];
        for (int t = 0; t < n; t++) ppath[cur ^ 1][size_t(to) * n + t] = ppath[cur][size_t(i) * n + t];
      }
      // each split prefix: a warp expands it and writes its children
      __shared__ int todo[kEnumItems], todo_at[kEnumItems], n_todo;
      if (i == 0) n_todo = 0;
      __syncthreads();
      if (i < ni && want && fits) {
        const int k = atomicAdd(&n_todo, 1);
        todo[k] = i;
        todo_at[k] = to;
      }
      __syncthreads();
      for (int k = warp < W ? warp : n_todo; k < n_todo; k += W) {
        const EnumPiece q = piece[cur][todo[k]];
        const uint8_t* pp = ppath[cur] + size_t(todo[k]) * n;
        const uint64_t pnb = S.neighbours(q.mask);
        const int slots = 1 + __popcll(pnb & ~q.mask);  // the room reserved for it
        // (warp 0's frames hold the open search: candidates go to the row of the last prefix
        // length, n - 1, whose frame has none of its own)
        S.missing = false;
        const int nc = S.expand(n - 1, q.mask, pnb, q.cost);
        int live = 0;
        for (int c = lane; c < nc; c += 32) live += S.fe[(n - 1) * n + c] <= R.min_cost;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) live += __shfl_xor_sync(0xffffffffu, live, o);
        for (int c = lane; c < slots; c += 32) {
          EnumPiece r = {};
          const size_t o = size_t(todo_at[k] + c);
          if (c < live) {
            const int v = S.fcand[(n - 1) * n + c];
            r.mask = q.mask | (1ull << v);
            r.cost = S.fe[(n - 1) * n + c];
            r.kind = r.mask == S.full ? kPlan : kTask;
            r.len = uint8_t(q.len + 1);
            for (int t = 0; t < q.len; t++) ppath[cur ^ 1][o * n + t] = pp[t];
            ppath[cur ^ 1][o * n + q.len] = uint8_t(v);
          } else if (c == live) {  // its pruned candidates (or nothing): the prefix itself counts here at the latest
            r.kind = kPruned;
            r.count = nc - live;
          }
          if (c == 0) {  // the prefix's own extension comes right before its first piece
            r.pre = q.pre + 1;
            r.missing = q.missing | uint8_t(S.missing);
          }
          piece[cur ^ 1][o] = r;
        }
        __syncwarp();
      }
      __syncthreads();
      if (i == 0) {
        R.n_items = ni + grown;
        R.cur = cur ^ 1;
      }
      __syncthreads();
    }
    // the first complete plan among the pieces ends the round's useful part
    {
      const int i = threadIdx.x;
      __syncthreads();
      if (i == 0) R.first = INT32_MAX;
      __syncthreads();
      if (i < R.n_items && i < kEnumItems && piece[R.cur][i].kind == kPlan) atomicMin(&R.first, i);
      __syncthreads();
    }
    const EnumPiece* list = piece[R.cur];
    const uint8_t* lpath = ppath[R.cur];
    const int n_items = R.n_items;
    // Search the pieces in order.  Warp 0 keeps the open search's frames: it takes no piece.
    if (warp > 0 && warp < W) {
      for (;;) {
        int k = 0;
        if (lane == 0) {
          k = atomicAdd(&R.next, 1);
          if (k >= n_items || k > *const_cast<volatile int*>(&R.first)) k = -1;
        }
        k = __shfl_sync(0xffffffffu, k, 0);
        if (k < 0) break;
        const EnumPiece q = list[k];
        if (q.kind != kTask) continue;
        S.d = q.len - 1;
        S.m = q.mask;
        S.nb = S.neighbours(q.mask);
        S.cost = q.cost;
        S.nx = 0;
        S.missing = false;
        __syncwarp();
        for (int t = lane; t < q.len; t += 32) S.path[t] = lpath[size_t(k) * n + t];
        __syncwarp();
        S.nc = S.expand(S.d, S.m, S.nb, S.cost);
        int64_t wn = 1, wp = 0, wplans = R.plans, wquiet = 0;
        uint64_t wcost = R.min_cost;
        bool improved = false;
        // (limit + 1: reaching it means more than the budget is left for)
        const int why = S.run(S.d, R.limit + 1, INT64_MAX, A.max_plans, wn, wp, wplans, wcost, improved, &R.first, k, wquiet);
        if (lane == 0) {
          EnumResult& r = result[k];
          r.nodes = wn;
          r.pruned = wp;
          r.cost = wcost;
          r.plans = int32_t(wplans - R.plans);
          r.warp = uint8_t(warp);
          r.missing = S.missing;
          r.over = why == EnumWarp::kLimit;
          r.improved = improved;
          __threadfence_block();
          if (wplans > R.plans) atomicMin(&R.first, k);
        }
        __syncwarp();
        if (wplans > R.plans) break;  // its best plan stays in this warp's frames
      }
    }
    __syncthreads();
    if (warp == 0) {  // take the results in search order, up to the first piece with a plan
      const int first = R.first;  // INT32_MAX: none
      int64_t rn = 0, rp = 0;
      bool over = false, miss = false;
      for (int k = lane; k < n_items && k <= first; k += 32) {
        const EnumPiece q = list[k];
        rn += q.pre;
        miss |= q.missing != 0;
        if (q.kind == kTask) {
          const EnumResult r = result[k];
          rn += r.nodes;
          rp += r.pruned;
          miss |= r.missing != 0;
          over |= r.over != 0;
        } else if (q.kind == kPruned) {
          rn += q.count;
          rp += q.count;
        } else if (q.kind == kPlan) {
          rn += 1;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        rn += __shfl_xor_sync(0xffffffffu, (long long)rn, o);
        rp += __shfl_xor_sync(0xffffffffu, (long long)rp, o);
      }
      over = __any_sync(0xffffffffu, over);
      miss = __any_sync(0xffffffffu, miss);
      if (over || rn > A.max_nodes - nodes) {  // the budget ends inside: the sequential search finds where
        alone = true;
        S.load(S.d);
      } else {
        nodes += rn;
        pruned += rp;
        missing |= miss;
        if (first == INT32_MAX) {
          open = false;  // nothing left from this source
        } else {
          const EnumPiece q = list[first];
          const uint8_t* pp = lpath + size_t(first) * n;
          int64_t got = 1;
          if (q.kind == kPlan) {
            if (q.cost < min_cost) {
              min_cost = q.cost;
              have = true;
              __syncwarp();
              for (int t = lane; t < n; t += 32) S.best[t] = pp[t];
            }
          } else {
            const EnumResult r = result[first];
            got = r.plans;
            if (r.improved) {
              min_cost = r.cost;
              have = true;
              const int32_t* wb = reinterpret_cast<const int32_t*>(
                  smem + L.frame + size_t(enum_frame(A.n_max).bytes) * r.warp + enum_frame(A.n_max).best);
              __syncwarp();
              for (int t = lane; t < n; t += 32) S.best[t] = wb[t];
            }
          }
          plans += got;
          p += got;
          if (A.max_plans > 0 && p >= A.max_plans) {
            open = false;
          } else {  // go on after that piece: its path's frames, each past the table the path takes
            __syncwarp();
            for (int t = lane; t < q.len; t += 32) S.path[t] = pp[t];
            __syncwarp();
            uint64_t m = 1ull << S.path[0], nb = g.adj[S.path[0]], cost = 0;
            for (int fd = 0; fd + 1 < q.len; fd++) {
              const int nc = S.expand(fd, m, nb, cost), v = S.path[fd + 1];
              int at = 0;
              while (at < nc && S.fcand[fd * n + at] != v) at++;  // a candidate by construction
              S.d = fd, S.m = m, S.nb = nb, S.cost = cost, S.nx = at + 1, S.nc = nc;
              const uint64_t next = at < nc ? S.fe[fd * n + at] : cost;
              S.save();
              m |= 1ull << v;
              nb |= g.adj[v];
              cost = next;
            }
          }
        }
      }
      S.missing = false;  // (what counts is in `missing`)
    }
    __syncthreads();
  }
  if (warp == 0) finish();
}

namespace {

struct EnumPlanParts {
  std::vector<EnumGraph> graphs;
  std::vector<EnumSlot> slots;
  EnumPlanHdr hdr;
};

cmp_status enum_plan(const cmp_graph* graphs, int32_t n_graphs, int32_t n_sub, const int32_t* sub_graph,
                     const uint64_t* sub_mask, EnumPlanParts* P) {
  if (!graphs || n_graphs < 1 || n_sub < 0 || (n_sub && (!sub_graph || !sub_mask))) return CMP_EINVAL;
  P->graphs.assign(size_t(n_graphs), EnumGraph{});
  std::vector<std::vector<std::pair<uint64_t, int64_t>>> per(n_graphs);
  for (int32_t q = 0; q < n_sub; q++) {
    const int32_t gi = sub_graph[q];
    if (gi < 0 || gi >= n_graphs || sub_mask[q] == 0) return CMP_EINVAL;
    const int32_t nt = graphs[gi].n_tables;
    if (nt < 64 && (sub_mask[q] >> nt) != 0) return CMP_EINVAL;
    per[gi].push_back({sub_mask[q], q});
  }
  P->slots.clear();
  for (int32_t gi = 0; gi < n_graphs; gi++) {
    const cmp_graph& cg = graphs[gi];
    if (cg.n_tables < 1 || cg.n_tables > kEnumMaxN || cg.n_edges < 0 || !cg.survivors_dev) return CMP_EINVAL;
    if (cg.n_edges && (!cg.edge_u || !cg.edge_v)) return CMP_EINVAL;
    EnumGraph& g = P->graphs[gi];
    std::memset(&g, 0, sizeof(g));
    g.n = cg.n_tables;
    g.card = cg.survivors_dev;
    for (int32_t e = 0; e < cg.n_edges; e++) {
      const int u = cg.edge_u[e], v = cg.edge_v[e];
      if (u < 0 || u >= g.n || v < 0 || v >= g.n || u == v) return CMP_EINVAL;
      g.adj[u] |= 1ull << v;
      g.adj[v] |= 1ull << u;
      g.deg[u]++;
      g.deg[v]++;
    }
    auto& list = per[gi];
    std::sort(list.begin(), list.end());
    for (size_t i = 1; i < list.size(); i++)
      if (list[i].first == list[i - 1].first) return CMP_EINVAL;  // one estimate per sub-plan
    g.n_masks = int64_t(list.size());
    int lg = 4;
    while ((int64_t(1) << lg) < 2 * g.n_masks) lg++;
    g.h_log2 = lg;
    g.h_begin = int64_t(P->slots.size());
    P->slots.resize(P->slots.size() + (size_t(1) << lg), EnumSlot{0, 0});
    EnumSlot* tab = P->slots.data() + g.h_begin;
    const uint64_t size = uint64_t(1) << lg;
    for (const auto& x : list) {
      uint64_t i = enum_hash(x.first, lg);
      while (tab[i].mask != 0) i = (i + 1) & (size - 1);
      tab[i] = EnumSlot{x.first, x.second};
    }
  }
  EnumPlanHdr& H = P->hdr;
  std::memset(&H, 0, sizeof(H));
  H.magic = kEnumPlanMagic;
  H.version = kEnumPlanVersion;
  H.n_graphs = n_graphs;
  H.n_sub = n_sub;
  H.n_slots = int64_t(P->slots.size());
  size_t off = align16(sizeof(EnumPlanHdr));
  H.off_graphs = int64_t(off);
  off += align16(sizeof(EnumGraph) * P->graphs.size());
  H.off_slots = int64_t(off);
  off += align16(sizeof(EnumSlot) * P->slots.size());
  H.total_bytes = int64_t(off);
  H.n_max = 1;
  H.stage_slots = 0;
  for (const EnumGraph& g : P->graphs) {
    H.n_max = std::max(H.n_max, g.n);
    if ((int64_t(1) << g.h_log2) <= kEnumStageSlots) H.stage_slots = std::max(H.stage_slots, 1 << g.h_log2);
  }
  H.ws_bytes = int64_t(n_graphs > kEnumBatch ? enum_saved_bytes(H.n_max) * size_t(n_graphs) + 15 : kEnumWsBytes);
  return CMP_OK;
}

}  // namespace
}  // namespace cmpk

using namespace cmpk;

extern "C" {

cmp_status cmp_enum_plan_bytes(const cmp_graph* graphs, int32_t n_graphs, int32_t n_sub, const int32_t* sub_graph,
                               const uint64_t* sub_mask, size_t* plan_bytes, size_t* ws_bytes) {
  if (!plan_bytes || !ws_bytes) return CMP_EINVAL;
  EnumPlanParts P;
  const cmp_status st = enum_plan(graphs, n_graphs, n_sub, sub_graph, sub_mask, &P);
  if (st != CMP_OK) return st;
  *plan_bytes = size_t(P.hdr.total_bytes);
  *ws_bytes = size_t(P.hdr.ws_bytes);
  return CMP_OK;
}

cmp_status cmp_enum_plan_encode(const cmp_graph* graphs, int32_t n_graphs, int32_t n_sub, const int32_t* sub_graph,
                                const uint64_t* sub_mask, void* plan_host, size_t plan_bytes) {
  if (!plan_host) return CMP_EINVAL;
  EnumPlanParts P;
  const cmp_status st = enum_plan(graphs, n_graphs, n_sub, sub_graph, sub_mask, &P);
  if (st != CMP_OK) return st;
  if (plan_bytes < size_t(P.hdr.total_bytes)) return CMP_EWORKSPACE;
  unsigned char* b = static_cast<unsigned char*>(plan_host);
  std::memset(b, 0, size_t(P.hdr.total_bytes));
  std::memcpy(b, &P.hdr, sizeof(P.hdr));
  std::memcpy(b + P.hdr.off_graphs, P.graphs.data(), sizeof(EnumGraph) * P.graphs.size());
  if (!P.slots.empty()) std::memcpy(b + P.hdr.off_slots, P.slots.data(), sizeof(EnumSlot) * P.slots.size());
  return CMP_OK;
}

cmp_status cmp_enumerate(const void* plan_host, const void* plan_dev, const double* est_dev, const cmp_enum_cfg* cfg,
                         void* ws_dev, size_t ws_bytes, int32_t* order_dev, double* cost_dev, int64_t* stats_dev,
                         int32_t* status_dev, void* stream) {
  if (!plan_host || !plan_dev) return CMP_EINVAL;
  EnumPlanHdr H;
  std::memcpy(&H, plan_host, sizeof(H));
  if (H.magic != kEnumPlanMagic || H.version != kEnumPlanVersion) return CMP_EINVAL;
  if (!order_dev || !cost_dev || !stats_dev || (H.n_sub > 0 && !est_dev)) return CMP_EINVAL;
  if (!ws_dev || ws_bytes < size_t(H.ws_bytes)) return CMP_EWORKSPACE;
  double alpha = 0.5, beta = 0.5;
  int64_t max_plans = 10, max_nodes = int64_t(1) << 26;
  if (cfg) {
    if (!(cfg->alpha >= 0.0) || !(cfg->beta >= 0.0) || cfg->max_plans < -1 || cfg->max_nodes < 0) return CMP_EINVAL;
    if (cfg->alpha != 0.0 || cfg->beta != 0.0) alpha = cfg->alpha, beta = cfg->beta;
    if (cfg->max_plans != 0) max_plans = cfg->max_plans;  // -1: no limit
    if (cfg->max_nodes > 0) max_nodes = cfg->max_nodes;
  }
  const unsigned char* pd = static_cast<const unsigned char*>(plan_dev);
  EnumArgs a;
  a.graphs = reinterpret_cast<const EnumGraph*>(pd + H.off_graphs);
  a.slots = reinterpret_cast<const EnumSlot*>(pd + H.off_slots);
  a.est = est_dev;
  a.n_graphs = H.n_graphs;
  a.alpha = alpha;
  a.beta = beta;
  a.max_plans = max_plans;
  a.max_nodes = max_nodes;
  a.n_max = H.n_max;
  a.stage_slots = H.stage_slots;
  a.order = order_dev;
  a.cost = cost_dev;
  a.stats = stats_dev;
  a.status = status_dev;
  a.saved = nullptr;
  a.first_nodes = 0;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (H.n_graphs > kEnumBatch) {  // a batch: every graph by one warp first
    a.saved = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(ws_dev) + 15) & ~uintptr_t(15));
    a.first_nodes = std::max(kEnumFirstLeast, kEnumFirstNodes * H.n_graphs / kEnumBatch);
    a.warps = 1;
    const size_t base = size_t(enum_smem(H.n_max, 1, true).table);
    const size_t room = base < kEnumFirstSmem ? (kEnumFirstSmem - base) / 16 : 0;
    a.stage_slots = int32_t(std::min<size_t>(size_t(H.stage_slots), room));
    static SmemLimit limit;
    if (limit.allow(k_enumerate<true>) != cudaSuccess) return CMP_ECUDA;
    k_enumerate<true><<<unsigned(H.n_graphs), 32, base + 16 * size_t(a.stage_slots), st>>>(a);
    if (cudaGetLastError() != cudaSuccess) return CMP_ECUDA;
  }
  // as many warps as their frames leave room for beside the lists and the staged table
  a.stage_slots = H.stage_slots;
  int warps = kEnumMaxWarps;
  auto smem_of = [&](int k) { return size_t(enum_smem(H.n_max, k).table) + 16 * size_t(H.stage_slots); };
  while (warps > 8 && smem_of(warps) > size_t(200) * 1024) warps >>= 1;  // 256 threads at least: one per piece
  a.warps = warps;
  while (a.warps > 1 && smem_of(a.warps) > size_t(200) * 1024) a.warps--;  // those beyond search nothing
  const size_t smem = smem_of(a.warps);
  static SmemLimit limit;
  if (limit.allow(k_enumerate<false>) != cudaSuccess) return CMP_ECUDA;
  k_enumerate<false><<<unsigned(H.n_graphs), 32 * warps, smem, st>>>(a);
  return cudaGetLastError() == cudaSuccess ? CMP_OK : CMP_ECUDA;
}

}  // extern "C"
