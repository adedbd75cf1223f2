// Counting pass of key aggregation over tables without predicates: every (sampled) row of every
// aggregated key column counts its key's slot (key - base) & mask in the CTA's shared-memory
// hot-key cache or, on a miss, with a global reduction on the count array; a presence column
// sets its key's bit.  Tables with predicates are counted by k_agg_count (build.cu).
//
// Bound by the shared-memory and L2 reductions of the keys (about one 32-key group per 50
// cycles and SM), so the kernel keeps everything else out of their way: a column's
// parameters and eight keys per thread in registers (131 instructions per
// key when the descriptors were read from shared memory for each key, 49 now, caches and
// flushes included), no selection code in
// the kernel (its registers spilled, and with the whole SM's L1 given to shared memory a
// spill is an L2 access), and the next chunk's rows bulk-prefetched into L2 while this chunk
// is counted, since a chunk is only four steps long.
// 81 M int32 keys of two fact tables (domains of 0.13 to 4 M): 592 us before, 259 us now, the
// unique-key kernel beside it both times; 165 M keys of 96 tables without declared domains (164
// instructions per key before, 89 now): 1158 us before, for the 58 largest, 859 us now.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "tile.cuh"

namespace cmpk {

namespace {

// ---- one aggregated column of the counting pass, in registers
constexpr uint32_t kCntEmpty = 0xFFFFFFFFu;  // never a slot index: cap <= 2^31 - 1
struct CntCol {
  int32_t* cnt;         // count array, or presence bitmap
  uint64_t base;
  uint32_t ckey, ccnt;  // its hot-key cache (shared addresses; ckey 0xFFFFFFFF: not cached)
  uint32_t last, mask;  // last slot (cap - 1), slot mask
  uint32_t hshift;
  bool declared;
};
constexpr uint32_t kNoCache = 0xFFFFFFFFu;

// The hot-key cache of one column: H / 2 sets of two (key, count) slots, a set chosen by a
// multiplicative hash of the slot index x.  x is counted in the way that holds it, else in
// an empty way it claims (compare-and-swap; a way once claimed keeps its key until the
// flush), else not at all (false: the caller counts it in the global array).  A set is its
// byte offset in the key (and count) array.
__device__ __forceinline__ uint32_t cache_set(const CntCol& cc, uint32_t x) {
  return ((x * 0x9E3779B1u) >> (cc.hshift + 1)) * 8;
}
__device__ __forceinline__ uint2 cache_read(const CntCol& cc, uint32_t set) {
  uint2 v;
  asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(cc.ckey + set));
  return v;
}
__device__ __forceinline__ void cache_inc(uint32_t addr) {
  asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool cache_claim(uint32_t keys, uint32_t cnts, uint32_t x, bool first_free) {
  for (uint32_t way = first_free ? 0 : 4; way < 8; way += 4) {
    uint32_t prev;
    asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(prev) : "r"(keys + way), "r"(kCntEmpty), "r"(x) : "memory");
    if (prev == kCntEmpty || prev == x) {
      cache_inc(cnts + way);
      return true;
    }
  }
  return false;
}
// x counted in its set, whose keys are `cur`; false: not in the cache.
__device__ __forceinline__ bool cache_hit(const CntCol& cc, uint32_t set, uint2 cur, uint32_t x) {
  if (cur.x == x || cur.y == x) {
    cache_inc(cc.ccnt + set + (cur.x == x ? 0 : 4));
    return true;
  }
  if (cur.x != kCntEmpty && cur.y != kCntEmpty) return false;
  return cache_claim(cc.ckey + set, cc.ccnt + set, x, cur.x == kCntEmpty);
}
__device__ __forceinline__ bool cache_count(const CntCol& cc, uint32_t x) {
  if (cc.ckey == kNoCache) return false;
  const uint32_t set = cache_set(cc, x);
  return cache_hit(cc, set, cache_read(cc, set), x);
}

// Every key of n rows of a column, by the whole CTA; the smallest and largest key are kept for
// undeclared columns, and false is returned when a key lies outside a declared domain (its
// counts are then discarded).  Two 16-byte loads per thread and step, the next step's issued
// before this step's keys are counted; the cache sets of one load's keys are read before any
// is compared.  The rows before the first 16-byte boundary and after the last whole load go
// straight to the count array.  KT: the key type; SMALL: every value of the declared domain
// is an int32 (or none is declared), so that slots are 32-bit sums.
template <typename KT, bool SMALL, bool PRESENCE>
__device__ __forceinline__ bool count_rows(const CntCol& cc, const KT* __restrict__ col, uint32_t n, KT* mn_out,
                                           KT* mx_out) {
  typedef typename std::conditional<SMALL, uint32_t, uint64_t>::type U;  // key - base
  constexpr uint32_t V = 16 / sizeof(KT);                                // keys per load
  const uint32_t tid = threadIdx.x, T = blockDim.x;
  const U base = U(cc.base), last = U(cc.last);
  bool ok = true;
  KT mn = *mn_out, mx = *mx_out;
  const uint32_t head = min(n, uint32_t((16 - (reinterpret_cast<uintptr_t>(col) & 15)) & 15) / uint32_t(sizeof(KT)));
  const uint32_t groups = (n - head) / V, tail = head + groups * V;
  if (tid < head + (n - tail)) {  // fewer than 2 V rows
    const KT key = __ldg(col + (tid < head ? tid : tail + tid - head));
    const U off = U(key) - base;
    mn = min(mn, key);
    mx = max(mx, key);
    if (cc.declared && off > last) ok = false;
    else if (PRESENCE) red_or(reinterpret_cast<uint32_t*>(cc.cnt) + (off >> 5), 1u << (uint32_t(off) & 31));
    else red_add(cc.cnt + (uint32_t(off) & cc.mask), 1);
  }
  const int4* p = reinterpret_cast<const int4*>(col + head);
  int4 cur[2], next[2];
  cur[0] = cur[1] = make_int4(0, 0, 0, 0);
  if (tid < groups) cur[0] = __ldg(p + tid);
  if (tid + T < groups) cur[1] = __ldg(p + tid + T);
  for (uint32_t g = tid; g < groups; g += 2 * T) {
    next[0] = next[1] = cur[1];
    if (g + 2 * T < groups) next[0] = __ldg(p + g + 2 * T);
    if (g + 3 * T < groups) next[1] = __ldg(p + g + 3 * T);
#pragma unroll
    for (int h = 0; h < 2; h++) {
      if (h == 1 && g + T >= groups) break;
      KT key[V];
      if (V == 4) {
        key[0] = KT(cur[h].x), key[1] = KT(cur[h].y), key[V - 2] = KT(cur[h].z), key[V - 1] = KT(cur[h].w);
      } else {
        key[0] = KT((uint64_t(uint32_t(cur[h].y)) << 32) | uint32_t(cur[h].x));
        key[1] = KT((uint64_t(uint32_t(cur[h].w)) << 32) | uint32_t(cur[h].z));
      }
      uint32_t x[V];
      bool in = true;
#pragma unroll
      for (uint32_t q = 0; q < V; q++) {
        const U off = U(key[q]) - base;
        if (PRESENCE) {
          if (off <= last) red_or(reinterpret_cast<uint32_t*>(cc.cnt) + (off >> 5), 1u << (uint32_t(off) & 31));
          else ok = false;
        } else {
          if (cc.declared) in &= off <= last;
          x[q] = uint32_t(off) & cc.mask;
          mn = min(mn, key[q]);
          mx = max(mx, key[q]);
        }
      }
      if (PRESENCE) continue;
      if (!in) {
        ok = false;  // the column's counts are discarded
      } else if (cc.ckey == kNoCache) {
#pragma unroll
        for (uint32_t q = 0; q < V; q++) red_add(cc.cnt + x[q], 1);
      } else {
        uint32_t set[V];
        uint2 way[V];
#pragma unroll
        for (uint32_t q = 0; q < V; q++) {
          set[q] = cache_set(cc, x[q]);
          way[q] = cache_read(cc, set[q]);
        }
#pragma unroll
        for (uint32_t q = 0; q < V; q++)
          if (!cache_hit(cc, set[q], way[q], x[q])) red_add(cc.cnt + x[q], 1);
      }
    }
    cur[0] = next[0];
    cur[1] = next[1];
  }
  *mn_out = mn;
  *mx_out = mx;
  return ok;
}

// Rows [r0, r0 + n) of a sampled table, by the whole CTA: each warp tries 64 rows at a time, keeps
// the sampled ones' offsets in its buffer (128 entries) and counts 64 of them, two per lane, in
// one or two columns whenever it holds 64.  The trials are the bulk of it: with the keys counted
// by the few lanes whose row is kept, every column cost a whole warp's work per 32 rows.  The
// columns' descriptors stay in shared memory: they are needed once in 64 kept rows, and in
// registers they spilled.  40 M rows at 10%, two columns: 386 us as filtered tiles, 216 us now.
// Returns the rows kept by this warp; key ranges as in count_rows.
struct SampledCol {
  CntCol cc;
  const void* col;
  int32_t dtype;
};
struct SampledRange {
  int64_t mn, mx;
  bool ok;
};
__device__ __forceinline__ uint32_t count_sampled(const volatile SampledCol* scv, SampledRange (&sr)[2], int ncol,
                                                  int64_t r0, uint32_t n, uint64_t seed, uint64_t keep, uint32_t* buf) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t nb = 0, kept = 0;  // warp-uniform
  auto count = [&](uint32_t m) {  // the first m <= 64 entries
#pragma unroll
    for (int c = 0; c < 2; c++) {
      if (c >= ncol) break;
      const volatile SampledCol& v = scv[c];
      const void* col = v.col;
      const int32_t dtype = v.dtype;
      int64_t key[2];
#pragma unroll
      for (int e = 0; e < 2; e++)
        if (lane + 32 * e < m) key[e] = load1(col, dtype, r0 + buf[lane + 32 * e]);
      CntCol cc;
      cc.cnt = v.cc.cnt, cc.base = v.cc.base, cc.ckey = v.cc.ckey, cc.ccnt = v.cc.ccnt;
      cc.last = v.cc.last, cc.mask = v.cc.mask, cc.hshift = v.cc.hshift, cc.declared = v.cc.declared;
#pragma unroll
      for (int e = 0; e < 2; e++) {
        if (lane + 32 * e >= m) continue;
        const uint64_t off = uint64_t(key[e]) - cc.base;
        sr[c].mn = min(sr[c].mn, key[e]);
        sr[c].mx = max(sr[c].mx, key[e]);
        if (cc.declared && off > cc.last) {
          sr[c].ok = false;
          continue;
        }
        const uint32_t x = uint32_t(off) & cc.mask;
        if (!cache_count(cc, x)) red_add(cc.cnt + x, 1);
      }
    }
    __syncwarp();
  };
  for (uint32_t b = 64 * warp; b < n; b += 64 * nw) {
    bool in[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const uint32_t r = b + 32 * h + lane;
      in[h] = r < n && splitmix64_at(seed, uint64_t(r0) + r) < keep;
    }
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const unsigned m = __ballot_sync(0xffffffffu, in[h]);
      if (in[h]) buf[nb + __popc(m & lt)] = b + 32 * h + lane;
      nb += __popc(m);
    }
    __syncwarp();
    if (nb >= 64) {
      count(64);
      nb -= 64;  // fewer than 64 left: to the front
      uint32_t v0 = 0, v1 = 0;
      if (lane < nb) v0 = buf[64 + lane];
      if (lane + 32 < nb) v1 = buf[96 + lane];
      __syncwarp();
      if (lane < nb) buf[lane] = v0;
      if (lane + 32 < nb) buf[32 + lane] = v1;
      kept += 64;
      __syncwarp();
    }
  }
  if (nb) count(nb);
  return kept + nb;
}

}  // namespace

// Persistent CTAs take chunks of a table's rows in order from an atomic counter, one ahead.
// SAMPLED: the tables with a row sample (a kernel of their own: in one, the sample's registers
// made the other loops spill).
template <bool SAMPLED>
__global__ void __launch_bounds__(512, 2) k_count_rows(const __grid_constant__ BuildArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  // the unique-key kernel or the dense kernel, launched next as a programmatic dependent, reads
  // nothing this launch writes: let it start now and share the SMs
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ int32_t acol[CMP_MAX_SKETCHES], aidx[CMP_MAX_SKETCHES], n_ac;
  __shared__ unsigned long long amax[CMP_MAX_SKETCHES], amin[CMP_MAX_SKETCHES];  // encoded
  __shared__ uint32_t sbuf[SAMPLED ? 512 / 32 : 1][128];  // sampled rows, per warp
  __shared__ SampledCol scol[SAMPLED ? CMP_MAX_SKETCHES : 1];  // the current table's columns
  __shared__ uint32_t akeys;  // the current table's aggregated key columns (bit c: column c)
  __shared__ long long next_chunk;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
  const int n_cache = A.cnt_cache_cols;
  int H = 0;  // the current table's cache slots per column (block-uniform)
  uint32_t* ckey = reinterpret_cast<uint32_t*>(smem);  // [n_cache][H] cached slot index
  uint32_t* ccnt = ckey;                                // [n_cache][H] its count so far
  unsigned long long* work = reinterpret_cast<unsigned long long*>(A.ws) + 2 * int64_t(A.n_agg) + A.cnt_work_slot;
  auto item_of = [&](int64_t c) {  // the item of chunk c (items are in chunk order)
    int it = 0;
    while (it + 1 < A.n_cnt_items && A.cnt_items[it + 1].chunk_begin <= c) it++;
    return it;
  };
  auto agg_of = [&](int a) -> const AggCol& { return A.agg[aidx[a]]; };
  // adds the caches and key ranges of the current table to the global arrays (block-wide)
  auto flush = [&]() {
    __syncthreads();
    for (int a = 0; a < min(int(n_ac), n_cache); a++) {
      if (agg_of(a).kind != kAggCount) continue;
      int32_t* cnt = reinterpret_cast<int32_t*>(A.ws + agg_of(a).off);
      for (int s = tid; s < H; s += T) {
        const uint32_t k = ckey[size_t(a) * H + s];
        if (k != kCntEmpty) red_add(cnt + k, int32_t(ccnt[size_t(a) * H + s]));
      }
    }
    if (tid < n_ac && amax[tid] != 0) {
      unsigned long long* st = reinterpret_cast<unsigned long long*>(A.ws) + 2 * int64_t(aidx[tid]);
      atomicMax(st, amax[tid]);
      atomicMax(st + 1, amin[tid]);
    }
    __syncthreads();
  };
  int item = -1;  // block-uniform
  if (tid == 0) next_chunk = A.cnt_chunk_begin + (long long)atomicAdd(work, 1ull);
  __syncthreads();
  int64_t c = next_chunk;
  while (c < A.cnt_chunk_end) {  // block-uniform
    const int it = item_of(c);
    const CountItem ci = A.cnt_items[it];
    const DevTable* tb = A.tables + ci.table;
    __syncthreads();  // every thread has read next_chunk
    if (tid == 0) next_chunk = A.cnt_chunk_begin + (long long)atomicAdd(work, 1ull);
    const bool new_table = it != item;  // block-uniform
    if (new_table) {  // flush the caches, then set them up for its columns
      if (item >= 0) flush();
      H = ci.cache_slots;
      ccnt = ckey + size_t(H) * n_cache;
      if (tid == 0) {
        int n = 0;
        uint32_t keys = 0;
        // count arrays first (they take the hot-key caches), then presence bitmaps
        for (int kind = kAggCount; kind <= kAggPresence; kind++)
          for (int col = 0; col < tb->n_cols && n < CMP_MAX_SKETCHES; col++) {
            const int ai = tb->agg[col];
            if (ai < 0 || A.agg[ai].kind != kind) continue;
            keys |= 1u << col;
            acol[n] = col;
            aidx[n] = ai;
            amax[n] = 0;
            amin[n] = 0;
            n++;
          }
        akeys = keys;
        n_ac = n;
      }
      for (int s = tid; s < H * n_cache; s += T) {
        ckey[s] = kCntEmpty;
        ccnt[s] = 0;
      }
      item = it;
    }
    __syncthreads();
    const int64_t c_next = next_chunk;
    if (tid < 32 && c_next < A.cnt_chunk_end && c_next < ci.chunk_begin + ci.n_chunks)  // (of the same table)
      prefetch_rows(tb, akeys, (c_next - ci.chunk_begin) * ci.chunk_rows,
                    (c_next - ci.chunk_begin + 1) * ci.chunk_rows, lane, 32);
    const int nac = n_ac;
    const int64_t r_begin = (c - ci.chunk_begin) * ci.chunk_rows;
    const int64_t r_end = min(int64_t(tb->n_rows), r_begin + ci.chunk_rows);
    auto cnt_col = [&](int a) {
      const AggCol& ac = agg_of(a);
      CntCol cc;
      cc.cnt = reinterpret_cast<int32_t*>(A.ws + ac.off);
      cc.ckey = a < n_cache ? uint32_t(__cvta_generic_to_shared(ckey + size_t(a) * H)) : kNoCache;
      cc.ccnt = uint32_t(__cvta_generic_to_shared(ccnt + size_t(a) * H));
      cc.base = uint64_t(ac.base);
      cc.last = uint32_t(ac.cap - 1);  // cap <= 2^32
      cc.mask = uint32_t(ac.mask);
      cc.hshift = uint32_t(32 - (31 - __clz(H)));  // H is a power of two >= 256
      cc.declared = ac.mask == ~0ull;
      return cc;
    };
    // key ranges of column a, over the warp, into the table's
    auto fold_range = [&](int a, const CntCol& cc, bool ok, int64_t mn, int64_t mx) {
      const AggCol& ac = agg_of(a);
      // a declared domain stands for its keys, unless one left it: out of range
      if (cc.declared) mn = ac.base, mx = ac.base + (ac.cap - 1);
      if (!ok) mn = INT64_MIN, mx = INT64_MAX;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)mn, o));
        mx = max(mx, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)mx, o));
      }
      if (lane == 0 && mx >= mn) {
        atomicMax(&amax[a], (unsigned long long)enc_max(mx));
        atomicMax(&amin[a], (unsigned long long)enc_min(mn));
      }
    };
    if constexpr (SAMPLED) {
      if (new_table) {
        if (tid < nac) {
          scol[tid].cc = cnt_col(tid);
          scol[tid].col = tb->col[acol[tid]];
          scol[tid].dtype = tb->dtype[acol[tid]];
        }
        __syncthreads();
      }
      unsigned long long kept = 0;
      for (int a = 0; a < nac; a += 2) {  // (a sampled table has no presence columns)
        const int ncol = min(2, nac - a);
        SampledRange sr[2] = {{INT64_MAX, INT64_MIN, true}, {INT64_MAX, INT64_MIN, true}};
        kept = count_sampled(scol + a, sr, ncol, r_begin, uint32_t(r_end - r_begin), tb->sample_seed, tb->sample_keep,
                             sbuf[tid >> 5]);
#pragma unroll
        for (int q = 0; q < 2; q++)
          if (q < ncol) fold_range(a + q, scol[a + q].cc, sr[q].ok, sr[q].mn, sr[q].mx);
      }
      if (lane == 0 && kept) atomicAdd(reinterpret_cast<unsigned long long*>(tb->survivors), kept);
    } else {
      if (tid == 0 && r_end > r_begin)
        atomicAdd(reinterpret_cast<unsigned long long*>(tb->survivors), (unsigned long long)(r_end - r_begin));
      for (int a = 0; a < nac; a++) {
        const AggCol& ac = agg_of(a);
        const CntCol cc = cnt_col(a);
        const bool i32 = tb->dtype[acol[a]] == CMP_I32, presence = ac.kind == kAggPresence;
        // the slots of an int32 column are 32-bit sums when its domain lies in int32
        const bool small = !cc.declared || (ac.base >= INT32_MIN && ac.base + ac.cap <= int64_t(INT32_MAX) + 1);
        const int32_t* k32 = reinterpret_cast<const int32_t*>(tb->col[acol[a]]) + r_begin;
        const int64_t* k64 = reinterpret_cast<const int64_t*>(tb->col[acol[a]]) + r_begin;
        const uint32_t n = uint32_t(r_end - r_begin);  // a chunk is at most 64 tiles
        int64_t mn = INT64_MAX, mx = INT64_MIN;
        bool ok = true;
        if (i32 && small) {
          int32_t mn32 = INT32_MAX, mx32 = INT32_MIN;
          ok = presence ? count_rows<int32_t, true, true>(cc, k32, n, &mn32, &mx32)
                        : count_rows<int32_t, true, false>(cc, k32, n, &mn32, &mx32);
          if (mx32 >= mn32) mn = mn32, mx = mx32;  // (else: no key seen)
        } else if (!i32) {
          ok = presence ? count_rows<int64_t, false, true>(cc, k64, n, &mn, &mx)
                        : count_rows<int64_t, false, false>(cc, k64, n, &mn, &mx);
        } else {  // int32 keys with a domain beyond int32: one by one (declared)
          for (uint32_t r = tid; r < n; r += T) {
            const uint64_t off = uint64_t(int64_t(__ldg(k32 + r))) - cc.base;
            if (off > cc.last) ok = false;
            else if (presence) red_or(reinterpret_cast<uint32_t*>(cc.cnt) + (off >> 5), 1u << (off & 31));
            else red_add(cc.cnt + off, 1);
          }
        }
        fold_range(a, cc, ok, mn, mx);
      }
    }
    c = c_next;
  }
  if (item >= 0) flush();
}

size_t count_rows_smem_bytes(int32_t cache_slots, int32_t cache_cols) {
  return align16(sizeof(uint32_t) * 2 * size_t(cache_slots) * size_t(cache_cols));
}

// One launch over chunks [chunk_begin, chunk_end) of tables without predicates, all with a row
// sample or all without, taken from chunk counter `work_slot` of the workspace header (zeroed
// before the build).
cudaError_t launch_count_rows(const BuildArgs& a, bool sampled, int32_t grid, int32_t work_slot, int64_t chunk_begin,
                              int64_t chunk_end, cudaStream_t st) {
  if (a.n_agg <= 0 || grid <= 0 || chunk_end <= chunk_begin) return cudaSuccess;
  auto k = sampled ? k_count_rows<true> : k_count_rows<false>;
  const size_t smem = count_rows_smem_bytes(a.cnt_cache_slots, a.cnt_cache_cols);
  static SmemLimit limit[2];
  cudaError_t e = limit[sampled].allow(k);
  if (e != cudaSuccess) return e;
  // the whole shared memory of the SM, so that a CTA of the unique-key or the dense kernel
  // (launched next, as a programmatic dependent) fits beside one of this pass
  e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e != cudaSuccess) return e;
  BuildArgs b = a;
  b.cnt_work_slot = work_slot;
  b.cnt_chunk_begin = chunk_begin;
  b.cnt_chunk_end = chunk_end;
  k<<<unsigned(std::min<int64_t>(grid, chunk_end - chunk_begin)), 512, smem, st>>>(b);
  return cudaGetLastError();
}

}  // namespace cmpk
