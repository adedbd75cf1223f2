// Internal device/host definitions of libcompass (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <type_traits>

#include "compass.h"

namespace cmpk {

// ------------------------------------------------------------------ constants
constexpr uint64_t kP61 = (1ull << 61) - 1;     // Mersenne prime of the CW hash family
constexpr uint32_t kM31 = 0x7FFFFFFFu;
constexpr uint64_t kM30 = (1ull << 30) - 1;
constexpr unsigned long long kEmptyKey = ~0ull;  // never a field element (< 2^61)

// ------------------------------------------------------- arithmetic mod 2^61-1
// A field element v < 2^61 is held as two limbs v = hi * 2^31 + lo (lo < 2^31,
// hi < 2^30) so that every partial product fits 62 bits and three of them can be
// summed in one uint64 before a single Mersenne fold (2^61 = 1, 2^62 = 2 mod p).
struct Limb {
  uint32_t lo, hi;
};

__device__ __forceinline__ Limb limb(uint64_t v) { return {uint32_t(v) & kM31, uint32_t(v >> 31)}; }
__device__ __forceinline__ uint64_t fold61(uint64_t v) { return (v & kP61) + (v >> 61); }
__device__ __forceinline__ uint64_t canon61(uint64_t v) { return v >= kP61 ? v - kP61 : v; }

// key -> residue of the sign-extended key mod p, in [0, p).  For k < 0 write
// k = -1 - m with m = ~k >= 0; then k mod p = p - 1 - (m mod p).
__device__ __forceinline__ uint64_t key_field(int64_t k) {
  const uint64_t s = uint64_t(k >> 63);
  const uint64_t m = uint64_t(k) ^ s;
  const uint64_t y = canon61(fold61(m));  // m < 2^64: fold < p + 8, one subtraction
  return s ? (kP61 - 1 - y) : y;
}

// (a * b) mod p from limbs.  t0 < 2^62, t1 < 2^62, t2 < 2^60 and
// a*b = t2 2^62 + t1 2^31 + t0 = 2 t2 + (t1 >> 30) + (t1 & (2^30-1)) 2^31 + t0 (mod p);
// the sum is < 2^63 + 2^32.
__device__ __forceinline__ uint64_t mulmod61(Limb a, Limb b) {
  const uint64_t t0 = uint64_t(a.lo) * b.lo;
  const uint64_t t1 = uint64_t(a.lo) * b.hi + uint64_t(a.hi) * b.lo;
  const uint64_t t2 = uint64_t(a.hi) * b.hi;
  const uint64_t s = t0 + (t1 >> 30) + ((t1 & kM30) << 31) + 2 * t2;
  return canon61(fold61(s));
}

// Hash parameters of one (edge, row), 16-aligned for shared-memory reads.
struct __align__(16) PairParam {
  uint64_t a, b, c0, c1, c2, c3;
};

__host__ __device__ inline PairParam make_pair_param(const cmp_hash& h) { return {h.a, h.b, h.c0, h.c1, h.c2, h.c3}; }

// Their coefficients in limbs, for the any-key forms.
struct __align__(16) PairLimb {
  Limb a, c1, c2, c3;
};
__device__ __forceinline__ PairLimb pair_limbs(const PairParam& q) {
  return {limb(q.a), limb(q.c1), limb(q.c2), limb(q.c3)};
}

// ---- Small keys: Horner steps of two multiplications, in two forms, kSmall29 for keys below
// 2^29 and kSmall31 for keys below 2^31 (every non-negative int32 key).
// sx_step: a value congruent to y x + c (mod p), below 2^64 - 8, for any y < 2^64 and c < 2^61.
// With y = yh 2^32 + yl and u = yh x, u 2^32 = (u >> 29) 2^61 + (u mod 2^29) 2^32 and 2^61 = 1:
//   y x + c = yl x + c + (u >> 29) + (u mod 2^29) 2^32,
// at most 2^63 + 2^61 + 2^34 + 2^61; the sum of one step is the next one's y as it is.  For x <
// 2^29, u >> 29 is the high word of yh (8 x), and u mod 2^29 the low word over 8.
// Bound by the integer ALU (64 lanes per cycle and SM, half the issue rate), so what counts is
// additions, shifts and masks; the carries are written out because the compiler's 64-bit sums
// took more of them.  Bucket and sign of a key, in registers: 389 G/s with every step's result
// folded below 2^61 + 8 (59 instructions), 430 G/s (kSmall31, 45), 550 G/s (kSmall29, 38).
enum KeyForm { kSmall29, kSmall31, kAnyKey };
template <int FORM>
__device__ __forceinline__ uint64_t sx_step(uint64_t y, uint32_t x, uint64_t c) {
  uint64_t s;
  if (FORM == kSmall29)
    asm("{\n\t.reg .u64 u, v;\n\t.reg .u32 yl, yh, ul, uh, vl, vh;\n\t"
        "mov.b64 {yl, yh}, %1;\n\t"
        "mul.wide.u32 u, yh, %4;\n\t"
        "mad.wide.u32 v, yl, %2, %3;\n\t"
        "mov.b64 {ul, uh}, u;\n\t"
        "mov.b64 {vl, vh}, v;\n\t"
        "shr.u32 ul, ul, 3;\n\t"
        "add.cc.u32 vl, vl, uh;\n\t"
        "addc.u32 vh, vh, ul;\n\t"
        "mov.b64 %0, {vl, vh};\n\t}"
        : "=l"(s)
        : "l"(y), "r"(x), "l"(c), "r"(x << 3));
  else
    asm("{\n\t.reg .u64 u, v;\n\t.reg .u32 yl, yh, ul, uh, vl, vh, t, m, h;\n\t"
        "mov.b64 {yl, yh}, %1;\n\t"
        "mul.wide.u32 u, yh, %2;\n\t"
        "mad.wide.u32 v, yl, %2, %3;\n\t"
        "mov.b64 {ul, uh}, u;\n\t"
        "mov.b64 {vl, vh}, v;\n\t"
        "shf.r.clamp.b32 t, ul, uh, 29;\n\t"
        "and.b32 m, ul, 0x1fffffff;\n\t"
        "shr.u32 h, uh, 29;\n\t"
        "add.u32 m, m, h;\n\t"
        "add.cc.u32 vl, vl, t;\n\t"
        "addc.u32 vh, vh, m;\n\t"
        "mov.b64 %0, {vl, vh};\n\t}"
        : "=l"(s)
        : "l"(y), "r"(x), "l"(c));
  return s;
}
// How often p goes into s < 2^64 - 8: s = q 2^61 + r = q p + (q + r), and q + r < 2p.  The
// residue is then s - k p = (s + k) mod 2^61.
__device__ __forceinline__ uint32_t sx_floor(uint64_t s) { return uint32_t((s + (s >> 61) + 1) >> 61); }

// Bucket ((a x + b) mod p) mod w of a small key (w a power of two divides 2^61).
template <bool POW2, int FORM>
__device__ __forceinline__ uint32_t sx_bucket(const PairParam& q, uint32_t x, uint32_t w) {
  const uint64_t s = sx_step<FORM>(q.a, x, q.b);
  const uint32_t k = sx_floor(s);
  if (POW2) return (uint32_t(s) + k) & (w - 1);
  return uint32_t(((s + k) & kP61) % w);
}
// Parity of (((c3 x + c2) x + c1) x + c0) mod p of a small key: 1 where the sign is -1.
template <int FORM>
__device__ __forceinline__ uint32_t sx_odd(const PairParam& q, uint32_t x) {
  uint64_t y = sx_step<FORM>(q.c3, x, q.c2);
  y = sx_step<FORM>(y, x, q.c1);
  y = sx_step<FORM>(y, x, q.c0);
  return (uint32_t(y) ^ sx_floor(y)) & 1u;  // p is odd
}
// The form every lane's keys fit, given the bits set in any of this lane's (active lanes only).
__device__ __forceinline__ int key_form(uint64_t bits) {
  const unsigned m = __activemask();
  if (__all_sync(m, (bits >> 29) == 0)) return kSmall29;
  return __all_sync(m, (bits >> 31) == 0) ? kSmall31 : kAnyKey;
}
// f(integral constant of the form); SMALL29: it may be kSmall29.
template <bool SMALL29 = true, typename F>
__device__ __forceinline__ void with_form(int form, F&& f) {
  if constexpr (SMALL29) {
    if (form == kSmall29) return f(std::integral_constant<int, kSmall29>{});
  }
  if (form == kSmall31) f(std::integral_constant<int, kSmall31>{});
  else f(std::integral_constant<int, kAnyKey>{});
}

// Powers of the key, shared by every (sketch, row) that hashes the same key.
struct KeyPow {
  Limb x, x2, x3;
};

__device__ __forceinline__ KeyPow key_powers(uint64_t x) {
  KeyPow k;
  k.x = limb(x);
  const uint64_t x2 = mulmod61(k.x, k.x);
  k.x2 = limb(x2);
  k.x3 = limb(mulmod61(k.x2, k.x));
  return k;
}

// Bucket: ((a x + b) mod p) mod w.  Sum bound: t0 + (t1>>30) + ((t1&M30)<<31) + 2 t2 + b
// < 2^62 + 2^32 + 3 * 2^61 < 2^64.
// The folded sums y are below 2^61 + 8 and congruent to the residue, which is y - p where y >= p;
// modulo a power of two that divides 2^61, and for the parity (p is odd), that is a bit
// added to y.  (Coefficients are split into limbs at each use, for the small-key steps take them
// whole.  2 M rows of keys near 2^45 in 64 x 64 partitions: 473 us with limbs stored, 494 split
// at each use with the residue formed, 486 like this.)
__device__ __forceinline__ uint32_t ge_p(uint64_t y) { return uint32_t((y + 1) >> 61); }  // 1 if y >= p, else 0
__device__ __forceinline__ uint64_t cw_bucket_fold(const PairParam& q, const PairLimb& l, const KeyPow& k) {
  const Limb a = l.a;
  const uint64_t t0 = uint64_t(a.lo) * k.x.lo;
  const uint64_t t1 = uint64_t(a.lo) * k.x.hi + uint64_t(a.hi) * k.x.lo;
  const uint64_t t2 = uint64_t(a.hi) * k.x.hi;
  const uint64_t s = t0 + (t1 >> 30) + ((t1 & kM30) << 31) + 2 * t2 + q.b;
  return fold61(s);
}
__device__ __forceinline__ uint64_t cw_bucket_residue(const PairParam& q, const PairLimb& l, const KeyPow& k) {
  return canon61(cw_bucket_fold(q, l, k));
}
template <bool POW2>
__device__ __forceinline__ uint32_t cw_bucket(const PairParam& q, const PairLimb& l, const KeyPow& k, uint32_t w) {
  const uint64_t y = cw_bucket_fold(q, l, k);
  if (POW2) return (uint32_t(y) + ge_p(y)) & (w - 1);
  return uint32_t(canon61(y) % w);
}

// Sign: parity of (c3 x^3 + c2 x^2 + c1 x + c0) mod p, as +1 / -1.  The three products
// are summed by limb position: S0 < 3 * 2^62, S1 < 6 * 2^61, S2 < 3 * 2^60, and
// fold(S0) + (S1>>30) + ((S1&M30)<<31) + 2 S2 + c0 < 6 * 2^61 + 2^35 < 2^64.
__device__ __forceinline__ uint64_t cw_sign_fold(const PairParam& q, const PairLimb& l, const KeyPow& k) {
  const Limb c1 = l.c1, c2 = l.c2, c3 = l.c3;
  const uint64_t S0 = uint64_t(c1.lo) * k.x.lo + uint64_t(c2.lo) * k.x2.lo + uint64_t(c3.lo) * k.x3.lo;
  const uint64_t S1 = uint64_t(c1.lo) * k.x.hi + uint64_t(c1.hi) * k.x.lo + uint64_t(c2.lo) * k.x2.hi +
                      uint64_t(c2.hi) * k.x2.lo + uint64_t(c3.lo) * k.x3.hi + uint64_t(c3.hi) * k.x3.lo;
  const uint64_t S2 = uint64_t(c1.hi) * k.x.hi + uint64_t(c2.hi) * k.x2.hi + uint64_t(c3.hi) * k.x3.hi;
  const uint64_t v = fold61(S0) + (S1 >> 30) + ((S1 & kM30) << 31) + 2 * S2 + q.c0;
  return fold61(v);
}
__device__ __forceinline__ uint64_t cw_sign_residue(const PairParam& q, const PairLimb& l, const KeyPow& k) {
  return canon61(cw_sign_fold(q, l, k));
}
__device__ __forceinline__ uint32_t cw_odd(const PairParam& q, const PairLimb& l, const KeyPow& k) {  // 1: the sign is -1
  const uint64_t y = cw_sign_fold(q, l, k);
  return (uint32_t(y) ^ ge_p(y)) & 1u;
}
__device__ __forceinline__ int cw_sign(const PairParam& q, const PairLimb& l, const KeyPow& k) {
  return 1 - 2 * int(cw_odd(q, l, k));
}

// ---- Horner form (one (sketch, row) pair per key: no powers to share).  The same two
// residues, (a x + b) mod p and (c3 x^3 + c2 x^2 + c1 x + c0) mod p = ((c3 x + c2) x + c1) x
// + c0, with intermediates kept only partly reduced: every step's result y satisfies
// y < 2^61 + 5 and y = the exact residue (mod p).
struct KeyX {
  uint32_t lo, hi, hi2;  // x < p as lo + hi 2^31 (lo < 2^31, hi < 2^30), hi2 = 2 hi
};
__device__ __forceinline__ KeyX key_x(uint64_t x) {
  return {uint32_t(x) & kM31, uint32_t(x >> 31), uint32_t(x >> 30) & ~1u};
}

// y x + c folded once, for y < 2^61 + 8 (ylo < 2^31, yhi <= 2^30), x < p, c < 2^61.
// y x = ylo xlo + (ylo xhi + yhi xlo) 2^31 + yhi xhi 2^62 and 2^62 = 2, 2^61 = 1 (mod p), so with
// t1 = ylo xhi + yhi xlo (< 2^62 + 2^31):
//   y x + c = ylo xlo + yhi (2 xhi) + c + (t1 >> 30) + (t1 & (2^30-1)) 2^31   (mod p),
// a sum below 2^62 + 2^61 + 2^61 + 2^33 + 2^61 < 2^64; one fold leaves it below 2^61 + 5.
__device__ __forceinline__ uint64_t mul_add_fold(Limb l, const KeyX& x, uint64_t c) {
  const uint64_t t1 = uint64_t(l.lo) * x.hi + uint64_t(l.hi) * x.lo;
  const uint64_t s = uint64_t(l.lo) * x.lo + uint64_t(l.hi) * x.hi2 + c + (t1 >> 30) + ((t1 & kM30) << 31);
  return fold61(s);
}

// Bucket ((a x + b) mod p) mod w; the same value as cw_bucket.  For w a power of two (w <=
// 2^31 divides 2^61), y - p = y + 1 (mod w).
template <bool POW2>
__device__ __forceinline__ uint32_t cw_bucket_h(const PairParam& q, const PairLimb& l, const KeyX& x, uint32_t w) {
  const uint64_t y = mul_add_fold(l.a, x, q.b);
  if (POW2) return (uint32_t(y) + ge_p(y)) & (w - 1);
  return uint32_t((ge_p(y) ? y - kP61 : y) % w);
}

// Sign: parity of ((c3 x + c2) x + c1) x + c0 mod p, as +1 / -1; the same value as cw_sign.
// The residue of the last y is y - p when y >= p, whose parity is flipped (p is odd).
__device__ __forceinline__ int cw_sign_h(const PairParam& q, const PairLimb& l, const KeyX& x) {
  uint64_t y = mul_add_fold(l.c3, x, q.c2);
  y = mul_add_fold(limb(y), x, q.c1);
  y = mul_add_fold(limb(y), x, q.c0);
  return 1 - 2 * int((uint32_t(y) ^ ge_p(y)) & 1u);
}

// Output r (0-based) of SplitMix64 (Steele, Lea & Flood 2014) seeded with `seed`: the
// generator's state after r + 1 steps, through its finaliser.
__host__ __device__ inline uint64_t splitmix64_at(uint64_t seed, uint64_t r) {
  uint64_t z = seed + (r + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Sample threshold of a rate: 0 (no sample) for 0 or 1, else floor(rate * 2^64), at least 1.
inline uint64_t sample_keep_of(double rate) {
  if (!(rate > 0.0 && rate < 1.0)) return 0;
  const uint64_t k = uint64_t(rate * 18446744073709551616.0);
  return k ? k : 1;
}

// ------------------------------------------------------------ build structures
struct DevPred {
  int32_t col, op;
  int64_t lo, hi;
  const uint32_t* bitmap;
  int64_t nbits;
};

struct DevTable {
  int64_t n_rows;
  int32_t n_cols, n_preds, n_sketches;
  int32_t vec_ok;  // every column 16-byte aligned: 128-bit loads allowed
  int32_t filtered;  // predicates or a row sample: tiles go through the survivor compaction
  int32_t surv_by;   // batched build: kernel that counts the survivors (kSurvRow / kSurvCount / kSurvUniq)
  uint64_t sample_seed, sample_keep;  // row r is sampled iff splitmix64_at(seed, r) < keep (keep 0: no sample)
  const void* col[CMP_MAX_COLS];
  int32_t dtype[CMP_MAX_COLS];
  DevPred pred[CMP_MAX_PREDS];
  int32_t key_col[CMP_MAX_SKETCHES];
  int32_t edge_id[CMP_MAX_SKETCHES];
  int32_t* counters;   // [n_sketches][d][w]
  int64_t* survivors;  // one int64
  int32_t agg[CMP_MAX_COLS];  // batched build: AggCol index of each aggregated key column, else -1
  uint32_t uniq_mask;         // batched build: key columns hashed by the unique-key kernel (bit c)
  int32_t pad1;
};
enum { kSurvRow = 0, kSurvCount = 1, kSurvUniq = 2 };

// Key aggregation of the batched build.  A key column of a large table is reduced to one
// (key, survivor count) entry per distinct key before hashing: the Fast-AGMS update is
// linear and the int32 counters wrap exactly, so count * xi(key) added once per entry
// gives the counters of one update per tuple.  The counting pass adds each surviving key
// to slot (key - base) & mask of the column's count array (cap slots, cleared before the
// pass) and records the smallest and largest surviving key.  Two layouts:
//  - declared domain [base, base + cap): mask = ~0; a key outside it marks the column as
//    out of range (its counts are then discarded);
//  - no declaration: cap is a power of two and mask = cap - 1, so any cap consecutive
//    keys occupy distinct slots.
// After the pass, a column whose surviving keys span at most cap values is "active" and
// its entries are hashed by k_agg_hash; otherwise it keeps the per-row path.  Workspace:
// [n_agg] x (max, min) encoded as uint64 pairs, then the chunk counters of the counting
// and hashing passes (two uint64; all zeroed before each build, 256-aligned area), then
// each column's int32 count array at byte offset `off`.
// A third kind, the presence bitmap, serves a unique key column with a declared domain in
// a table without predicates: the counting pass sets bit (key - base) of a bitmap instead
// of counting, and k_dense_hash walks the domain in key order.  A key outside the domain
// makes the column inactive, and so does a bitmap with fewer set bits than the table has
// rows (a key seen twice: the column is not unique after all), checked by
// k_presence_check; an inactive column keeps the per-row path.  After the bitmap's whole
// runs, its allocation holds the check's set-bit total and CTA ticket (PresenceCheck).
enum { kAggCount = 0, kAggPresence = 1 };
struct AggCol {
  int32_t table, col;
  int64_t cap;   // count slots (presence: domain keys)
  int64_t off;   // byte offset of the count array (presence: the bitmap) in the workspace
  int64_t base;  // key of slot 0 (declared domain) or 0
  uint64_t mask; // ~0 (declared domain) or cap - 1 (power of two)
  // hashing pass: the column's pairs are hashed in slabs of hash_pairs, and each slab's slots are
  // dealt to at most hash_groups items; its items begin at hash_item0
  int64_t hash_item0;
  int32_t kind;  // kAggCount / kAggPresence
  int32_t hash_pairs, hash_groups, hash_slabs;
};
// Hashing pass (k_agg_hash): threads, pairs of a slab at most, slots a warp reads at a time; the
// shared memory of a slab's counters (192 KB and one CTA per SM instead: 50 us more on five
// tables, 356 us instead of 295 on a batch of graphs); items per resident CTA, so that the
// CTAs end together: few where counters have to be written out (4 / 8 / 16: 123 / 132 / 144 us
// on the sparse counts of a 10% sample, 492 / 401 / 380 us on the dense ones of 48 joins), more
// where not (24 / 48: 637 / 490 us).
constexpr int kHashThreads = 512, kHashMaxPairs = 64;
constexpr int64_t kHashStep = 128;
constexpr int64_t kHashBudget = 76 << 10;      // two CTAs per SM
constexpr int64_t kHashItems = 6, kHashDirectItems = 48;
// Where that many items are too short for private counters, updates of few counters in global
// memory get in each other's way (3 M keys of a domain of 1 M, w = 1024, 5 pairs: 185 us), and
// fewer items with private ones pay (34 us): in plans of at most kHashFewCounters counters of
// counted columns (12 columns of 300,000 skewed keys, 61,000 counters: 55 us shared, 66 private)
// and for a key range of at least kHashFewRange (100,000 keys are too few for the CTAs: 10 us
// shared, 21 private).  Several slabs read the slots as often, so they also want two
// survivors for each (3 M keys, w = 4096, 5 pairs: 70 and 38 us; 1 M skewed ones 16 and 21).  The
// kernel of such plans is one of its own: the rule's registers cost the others 0.5%.
constexpr int64_t kHashFewCounters = 48 << 10, kHashFewRange = 1 << 18;
// Presence bitmaps are walked in runs of kDenseRun keys (8 words); a bitmap holds whole runs.
constexpr int64_t kDenseRun = 256;
__host__ __device__ inline int64_t presence_words(int64_t cap) { return (cap + kDenseRun - 1) / kDenseRun * (kDenseRun / 32); }
struct PresenceCheck {
  unsigned long long bits;  // set bits counted so far
  unsigned int ticket;      // CTAs done
  unsigned int pad;
};

// Order-preserving maps of an int64 to uint64, for atomicMax on the stats pairs (both
// zero-initialised: an empty column decodes as max < min).
__host__ __device__ inline uint64_t enc_max(int64_t v) { return uint64_t(v) ^ (1ull << 63); }
__host__ __device__ inline uint64_t enc_min(int64_t v) { return ~(uint64_t(v) ^ (1ull << 63)); }
__host__ __device__ inline int64_t dec_max(uint64_t e) { return int64_t(e ^ (1ull << 63)); }
__host__ __device__ inline int64_t dec_min(uint64_t e) { return int64_t(~e ^ (1ull << 63)); }

// Whether aggregated column `a` (index ai) takes the aggregated path in this run (read
// after the counting pass), with its smallest surviving key and key range (otherwise the
// first slot's key and an empty range: never another column's).
__host__ __device__ __forceinline__ bool agg_active(const AggCol& a, int ai, const unsigned char* ws, int64_t* kmin,
                                                    int64_t* range) {
  const unsigned long long* st = reinterpret_cast<const unsigned long long*>(ws) + 2 * int64_t(ai);
  const int64_t mx = dec_max(st[0]), mn = dec_min(st[1]);
  *kmin = a.base;
  *range = 0;
  if (mx < mn) return false;
  const uint64_t r = uint64_t(mx) - uint64_t(mn);
  if (r >= uint64_t(a.cap)) return false;
  *kmin = mn;
  *range = int64_t(r) + 1;
  return true;
}

// The keys kmin + j, begin <= j < end, of item `group` of a column's `groups` items of `len` keys
// each in the hashing pass.  Key kmin + j sits in slot (kmin - base + j) & mask, and a load
// takes four slots from a multiple of four (count arrays are whole int4 words, a masked one at
// least 8 slots), so the first item begins at j = -((kmin - base) & 3).  A column without a
// range (inactive) has no items: its kmin says nothing about its array.
struct HashSpan {
  int64_t begin, end;
};
__host__ __device__ __forceinline__ HashSpan hash_span(const AggCol& a, int64_t kmin, int64_t range, int64_t len,
                                                       int group, int groups) {
  if (range <= 0 || group >= groups) return {0, 0};
  const int64_t begin = group * len - int64_t((uint64_t(kmin) - uint64_t(a.base)) & 3);
  return {begin, begin + len < range ? begin + len : range};
}

// Unique key columns (declared distinct, e.g. primary keys) of the batched build: no key
// repeats, so aggregation cannot reduce the hashing.  k_uniq_hash hashes each surviving
// row once per (sketch, row) pair with a slab of the column's pairs held in shared
// memory.  A slab is up to kUniqMaxPairs pairs of one column; an item is one slab over a
// range of the table's rows.
constexpr int32_t kUniqMaxPairs = 32;
struct UniqSlab {
  int32_t table, col, n_pairs, pad;
  int32_t pair[kUniqMaxPairs];  // pair = sketch * d + row of the table
};
struct UniqItem {
  int32_t slab, count_surv;  // count_surv: this item adds its range's survivors to the table's count
  int64_t row_begin, row_end;
};
// k_dense_hash reuses both: a slab's pad is the AggCol index of its presence column, and an
// item's [row_begin, row_end) is a range of domain offsets (key - base), whole runs.

// One (table, slab of (sketch,row) pairs) handled by n_ctas consecutive CTAs walking tiles
// of the table's rows (aggregated key columns are hashed by k_agg_hash instead).
struct BuildItem {
  int32_t table;
  int32_t pair_begin, pair_end;
  int32_t n_ctas;
  int32_t first_cta;
  int32_t pad;
};

// Counting pass of key aggregation: the rows of one table as chunks [chunk_begin,
// chunk_begin + n_chunks) of the pass's global chunk sequence (chunk_rows each), handed out
// to the persistent CTAs in order by an atomic counter.
struct CountItem {
  int32_t table, cache_slots;  // cache_slots: hot-key cache slots per column (a power of two)
  int64_t chunk_begin, n_chunks;
  int64_t chunk_rows;  // a multiple of 4 tiles
};

struct BuildShape {
  int32_t mode;            // 1 smem, 2 global
  int32_t dedupe;          // 0 / 1
  int32_t threads;
  int32_t tile_rows;
  int32_t map_slots;       // power of two >= 2 * tile_rows (dedupe only)
  int32_t max_pairs;       // max pairs of any item (sizes the parameter area)
  int32_t smem_pairs;      // pairs whose counters live in shared memory (mode 1)
  int32_t pairs_per_slab;  // single-table launches
  int32_t ctas_per_slab;   // single-table launches
  int32_t grid;
  size_t smem_bytes;
};

struct BuildArgs {
  DevTable table;             // single-table launch (items == nullptr)
  const DevTable* tables;     // batched launch
  const BuildItem* items;
  const int32_t* cta_item;    // [grid] item of each CTA
  const cmp_hash* hash;       // [n_edges * d]
  int32_t* status;
  int32_t d, w, n_edges;
  int32_t threads, tile_rows, map_slots, max_pairs, smem_pairs;
  int32_t pairs_per_slab, ctas_per_slab;
  const AggCol* agg;  // key aggregation (batched build only)
  int32_t n_agg;
  unsigned char* ws;
  const CountItem* cnt_items;
  int32_t n_cnt_items;
  int32_t cnt_work_slot;                      // chunk counter of this launch of the counting pass
  int64_t cnt_chunk_begin, cnt_chunk_end;     // its chunks
  int32_t cnt_cache_slots, cnt_cache_cols;  // counting pass: hot-key cache slots per column, columns cached
  int64_t cnt_total_chunks;
  int64_t hash_items;   // hashing pass of the aggregated columns: its items,
  int32_t hash_private;  // words of the CTA's own counters (0: counters in global memory)
  int32_t hash_few;      // 1: at most kHashFewCounters counters
  // unique-key kernel
  const UniqSlab* uslab;
  const UniqItem* uitem;
  const int32_t* u_cta_item;  // [grid + 1] first item of each CTA
  int64_t n_uitems;
  int32_t u_pack16;  // 1: one pair per slab, counters as two 16-bit halves per word
  int32_t u_words;   // shared-memory counter words of a slab
  // dense (presence-bitmap) kernel: slabs, items and CTA map as for the unique-key kernel
  const UniqSlab* dslab;
  const UniqItem* ditem;
  const int32_t* d_cta_item;
  int64_t n_ditems;
  int32_t d_pack16, d_words;
  // the dense kernel's share of each item's runs: 0 all; 1 the first ceil(n d_cut / 1024);
  // 2 the rest
  int32_t dense_part, dense_cut;
};

// Plan blob (host-encoded, device-read) for the batched build.
struct BuildPlanHdr {
  uint64_t magic;
  int32_t version, n_tables, n_items, d, w, n_edges;
  BuildShape shape;
  int64_t off_tables, off_items, off_cta_item, off_zero, n_zero;  // byte offsets in the blob
  int64_t total_bytes;
  int64_t n_agg, off_agg;                            // aggregated key columns
  int64_t n_cnt_items, off_cnt_items, cnt_total_chunks;  // counting pass
  int32_t cnt_grid[4], cnt_threads;  // CTAs of each launch of the counting pass (kCnt*)
  int64_t ws_bytes;
  int32_t cnt_cache_slots, cnt_cache_cols;
  int64_t hash_items;
  int32_t hash_private;
  int32_t hash_grid;
  int64_t n_uslab, off_uslab, n_uitems, off_uitems, off_u_cta;  // unique-key kernel
  int32_t u_grid, u_pack16, u_words, u_tile_rows;
  int64_t n_dslab, off_dslab, n_ditems, off_ditems, off_d_cta;  // dense kernel
  int32_t d_grid, d_pack16, d_words, n_presence;
  // split counting pass (cnt_split > 0): chunks [0, cnt_split) of the tables with presence
  // columns first, then [cnt_split, total) with the dense kernel beside their last launch
  int64_t cnt_split;
  // split pass: the dense kernel walks the first d_cut / 1024 of each item's runs beside the
  // last counting launch, the rest after it with 512 threads (d_cut = 1024: all beside)
  int32_t d_cut, hash_few;  // (hash_few: of the hashing pass)
  // chunks: tables with presence columns and without a selection, from cnt_sampled on tables with a
  // row sample only (k_count_rows), from cnt_filtered on tables with predicates (k_agg_count)
  int64_t cnt_sampled;
  int64_t cnt_filtered;
};
constexpr int32_t kBuildPlanVersion = 14;
// Launches of the counting pass: tables with presence columns (of a split pass; else they are
// counted with the whole ones), every row, a row sample, predicates.
enum { kCntPresence = 0, kCntWhole = 1, kCntSampled = 2, kCntFiltered = 3 };
struct ZeroSpan {
  void* ptr;
  int64_t bytes;
};
constexpr uint64_t kBuildPlanMagic = 0x434d504255494c44ull;  // "CMPBUILD"

// Fire-and-forget atomic additions (PTX red, relaxed): the same update as atomicAdd, with
// no result register, so no instruction waits for the reply.
__device__ __forceinline__ void red_or(uint32_t* p, uint32_t v) {
  asm volatile("red.relaxed.gpu.global.or.b32 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void red_add(int32_t* p, int32_t v) {
  asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void red_add_shared(int32_t* p, int32_t v) {
  asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(uint32_t(__cvta_generic_to_shared(p))), "r"(v) : "memory");
}
__device__ __forceinline__ void red_add_shared(uint32_t* p, uint32_t v) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(uint32_t(__cvta_generic_to_shared(p))), "r"(v) : "memory");
}

// device status helper: first error wins
__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
  if (status) atomicCAS(status, 0, code);
}

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// launchers implemented in the .cu files
size_t build_smem_bytes(const BuildShape& s, int w);
cudaError_t launch_build(const BuildArgs& a, const BuildShape& s, cudaStream_t st);
size_t agg_count_smem_bytes(int32_t tile_rows, int32_t cache_slots, int32_t cache_cols, int32_t threads);
cudaError_t launch_agg_zero(const BuildArgs& a, cudaStream_t st);
cudaError_t launch_presence_check(const BuildArgs& a, cudaStream_t st);
cudaError_t launch_agg_count(const BuildArgs& a, int32_t tile_rows, int32_t cnt_threads, int32_t cnt_grid,
                             int32_t work_slot, int64_t chunk_begin, int64_t chunk_end, cudaStream_t st);
cudaError_t launch_count_rows(const BuildArgs& a, bool sampled, int32_t grid, int32_t work_slot, int64_t chunk_begin,
                              int64_t chunk_end, cudaStream_t st);
size_t uniq_smem_bytes(int32_t words, int32_t tile_rows);
cudaError_t launch_uniq(const BuildArgs& a, int32_t grid, int32_t threads, int32_t tile_rows, cudaStream_t st);
cudaError_t launch_zero_spans(const ZeroSpan* spans_dev, int32_t n, cudaStream_t st);
cudaError_t launch_agg_hash(const BuildArgs& a, int32_t grid, cudaStream_t st);
size_t dense_smem_bytes(int32_t words);
cudaError_t launch_dense(const BuildArgs& a, int32_t grid, bool pdl, int32_t threads, cudaStream_t st);
constexpr int32_t kDenseThreadsAlone = 512, kDenseThreadsBeside = 256;

int sm_count();
size_t smem_optin_bytes();

// Dynamic shared memory beyond 48 KB has to be allowed per kernel, and the limit is the
// process's, not the call's: set to what one call needs, it could be lowered by another host
// thread's smaller call before this one's launch, which then failed.  So every call allows the
// most the kernel can be given, the same value each time (one object per kernel; a failed
// query is not kept).
class SmemLimit {
 public:
  template <typename... A>
  cudaError_t allow(void (*kernel)(A...)) {
    const void* const f = reinterpret_cast<const void*>(kernel);
    int n = most_.load(std::memory_order_relaxed);
    if (n == 0) {
      cudaFuncAttributes a;
      const cudaError_t e = cudaFuncGetAttributes(&a, f);
      if (e != cudaSuccess) return e;
      n = int(smem_optin_bytes()) - int(a.sharedSizeBytes);
      most_.store(n, std::memory_order_relaxed);
    }
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
  }

 private:
  std::atomic<int> most_{0};
};
// host checks and device descriptor of one cmp_table (api_build.cu)
cmp_status check_table(const cmp_table* t, int32_t d, int32_t w, int32_t n_edges);
DevTable to_dev(const cmp_table* t, int32_t* counters, int64_t* survivors);

}  // namespace cmpk
