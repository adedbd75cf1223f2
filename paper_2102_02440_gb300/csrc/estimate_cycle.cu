// Cyclic sub-plans whose tables form one simple cycle (four or more tables, each joined to its
// two neighbours): the row estimate without one block-wide tree contraction per conditioning
// value.
//
// With M_t[j][k] the merged sketch of table t (its sketch value on the cycle's edge before t
// at bucket j, or on the edge after t at bucket k, whichever has the smaller magnitude, the
// lower edge id on ties; Sec. 4.2), the row estimate is the trace of the product of the n
// matrices M_t along the cycle.  Three facts make it cheap:
//  - Row M_0[j] of the first table depends on its sketch value v at bucket j only, so buckets
//    with equal v share the whole product vector x_v = M_0[j] M_1 ... M_{n-1}; the trace is
//    the sum over the distinct nonzero values v of x_v summed over v's buckets.  The cycle is
//    cut at the sketch (of its 2n) with the fewest distinct magnitudes, in either direction.
//  - x M_t is one pass over the merged order of the table's two sorted sketches: with P0 and
//    P1 the prefix sums of x and of a x in a's sorted order (a: the sketch on the incoming
//    edge), out[k] = p_k (total - P0[q]) + P1[q] at p_k's cross rank q.
//  - Everything is a ring expression in the counters, so it is exact modulo 2^(32 L) for
//    any L with |E| < 2^(32 L - 1): values are L-limb two's complement integers, L chosen per
//    row from the bound |E| <= prod_t sum_j min(|a_j|, max |p|) (the infinity norms).  Rows
//    beyond int128 come out exact as well; the exact tier only turns them into residues.
// Layout: a CTA of 256 or 512 threads holds C product vectors (columns) in shared memory, two
// buffers [w][C][L]; thread = (segment, column), the segments cutting the merged order of 2 w
// steps evenly (merge path), so a segment's running sums start from a scan over the
// segments.  The integers bound it (about 12 L + 20 instructions per merged pair and column),
// not the barriers: three per operation.
// Before: one contraction per conditioning value, a block scan per table each, and once more
// per prime for the rows beyond int128.  The cycles of 4, 5, 15 and 17 tables of a batch at
// w = 1024, d = 11: 74 ms of estimate kernels before, 1.4 ms now (0.85 here).
// A row whose L does not fit keeps the generic path (k_estimate_items), decided on the device;
// so does, in the plan, a cycle with w > kCycMaxW or with fewer conditioning chunks than
// kCycRowItems (a row's state is kept in their partial sums): w <= 7 cond_chunk, which is w <= 448
// at the default of 64 values.
#include <cuda_runtime.h>

#include <algorithm>

#include "est_arith.cuh"

namespace cmpk {
namespace {

// L-limb (32-bit) integers modulo 2^(32 L): a += b, a -= b, a -= b 2^32, a += b m, each one
// carry chain (the product as two chains of low / high pairs: even limbs, then odd).
template <int L>
struct Limbs;
template <> struct Limbs<2> {
  static __device__ __forceinline__ void add(uint32_t (&a)[2], const uint32_t (&b)[2]) {
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+r"(a[0]), "+r"(a[1]) : "r"(b[0]), "r"(b[1]));
  }
  static __device__ __forceinline__ void sub(uint32_t (&a)[2], const uint32_t (&b)[2]) {
    asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %3;" : "+r"(a[0]), "+r"(a[1]) : "r"(b[0]), "r"(b[1]));
  }
  static __device__ __forceinline__ void sub_shift(uint32_t (&a)[2], const uint32_t (&b)[2]) {
    asm("sub.u32 %0, %0, %1;" : "+r"(a[1]) : "r"(b[0]));
  }
  static __device__ __forceinline__ void mad(uint32_t (&a)[2], const uint32_t (&b)[2], uint32_t m) {
    asm(
        "mad.lo.cc.u32 %0, %2, %4, %0;\n\tmadc.hi.u32 %1, %2, %4, %1;\n\tmad.lo.u32 %1, %3, %4, %1;"
        : "+r"(a[0]), "+r"(a[1])
        : "r"(b[0]), "r"(b[1]), "r"(m));
  }
};
template <> struct Limbs<4> {
  static __device__ __forceinline__ void add(uint32_t (&a)[4], const uint32_t (&b)[4]) {
    asm(
        "add.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\taddc.cc.u32 %2, %2, %6;\n\taddc.u32 %3, %3, %7;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]));
  }
  static __device__ __forceinline__ void sub(uint32_t (&a)[4], const uint32_t (&b)[4]) {
    asm(
        "sub.cc.u32 %0, %0, %4;\n\tsubc.cc.u32 %1, %1, %5;\n\tsubc.cc.u32 %2, %2, %6;\n\tsubc.u32 %3, %3, %7;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]));
  }
  static __device__ __forceinline__ void sub_shift(uint32_t (&a)[4], const uint32_t (&b)[4]) {
    asm(
        "sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %4;\n\tsubc.u32 %2, %2, %5;"
        : "+r"(a[1]), "+r"(a[2]), "+r"(a[3])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]));
  }
  static __device__ __forceinline__ void mad(uint32_t (&a)[4], const uint32_t (&b)[4], uint32_t m) {
    asm(
        "mad.lo.cc.u32 %0, %4, %8, %0;\n\tmadc.hi.cc.u32 %1, %4, %8, %1;\n\tmadc.lo.cc.u32 %2, %6, %8, %2;\n\t"
        "madc.hi.u32 %3, %6, %8, %3;\n\tmad.lo.cc.u32 %1, %5, %8, %1;\n\tmadc.hi.cc.u32 %2, %5, %8, %2;\n\t"
        "madc.lo.u32 %3, %7, %8, %3;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(m));
  }
};
template <> struct Limbs<6> {
  static __device__ __forceinline__ void add(uint32_t (&a)[6], const uint32_t (&b)[6]) {
    asm(
        "add.cc.u32 %0, %0, %6;\n\taddc.cc.u32 %1, %1, %7;\n\taddc.cc.u32 %2, %2, %8;\n\t"
        "addc.cc.u32 %3, %3, %9;\n\taddc.cc.u32 %4, %4, %10;\n\taddc.u32 %5, %5, %11;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]));
  }
  static __device__ __forceinline__ void sub(uint32_t (&a)[6], const uint32_t (&b)[6]) {
    asm(
        "sub.cc.u32 %0, %0, %6;\n\tsubc.cc.u32 %1, %1, %7;\n\tsubc.cc.u32 %2, %2, %8;\n\t"
        "subc.cc.u32 %3, %3, %9;\n\tsubc.cc.u32 %4, %4, %10;\n\tsubc.u32 %5, %5, %11;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]));
  }
  static __device__ __forceinline__ void sub_shift(uint32_t (&a)[6], const uint32_t (&b)[6]) {
    asm(
        "sub.cc.u32 %0, %0, %5;\n\tsubc.cc.u32 %1, %1, %6;\n\tsubc.cc.u32 %2, %2, %7;\n\t"
        "subc.cc.u32 %3, %3, %8;\n\tsubc.u32 %4, %4, %9;"
        : "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]));
  }
  static __device__ __forceinline__ void mad(uint32_t (&a)[6], const uint32_t (&b)[6], uint32_t m) {
    asm(
        "mad.lo.cc.u32 %0, %6, %12, %0;\n\tmadc.hi.cc.u32 %1, %6, %12, %1;\n\t"
        "madc.lo.cc.u32 %2, %8, %12, %2;\n\tmadc.hi.cc.u32 %3, %8, %12, %3;\n\t"
        "madc.lo.cc.u32 %4, %10, %12, %4;\n\tmadc.hi.u32 %5, %10, %12, %5;\n\tmad.lo.cc.u32 %1, %7, %12, %1;\n\t"
        "madc.hi.cc.u32 %2, %7, %12, %2;\n\tmadc.lo.cc.u32 %3, %9, %12, %3;\n\t"
        "madc.hi.cc.u32 %4, %9, %12, %4;\n\tmadc.lo.u32 %5, %11, %12, %5;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(m));
  }
};
template <> struct Limbs<8> {
  static __device__ __forceinline__ void add(uint32_t (&a)[8], const uint32_t (&b)[8]) {
    asm(
        "add.cc.u32 %0, %0, %8;\n\taddc.cc.u32 %1, %1, %9;\n\taddc.cc.u32 %2, %2, %10;\n\t"
        "addc.cc.u32 %3, %3, %11;\n\taddc.cc.u32 %4, %4, %12;\n\taddc.cc.u32 %5, %5, %13;\n\t"
        "addc.cc.u32 %6, %6, %14;\n\taddc.u32 %7, %7, %15;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  }
  static __device__ __forceinline__ void sub(uint32_t (&a)[8], const uint32_t (&b)[8]) {
    asm(
        "sub.cc.u32 %0, %0, %8;\n\tsubc.cc.u32 %1, %1, %9;\n\tsubc.cc.u32 %2, %2, %10;\n\t"
        "subc.cc.u32 %3, %3, %11;\n\tsubc.cc.u32 %4, %4, %12;\n\tsubc.cc.u32 %5, %5, %13;\n\t"
        "subc.cc.u32 %6, %6, %14;\n\tsubc.u32 %7, %7, %15;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  }
  static __device__ __forceinline__ void sub_shift(uint32_t (&a)[8], const uint32_t (&b)[8]) {
    asm(
        "sub.cc.u32 %0, %0, %7;\n\tsubc.cc.u32 %1, %1, %8;\n\tsubc.cc.u32 %2, %2, %9;\n\t"
        "subc.cc.u32 %3, %3, %10;\n\tsubc.cc.u32 %4, %4, %11;\n\tsubc.cc.u32 %5, %5, %12;\n\t"
        "subc.u32 %6, %6, %13;"
        : "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]));
  }
  static __device__ __forceinline__ void mad(uint32_t (&a)[8], const uint32_t (&b)[8], uint32_t m) {
    asm(
        "mad.lo.cc.u32 %0, %8, %16, %0;\n\tmadc.hi.cc.u32 %1, %8, %16, %1;\n\t"
        "madc.lo.cc.u32 %2, %10, %16, %2;\n\tmadc.hi.cc.u32 %3, %10, %16, %3;\n\t"
        "madc.lo.cc.u32 %4, %12, %16, %4;\n\tmadc.hi.cc.u32 %5, %12, %16, %5;\n\t"
        "madc.lo.cc.u32 %6, %14, %16, %6;\n\tmadc.hi.u32 %7, %14, %16, %7;\n\tmad.lo.cc.u32 %1, %9, %16, %1;\n\t"
        "madc.hi.cc.u32 %2, %9, %16, %2;\n\tmadc.lo.cc.u32 %3, %11, %16, %3;\n\t"
        "madc.hi.cc.u32 %4, %11, %16, %4;\n\tmadc.lo.cc.u32 %5, %13, %16, %5;\n\t"
        "madc.hi.cc.u32 %6, %13, %16, %6;\n\tmadc.lo.u32 %7, %15, %16, %7;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(m));
  }
};
template <> struct Limbs<10> {
  static __device__ __forceinline__ void add(uint32_t (&a)[10], const uint32_t (&b)[10]) {
    asm(
        "add.cc.u32 %0, %0, %10;\n\taddc.cc.u32 %1, %1, %11;\n\taddc.cc.u32 %2, %2, %12;\n\t"
        "addc.cc.u32 %3, %3, %13;\n\taddc.cc.u32 %4, %4, %14;\n\taddc.cc.u32 %5, %5, %15;\n\t"
        "addc.cc.u32 %6, %6, %16;\n\taddc.cc.u32 %7, %7, %17;\n\taddc.cc.u32 %8, %8, %18;\n\t"
        "addc.u32 %9, %9, %19;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
          "+r"(a[8]), "+r"(a[9])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(b[8]),
          "r"(b[9]));
  }
  static __device__ __forceinline__ void sub(uint32_t (&a)[10], const uint32_t (&b)[10]) {
    asm(
        "sub.cc.u32 %0, %0, %10;\n\tsubc.cc.u32 %1, %1, %11;\n\tsubc.cc.u32 %2, %2, %12;\n\t"
        "subc.cc.u32 %3, %3, %13;\n\tsubc.cc.u32 %4, %4, %14;\n\tsubc.cc.u32 %5, %5, %15;\n\t"
        "subc.cc.u32 %6, %6, %16;\n\tsubc.cc.u32 %7, %7, %17;\n\tsubc.cc.u32 %8, %8, %18;\n\t"
        "subc.u32 %9, %9, %19;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
          "+r"(a[8]), "+r"(a[9])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(b[8]),
          "r"(b[9]));
  }
  static __device__ __forceinline__ void sub_shift(uint32_t (&a)[10], const uint32_t (&b)[10]) {
    asm(
        "sub.cc.u32 %0, %0, %9;\n\tsubc.cc.u32 %1, %1, %10;\n\tsubc.cc.u32 %2, %2, %11;\n\t"
        "subc.cc.u32 %3, %3, %12;\n\tsubc.cc.u32 %4, %4, %13;\n\tsubc.cc.u32 %5, %5, %14;\n\t"
        "subc.cc.u32 %6, %6, %15;\n\tsubc.cc.u32 %7, %7, %16;\n\tsubc.u32 %8, %8, %17;"
        : "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]), "+r"(a[8]),
          "+r"(a[9])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(b[8]));
  }
  static __device__ __forceinline__ void mad(uint32_t (&a)[10], const uint32_t (&b)[10], uint32_t m) {
    asm(
        "mad.lo.cc.u32 %0, %10, %20, %0;\n\tmadc.hi.cc.u32 %1, %10, %20, %1;\n\t"
        "madc.lo.cc.u32 %2, %12, %20, %2;\n\tmadc.hi.cc.u32 %3, %12, %20, %3;\n\t"
        "madc.lo.cc.u32 %4, %14, %20, %4;\n\tmadc.hi.cc.u32 %5, %14, %20, %5;\n\t"
        "madc.lo.cc.u32 %6, %16, %20, %6;\n\tmadc.hi.cc.u32 %7, %16, %20, %7;\n\t"
        "madc.lo.cc.u32 %8, %18, %20, %8;\n\tmadc.hi.u32 %9, %18, %20, %9;\n\t"
        "mad.lo.cc.u32 %1, %11, %20, %1;\n\tmadc.hi.cc.u32 %2, %11, %20, %2;\n\t"
        "madc.lo.cc.u32 %3, %13, %20, %3;\n\tmadc.hi.cc.u32 %4, %13, %20, %4;\n\t"
        "madc.lo.cc.u32 %5, %15, %20, %5;\n\tmadc.hi.cc.u32 %6, %15, %20, %6;\n\t"
        "madc.lo.cc.u32 %7, %17, %20, %7;\n\tmadc.hi.cc.u32 %8, %17, %20, %8;\n\tmadc.lo.u32 %9, %19, %20, %9;"
        : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
          "+r"(a[8]), "+r"(a[9])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(b[8]),
          "r"(b[9]), "r"(m));
  }
};

constexpr int kCycThreads = 256;       // two CTAs per SM
constexpr int kCycWideThreads = 512;   // one
constexpr int kCycBlk = 16;     // sorted positions of the cut sketch per job
constexpr int kCycMaxCols = 8;

// Shared memory of k_cycle: two buffers of product vectors, then the operation's two sorted
// sketches: a as (bucket, value), p as (bucket, value), p's cross ranks in a.
__host__ __device__ inline size_t cyc_fixed_bytes(int w) { return align16(size_t(20) * size_t(w)); }
__host__ __device__ inline size_t cyc_col_bytes(int w, int L) { return size_t(2) * size_t(w) * size_t(L) * 4; }
// (5 KB of static shared memory beside it) Two CTAs per SM while a column of eight limbs fits
// beside the sketches, else one.
__host__ __device__ inline bool cyc_two_per_sm(int w) {
  return cyc_fixed_bytes(w) + cyc_col_bytes(w, 8) <= size_t(104) * 1024;
}
__host__ __device__ inline size_t cyc_smem_bytes(int w) {
  return cyc_two_per_sm(w) ? size_t(104) * 1024 : size_t(220) * 1024;
}
// Columns per CTA for L limbs: a power of two, 0 when not even one fits.
__device__ __forceinline__ int cyc_cols(int w, int L) {
  const size_t room = cyc_smem_bytes(w);
  if (cyc_fixed_bytes(w) >= room) return 0;
  int c = int((room - cyc_fixed_bytes(w)) / cyc_col_bytes(w, L));
  c = c > kCycMaxCols ? kCycMaxCols : c;
  while (c & (c - 1)) c &= c - 1;
  return c;
}
__device__ __forceinline__ int cyc_limbs(double bits) {  // fewest limbs with |E| < 2^(32 L - 1); 0: too many
  for (int L = 2; L <= kCycMaxLimbs; L += 2)
    if (bits < double(32 * L - 1)) return L;
  return 0;
}

// The sketches of position t of the cycle walked from `start` in direction `back`: the one on
// the edge it is entered by, and the one on the edge it is left by.
__device__ __forceinline__ const EstIn* cyc_in(const EstArgs& A, const CycSub& cs, int start, int back, int t,
                                               int leaving) {
  const int n = cs.n, pos = back ? (start + n - t) % n : (start + t) % n;
  return A.inputs + cs.in_begin + 2 * pos + (leaving ^ back);
}

// One CTA per (cycle, sketch row): where to cut the cycle, the limbs its row needs, and the
// row's state (CycRow) cleared.  A warp per sketch counts distinct magnitudes.
__global__ void __launch_bounds__(1024) k_cycle_prep(const __grid_constant__ EstArgs A) {
  __shared__ int distinct[2 * CMP_MAX_TABLES];
  __shared__ double bits[2 * CMP_MAX_TABLES];
  __shared__ int s_ok;
  const CycSub cs = A.cyc[blockIdx.x / A.d];
  const int row = int(blockIdx.x % A.d), w = A.w;
  const int64_t ro = int64_t(row) * w;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = warp; q < 2 * cs.n; q += 32) {
    const EstIn& x = A.inputs[cs.in_begin + q];
    const uint32_t* abs = x.abs + ro;
    const uint32_t cap = __ldg(A.inputs[cs.in_begin + (q ^ 1)].abs + ro + w - 1);  // the other sketch's largest
    int n = 0;
    uint64_t sum = 0;
    for (int r = lane; r < w; r += 32) {
      const uint32_t v = __ldg(abs + r);
      n += v != 0 && (r == 0 || __ldg(abs + r - 1) != v);
      sum += min(v, cap);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n += __shfl_xor_sync(0xffffffffu, n, o);
      sum += __shfl_xor_sync(0xffffffffu, (unsigned long long)sum, o);
    }
    if (lane == 0) {
      distinct[q] = n;
      bits[q] = sum ? log2(double(sum)) + 1e-9 : 0.0;
    }
  }
  __syncthreads();
  const EstSub& sb = A.subs[cs.sub];
  const int64_t it0 = sb.item_begin + int64_t(row) * sb.n_chunks;
  if (threadIdx.x == 0) {
    double fwd = 0.0, bwd = 0.0;  // infinity norms entered by sketch 2t, or by 2t + 1
    int best = 0;
    for (int t = 0; t < cs.n; t++) {
      fwd += bits[2 * t];
      bwd += bits[2 * t + 1];
    }
    for (int q = 1; q < 2 * cs.n; q++)
      if (distinct[q] < distinct[best]) best = q;
    const int L = cyc_limbs(min(fwd, bwd) + 0.01);
    const int C = L ? cyc_cols(w, L) : 0;
    CycRow* cr = cyc_row(A, it0);
    for (int l = 0; l < kCycMaxLimbs; l++) cr->acc[l] = 0;
    cr->limbs = L;
    cr->cols = C;
    cr->start = best >> 1;
    cr->back = best & 1;
    s_ok = C > 0;
  }
  __syncthreads();
  for (int ch = threadIdx.x; ch < sb.n_chunks; ch += blockDim.x) A.partial_ovf[it0 + ch] = s_ok ? kCycDone : 0;
}

// One operation's walk state of a thread: the prefix of its column over a's sorted order.
template <int L>
struct CycSum {
  uint32_t x[L], neg[L], ax[L];  // sums of x, of x where a < 0, of (a mod 2^32) x
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int l = 0; l < L; l++) x[l] = neg[l] = ax[l] = 0;
  }
  __device__ __forceinline__ void step(const uint32_t (&v)[L], int32_t a) {
    Limbs<L>::add(x, v);
    Limbs<L>::mad(ax, v, uint32_t(a));
    if (a < 0) Limbs<L>::add(neg, v);  // a x = (a mod 2^32) x - 2^32 x
  }
};

template <int L>
__device__ __forceinline__ void cyc_load(const uint32_t* p, uint32_t (&v)[L]) {
#pragma unroll
  for (int l = 0; l < L; l += 2) {
    const uint2 u = *reinterpret_cast<const uint2*>(p + l);
    v[l] = u.x;
    v[l + 1] = u.y;
  }
}
template <int L>
__device__ __forceinline__ void cyc_store(uint32_t* p, const uint32_t (&v)[L]) {
#pragma unroll
  for (int l = 0; l < L; l += 2) *reinterpret_cast<uint2*>(p + l) = make_uint2(v[l], v[l + 1]);
}

// The product vectors of the values vals[0..n_val) of the cut sketch (C at a time), and the
// trace's share of them added to the row's accumulators.
template <int L, int T>
__device__ __noinline__ void cyc_run(const EstArgs& A, const CycSub& cs, int row, const CycRow& cr, CycRow* out,
                                     const int32_t* vals, int n_val, unsigned char* smem, uint32_t* tot) {
  const int w = A.w, C = cr.cols, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = T / 32;
  const int nseg = T / C, c = tid & (C - 1), seg = tid / C;
  const int64_t ro = int64_t(row) * w;
  uint32_t* X = reinterpret_cast<uint32_t*>(smem);
  uint32_t* Y = X + size_t(w) * C * L;
  int2* sa = reinterpret_cast<int2*>(smem + size_t(C) * cyc_col_bytes(w, L));
  int2* sp = sa + w;
  int32_t* sq = reinterpret_cast<int32_t*>(sp + w);
  const EstIn* cut = cyc_in(A, cs, cr.start, cr.back, 0, 0);
  uint32_t E[L];
#pragma unroll
  for (int l = 0; l < L; l++) E[l] = 0;
  for (int v0 = 0; v0 < n_val; v0 += C) {
    const bool live = v0 + c < n_val;
    const int32_t val = live ? vals[v0 + c] : 0;
    {  // the first table: row M_0[j] of a bucket with value val (0: a zero column)
      const EstIn* p = cyc_in(A, cs, cr.start, cr.back, 0, 1);
      const uint32_t m = val < 0 ? uint32_t(-int64_t(val)) : uint32_t(val);
      const bool first = cut->slot < p->slot;  // the cut sketch wins ties
      for (int k = seg; k < w; k += nseg) {
        const int32_t s = __ldg(p->s + ro + k);
        const uint32_t ms = s < 0 ? uint32_t(-int64_t(s)) : uint32_t(s);
        const int32_t e = (first ? m <= ms : m < ms) ? val : s;
        uint32_t v[L];
        v[0] = live ? uint32_t(e) : 0u;
#pragma unroll
        for (int l = 1; l < L; l++) v[l] = live && e < 0 ? ~0u : 0u;
        cyc_store<L>(X + (size_t(k) * C + c) * L, v);
      }
    }
    for (int t = 1; t < cs.n; t++) {
      const bool last = t == cs.n - 1;
      const EstIn* a = cyc_in(A, cs, cr.start, cr.back, t, 0);
      const EstIn* p = cyc_in(A, cs, cr.start, cr.back, t, 1);
      const int32_t* rk = p->rk + (int64_t(a->tslot) * A.d + row) * w;
      for (int r = tid; r < w; r += T) {
        const int ja = __ldg(a->perm + ro + r), jp = __ldg(p->perm + ro + r);
        sa[r] = make_int2(ja, __ldg(a->s + ro + ja));
        // (the last table's buckets are the cut edge's: the cut sketch's value at jp decides)
        sp[r] = make_int2(last ? __ldg(cut->s + ro + jp) : jp, __ldg(p->s + ro + jp));
        sq[r] = __ldg(rk + r);
      }
      __syncthreads();  // (also: X is complete)
      // merge path: output r comes after a's first sq[r] entries, i.e. at step r + sq[r]
      auto outputs_before = [&](int D) {
        int lo = 0, hi = w;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (mid + sq[mid] < D) lo = mid + 1;
          else hi = mid;
        }
        return lo;
      };
      const int D0 = int(int64_t(2) * w * seg / nseg), D1 = int(int64_t(2) * w * (seg + 1) / nseg);
      const int r0 = outputs_before(D0), r1 = outputs_before(D1);
      const int i0 = D0 - r0, i1 = D1 - r1;
      CycSum<L> s;
      s.clear();
      for (int i = i0; i < i1; i++) {
        const int2 e = sa[i];
        uint32_t v[L];
        cyc_load<L>(X + (size_t(e.x) * C + c) * L, v);
        s.step(v, e.y);
      }
      Limbs<L>::sub_shift(s.ax, s.neg);
      // exclusive scan over the column's segments: lanes C apart, then the warps before
      uint32_t own_x[L], own_a[L];
#pragma unroll
      for (int l = 0; l < L; l++) {
        own_x[l] = s.x[l];
        own_a[l] = s.ax[l];
      }
      for (int o = C; o < 32; o <<= 1) {
        uint32_t ox[L], oa[L];
#pragma unroll
        for (int l = 0; l < L; l++) {
          ox[l] = __shfl_up_sync(0xffffffffu, s.x[l], o);
          oa[l] = __shfl_up_sync(0xffffffffu, s.ax[l], o);
          if (lane < o) ox[l] = oa[l] = 0;
        }
        Limbs<L>::add(s.x, ox);
        Limbs<L>::add(s.ax, oa);
      }
      if (lane >= 32 - C) {
        cyc_store<L>(tot + (warp * C + c) * 2 * L, s.x);
        cyc_store<L>(tot + (warp * C + c) * 2 * L + L, s.ax);
      }
      Limbs<L>::sub(s.x, own_x);
      Limbs<L>::sub(s.ax, own_a);
      __syncthreads();
      uint32_t total[L];
#pragma unroll
      for (int l = 0; l < L; l++) {
        total[l] = 0;
        s.neg[l] = 0;
      }
      for (int k = 0; k < NW; k++) {
        uint32_t u[L];
        cyc_load<L>(tot + (k * C + c) * 2 * L, u);
        Limbs<L>::add(total, u);
        if (k < warp) {
          Limbs<L>::add(s.x, u);
          cyc_load<L>(tot + (k * C + c) * 2 * L + L, u);
          Limbs<L>::add(s.ax, u);
        }
      }
      int i = i0;
      for (int r = r0; r < r1; r++) {
        const int q = sq[r];
        for (; i < q; i++) {
          const int2 e = sa[i];
          uint32_t v[L];
          cyc_load<L>(X + (size_t(e.x) * C + c) * L, v);
          s.step(v, e.y);
        }
        const int2 e = sp[r];
        if (last && e.x != val) continue;
        // p (total - P0) + P1, with the 2^32 parts of the negative factors taken off together
        uint32_t rest[L], o[L], n[L];
#pragma unroll
        for (int l = 0; l < L; l++) {
          rest[l] = total[l];
          o[l] = s.ax[l];
          n[l] = s.neg[l];
        }
        Limbs<L>::sub(rest, s.x);
        Limbs<L>::mad(o, rest, uint32_t(e.y));
        if (e.y < 0) Limbs<L>::add(n, rest);
        Limbs<L>::sub_shift(o, n);
        if (last) {
          if (live) Limbs<L>::add(E, o);
        } else {
          cyc_store<L>(Y + (size_t(e.x) * C + c) * L, o);
        }
      }
      __syncthreads();  // Y is complete; sa, sp, sq and tot are rewritten next
      uint32_t* z = X;
      X = Y;
      Y = z;
    }
  }
  // sum over the CTA's threads, limb sums added to the row (carries are resolved at the end)
  for (int o = 16; o > 0; o >>= 1) {
    uint32_t u[L];
#pragma unroll
    for (int l = 0; l < L; l++) u[l] = __shfl_xor_sync(0xffffffffu, E[l], o);
    Limbs<L>::add(E, u);
  }
  if (lane == 0)
#pragma unroll
    for (int l = 0; l < L; l++)
      if (E[l]) atomicAdd(out->acc + l, (unsigned long long)E[l]);
}

// Persistent over jobs (cycle, row, block of kCycBlk sorted positions of the cut sketch): the
// block's positions that are the first of their value.
// T threads: with one CTA per SM, twice as many keep its latencies covered (the sums' carry chains
// and their shared-memory operands; five rows of four tables of w = 4096, all values distinct:
// 12.5 ms with 256, 8.5 with 512, 9.7 on the generic path; eleven rows of five of w = 2048 10.2,
// 8.0 and 7.7).
template <int T>
__global__ void __launch_bounds__(T, 512 / T) k_cycle(const __grid_constant__ EstArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  // [T / 32][columns][2][limbs] (512 threads: columns x limbs <= 19 by the shared memory there is)
  __shared__ __align__(16) uint32_t tot[(kCycThreads / 32) * kCycMaxCols * 2 * kCycMaxLimbs];
  __shared__ int32_t vals[kCycBlk];
  __shared__ int32_t n_val;
  const int w = A.w;
  const int nblk = (w + kCycBlk - 1) / kCycBlk;
  const int64_t jobs = A.n_cyc * A.d * nblk;
  for (int64_t g = blockIdx.x; g < jobs; g += gridDim.x) {
    const int blk = int(g % nblk), row = int((g / nblk) % A.d);
    const CycSub cs = A.cyc[g / (int64_t(nblk) * A.d)];
    const EstSub& sb = A.subs[cs.sub];
    const int64_t it0 = sb.item_begin + int64_t(row) * sb.n_chunks;
    if (A.partial_ovf[it0] != kCycDone) continue;  // block-uniform: the generic path takes the row
    CycRow* out = cyc_row(A, it0);
    CycRow cr;
    cr.limbs = out->limbs, cr.cols = out->cols, cr.start = out->start, cr.back = out->back;
    if (threadIdx.x < 32) {
      const EstIn* cut = cyc_in(A, cs, cr.start, cr.back, 0, 0);
      const int64_t ro = int64_t(row) * w;
      const int r = blk * kCycBlk + int(threadIdx.x);
      bool rep = false;
      int32_t v = 0;
      if (int(threadIdx.x) < kCycBlk && r < w) {
        v = __ldg(cut->s + ro + __ldg(cut->perm + ro + r));
        const uint32_t m = __ldg(cut->abs + ro + r);
        rep = v != 0;
        for (int q = r - 1; rep && q >= 0 && __ldg(cut->abs + ro + q) == m; q--)
          rep = __ldg(cut->s + ro + __ldg(cut->perm + ro + q)) != v;
      }
      const unsigned b = __ballot_sync(0xffffffffu, rep);
      if (rep) vals[__popc(b & ((1u << threadIdx.x) - 1u))] = v;
      if (threadIdx.x == 0) n_val = __popc(b);
    }
    __syncthreads();
    const int n = n_val;
    if (n > 0) {
      switch (cr.limbs) {
        case 2: cyc_run<2, T>(A, cs, row, cr, out, vals, n, smem, tot); break;
        case 4: cyc_run<4, T>(A, cs, row, cr, out, vals, n, smem, tot); break;
        case 6: cyc_run<6, T>(A, cs, row, cr, out, vals, n, smem, tot); break;
        case 8: cyc_run<8, T>(A, cs, row, cr, out, vals, n, smem, tot); break;
        default: cyc_run<10, T>(A, cs, row, cr, out, vals, n, smem, tot); break;
      }
    }
    __syncthreads();  // vals and the buffers are rewritten by the next job
  }
}

}  // namespace

// Before the generic items: every row it takes has its items marked kCycDone.
cudaError_t launch_estimate_cycle(const EstArgs& a, cudaStream_t st) {
  if (a.n_cyc <= 0) return cudaSuccess;
  const size_t smem = cyc_smem_bytes(a.w);
  const bool two = cyc_two_per_sm(a.w);
  auto k = two ? k_cycle<kCycThreads> : k_cycle<kCycWideThreads>;
  static SmemLimit limit[2];
  cudaError_t e = limit[two].allow(k);
  if (e != cudaSuccess) return e;
  k_cycle_prep<<<unsigned(a.n_cyc * a.d), 1024, 0, st>>>(a);
  const int64_t jobs = a.n_cyc * a.d * ((a.w + kCycBlk - 1) / kCycBlk);
  k<<<unsigned(std::min<int64_t>(jobs, int64_t(sm_count()) * (two ? 2 : 1))), two ? kCycThreads : kCycWideThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace cmpk
