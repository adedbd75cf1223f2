// Star families of the estimate: every sub-plan made of one root table joined to leaves,
// for all leaf subsets of one (graph, root) at once (Sec. 5: products of sketches cached
// across the sub-plans of an enumeration; Sec. 4.2: the merged root sketch contracted with
// the leaf sketches).
//
// With the root's sketches on its leaf edges U (ascending id), a star over leaf set S has,
// in sketch row i, the exact row estimate
//   E(S) = sum_{a in S} sum_r w_a(r) prod_{b in S, b != a} f_ab(r),
// where r runs over a's sorted order (the merged entry takes a's value where a's |value|
// is the minimum), w_a(r) = s_a[pi_a(r)] m_a[pi_a(r)] (root sketch times leaf sketch) and
// f_ab(r) is the suffix sum of leaf b's sketch in b's sorted order from the cross rank of
// a's position r.  The factors f_ab(r) do not depend on S, so the sums
//   T_a(V) = sum_r w_a(r) prod_{b in V} f_ab(r)   for every V in U \ {a}
// are a product of two tables over r: A[V1][r] = w_a(r) prod_{V1} f (the k1 low positions)
// and B[V2][r] = prod_{V2} f (the k2 high positions), T_a(V1 | V2 << k1) = sum_r A B.  Each
// table entry is built from a smaller one by one multiplication, each T entry costs one
// multiply-add per r, and E(S) is a gather of |S| entries (k_estimate_finalize).
//
// Every value is an exact int128.  A table entry whose exact value leaves int128 is flagged
// (it stays flagged through further nonzero factors; a zero factor makes it an exact 0); a
// T entry is flagged when one of its terms or partial sums leaves int128, and the gather
// flags the row, so a row that is not flagged is exact.
#include <cuda_runtime.h>

#include <algorithm>

#include "est_arith.cuh"

namespace cmpk {
namespace {

__device__ __forceinline__ const int32_t* star_rank_row(const EstIn& x, const EstIn& y, int d, int row, int w) {
  return x.rk + (int64_t(y.tslot) * d + row) * w;
}

// An upper bound of |v| in float (+inf for an out-of-range entry): the high word plus one,
// or the low word, rounded up.
__device__ __forceinline__ float star_mag(i128 v, bool fl) {
  if (fl) return __int_as_float(0x7f800000);
  const u128 m = v < 0 ? u128(0) - u128(v) : u128(v);
  const uint64_t hi = uint64_t(m >> 64);
  return hi ? __ull2float_ru(hi + 1) * 0x1p64f : __ull2float_ru(uint64_t(m));
}

// v *= f with the out-of-range flag carried (see the file comment).
__device__ __forceinline__ void star_step(i128& v, bool& fl, int64_t f) {
  if (f == 0) {
    v = 0;
    fl = false;
  } else if (!fl) {
    fl = mul_ovf(v, i128(f), &v);
  }
}

// One CTA per (family, row, leaf b): b's suffix sums in b's sorted order, [w + 1] int64
// (|m| < 2^31 and w <= 2^20: no overflow).
__global__ void __launch_bounds__(kStarThreads) k_star_suf(const __grid_constant__ EstArgs A) {
  __shared__ i128 sh_i128[33];
  __shared__ int32_t sh_flag[1];
  BlockScratch bs{sh_i128, sh_flag};
  const StarUnit u = A.star_units[blockIdx.x];
  const StarFam F = A.star[u.fam];
  const EstIn x = A.inputs[F.in_begin + u.a];
  const int w = A.w;
  const int64_t ro = int64_t(u.row) * w;
  int64_t* sl = A.star_suf + F.suf_off + (int64_t(u.row) * F.K + u.a) * (int64_t(w) + 1);
  for (int r = threadIdx.x; r < w; r += blockDim.x) sl[r] = int64_t(__ldg(x.msk + ro + __ldg(x.perm + ro + r)));
  if (threadIdx.x == 0) {
    sl[w] = 0;
    sh_flag[0] = 0;
  }
  __syncthreads();
  block_scan(sl, w, /*reverse=*/true, bs);
}

// A unit evaluated in int128 with overflow flags (any magnitude): E = 2^(m1+k2) entries, Ep =
// min(E, 256) entry slots, L = 256 / Ep lanes per slot splitting the sorted positions
// (reduced at the end), J = E / Ep entries per thread.  Shared memory per chunk of kStarR
// positions: B[r][v2], A[r][v1] (int128 with byte flags), the factors f[j][r] and w[r].
// Bound by integer issue: 52 instructions per multiply-add.
__device__ __forceinline__ void star_unit_int128(const EstArgs& A, const StarUnit& u, unsigned char* smem) {
  constexpr int R = kStarR, NB = 1 << kStarMaxK2;
  i128* Bs = reinterpret_cast<i128*>(smem);                      // [R][256]
  i128* As = Bs + R * NB;                                          // [R][16]
  i128* red = As + R * 16;                                         // [256]
  int64_t* fv = reinterpret_cast<int64_t*>(red + kStarThreads);  // [15][R]
  int64_t* wv = fv + 15 * R;                                       // [R]
  uint8_t* Bf = reinterpret_cast<uint8_t*>(wv + R);               // [R][256]
  uint8_t* Af = Bf + R * NB;                                       // [R][16]
  uint8_t* redf = Af + R * 16;                                     // [256]
  float* Bm = reinterpret_cast<float*>(redf + kStarThreads);      // [R][256] magnitude bounds
  float* Am = Bm + R * NB;                                         // [R][16]
  const int tid = threadIdx.x;
  const int w = A.w, d = A.d;
  const StarFam F = A.star[u.fam];
  const int K = F.K, k = K - 1, k1 = F.k1, k2 = F.k2, m1 = F.m1;
  const int NV2 = 1 << k2, E = 1 << (m1 + k2);
  const int Ep = E < kStarThreads ? E : kStarThreads;
  const int L = kStarThreads / Ep, J = E / Ep;
  const int es = tid % Ep, lane = tid / Ep;
  const int64_t ro = int64_t(u.row) * w;
  const EstIn xa = A.inputs[F.in_begin + u.a];
  const int64_t* suf0 = A.star_suf + F.suf_off + int64_t(u.row) * K * (int64_t(w) + 1);
  i128 acc[16];
  uint32_t accf = 0;
#pragma unroll
  for (int j = 0; j < 16; j++) acc[j] = 0;

  for (int r0 = 0; r0 < w; r0 += R) {
    // 1. the chunk's factors f[j][r] (position j of U \ {a}) and w[r]
    for (int q = tid; q < (k + 1) * R; q += kStarThreads) {
      const int j = q / R, rr = q % R, r = r0 + rr;
      if (j < k) {
        int64_t f = 0;
        if (r < w) {
          const int ub = j < u.a ? j : j + 1;
          const EstIn& xb = A.inputs[F.in_begin + ub];
          const int32_t pos = __ldg(star_rank_row(xa, xb, d, u.row, w) + r);
          f = suf0[int64_t(ub) * (w + 1) + pos];
        }
        fv[j * R + rr] = f;
      } else {
        int64_t wr = 0;
        if (r < w) {
          const int32_t jj = __ldg(xa.perm + ro + r);
          wr = int64_t(__ldg(xa.s + ro + jj)) * int64_t(__ldg(xa.msk + ro + jj));  // |int32 int32| < 2^62
        }
        wv[rr] = wr;
      }
    }
    __syncthreads();
    // 2. table roots: B[r][0] = 1, A[r][0] = w(r) times the factors of blk's bits
    for (int rr = tid; rr < R; rr += kStarThreads) {
      Bs[rr * NB] = 1;
      Bf[rr * NB] = 0;
      Bm[rr * NB] = 1.0f;
      i128 v = i128(wv[rr]);
      bool fl = false;
      for (int i = 0; i < k1 - m1; i++)
        if ((u.blk >> i) & 1) star_step(v, fl, fv[(m1 + i) * R + rr]);
      As[rr * 16] = v;
      Af[rr * 16] = fl;
      Am[rr * 16] = star_mag(v, fl);
    }
    __syncthreads();
    // 3. doubling: entries [h, 2h) from [0, h) times the factor of bit jj
    const int steps = k2 > m1 ? k2 : m1;
    for (int jj = 0; jj < steps; jj++) {
      const int h = 1 << jj;
      if (jj < k2)
        for (int q = tid; q < h * R; q += kStarThreads) {
          const int rr = q / h, idx = h + q % h;
          i128 v = Bs[rr * NB + idx - h];
          bool fl = Bf[rr * NB + idx - h];
          star_step(v, fl, fv[(k1 + jj) * R + rr]);
          Bs[rr * NB + idx] = v;
          Bf[rr * NB + idx] = fl;
          Bm[rr * NB + idx] = star_mag(v, fl);
        }
      if (jj < m1)
        for (int q = tid; q < h * R; q += kStarThreads) {
          const int rr = q / h, idx = h + q % h;
          i128 v = As[rr * 16 + idx - h];
          bool fl = Af[rr * 16 + idx - h];
          star_step(v, fl, fv[jj * R + rr]);
          As[rr * 16 + idx] = v;
          Af[rr * 16 + idx] = fl;
          Am[rr * 16 + idx] = star_mag(v, fl);
        }
      __syncthreads();
    }
    // 4. multiply-add over the chunk's positions.  When the magnitude bounds keep the product
    //    below 2^126 (float rounding stays far from 2^127), the product modulo 2^128 is exact.
#pragma unroll
    for (int j = 0; j < 16; j++) {
      if (j >= J) break;
      const int e = es + Ep * j;
      const int v1 = e >> k2, v2 = e & (NV2 - 1);
      i128 s = acc[j];
      bool sf = (accf >> j) & 1u;
      for (int rr = lane; rr < R; rr += L) {
        const i128 a = As[rr * 16 + v1], b = Bs[rr * NB + v2];
        if (Am[rr * 16 + v1] * Bm[rr * NB + v2] < 0x1p126f) {
          sf |= add_ovf(s, i128(u128(a) * u128(b)), &s);
          continue;
        }
        const bool fa = Af[rr * 16 + v1], fb = Bf[rr * NB + v2];
        if ((!fa && a == 0) || (!fb && b == 0)) continue;  // an exact zero factor
        if (fa || fb) {
          sf = true;
          continue;
        }
        i128 p;
        sf |= mul_ovf(a, b, &p);
        sf |= add_ovf(s, p, &s);
      }
      acc[j] = s;
      accf = (accf & ~(1u << j)) | (uint32_t(sf) << j);
    }
    __syncthreads();
  }
  // 5. lanes of one slot (L > 1 means J = 1): exact sum of their partial sums
  if (L > 1) {
    red[tid] = acc[0];
    redf[tid] = uint8_t(accf & 1u);
    __syncthreads();
    if (lane == 0) {
      i128 s = 0;
      bool sf = false;
      for (int l = 0; l < L; l++) {
        const int t = es + Ep * l;
        if (redf[t]) sf = true;
        else sf |= add_ovf(s, red[t], &s);
      }
      acc[0] = s;
      accf = sf ? 1u : 0u;
    }
    __syncthreads();
  }
  if (lane == 0) {
    const int64_t base = F.t_off + ((int64_t(u.row) * K + u.a) << k);
#pragma unroll
    for (int j = 0; j < 16; j++) {
      if (j >= J) break;
      const int e = es + Ep * j;
      const int v1 = e >> k2, v2 = e & (NV2 - 1);
      const int64_t V = int64_t((u.blk << m1) | v1) | (int64_t(v2) << k1);
      A.star_t[base + V] = acc[j];
      A.star_tf[base + V] = uint8_t((accf >> j) & 1u);
    }
  }
}

// ---------------------------------------------------------------- residues
// A unit whose sums are bounded below 2^138 is evaluated modulo n <= 5 primes just below 2^28
// and each entry rebuilt as an int128 (flagged when it does not fit).  A product of two
// residues is below 2^56, so a 64-bit accumulator takes 128 of them before it is reduced: a
// multiply-add is one 32 x 32 + 64 bit instruction per prime instead of about 52
// instructions on int128.  (This is the same exact integer: |T| < 2^138 < P / 4.)
constexpr int kRnsMax = 5;
__host__ __device__ constexpr uint32_t rns_c(int j) { return j == 0 ? 57 : j == 1 ? 89 : j == 2 ? 95 : j == 3 ? 119 : 125; }
__host__ __device__ constexpr uint32_t rns_p(int j) { return (1u << 28) - rns_c(j); }
constexpr uint32_t kM28 = (1u << 28) - 1;
constexpr float kRnsBits = 27.999f;  // log2 of each prime, rounded down

// x mod p = 2^28 - c, for any x: 2^28 = c folds 64 -> 45 -> 29 bits (c < 2^7).
__device__ __forceinline__ uint32_t rns_reduce(uint64_t x, uint32_t p, uint32_t c) {
  const uint64_t y = (x & kM28) + (x >> 28) * c;                           // < 2^43 + 2^28
  const uint32_t z = uint32_t(y & kM28) + uint32_t(y >> 28) * c;           // < 2^28 + 2^23
  return min(z, z - p);
}
__device__ __forceinline__ uint32_t rns_mul(uint32_t a, uint32_t b, uint32_t p, uint32_t c) {
  return rns_reduce(uint64_t(a) * b, p, c);
}
__device__ __forceinline__ uint32_t rns_from(int64_t v, uint32_t p, uint32_t c) {
  const uint32_t m = rns_reduce(v < 0 ? uint64_t(0) - uint64_t(v) : uint64_t(v), p, c);
  return v < 0 && m ? p - m : m;
}
constexpr uint32_t rns_pow(uint64_t a, uint32_t e, uint32_t p) {
  uint64_t r = 1;
  for (a %= p; e; e >>= 1) {
    if (e & 1) r = r * a % p;
    a = a * a % p;
  }
  return uint32_t(r);
}
// p_i^-1 mod p_j (Fermat)
__host__ __device__ constexpr uint32_t rns_inv(int i, int j) { return rns_pow(rns_p(i), rns_p(j) - 2, rns_p(j)); }

// The integer of (-P/4, P/4) with residues r[0..n), P the product of the first n primes, as
// an int128; true when it does not fit.  Garner's mixed-radix digits v; the value is negative
// when the top digit lies in the upper half of its range.
__device__ bool rns_value(const uint32_t* r, int n, i128* out) {
  constexpr uint32_t inv[kRnsMax][kRnsMax] = {
      {0, rns_inv(0, 1), rns_inv(0, 2), rns_inv(0, 3), rns_inv(0, 4)},
      {0, 0, rns_inv(1, 2), rns_inv(1, 3), rns_inv(1, 4)},
      {0, 0, 0, rns_inv(2, 3), rns_inv(2, 4)},
      {0, 0, 0, 0, rns_inv(3, 4)},
      {0, 0, 0, 0, 0}};
  uint32_t v[kRnsMax];
  bool neg = false;
#pragma unroll
  for (int j = 0; j < kRnsMax; j++) {
    v[j] = 0;
    if (j < n) {
      const uint32_t p = rns_p(j), c = rns_c(j);
      uint32_t t = r[j];
#pragma unroll
      for (int i = 0; i < j; i++) {
        const uint32_t vi = min(v[i], v[i] - p);  // v[i] < p_i < 2 p
        t = rns_mul(t >= vi ? t - vi : t + p - vi, inv[i][j], p, c);
      }
      v[j] = t;
      neg = t > p / 2;
    }
  }
  // x (or P - x: the digits' complements) as 64 x 3 limbs; below 2^138
  u128 lo = 0;
  uint64_t hi = 0;
  uint32_t carry = neg ? 1 : 0;  // P - x = 1 + sum (p_j - 1 - v_j) p_0 ... p_{j-1}
#pragma unroll
  for (int j = kRnsMax - 1; j >= 0; j--) {
    if (j >= n) continue;
    const uint32_t p = rns_p(j), dgt = neg ? p - 1 - v[j] : v[j];
    const u128 l = u128(uint64_t(lo)) * p + dgt;
    const u128 h = (lo >> 64) * p + uint64_t(l >> 64);
    lo = (h << 64) | uint64_t(l);
    hi = hi * p + uint64_t(h >> 64);
  }
  lo += carry;
  if (carry && lo == 0) hi++;
  *out = neg ? i128(u128(0) - lo) : i128(lo);
  return hi != 0 || (lo >> 127) != 0;  // (-2^127 itself is left to the exact tier)
}

// Shared memory of a residue unit.  Its free leaf bits are split into an X and a Y side of at
// most 64 subsets each; G = 32, 64 or 128 threads (a group) hold all entries as 8 x 4 tiles, the
// 256 / G groups take the chunks of 16 sorted positions in turn, and when the tiles take
// fewer threads than a warp, the rest of the warp shares a chunk's positions.
struct RnsUnit {
  const int32_t* rank[16];   // per factor: a's ranks in leaf b's order ...
  const int64_t* suf[16];    // ... and b's suffix sums
  const int32_t *perm, *s, *msk;
  float bits[kStarThreads / 32];
};
constexpr int kRnsR = 16;  // positions per chunk

template <int G>
__device__ __forceinline__ void group_sync(int g) {
  if (G == 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(G) : "memory");
}

// Bytes of one group's tables: factors [16][16], sub-tables [4][16][8], X [16][NX], Y [16][NY].
__host__ __device__ constexpr int rns_group_words(int nx, int ny) { return 256 + 512 + 16 * (nx + ny); }

template <int G>
__device__ __forceinline__ void star_unit_rns(const EstArgs& A, const StarUnit& u, const StarFam& F, const RnsUnit& U,
                                           int n_primes, unsigned char* smem) {
  constexpr int NG = kStarThreads / G, NQ = 256 / G;  // NQ: factor values per thread and chunk
  const int tid = threadIdx.x, g = tid / G, l = tid % G, w = A.w;
  const int k = F.K - 1, k1 = F.k1, k2 = F.k2, m1 = F.m1, nf = m1 + k2;
  const int hx = (nf + 1) / 2, hy = nf - hx;                     // bits of the two sides
  const int nx = max(8, 1 << hx), ny = max(4, 1 << hy);          // (padded to a tile)
  const int tx = nx / 8, ty = ny / 4, tiles = tx * ty;           // <= G
  const int sub = l / tiles, subs = G / tiles, tix = l % tiles % tx, tiy = l % tiles / tx;
  const bool busy = sub < subs;
  const int E = 1 << nf;
  uint32_t* stash = reinterpret_cast<uint32_t*>(smem);           // [n_primes][E] residue sums of the groups
  uint32_t* fr = stash + kRnsMax * E + g * rns_group_words(nx, ny);
  uint32_t* st = fr + 256;                                       // Xlo, Xhi, Ylo, Yhi: [16][8] each
  uint32_t* X = st + 512;
  uint32_t* Y = X + 16 * nx;
  // position among the k factors of free bit i, of side bits and of the fixed bits
  auto free_pos = [&](int i) { return i < m1 ? i : k1 + i - m1; };
  for (int q = tid; q < n_primes * E; q += kStarThreads) stash[q] = 0;
  __syncthreads();
  const int chunks = (w + kRnsR - 1) / kRnsR;
  for (int pj = 0; pj < n_primes; pj++) {
    const uint32_t p = rns_p(pj), c = rns_c(pj);
    uint64_t acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) acc[i][j] = 0;
    int pending = 0;
    int32_t idx[NQ];
    int64_t val[NQ];
    auto load_ranks = [&](int ch) {
#pragma unroll
      for (int i = 0; i < NQ; i++) {
        const int q = l + i * G, j = q / 16, r = ch * kRnsR + q % 16;
        idx[i] = ch < chunks && j <= k && r < w ? __ldg((j < k ? U.rank[j] : U.perm) + r) : -1;
      }
    };
    auto load_values = [&]() {
#pragma unroll
      for (int i = 0; i < NQ; i++) {
        const int j = (l + i * G) / 16;
        val[i] = 0;
        if (idx[i] >= 0)
          val[i] = j < k ? __ldg(reinterpret_cast<const long long*>(U.suf[j]) + idx[i])
                         : int64_t(__ldg(U.s + idx[i])) * int64_t(__ldg(U.msk + idx[i]));  // |int32 int32| < 2^62
      }
    };
    load_ranks(g);
    load_values();
    for (int ch = g; ch < chunks; ch += NG) {
      // 1. the chunk's factors and w, as residues (row k: w)
#pragma unroll
      for (int i = 0; i < NQ; i++)
        if (l + i * G < (k + 1) * 16) fr[l + i * G] = rns_from(val[i], p, c);
      load_ranks(ch + NG);
      group_sync<G>(g);
      // 2. sub-tables: subsets of the low and of the high three bits of each side; Xlo carries w
      //    and the factors of the block's fixed bits
      for (int q = l; q < 512; q += G) {
        const int t = q / 128, rr = (q / 8) % 16, m = q % 8;
        const int b0 = (t < 2 ? 0 : hx) + (t & 1) * 3, nb = max(0, min(3, (t < 2 ? hx : nf) - b0));
        uint32_t v = 1;
        if (t == 0) {
          v = fr[k * 16 + rr];
          for (int i = 0; i < k1 - m1; i++)
            if ((u.blk >> i) & 1) v = rns_mul(v, fr[(m1 + i) * 16 + rr], p, c);
        }
        for (int i = 0; i < nb; i++)
          if ((m >> i) & 1) v = rns_mul(v, fr[free_pos(b0 + i) * 16 + rr], p, c);
        st[q] = v;
      }
      group_sync<G>(g);
      // 3. the two sides
      for (int q = l; q < 16 * nx; q += G) {
        const int rr = q / nx, x = q % nx;
        X[q] = rns_mul(st[rr * 8 + (x & 7)], st[128 + rr * 8 + (x >> 3)], p, c);
      }
      for (int q = l; q < 16 * ny; q += G) {
        const int rr = q / ny, y = q % ny;
        Y[q] = rns_mul(st[256 + rr * 8 + (y & 7)], st[384 + rr * 8 + (y >> 3)], p, c);
      }
      load_values();  // of the next chunk: in flight during the multiply-adds
      group_sync<G>(g);
      // 4. multiply-adds: X entries 4 tix .. + 3 of both halves times Y entries 4 tiy .. + 3
      if (busy) {
#pragma unroll 2
        for (int rr = sub; rr < 16; rr += subs) {
          const uint4 x0 = *reinterpret_cast<const uint4*>(X + rr * nx + 4 * tix);
          const uint4 x1 = *reinterpret_cast<const uint4*>(X + rr * nx + nx / 2 + 4 * tix);
          const uint4 y = *reinterpret_cast<const uint4*>(Y + rr * ny + 4 * tiy);
          const uint32_t xs[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
          for (int i = 0; i < 8; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) acc[i][j] += uint64_t(xs[i]) * ys[j];
        }
      }
      if (++pending == 7) {  // at most 7 x 16 products below 2^56 and a remainder below 2^28
        pending = 0;
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
          for (int j = 0; j < 4; j++) acc[i][j] = rns_reduce(acc[i][j], p, c);
      }
    }
    // residues of the tile: the sub-teams of a warp meet by shuffles, the groups in the stash
    // (at most 8 groups of residues below 2^28)
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) {
        uint32_t v = busy ? rns_reduce(acc[i][j], p, c) : 0;
        if (G == 32)
          for (int o = tiles; o < 32; o <<= 1) {
            const uint32_t s = v + __shfl_xor_sync(0xffffffffu, v, o);
            v = min(s, s - p);
          }
        const int x = 4 * tix + (i & 3) + (i >> 2) * (nx / 2), y = 4 * tiy + j;
        if (busy && sub == 0 && x < (1 << hx) && y < (1 << hy)) atomicAdd(stash + pj * E + (x | (y << hx)), v);
      }
    group_sync<G>(g);  // the group's tables are rewritten for the next prime
  }
  __syncthreads();
  const int64_t base = F.t_off + ((int64_t(u.row) * F.K + u.a) << k);
  for (int e = tid; e < E; e += kStarThreads) {
    uint32_t r[kRnsMax];
#pragma unroll
    for (int j = 0; j < kRnsMax; j++)
      r[j] = j < n_primes ? rns_reduce(stash[j * E + e], rns_p(j), rns_c(j)) : 0;
    i128 v;
    const bool fl = rns_value(r, n_primes, &v);
    const int64_t V = (int64_t(u.blk) << m1) | (e & ((1 << m1) - 1)) | (int64_t(e >> m1) << k1);
    A.star_t[base + V] = v;
    A.star_tf[base + V] = uint8_t(fl);
  }
  __syncthreads();
}

// The most primes with which a unit of 2^nf entries is faster on residues than in int128.  A prime
// costs its chunks' tables and barriers whatever the entries, and a group's first chunk (w / (w +
// 180): the width spread over the groups); int128 costs 52 instructions an entry and position.
// 20 stars of 3, 5 and 6 leaves at w = 1024, d = 11 on 3, 5 and 5 primes: 371, 1064 and 1336 us,
// in int128 346, 682 and 1237; of 5 leaves at w = 512 on 5 primes 612 and 347; one of 6 at w = 64
// on 4 primes 56 and 16.
__device__ __forceinline__ float rns_most(int nf, int w) {
  const float wide =
      nf <= 2 ? 3.4f : nf == 3 ? 4.2f : nf == 4 ? 4.05f : nf == 5 ? 4.8f : nf == 6 ? 5.5f : 3.0f * float(nf) - 11.5f;
  return wide * float(w) / float(w + 180);
}

// Lattice units (family, row, a, blk), persistent over the unit list.  A unit computes
// T_a(V) for the 2^m1 A-side subsets of block blk (bits m1..k1-1 of V1 = blk) and all 2^k2
// B-side subsets.  Its sums are bounded by w max_r |w_a(r)| prod_b max(1, |f_ab(r)|): below
// 2^138 it runs on residues, on as many primes as the bound asks for, if that pays (rns_most),
// else in int128.
// Stars of 10, 14 and 15 tables (2.0 G multiply-adds at w = 1024, d = 11): 6.16 ms all in int128,
// 2.53 to 2.82 ms on four and five residues.  The units are inlined: as functions of their own
// they spilled, and stars beyond 2^138 (three of 10 to 13 tables, up to 8 M rows) took 9.03 ms,
// 8.30 now (8.68 with an int128 kernel alone).
__global__ void __launch_bounds__(kStarThreads, 2) k_star_lattice(const __grid_constant__ EstArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RnsUnit U;
  const int tid = threadIdx.x, w = A.w, d = A.d;
  for (int64_t ui = A.n_star_suf_units + blockIdx.x; ui < A.n_star_units; ui += gridDim.x) {
    const StarUnit u = A.star_units[ui];
    const StarFam F = A.star[u.fam];
    const int K = F.K, k = K - 1;
    const int64_t ro = int64_t(u.row) * w;
    if (tid < K) {
      const EstIn& xa = A.inputs[F.in_begin + u.a];
      if (tid < k) {
        const int ub = tid < u.a ? tid : tid + 1;
        U.rank[tid] = star_rank_row(xa, A.inputs[F.in_begin + ub], d, u.row, w);
        U.suf[tid] = A.star_suf + F.suf_off + (int64_t(u.row) * K + ub) * (int64_t(w) + 1);
      } else {
        U.perm = xa.perm + ro;
        U.s = xa.s + ro;
        U.msk = xa.msk + ro;
      }
    }
    __syncthreads();
    // the bound: per position, mantissas multiplied (rounded up) and exponents added
    float bits = 0.0f;
    for (int r = tid; r < w; r += kStarThreads) {
      const int jj = __ldg(U.perm + r);
      float m = star_mag(i128(int64_t(__ldg(U.s + jj)) * int64_t(__ldg(U.msk + jj))), false);
      if (m == 0.0f) continue;  // no term at this position
      int e = 0;
      for (int j = 0; j < k; j++) {
        const int64_t f = U.suf[j][__ldg(U.rank[j] + r)];
        m = __fmul_ru(m, fmaxf(1.0f, __ull2float_ru(f < 0 ? uint64_t(0) - uint64_t(f) : uint64_t(f))));
        const int x = ((__float_as_int(m) >> 23) & 255) - 127;  // keep m in [1, 2)
        e += x;
        m = __int_as_float(__float_as_int(m) - (x << 23));
      }
      bits = fmaxf(bits, float(e) + log2f(m) + 0.001f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bits = fmaxf(bits, __shfl_xor_sync(0xffffffffu, bits, o));
    if ((tid & 31) == 0) U.bits[tid >> 5] = bits;
    __syncthreads();
    bits = 0.0f;
    for (int i = 0; i < kStarThreads / 32; i++) bits = fmaxf(bits, U.bits[i]);
    bits += float(32 - __clz(w - 1)) + 2.01f;  // w terms; |T| < P / 4
    const int n_primes = max(1, int(ceilf(bits / kRnsBits)));
    const int nf = F.m1 + F.k2;
    const int tiles = max(1, (1 << ((nf + 1) / 2)) / 8) * max(1, (1 << (nf / 2)) / 4);
    if (n_primes > kRnsMax || float(n_primes) > rns_most(nf, w)) star_unit_int128(A, u, smem);
    else if (tiles <= 32) star_unit_rns<32>(A, u, F, U, n_primes, smem);
    else if (tiles <= 64) star_unit_rns<64>(A, u, F, U, n_primes, smem);
    else star_unit_rns<128>(A, u, F, U, n_primes, smem);
    __syncthreads();  // U is rewritten
  }
}

}  // namespace

cudaError_t launch_estimate_star(const EstArgs& a, cudaStream_t st) {
  if (a.n_star_units <= 0) return cudaSuccess;
  if (a.n_star_suf_units > 0) k_star_suf<<<unsigned(a.n_star_suf_units), kStarThreads, 0, st>>>(a);
  const int64_t lat = a.n_star_units - a.n_star_suf_units;
  if (lat > 0) {
    const size_t smem = star_smem_bytes();
    static SmemLimit limit;
    cudaError_t e = limit.allow(k_star_lattice);
    if (e != cudaSuccess) return e;
    const int64_t grid = std::min<int64_t>(lat, int64_t(sm_count()) * 2);  // two 102 KB CTAs per SM
    k_star_lattice<<<unsigned(grid), kStarThreads, smem, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace cmpk
