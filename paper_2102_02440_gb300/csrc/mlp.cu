// Learned estimate combiner (not in the paper, which takes the median over the d row
// estimates, Sec. 3.2): features from the exact row estimates and the sketches' self-join
// sizes, a 2-layer perceptron y = base + W2 relu(W1 x + b1) + b2 (base = max(x[skip], 0),
// a skip connection from the median row feature) with bfloat16 weights and fp32
// accumulation, and its training step (forward, backward, Adam) on the GPU.
//
// Parameters (fp32 master copy): W1[nh][nin], b1[nh], W2[nh], b2[1].  Every forward and
// backward pass uses their bfloat16 (nearest-even) roundings.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "estimate.cuh"

namespace cmpk {

constexpr int kMlpMaxIn = 66;      // d <= 64 row features + 2 self-join features
constexpr int kMlpMaxHidden = 64;
constexpr int kTrainSamples = 128;  // samples per CTA in the training kernel
constexpr float kFeatScale = 1.0f / 32.0f;

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// Thread-block cluster helpers: this CTA's rank in its cluster, a barrier of every thread of
// the cluster (release / acquire: shared-memory writes before it are visible after it), and
// the address of a shared variable in another CTA of the cluster.
__device__ __forceinline__ unsigned cluster_ctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <class T>
__device__ __forceinline__ T* cluster_map_shared(T* p, unsigned rank) {
  uint64_t out;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
  return reinterpret_cast<T*>(out);
}

// ---------------------------------------------------------------- self-join sizes
// f2[s] = median over rows i of sum_j C[s][i][j]^2 (the Fast-AGMS self-join estimate of
// Sec. 3.2 applied to one sketch), exact per row, rounded once.  One cluster of kF2Cluster
// CTAs per sketch: CTA r of the cluster takes rows r, r + kF2Cluster, ..., its warps split
// each of them into contiguous parts, each lane streaming its part with four independent
// accumulators; after a cluster barrier the first CTA reads every row's exact sum from the
// other CTAs' shared memory (distributed shared memory) and takes the median.
constexpr int kF2Threads = 1024;
constexpr int kF2Cluster = 8;

__global__ void __launch_bounds__(kF2Threads) k_sketch_f2(const int32_t* __restrict__ C, int64_t n_sketches,
                                                          int32_t d, int32_t w, double* __restrict__ f2) {
  __shared__ u128 part[32];
  __shared__ i128 rows[CMP_MAX_D];  // this CTA's rows (the others: unused)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned rank = cluster_ctarank();
  const int64_t s = int64_t(blockIdx.x) / kF2Cluster;
  const int my_rows = (d - int(rank) + kF2Cluster - 1) / kF2Cluster;  // rows rank, rank + kF2Cluster, ...
  if (my_rows > 0) {
    const int split = nw / my_rows > 0 ? nw / my_rows : 1;
    const int units = my_rows * split;
    const int64_t len = (int64_t(w) + split - 1) / split;
    for (int u0 = 0; u0 < units; u0 += nw) {  // rounds of at most nw parts
      const int u = u0 + warp;
      if (u < units) {
        const int i = int(rank) + (u / split) * kF2Cluster, p = u % split;
        const int64_t b = int64_t(p) * len, e = b + len < w ? b + len : int64_t(w);
        const int32_t* src = C + (s * d + i) * int64_t(w);
        u128 a0 = 0, a1 = 0, a2 = 0, a3 = 0;  // each term < 2^62
        int64_t j = b + lane;
        for (; j + 96 < e; j += 128) {
          const int64_t v0 = __ldg(src + j), v1 = __ldg(src + j + 32), v2 = __ldg(src + j + 64),
                        v3 = __ldg(src + j + 96);
          a0 += u128(uint64_t(v0 * v0));
          a1 += u128(uint64_t(v1 * v1));
          a2 += u128(uint64_t(v2 * v2));
          a3 += u128(uint64_t(v3 * v3));
        }
        for (; j < e; j += 32) {
          const int64_t v = __ldg(src + j);
          a0 += u128(uint64_t(v * v));
        }
        u128 acc = a0 + a1 + a2 + a3;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          const uint64_t lo = __shfl_down_sync(0xffffffffu, uint64_t(acc), off);
          const uint64_t hi = __shfl_down_sync(0xffffffffu, uint64_t(acc >> 64), off);
          acc += (u128(hi) << 64) | lo;
        }
        if (lane == 0) part[warp] = acc;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int q = 0; q < nw && u0 + q < units; q++) {
          const int uu = u0 + q, i = int(rank) + (uu / split) * kF2Cluster;
          if (uu % split == 0) rows[i] = 0;
          rows[i] = i128(u128(rows[i]) + part[q]);
        }
      }
      __syncthreads();
    }
  }
  cluster_sync_all();  // every row sum of the sketch is in its CTA's shared memory
  if (rank == 0 && threadIdx.x == 0) {
    i128 all[CMP_MAX_D];
    for (int i = 0; i < d; i++) all[i] = *cluster_map_shared(&rows[i], unsigned(i % kF2Cluster));
    for (int i = 1; i < d; i++) {  // insertion sort of exact integers
      const i128 v = all[i];
      int j = i - 1;
      while (j >= 0 && all[j] > v) {
        all[j + 1] = all[j];
        j--;
      }
      all[j + 1] = v;
    }
    const double r = (d & 1) ? i128_to_double(all[d / 2])
                             : 0.5 * mag_to_double(false, 0, u128(all[d / 2 - 1]) + u128(all[d / 2]));
    f2[s] = r;
  }
  cluster_sync_all();  // the other CTAs' shared memory stays until the first has read it
}

// ---------------------------------------------------------------- features
// v = sorted_i sign(E_i) ln(1 + |E_i|) / 32, m = d / 2 (the median slot):
// feat[q] = ( v_0 - v_m, ..., v_m, ..., v_{d-1} - v_m,  ln(1 + f2a[q]) / 32,  ln(1 + f2b[q]) / 32 )
// Centring the order statistics on the median keeps the inputs of a correction to the
// median small, so bfloat16 weights do not swamp it with rounding noise.
// f2a / f2b per sample, or (f2_idx != nullptr) both read from one per-sketch f2 array at
// f2_idx[2q], f2_idx[2q + 1] (-1: no sketch, feature of 0).
__global__ void k_mlp_features(const int64_t* __restrict__ row_est, int64_t n, int32_t d,
                               const double* __restrict__ f2a, const double* __restrict__ f2b,
                               const int32_t* __restrict__ f2_idx, float* __restrict__ feat) {
  const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q >= n) return;
  float v[CMP_MAX_D];
  for (int i = 0; i < d; i++) {
    const u128 lo = uint64_t(row_est[(q * d + i) * 2]);
    const u128 hi = uint64_t(row_est[(q * d + i) * 2 + 1]);
    const double e = i128_to_double(i128((hi << 64) | lo));
    v[i] = float(copysign(log1p(fabs(e)), e)) * kFeatScale;
  }
  for (int i = 1; i < d; i++) {
    const float x = v[i];
    int j = i - 1;
    while (j >= 0 && v[j] > x) {
      v[j + 1] = v[j];
      j--;
    }
    v[j + 1] = x;
  }
  float* out = feat + q * (d + 2);
  const float vm = v[d / 2];
  for (int i = 0; i < d; i++) out[i] = i == d / 2 ? vm : v[i] - vm;
  double fa, fb;
  if (f2_idx) {
    const int32_t ia = f2_idx[2 * q], ib = f2_idx[2 * q + 1];
    fa = ia >= 0 ? f2a[ia] : 0.0;
    fb = ib >= 0 ? f2a[ib] : 0.0;
  } else {
    fa = f2a[q];
    fb = f2b[q];
  }
  out[d] = float(log1p(fmax(fa, 0.0))) * kFeatScale;
  out[d + 1] = float(log1p(fmax(fb, 0.0))) * kFeatScale;
}

// ---------------------------------------------------------------- inference
__global__ void k_mlp_infer(const float* __restrict__ P, int32_t nin, int32_t nh, int32_t skip,
                            const float* __restrict__ x, int64_t n, float* __restrict__ y) {
  __shared__ float W[kMlpMaxHidden * kMlpMaxIn + 2 * kMlpMaxHidden + 1];
  const int np = nh * nin + 2 * nh + 1;
  for (int k = threadIdx.x; k < np; k += blockDim.x) W[k] = bf16r(P[k]);
  __syncthreads();
  const float* W1 = W;
  const float* b1 = W1 + nh * nin;
  const float* W2 = b1 + nh;
  const float b2 = W2[nh];
  for (int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; s < n; s += int64_t(gridDim.x) * blockDim.x) {
    float xs[kMlpMaxIn];
    for (int c = 0; c < nin; c++) xs[c] = x[s * nin + c];
    float acc = b2 + (skip >= 0 ? fmaxf(xs[skip], 0.f) : 0.f);
    for (int h = 0; h < nh; h++) {
      float z = b1[h];
      for (int c = 0; c < nin; c++) z = fmaf(W1[h * nin + c], xs[c], z);
      if (z > 0.f) acc = fmaf(W2[h], z, acc);
    }
    y[s] = acc;
  }
}

// ---------------------------------------------------------------- training
// One CTA per chunk of kTrainSamples samples (persistent beyond kTrainMaxCtas).  Phase 1
// (thread = sample): forward pass in blocks of kHidBlock hidden units, d(loss)/dy and the
// activations to shared memory.  Phase 2 (thread = hidden unit x every G-th input): the
// chunk's gradient, summed over its samples in a fixed order -> partial[cta][k].
// Bound: shared-memory wavefronts.  Both x and act are kept [feature][sample] with rows of
// kTrainStride = 132 floats: phase 1's lanes (samples) touch consecutive words, and phase
// 2's 16-byte loads of eight hidden units fall on eight different bank groups; the weights,
// x and dy are read as 16-byte broadcasts.  The hidden gradient dy W2[h] [act > 0] is formed
// from act instead of being stored.  Rows of 64 floats per sample made every access of both
// phases a 32-way conflict: a step on 80,000 samples of 13 -> 64 -> 1 took 189 us (143 of them
// here, 40 in k_mlp_adam) and takes 31 us.
constexpr int kTrainStride = kTrainSamples + 4;  // floats: 16-byte aligned rows, 4 banks apart
constexpr int kHidBlock = 16;
constexpr int kColBlock = 8;                     // gradient columns per thread and pass over the samples
constexpr int kTrainMaxCtas = 4096;

struct TrainSmem {  // offsets in floats
  int w1, b1, w2, xs, act, dys, total;
};
__host__ __device__ inline TrainSmem train_smem(int nin, int nh) {
  const int nhp = (nh + kHidBlock - 1) / kHidBlock * kHidBlock;
  TrainSmem L;
  L.w1 = 0;                            // [nin][nhp], zero beyond nh
  L.b1 = L.w1 + nin * nhp;             // [nhp]
  L.w2 = L.b1 + nhp;                   // [nhp], then b2
  L.xs = L.w2 + nhp + 4;               // [nin][kTrainStride]
  L.act = L.xs + nin * kTrainStride;   // [nhp][kTrainStride]
  L.dys = L.act + nhp * kTrainStride;  // dy[kTrainSamples], loss terms[kTrainSamples]
  L.total = L.dys + 2 * kTrainSamples;
  return L;
}

__global__ void __launch_bounds__(kTrainSamples) k_mlp_grad(const float* __restrict__ P, int32_t nin, int32_t nh,
                                                           int32_t skip, const float* __restrict__ x,
                                                           const float* __restrict__ t,
                                                           int64_t n, float huber_delta, int64_t chunks,
                                                           float* __restrict__ partial,
                                                           float* __restrict__ partial_loss) {
  extern __shared__ __align__(16) float shm[];
  const TrainSmem L = train_smem(nin, nh);
  const int np = nh * nin + 2 * nh + 1;
  const int nhp = (nh + kHidBlock - 1) / kHidBlock * kHidBlock;
  float *W1 = shm + L.w1, *B1 = shm + L.b1, *W2 = shm + L.w2, *xs = shm + L.xs, *act = shm + L.act,
        *dys = shm + L.dys, *err = dys + kTrainSamples;
  const int tid = threadIdx.x;
  for (int k = tid; k < nin * nhp; k += kTrainSamples) {
    const int c = k / nhp, h = k % nhp;
    W1[k] = h < nh ? bf16r(P[h * nin + c]) : 0.f;
  }
  for (int h = tid; h < nhp; h += kTrainSamples) {
    B1[h] = h < nh ? bf16r(P[nh * nin + h]) : 0.f;
    W2[h] = h < nh ? bf16r(P[nh * nin + nh + h]) : 0.f;
  }
  const float b2 = bf16r(P[np - 1]);
  // phase 2's share of this thread: hidden unit h, inputs g, g + G, ...
  int hp2 = 1;
  while (hp2 < nh) hp2 <<= 1;  // <= 64
  const int G = kTrainSamples / hp2, h = tid & (hp2 - 1), g = tid / hp2;
  for (int64_t chunk = blockIdx.x; chunk < chunks; chunk += gridDim.x) {
    const int64_t s0 = chunk * kTrainSamples;
    const int ns = int(min(int64_t(kTrainSamples), n - s0));
    for (int i = tid; i < kTrainSamples * nin; i += kTrainSamples) {  // coalesced; samples beyond n are 0
      const int si = i / nin, c = i - si * nin;
      xs[c * kTrainStride + si] = si < ns ? __ldg(x + s0 * nin + i) : 0.f;
    }
    __syncthreads();
    {
      float acc = b2 + (skip >= 0 ? fmaxf(xs[skip * kTrainStride + tid], 0.f) : 0.f);
      for (int h0 = 0; h0 < nhp; h0 += kHidBlock) {
        float z[kHidBlock];
#pragma unroll
        for (int j = 0; j < kHidBlock; j += 4) {
          const float4 b = *reinterpret_cast<const float4*>(B1 + h0 + j);
          z[j] = b.x, z[j + 1] = b.y, z[j + 2] = b.z, z[j + 3] = b.w;
        }
        for (int c = 0; c < nin; c++) {
          const float xv = xs[c * kTrainStride + tid];
          const float4* wr = reinterpret_cast<const float4*>(W1 + c * nhp + h0);
#pragma unroll
          for (int j = 0; j < kHidBlock; j += 4) {
            const float4 wv = wr[j / 4];
            z[j] = fmaf(wv.x, xv, z[j]);
            z[j + 1] = fmaf(wv.y, xv, z[j + 1]);
            z[j + 2] = fmaf(wv.z, xv, z[j + 2]);
            z[j + 3] = fmaf(wv.w, xv, z[j + 3]);
          }
        }
#pragma unroll
        for (int j = 0; j < kHidBlock; j++) {
          const bool on = z[j] > 0.f && tid < ns;
          act[(h0 + j) * kTrainStride + tid] = on ? z[j] : 0.f;
          if (on) acc = fmaf(W2[h0 + j], z[j], acc);
        }
      }
      float dy = 0.f, l = 0.f;
      if (tid < ns) {
        const float e = acc - __ldg(t + s0 + tid);
        if (huber_delta > 0.f) {  // Huber: quadratic within delta, linear beyond
          const float a = fabsf(e);
          dy = (a <= huber_delta ? e : copysignf(huber_delta, e)) / float(n);
          l = a <= huber_delta ? 0.5f * e * e : huber_delta * (a - 0.5f * huber_delta);
        } else {
          dy = 2.f * e / float(n);
          l = e * e;
        }
      }
      dys[tid] = dy;
      err[tid] = l;
    }
    __syncthreads();
    float* out = partial + int64_t(blockIdx.x) * np;
    const bool first = chunk == blockIdx.x;  // a later chunk of this CTA adds to its partial
    auto put = [&](int k, float v) { out[k] = first ? v : out[k] + v; };
    if (h < nh) {
      const float4* ar = reinterpret_cast<const float4*>(act + h * kTrainStride);
      const float4* dr = reinterpret_cast<const float4*>(dys);
      const float w2 = W2[h];
      for (int c0 = g; c0 < nin; c0 += G * kColBlock) {
        float acc[kColBlock];
#pragma unroll
        for (int q = 0; q < kColBlock; q++) acc[q] = 0.f;
#pragma unroll 2
        for (int s4 = 0; s4 < kTrainSamples / 4; s4++) {
          const float4 a = ar[s4], dy = dr[s4];
          const float d0 = a.x > 0.f ? dy.x * w2 : 0.f, d1 = a.y > 0.f ? dy.y * w2 : 0.f,
                      d2 = a.z > 0.f ? dy.z * w2 : 0.f, d3 = a.w > 0.f ? dy.w * w2 : 0.f;
#pragma unroll
          for (int q = 0; q < kColBlock; q++) {
            if (c0 + q * G < nin) {  // uniform over the threads of a group
              const float4 v = *reinterpret_cast<const float4*>(xs + (c0 + q * G) * kTrainStride + 4 * s4);
              acc[q] = fmaf(d0, v.x, acc[q]);
              acc[q] = fmaf(d1, v.y, acc[q]);
              acc[q] = fmaf(d2, v.z, acc[q]);
              acc[q] = fmaf(d3, v.w, acc[q]);
            }
          }
        }
#pragma unroll
        for (int q = 0; q < kColBlock; q++)
          if (c0 + q * G < nin) put(h * nin + c0 + q * G, acc[q]);
      }
      if (g == 0 || g == G - 1) {  // b1 and W2 (one thread of each hidden unit for either)
        float gb = 0.f, gw = 0.f;
        for (int s4 = 0; s4 < kTrainSamples / 4; s4++) {
          const float4 a = ar[s4], dy = dr[s4];
          gb += a.x > 0.f ? dy.x * w2 : 0.f;
          gb += a.y > 0.f ? dy.y * w2 : 0.f;
          gb += a.z > 0.f ? dy.z * w2 : 0.f;
          gb += a.w > 0.f ? dy.w * w2 : 0.f;
          gw = fmaf(dy.x, a.x, gw);
          gw = fmaf(dy.y, a.y, gw);
          gw = fmaf(dy.z, a.z, gw);
          gw = fmaf(dy.w, a.w, gw);
        }
        if (g == 0) put(nh * nin + h, gb);
        if (g == G - 1) put(nh * nin + nh + h, gw);
      }
    }
    if (tid >= kTrainSamples - 32) {  // b2 and the loss: the last warp, a fixed tree
      const int lane = tid & 31;
      float sd = (dys[lane] + dys[lane + 32]) + (dys[lane + 64] + dys[lane + 96]);
      float sl = (err[lane] + err[lane + 32]) + (err[lane + 64] + err[lane + 96]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        sd += __shfl_xor_sync(0xffffffffu, sd, o);
        sl += __shfl_xor_sync(0xffffffffu, sl, o);
      }
      if (lane == 0) {
        put(np - 1, sd);
        partial_loss[blockIdx.x] = first ? sl : partial_loss[blockIdx.x] + sl;
      }
    }
    __syncthreads();  // xs, act and dys are rewritten by the next chunk
  }
}

// Sum of the CTA partials in a fixed order, then one Adam step (Kingma & Ba 2015) on the
// fp32 master parameters.  A CTA takes 32 parameters: warp y sums partials y, y + 32, ...
// (128-byte rows), then the 32 sums of a parameter meet in a fixed tree.  (One thread per
// parameter walking all 625 partials of 80,000 samples, on four CTAs, took 40 us.)  Column
// np is the loss, summed by the CTA after the last parameter block.
__global__ void __launch_bounds__(1024) k_mlp_adam(float* __restrict__ P, float* __restrict__ m, float* __restrict__ v,
                                                   int32_t np, const float* __restrict__ partial,
                                                   const float* __restrict__ partial_loss, int32_t n_cta,
                                                   int64_t n, float lr, int32_t step, float* __restrict__ loss,
                                                   float* __restrict__ grad) {
  __shared__ float part[32][33];
  const int lane = threadIdx.x & 31, y = threadIdx.x >> 5;
  const bool is_loss = int(blockIdx.x) == int(gridDim.x) - 1;
  if (is_loss) {
    float l = 0.f;
    for (int c = int(threadIdx.x); c < n_cta; c += 1024) l += partial_loss[c];
    part[lane][y] = l;
  } else {
    const int k = int(blockIdx.x) * 32 + lane;
    float g = 0.f;
    if (k < np)
      for (int c = y; c < n_cta; c += 32) g += partial[int64_t(c) * np + k];
    part[lane][y] = g;
  }
  __syncthreads();
  float s = part[y][lane];  // warp y now holds parameter y of the block (loss: a 32nd of the terms)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (is_loss) {
    __syncthreads();
    if (lane == 0) part[0][y] = s;
    __syncthreads();
    if (y != 0) return;
    s = part[0][lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0 && loss) *loss = s / float(n);
    return;
  }
  const int k = int(blockIdx.x) * 32 + y;
  if (lane != 0 || k >= np) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.f - powf(b1, float(step)), c2 = 1.f - powf(b2, float(step));
  if (grad) grad[k] = s;
  const float mk = b1 * m[k] + (1.f - b1) * s;
  const float vk = b2 * v[k] + (1.f - b2) * s * s;
  m[k] = mk;
  v[k] = vk;
  P[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

// Combined estimate: the plain median where it is a usable join size (>= 1 tuple), the
// network's prediction exp(32 y) - 1 where the median is below one tuple.
__global__ void k_mlp_combine(const double* __restrict__ median, const float* __restrict__ y,
                              const uint8_t* __restrict__ eligible, int64_t n, double use_median_at,
                              double* __restrict__ out) {
  const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const double m = median[q];
  const bool net = (!eligible || eligible[q]) && !(m >= use_median_at);
  out[q] = net ? fmax(expm1(32.0 * double(y[q])), 0.0) : m;
}

cudaError_t launch_sketch_f2(const int32_t* C, int64_t n_sketches, int32_t d, int32_t w, double* f2,
                             cudaStream_t st) {
  if (n_sketches <= 0) return cudaSuccess;
  if (n_sketches > (int64_t(1) << 31) / kF2Cluster - 1) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(n_sketches * kF2Cluster));  // one cluster per sketch
  cfg.blockDim = dim3(unsigned(kF2Threads));
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kF2Cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_sketch_f2, C, n_sketches, d, w, f2);
}

cudaError_t launch_mlp_features(const int64_t* row_est, int64_t n, int32_t d, const double* f2a, const double* f2b,
                                float* feat, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_mlp_features<<<unsigned((n + 127) / 128), 128, 0, st>>>(row_est, n, d, f2a, f2b, nullptr, feat);
  return cudaGetLastError();
}

cudaError_t launch_mlp_features_indexed(const int64_t* row_est, int64_t n, int32_t d, const double* f2,
                                        const int32_t* f2_idx, float* feat, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_mlp_features<<<unsigned((n + 127) / 128), 128, 0, st>>>(row_est, n, d, f2, nullptr, f2_idx, feat);
  return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const float* P, int32_t nin, int32_t nh, int32_t skip, const float* x, int64_t n,
                             float* y, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t blocks = (n + 255) / 256;
  k_mlp_infer<<<unsigned(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(P, nin, nh, skip, x, n, y);
  return cudaGetLastError();
}

cudaError_t launch_mlp_combine(const double* median, const float* y, int64_t n, double* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_mlp_combine<<<unsigned((n + 255) / 256), 256, 0, st>>>(median, y, nullptr, n, 1.0, out);
  return cudaGetLastError();
}

int64_t mlp_train_ctas(int64_t n) { return (n + kTrainSamples - 1) / kTrainSamples; }

cudaError_t launch_mlp_train(float* P, float* m, float* v, int32_t nin, int32_t nh, int32_t skip, const float* x,
                             const float* t, int64_t n, float huber_delta, float lr, int32_t step, float* loss,
                             float* grad, float* partial,
                             float* partial_loss, cudaStream_t st) {
  const int64_t chunks = mlp_train_ctas(n);
  const int64_t ctas = chunks < kTrainMaxCtas ? chunks : kTrainMaxCtas;
  const int32_t np = nh * nin + 2 * nh + 1;
  if (ctas > 0) {
    const size_t smem = sizeof(float) * size_t(train_smem(nin, nh).total);
    static SmemLimit limit;
    cudaError_t e0 = limit.allow(k_mlp_grad);
    if (e0 != cudaSuccess) return e0;
    k_mlp_grad<<<unsigned(ctas), kTrainSamples, smem, st>>>(P, nin, nh, skip, x, t, n, huber_delta, chunks, partial,
                                                            partial_loss);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  k_mlp_adam<<<unsigned((np + 31) / 32 + 1), 1024, 0, st>>>(P, m, v, np, partial, partial_loss, int32_t(ctas), n, lr,
                                                            step, loss, grad);
  return cudaGetLastError();
}

}  // namespace cmpk

using namespace cmpk;

extern "C" {

int64_t cmp_mlp_param_count(int32_t nin, int32_t nh) {
  if (nin < 1 || nin > kMlpMaxIn || nh < 1 || nh > kMlpMaxHidden) return -1;
  return int64_t(nh) * nin + 2 * nh + 1;
}

cmp_status cmp_sketch_f2(const int32_t* counters_dev, int64_t n_sketches, int32_t d, int32_t w, double* f2_dev,
                         void* stream) {
  if (n_sketches < 0 || d < 1 || d > CMP_MAX_D || w < 1 || w > CMP_MAX_W) return CMP_EINVAL;
  if (n_sketches > 0 && (!counters_dev || !f2_dev)) return CMP_EINVAL;
  return launch_sketch_f2(counters_dev, n_sketches, d, w, f2_dev, reinterpret_cast<cudaStream_t>(stream)) ==
                 cudaSuccess
             ? CMP_OK
             : CMP_ECUDA;
}

cmp_status cmp_mlp_features(const int64_t* row_est_dev, int64_t n, int32_t d, const double* f2a_dev,
                            const double* f2b_dev, float* feat_dev, void* stream) {
  if (n < 0 || d < 1 || d > CMP_MAX_D) return CMP_EINVAL;
  if (n > 0 && (!row_est_dev || !f2a_dev || !f2b_dev || !feat_dev)) return CMP_EINVAL;
  return launch_mlp_features(row_est_dev, n, d, f2a_dev, f2b_dev, feat_dev, reinterpret_cast<cudaStream_t>(stream)) ==
                 cudaSuccess
             ? CMP_OK
             : CMP_ECUDA;
}

cmp_status cmp_mlp_features_indexed(const int64_t* row_est_dev, int64_t n, int32_t d, const double* f2_dev,
                                    const int32_t* f2_index_dev, float* feat_dev, void* stream) {
  if (n < 0 || d < 1 || d > CMP_MAX_D) return CMP_EINVAL;
  if (n > 0 && (!row_est_dev || !f2_dev || !f2_index_dev || !feat_dev)) return CMP_EINVAL;
  return launch_mlp_features_indexed(row_est_dev, n, d, f2_dev, f2_index_dev, feat_dev,
                                     reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess
             ? CMP_OK
             : CMP_ECUDA;
}

cmp_status cmp_mlp_infer(const float* params_dev, int32_t nin, int32_t nh, int32_t skip, const float* x_dev, int64_t n,
                         float* y_dev, void* stream) {
  if (cmp_mlp_param_count(nin, nh) < 0 || n < 0 || skip < -1 || skip >= nin) return CMP_EINVAL;
  if (!params_dev || (n > 0 && (!x_dev || !y_dev))) return CMP_EINVAL;
  return launch_mlp_infer(params_dev, nin, nh, skip, x_dev, n, y_dev, reinterpret_cast<cudaStream_t>(stream)) ==
                 cudaSuccess
             ? CMP_OK
             : CMP_ECUDA;
}

cmp_status cmp_mlp_combine_ex(const double* median_dev, const float* y_dev, const uint8_t* eligible_dev, int64_t n,
                              double use_median_at, double* est_dev, void* stream) {
  if (n < 0 || (n > 0 && (!median_dev || !y_dev || !est_dev)) || use_median_at != use_median_at) return CMP_EINVAL;
  if (n == 0) return CMP_OK;
  k_mlp_combine<<<unsigned((n + 255) / 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      median_dev, y_dev, eligible_dev, n, use_median_at, est_dev);
  return cudaGetLastError() == cudaSuccess ? CMP_OK : CMP_ECUDA;
}

cmp_status cmp_mlp_combine(const double* median_dev, const float* y_dev, int64_t n, double* est_dev, void* stream) {
  if (n < 0 || (n > 0 && (!median_dev || !y_dev || !est_dev))) return CMP_EINVAL;
  return launch_mlp_combine(median_dev, y_dev, n, est_dev, reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess
             ? CMP_OK
             : CMP_ECUDA;
}

size_t cmp_mlp_train_ws_bytes(int32_t nin, int32_t nh, int64_t n) {
  const int64_t np = cmp_mlp_param_count(nin, nh);
  if (np < 0 || n < 0) return 0;
  const int64_t ctas = mlp_train_ctas(n);
  return size_t(align16(sizeof(float) * size_t(ctas * np)) + align16(sizeof(float) * size_t(ctas > 0 ? ctas : 1)));
}

cmp_status cmp_mlp_train_step(float* params_dev, float* adam_m_dev, float* adam_v_dev, int32_t nin, int32_t nh,
                              int32_t skip, const float* x_dev, const float* y_dev, int64_t n, float huber_delta,
                              float lr, int32_t step, float* loss_dev, float* grad_dev, void* ws_dev, size_t ws_bytes,
                              void* stream) {
  const int64_t np = cmp_mlp_param_count(nin, nh);
  if (np < 0 || n < 1 || step < 1 || !(lr > 0.f) || skip < -1 || skip >= nin || !(huber_delta >= 0.f))
    return CMP_EINVAL;
  if (!params_dev || !adam_m_dev || !adam_v_dev || !x_dev || !y_dev) return CMP_EINVAL;
  if (ws_bytes < cmp_mlp_train_ws_bytes(nin, nh, n) || !ws_dev) return CMP_EWORKSPACE;
  const int64_t ctas = mlp_train_ctas(n);
  float* partial = static_cast<float*>(ws_dev);
  float* partial_loss =
      reinterpret_cast<float*>(static_cast<unsigned char*>(ws_dev) + align16(sizeof(float) * size_t(ctas * np)));
  return launch_mlp_train(params_dev, adam_m_dev, adam_v_dev, nin, nh, skip, x_dev, y_dev, n, huber_delta, lr, step,
                          loss_dev, grad_dev,
                          partial, partial_loss, reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess
             ? CMP_OK
             : CMP_ECUDA;
}

}  // extern "C"
