// prep.cu -- vector copies kept in HBM and per-layer preparation.
//
//  * padded FP32 master copy (rows of dpad = roundup(d, 32) floats, zero
//    tail, so every row is a whole number of 128-byte lines)
//  * inverse norms and unit-length copies for the angular metric (App. G:
//    cosine similarity works on vectors normalised to the unit sphere)
//  * insertion order of a layer (keyed Feistel permutation) and the layer's
//    centred vectors in that order, the operand of the distance tiles
//  * BF16 / FP8-E4M3 precision copies of the traversal vectors
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "kernels.cuh"

namespace henn {

__global__ void k_pad_copy(const float* __restrict__ X, int64_t n, int32_t d, int32_t dpad, float* __restrict__ x32) {
  int64_t total = n * dpad;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = i / dpad;
    int32_t k = (int32_t)(i - r * dpad);
    x32[i] = k < d ? X[r * d + k] : 0.f;
  }
}

void launch_pad_copy(const float* X, int64_t n, int32_t d, int32_t dpad, float* x32, cudaStream_t st) {
  k_pad_copy<<<152 * 8, 256, 0, st>>>(X, n, d, dpad, x32);
}

// one warp per row: 1/sqrt(sum x^2), correctly rounded division and sqrt
__global__ void k_inv_norms(const float* __restrict__ x32, int64_t n, int32_t dpad, float* __restrict__ inv) {
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < n;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const float* row = x32 + r * dpad;
    float acc = 0.f;
    for (int k = lane; k < dpad; k += 32) acc = fmaf(row[k], row[k], acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) inv[r] = acc > 0.f ? __fdiv_rn(1.f, __fsqrt_rn(acc)) : 0.f;
  }
}

void launch_inv_norms(const float* x32, int64_t n, int32_t dpad, float* inv_norm, cudaStream_t st) {
  k_inv_norms<<<152 * 8, 256, 0, st>>>(x32, n, dpad, inv_norm);
}

__global__ void k_normalise(const float* __restrict__ x32, const float* __restrict__ inv, int64_t n, int32_t dpad,
                            float* __restrict__ xn) {
  int64_t total = n * dpad;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
    xn[i] = x32[i] * inv[i / dpad];
}

void launch_normalise(const float* x32, const float* inv_norm, int64_t n, int32_t dpad, float* xn,
                      cudaStream_t st) {
  k_normalise<<<152 * 8, 256, 0, st>>>(x32, inv_norm, n, dpad, xn);
}

// Deterministic column means in two stages: each block sums kMeanChunk rows
// (its threads take 4 columns each, 256 / (dpad / 4) row groups side by side,
// added up in group order), then the chunks' partial sums are added in FP64,
// 8 strided runs per column, in run order.  Bound by the read of the rows:
// one block per 4,096 rows, each thread walking a column alone, was
// latency-bound (one load in flight per thread, 3 blocks for 10,000 rows):
// 1,000,000 x 128 rows with their upper layers 1.78 ms, now 0.19 ms; 10,000
// x 32 0.55 ms, now 0.02 ms.
constexpr int kMeanThreads = 256;
constexpr int kMeanChunk = 512;

__global__ void __launch_bounds__(kMeanThreads) k_mean_partial(const float* __restrict__ xw,
                                                               const int32_t* __restrict__ ids, int64_t s,
                                                               int32_t dpad, float* __restrict__ partial) {
  __shared__ float4 sums[kMeanThreads];
  const int64_t c = blockIdx.x;
  const int64_t r0 = c * kMeanChunk, r1 = min(s, r0 + kMeanChunk);
  const int quads = dpad / 4;             // 8 .. 256
  const int groups = kMeanThreads / quads;  // row groups (threads past them idle)
  const int g = threadIdx.x / quads, k4 = threadIdx.x - g * quads;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (g < groups) {
#pragma unroll 8
    for (int64_t r = r0 + g; r < r1; r += groups) {
      const int64_t gid = ids ? ids[r] : r;
      const float4 v = __ldg(reinterpret_cast<const float4*>(xw + gid * dpad) + k4);
      acc.x += v.x;
      acc.y += v.y;
      acc.z += v.z;
      acc.w += v.w;
    }
  }
  sums[threadIdx.x] = acc;
  __syncthreads();
  if (g == 0) {
    for (int o = 1; o < groups; ++o) {
      const float4 v = sums[o * quads + k4];
      acc.x += v.x;
      acc.y += v.y;
      acc.z += v.z;
      acc.w += v.w;
    }
    reinterpret_cast<float4*>(partial + c * dpad)[k4] = acc;
  }
}

__global__ void __launch_bounds__(256) k_mean_final(const float* __restrict__ partial, int64_t chunks, int64_t s,
                                                    int32_t dpad, float* __restrict__ mean) {
  __shared__ double sums[8][33];
  const int lane = threadIdx.x & 31, run = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + lane;  // dpad is a multiple of 32
  double acc = 0.0;
#pragma unroll 4
  for (int64_t c = run; c < chunks; c += 8) acc += (double)partial[c * dpad + k];
  sums[run][lane] = acc;
  __syncthreads();
  if (run == 0) {
    for (int o = 1; o < 8; ++o) acc += sums[o][lane];
    mean[k] = (float)(acc / (double)s);
  }
}

int64_t mean_chunks(int64_t s) { return (s + kMeanChunk - 1) / kMeanChunk; }

void launch_layer_mean(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, float* partial, float* mean,
                       cudaStream_t st) {
  const int64_t chunks = mean_chunks(s);
  k_mean_partial<<<(unsigned)chunks, kMeanThreads, 0, st>>>(xw, ids, s, dpad, partial);
  k_mean_final<<<dpad / 32, 256, 0, st>>>(partial, chunks, s, dpad, mean);
}

// Insertion order of a layer: point j (layer-local) is inserted at rank
// perm(j); the tiles work in rank order so that "inserted earlier" is
// "lower row index" (causal lower triangle).  For the kNN graph the order
// is irrelevant and the identity is used.
__global__ void k_order_gather(const float* __restrict__ xw, const int32_t* __restrict__ ids, int64_t s,
                               int32_t dpad, Feistel f, int32_t identity, const float* __restrict__ mean,
                               int32_t* __restrict__ inv, float* __restrict__ xo, float* __restrict__ norms) {
  const int lane = threadIdx.x & 31;
  for (int64_t j = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; j < s;
       j += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    int64_t rank = identity ? j : (int64_t)f.perm((uint64_t)j);
    int64_t g = ids ? ids[j] : j;
    const float* src = xw + g * dpad;
    float* dst = xo + rank * dpad;
    float acc = 0.f;
    for (int k = lane; k < dpad; k += 32) {
      float v = src[k] - mean[k];
      dst[k] = v;
      acc = fmaf(v, v, acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      inv[rank] = (int32_t)j;
      norms[rank] = acc;
    }
  }
}

void launch_order_gather(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, uint64_t seed, int32_t layer,
                         int32_t graph, const float* mean, int32_t* inv, float* xo, float* norms, cudaStream_t st) {
  Feistel f = Feistel::make(seed, layer, (uint64_t)s);
  k_order_gather<<<152 * 8, 256, 0, st>>>(xw, ids, s, dpad, f, graph == HENN_GRAPH_KNN ? 1 : 0, mean, inv, xo,
                                          norms);
}

// The same for the tensor-core tiles, straight to BF16 planes (no FP32 copy
// in between) with the largest norm on the way: one read of the rows, one
// write of the planes, 4 consecutive values per lane.  Bound by that traffic:
// 1,000,000 x 128 rows 0.25 ms against 0.36 + 0.34 + 0.01 ms in three passes.
__global__ void __launch_bounds__(256) k_order_split(const float* __restrict__ xw, const int32_t* __restrict__ ids,
                                                     int64_t s, int32_t dpad, Feistel f, int32_t identity,
                                                     const float* __restrict__ mean, int32_t dk,
                                                     __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                                     int32_t* __restrict__ inv, float* __restrict__ norms,
                                                     float* __restrict__ norm_max) {
  const int lane = threadIdx.x & 31;
  int most = 0;  // bits of the largest norm (a NaN is above +inf)
  for (int64_t j = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; j < s;
       j += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t rank = identity ? j : (int64_t)f.perm((uint64_t)j);
    const float* src = xw + (ids ? (int64_t)ids[j] : j) * dpad;
    float acc = 0.f;
    for (int k = 4 * lane; k < dk; k += 128) {
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (k < dpad) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(src + k));
        const float4 m = __ldg(reinterpret_cast<const float4*>(mean + k));
        v[0] = x.x - m.x;
        v[1] = x.y - m.y;
        v[2] = x.z - m.z;
        v[3] = x.w - m.w;
      }
      uint32_t h[2], l[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * i]), h1 = __float2bfloat16_rn(v[2 * i + 1]);
        const __nv_bfloat16 l0 = __float2bfloat16_rn(v[2 * i] - __bfloat162float(h0));
        const __nv_bfloat16 l1 = __float2bfloat16_rn(v[2 * i + 1] - __bfloat162float(h1));
        h[i] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        l[i] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
        acc = fmaf(v[2 * i], v[2 * i], acc);
        acc = fmaf(v[2 * i + 1], v[2 * i + 1], acc);
      }
      *reinterpret_cast<uint2*>(hi + rank * dk + k) = make_uint2(h[0], h[1]);
      *reinterpret_cast<uint2*>(lo + rank * dk + k) = make_uint2(l[0], l[1]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    most = max(most, __float_as_int(acc));
    if (lane == 0) {
      if (inv) inv[rank] = (int32_t)j;
      norms[rank] = acc;
    }
  }
  if (lane == 0) atomicMax(reinterpret_cast<int*>(norm_max), most);
}

void launch_order_split(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, uint64_t seed, int32_t layer,
                        bool identity, const float* mean, int32_t dk, void* hi, void* lo, int32_t* inv, float* norms,
                        float* norm_max, cudaStream_t st) {
  cudaMemsetAsync(norm_max, 0, sizeof(float), st);
  int grid = (int)((s + 7) / 8);
  if (grid > 152 * 8) grid = 152 * 8;
  const Feistel f = Feistel::make(seed, layer, (uint64_t)s);
  k_order_split<<<grid, 256, 0, st>>>(xw, ids, s, dpad, f, identity ? 1 : 0, mean, dk,
                                      static_cast<__nv_bfloat16*>(hi), static_cast<__nv_bfloat16*>(lo), inv, norms,
                                      norm_max);
}

__global__ void k_gather_rows32(const float* __restrict__ xw, const int32_t* __restrict__ ids, int64_t s,
                                int32_t dpad, float* __restrict__ out) {
  int64_t total = s * dpad;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = i / dpad;
    out[i] = xw[(int64_t)ids[r] * dpad + (i - r * dpad)];
  }
}

void launch_gather_rows32(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, float* out, cudaStream_t st) {
  k_gather_rows32<<<152 * 8, 256, 0, st>>>(xw, ids, s, dpad, out);
}

// BF16: round to nearest even.  FP8: scale = max|x|/448 per row (FP32),
// code = E4M3(x / scale) rounded to nearest even with saturation.
__global__ void k_quant_bf16(const float* __restrict__ x, int64_t n, int32_t d, int32_t din, int32_t dout,
                             __nv_bfloat16* __restrict__ out) {
  int64_t total = n * dout;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = i / dout;
    int32_t k = (int32_t)(i - r * dout);
    out[i] = __float2bfloat16_rn(k < d ? x[r * din + k] : 0.f);
  }
}

__global__ void k_quant_fp8(const float* __restrict__ x, int64_t n, int32_t d, int32_t din, int32_t dout,
                            __nv_fp8_storage_t* __restrict__ out, float* __restrict__ scales) {
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < n;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const float* row = x + r * din;
    float m = 0.f;
    for (int k = lane; k < d; k += 32) m = fmaxf(m, fabsf(row[k]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float scale = m > 0.f ? __fdiv_rn(m, 448.f) : 1.f;
    for (int k = lane; k < dout; k += 32) {
      float v = k < d ? __fdiv_rn(row[k], scale) : 0.f;
      out[r * dout + k] = __nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3);
    }
    if (lane == 0) scales[r] = scale;
  }
}

void launch_quantize(const float* x, int64_t n, int32_t d, int32_t dpad_in, int32_t dpad_out, int32_t storage,
                     void* out, float* scales, cudaStream_t st) {
  if (storage == HENN_BF16)
    k_quant_bf16<<<152 * 8, 256, 0, st>>>(x, n, d, dpad_in, dpad_out, (__nv_bfloat16*)out);
  else if (storage == HENN_FP8E4M3)
    k_quant_fp8<<<152 * 8, 256, 0, st>>>(x, n, d, dpad_in, dpad_out, (__nv_fp8_storage_t*)out, scales);
}

}  // namespace henn
