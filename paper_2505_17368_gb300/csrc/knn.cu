// knn.cu -- construction distance tiles with a running top-KP per row, the
// exact FP32 rerank that turns the KP candidates into forward lists, and
// the exact k-NN of a query batch (k-NN query of Sec. 2).
//
// Tile distances use |a|^2 + |b|^2 - 2<a,b> on centred vectors: a dense
// contraction.  This file holds the CUDA-core (SIMT FP32) engine; the
// tcgen05 tensor-core engine lives in knn_tc.cu and feeds the same
// candidate format.  Candidates are (distance, column) keys packed into
// uint64 so the integer order is the (distance, index) order.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace henn {

constexpr int kBM = 64, kBN = 64, kBK = 32;

template <int KP>
__global__ void __launch_bounds__(256) k_tile_topk_simt(const float* __restrict__ A, const float* __restrict__ An,
                                                        int64_t na, const float* __restrict__ B,
                                                        const float* __restrict__ Bn, int64_t nb, int32_t dpad,
                                                        int32_t mode, int32_t splits, uint64_t* __restrict__ out) {
  __shared__ __align__(16) float As[kBK][kBM + 4];
  __shared__ __align__(16) float Bs[kBK][kBN + 4];
  __shared__ float S[kBM][kBN + 1];

  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int warp = tid >> 5;
  const int64_t nblocks = (na + kBM - 1) / kBM;
  // causal rows: heaviest row blocks first
  const int64_t rb = (mode == 0) ? (nblocks - 1 - blockIdx.x) : blockIdx.x;
  const int64_t r0 = rb * kBM;
  const int split = blockIdx.y;

  int64_t cend = (mode == 0) ? min(nb, r0 + kBM) : nb;
  // columns of this split
  int64_t ctiles = (cend + kBN - 1) / kBN;
  int64_t per = (ctiles + splits - 1) / splits;
  int64_t ct0 = split * per, ct1 = min(ctiles, ct0 + per);

  WarpList<KP> lists[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) lists[i].clear();

  for (int64_t ct = ct0; ct < ct1; ++ct) {
    const int64_t c0 = ct * kBN;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    for (int k0 = 0; k0 < dpad; k0 += kBK) {
      // load A rows r0..r0+63, dims k0..k0+31 (8 threads per row, float4 each)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        int idx = tid + p * 256;  // 0..511
        int row = idx >> 3, kq = (idx & 7) * 4;
        int64_t gr = r0 + row;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (gr < na) v = *reinterpret_cast<const float4*>(A + gr * dpad + k0 + kq);
        As[kq + 0][row] = v.x;
        As[kq + 1][row] = v.y;
        As[kq + 2][row] = v.z;
        As[kq + 3][row] = v.w;
        int64_t gc = c0 + row;
        float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
        if (gc < nb) w = *reinterpret_cast<const float4*>(B + gc * dpad + k0 + kq);
        Bs[kq + 0][row] = w.x;
        Bs[kq + 1][row] = w.y;
        Bs[kq + 2][row] = w.z;
        Bs[kq + 3][row] = w.w;
      }
      __syncthreads();
#pragma unroll 8
      for (int k = 0; k < kBK; ++k) {
        float4 a = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
        float4 b = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
        float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
      }
      __syncthreads();
    }
    // epilogue: approximate distances with the validity mask
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int64_t gr = r0 + ty * 4 + i;
      float an = gr < na ? An[gr] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        int64_t gc = c0 + tx * 4 + j;
        bool valid = gr < na && gc < nb;
        if (mode == 0) valid = valid && gc < gr;
        if (mode == 1) valid = valid && gc != gr;
        float dv = valid ? fmaxf(an + Bn[gc] - 2.f * acc[i][j], 0.f) : __int_as_float(0x7f800000);
        S[ty * 4 + i][tx * 4 + j] = dv;
      }
    }
    __syncthreads();
    // running top-KP: warp w owns rows w*8 .. w*8+7
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = warp * 8 + i;
      const int lane = tid & 31;
      uint64_t thr = lists[i].worst();
      float d0 = S[row][lane], d1 = S[row][lane + 32];
      uint64_t k0v = isinf(d0) ? kEmpty : pack(d0, (uint32_t)(c0 + lane));
      uint64_t k1v = isinf(d1) ? kEmpty : pack(d1, (uint32_t)(c0 + lane + 32));
      unsigned m0 = __ballot_sync(0xffffffffu, k0v < thr);
      unsigned m1 = __ballot_sync(0xffffffffu, k1v < thr);
      while (m0 | m1) {
        uint64_t x;
        if (m0) {
          int src = __ffs(m0) - 1;
          m0 &= m0 - 1;
          x = shfl64(k0v, src);
        } else {
          int src = __ffs(m1) - 1;
          m1 &= m1 - 1;
          x = shfl64(k1v, src);
        }
        if (x < thr) {
          lists[i].insert(x);
          thr = lists[i].worst();
        }
      }
    }
    __syncthreads();
  }
  // write lists
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    int64_t gr = r0 + warp * 8 + i;
    if (gr < na) {
      uint64_t* dst = out + ((int64_t)split * na + gr) * KP;
#pragma unroll
      for (int r = 0; r < KP / 32; ++r) dst[r * 32 + (tid & 31)] = lists[i].v[r];
    }
  }
}

void launch_tile_topk_simt(const float* A, const float* An, int64_t na, const float* B, const float* Bn, int64_t nb,
                           int32_t dpad, int32_t mode, int32_t KP, int32_t splits, uint64_t* out, cudaStream_t st) {
  dim3 grid((unsigned)((na + kBM - 1) / kBM), (unsigned)splits);
  switch (KP) {
    case 32: k_tile_topk_simt<32><<<grid, 256, 0, st>>>(A, An, na, B, Bn, nb, dpad, mode, splits, out); break;
    case 64: k_tile_topk_simt<64><<<grid, 256, 0, st>>>(A, An, na, B, Bn, nb, dpad, mode, splits, out); break;
    default: k_tile_topk_simt<128><<<grid, 256, 0, st>>>(A, An, na, B, Bn, nb, dpad, mode, splits, out); break;
  }
}

// merge per-split lists (32 keys) of one row into one
__global__ void k_merge_splits(const uint64_t* __restrict__ in, int64_t rows, int32_t splits,
                               uint64_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < rows;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    WarpList<32> list;
    list.clear();
    for (int s = 0; s < splits; ++s) {
      const uint64_t v = in[((int64_t)s * rows + r) * 32 + lane];
      unsigned m = __ballot_sync(0xffffffffu, v < list.worst());
      while (m) {
        const uint64_t x = shfl64(v, __ffs(m) - 1);
        m &= m - 1;
        if (x < list.worst()) list.insert(x);
      }
    }
    out[r * 32 + lane] = list.v[0];
  }
}

void launch_merge_splits(const uint64_t* in, int64_t rows, int32_t splits, uint64_t* out, cudaStream_t st) {
  int grid = (int)((rows + 7) / 8);
  if (grid > 152 * 16) grid = 152 * 16;
  k_merge_splits<<<grid, 256, 0, st>>>(in, rows, splits, out);
}

// Exact FP32 distance from row `a` to 32 rows at once: lane c gives row c's
// index (count of them, lanes 0 .. count - 1) and gets its distance.  L2:
// squared distance; angular (unit vectors): |a-b|^2 / 2 = 1 - cos.  Per row,
// lane l sums the squared differences of elements l, l + 32, ... in order,
// and the lanes' sums are added up in the tree of an xor butterfly (offsets
// 16, 8, 4, 2, 1; addition commutes): symmetric in (a, b), so dist(a, b) and
// dist(b, a) are bitwise equal.  Eight rows' loads are in flight together,
// and the 32 sums over the lanes are formed by exchanging halves (31 shuffles
// for 32 rows instead of 160): lane l ends with row l's sum.  The rows come
// from L2 or HBM at random; one row at a time left one load in flight per
// lane and a butterfly per row (the rerank of 10,000 x 32 points' 32
// candidates: 104 us, now 64 us).
__device__ __forceinline__ float warp_exact_dist32(const float* __restrict__ a, const float* __restrict__ X,
                                                   int64_t row, int count, int32_t dpad, int32_t metric) {
  const int lane = threadIdx.x & 31;
  float acc[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) acc[c] = 0.f;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if (8 * g < count) {  // warp-uniform
      const float* p[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        // past the last row: the last one again (its sum is not used)
        const int64_t r = __shfl_sync(0xffffffffu, row, min(8 * g + i, count - 1));
        p[i] = X + r * dpad + lane;
      }
#pragma unroll 2
      for (int k = 0; k < dpad; k += 32) {
        const float x = a[k + lane];
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __ldg(p[i] + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float t = x - v[i];
          acc[8 * g + i] = fmaf(t, t, acc[8 * g + i]);
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float keep = up ? acc[i + o] : acc[i];
      const float send = up ? acc[i] : acc[i + o];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return metric == HENN_ANGULAR ? 0.5f * acc[0] : acc[0];
}

// ascending sort of a bitonic sequence, one key per lane
__device__ __forceinline__ uint64_t warp_bitonic_clean(uint64_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t x = shfl_xor64(v, o);
    v = (lane & o) == 0 ? (x < v ? x : v) : (x > v ? x : v);
  }
  return v;
}

// The 32 R smallest of a sorted list (element 32 r + lane in v[r]) and 32
// sorted keys: the keys' smaller half against the list's last 32, then down
// through the list, 32 and 32 merged into 64 at a time.
template <int R>
__device__ __forceinline__ void merge_sorted32(uint64_t (&v)[R], uint64_t keys) {
  if (!__any_sync(0xffffffffu, keys < shfl64(v[R - 1], 31))) return;
  uint64_t b = shfl64(keys, 31 - (threadIdx.x & 31));
  b = warp_bitonic_clean(b < v[R - 1] ? b : v[R - 1]);
#pragma unroll
  for (int r = R - 2; r >= 0; --r) {
    const uint64_t x = shfl64(b, 31 - (threadIdx.x & 31));
    const uint64_t lo = x < v[r] ? x : v[r], hi = x < v[r] ? v[r] : x;
    v[r + 1] = warp_bitonic_clean(hi);
    b = warp_bitonic_clean(lo);
  }
  v[0] = b;
}

template <int KP>
__global__ void __launch_bounds__(256) k_merge_lists(const uint64_t* __restrict__ in, const float* __restrict__ thr_in,
                                                     int64_t rows, int32_t splits, uint64_t* __restrict__ out,
                                                     float* __restrict__ thr) {
  const int lane = threadIdx.x & 31;
  const float kInf = __int_as_float(0x7f800000);
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < rows;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    uint64_t v[KP / 32];
#pragma unroll
    for (int i = 0; i < KP / 32; ++i) v[i] = kEmpty;
    float bound = kInf;
    for (int s = 0; s < splits; ++s) {
      bound = fminf(bound, __ldg(thr_in + (int64_t)s * rows + r));
      merge_sorted32(v, __ldg(in + ((int64_t)s * rows + r) * 32 + lane));
    }
    const uint64_t last = shfl64(v[KP / 32 - 1], 31);
    if (last != kEmpty) bound = fminf(bound, key_dist(last));
#pragma unroll
    for (int i = 0; i < KP / 32; ++i) out[r * KP + 32 * i + lane] = v[i];
    if (lane == 0) thr[r] = bound;
  }
}

void launch_merge_lists(const uint64_t* in, const float* thr_in, int64_t rows, int32_t splits, int32_t KP,
                        uint64_t* out, float* thr, cudaStream_t st) {
  int grid = (int)((rows + 7) / 8);
  if (grid > 152 * 16) grid = 152 * 16;
  if (KP == 32)
    k_merge_lists<32><<<grid, 256, 0, st>>>(in, thr_in, rows, splits, out, thr);
  else if (KP == 64)
    k_merge_lists<64><<<grid, 256, 0, st>>>(in, thr_in, rows, splits, out, thr);
  else
    k_merge_lists<128><<<grid, 256, 0, st>>>(in, thr_in, rows, splits, out, thr);
}

// The certificate of a candidate pool.  The tile distance of any column
// outside the pool is >= thr, so its true distance is >= thr - beta, beta
// bounding the tile error for this row; if that exceeds the wanted list's
// last exact distance dm, no outside column belongs to the list.  Else
// *collect is the tile distance at or under which every column of the list
// lies: their true distances are at most dm (the pool holds that many), so
// their tile distances at most dm + beta.  *collect is +inf where no bound
// holds: fewer than the wanted number in the pool, values that are no
// numbers, or norms so large that a column of the list may overflow in the
// tiles (its tile distance would be +inf or no number, and left out).
__device__ __forceinline__ bool pool_certified(double thr, double dm, float norm_row, float norm_max, double tile_u,
                                               int32_t dpad, float* collect) {
  // relative error bound of the exact FP32 distances (dpad / 32 FMA
  // steps per lane, five butterfly additions), doubled
  const double slack = (dpad / 32 + 8) * 0x1p-23;
  // Only columns whose true distance can reach dm matter, and those lie
  // within sqrt(dm) of this row, so their centred norm is at most
  // (|x_r| + sqrt(dm))^2 (widened for the centring rounding); the tile
  // error bound needs the column norm only up to that cap.
  const double nr = (double)norm_row;
  const double rad = sqrt(nr) * (1.0 + 1e-3) + sqrt(dm * (1.0 + 2.0 * slack)) * (1.0 + 1e-3);
  // a NaN among the columns' norms stays one (fmin would drop it)
  const double nc = norm_max != norm_max ? (double)norm_max : fmin((double)norm_max, rad * rad);
  const double beta = tile_u * 4.0 * (nr + nc) + 1e-30;
  *collect = __double2float_ru(dm * (1.0 + slack) + beta);
  // norms and products of columns within reach add up to (2 rad)^2 at most
  if (!(4.0 * rad * rad < 3.4e38)) {
    *collect = __int_as_float(0x7f800000);
    return false;
  }
  return thr - beta > dm * (1.0 + slack);
}

__device__ __forceinline__ void flag_row(const FlaggedRows& f, int32_t row, float thr) {
  if ((threadIdx.x & 31) == 0) {
    const int at = atomicAdd(f.count, 1);
    f.rows[at] = row;
    f.thr[at] = thr != thr ? __int_as_float(0x7f800000) : thr;  // +inf: no bound
  }
}

// key g of a sorted list
template <int R>
__device__ __forceinline__ uint64_t list_key(const uint64_t (&v)[R], int g) {
  uint64_t x = v[0];
#pragma unroll
  for (int r = 1; r < R; ++r)
    if (r == g >> 5) x = v[r];
  return shfl64(x, g & 31);
}

template <int R>
__device__ __forceinline__ void write_fwd(const uint64_t (&v)[R], int64_t j, int32_t M, int32_t* __restrict__ fwd,
                                          float* __restrict__ fwd_d) {
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int g = q * 32 + (threadIdx.x & 31);
    if (g < M) {
      fwd[j * M + g] = v[q] == kEmpty ? -1 : (int32_t)key_index(v[q]);
      fwd_d[j * M + g] = v[q] == kEmpty ? __int_as_float(0x7f800000) : key_dist(v[q]);
    }
  }
}

template <int R>
__device__ __forceinline__ void write_knn(const uint64_t (&v)[R], int64_t q, int32_t k, int32_t metric,
                                          int64_t* __restrict__ out_ids, float* __restrict__ out_d) {
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int g = r * 32 + (threadIdx.x & 31);
    if (g < k) {
      const bool e = v[r] == kEmpty;
      const float dv = e ? __int_as_float(0x7f800000) : key_dist(v[r]);
      out_ids[q * k + g] = e ? -1 : (int64_t)key_index(v[r]);
      out_d[q * k + g] = e ? dv : (metric == HENN_ANGULAR ? dv : sqrtf(dv));
    }
  }
}

// Forward lists from the KP tile candidates of each row (rank space), with
// the certificate above; a row that fails it is flagged.
constexpr int kTakeAll = 128;  // half a tile's columns
template <int KP>
__global__ void __launch_bounds__(256) k_rerank_fwd(const float* __restrict__ xw, const int32_t* __restrict__ ids,
                                                    int64_t nr, int64_t row0, int32_t dpad, int32_t metric,
                                                    const int32_t* __restrict__ inv, const uint64_t* __restrict__ cand,
                                                    const float* __restrict__ thr, int64_t nb, int32_t causal,
                                                    int32_t inserted, int32_t M, const float* __restrict__ norms,
                                                    const float* __restrict__ norm_max, double tile_u,
                                                    int32_t* __restrict__ fwd, float* __restrict__ fwd_d,
                                                    FlaggedRows flagged) {
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < nr;
       r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t j = inv ? (int64_t)inv[r] : row0 + r;
    const float* xj = xw + (ids ? (int64_t)ids[j] : j) * dpad;
    uint64_t v[KP / 32];
#pragma unroll
    for (int i = 0; i < KP / 32; ++i) v[i] = kEmpty;
    uint64_t last = kEmpty;  // the pool's last key, if it is full
    // a row with few columns takes them all: its two lists need not share
    // them evenly, and a bound from half of them seldom proves anything
    const int64_t ncols = causal ? row0 + r : nb;
    const bool all = ncols <= kTakeAll;
    const int pool = all ? (int)ncols : KP;
#pragma unroll 1
    for (int b = 0; b < pool; b += 32) {
      const int c = b + lane;
      const uint64_t key = !all ? __ldg(cand + r * KP + c) : (c < pool && (causal || c != r) ? pack(0.f, c) : kEmpty);
      last = shfl64(key, 31);
      const unsigned valid = __ballot_sync(0xffffffffu, key != kEmpty);
      if (valid == 0) break;  // only at the pool's end: its keys are sorted, the empty ones last
      int64_t qj = 0, gq = 0;
      if (key != kEmpty) {
        qj = inv ? (int64_t)inv[key_index(key)] : (int64_t)key_index(key);
        gq = ids ? (int64_t)ids[qj] : qj;
      }
      const float dv = warp_exact_dist32(xj, xw, gq, 32 - __clz(valid), dpad, metric);
      merge_sorted32(v, warp_sort_asc(key != kEmpty ? pack(dv, (uint32_t)qj) : kEmpty));
    }
    // what bounds the columns left out (+inf: there are none)
    const float bound = all ? __int_as_float(0x7f800000)
                        : thr ? thr[r] : (last == kEmpty ? __int_as_float(0x7f800000) : key_dist(last));
    // (an insertion's lists are exact: a pool that is not full lacks the
    // columns whose tile distances are no finite numbers)
    if (!isinf(bound) || (inserted && !all)) {
      const uint64_t mkey = list_key(v, M - 1);
      double dm = (mkey == kEmpty) ? 1e300 : (double)key_dist(mkey);
      // exact distances here are of raw vectors; tile distances of centred
      // ones: identical in exact arithmetic.  Angular: tile values are 2x.
      if (metric == HENN_ANGULAR) dm *= 2.0;
      float collect;
      if (!pool_certified((double)bound, dm, norms[r], *norm_max, tile_u, dpad, &collect))
        flag_row(flagged, (int32_t)r, collect);
    }
    write_fwd(v, j, M, fwd, fwd_d);
  }
}

void launch_rerank_fwd(const float* xw, const int32_t* ids, int64_t nr, int64_t row0, int32_t dpad, int32_t metric,
                       const int32_t* inv, const uint64_t* cand, const float* thr, int64_t nb, bool causal, bool inserted,
                       int32_t KP, int32_t M, const float* norms, const float* norm_max, double tile_u, int32_t* fwd, float* fwd_d,
                       const FlaggedRows& flagged, cudaStream_t st) {
  int grid = (int)((nr + 7) / 8);
  if (grid > 152 * 32) grid = 152 * 32;
  if (grid < 1) grid = 1;
  switch (KP) {
    case 32:
      k_rerank_fwd<32><<<grid, 256, 0, st>>>(xw, ids, nr, row0, dpad, metric, inv, cand, thr, nb, causal, inserted, M, norms,
                                              norm_max, tile_u, fwd,
                                             fwd_d, flagged);
      break;
    case 64:
      k_rerank_fwd<64><<<grid, 256, 0, st>>>(xw, ids, nr, row0, dpad, metric, inv, cand, thr, nb, causal, inserted, M, norms,
                                              norm_max, tile_u, fwd,
                                             fwd_d, flagged);
      break;
    default:
      k_rerank_fwd<128><<<grid, 256, 0, st>>>(xw, ids, nr, row0, dpad, metric, inv, cand, thr, nb, causal, inserted, M, norms,
                                              norm_max, tile_u,
                                              fwd, fwd_d, flagged);
      break;
  }
}

template <int KP>
__global__ void __launch_bounds__(256) k_rerank_knn(const float* __restrict__ Q, int64_t nq, const float* __restrict__ X,
                                                    int64_t n, int32_t dpad, int32_t metric,
                                                    const uint64_t* __restrict__ cand, const float* __restrict__ thr,
                                                    int32_t k, const float* __restrict__ qnorms,
                                                    const float* __restrict__ norm_max, double tile_u,
                                                    const int32_t* __restrict__ err, int64_t* __restrict__ out_ids,
                                                    float* __restrict__ out_d, FlaggedRows flagged) {
  const int lane = threadIdx.x & 31;
  for (int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; q < nq;
       q += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    uint64_t v[KP / 32];
#pragma unroll
    for (int i = 0; i < KP / 32; ++i) v[i] = kEmpty;
    int64_t total = 0;
#pragma unroll 1
    for (int b = 0; b < KP; b += 32) {
      const uint64_t key = __ldg(cand + q * KP + b + lane);
      const int cnt = __popc(__ballot_sync(0xffffffffu, key != kEmpty));
      if (cnt == 0) break;
      total += cnt;
      const int64_t col = lane < cnt ? (int64_t)key_index(key) : 0;
      const float dv = warp_exact_dist32(Q + q * dpad, X, col, cnt, dpad, metric);
      merge_sorted32(v, warp_sort_asc(lane < cnt ? pack(dv, (uint32_t)col) : kEmpty));
    }
    if (total < n || *err != 0) {
      const uint64_t mkey = list_key(v, k - 1);
      double dm = mkey == kEmpty ? 1e300 : (double)key_dist(mkey);
      if (metric == HENN_ANGULAR) dm *= 2.0;
      float collect;
      const bool ok = pool_certified((double)thr[q], dm, qnorms[q], *norm_max, tile_u, dpad, &collect);
      if (!ok || *err != 0) flag_row(flagged, (int32_t)q, collect);
    }
    write_knn(v, q, k, metric, out_ids, out_d);
  }
}

void launch_rerank_knn(const float* Q, int64_t nq, const float* X, int64_t n, int32_t dpad, int32_t metric,
                       const uint64_t* cand, const float* thr, int32_t KP, int32_t k, const float* qnorms,
                       const float* norm_max, double tile_u, const int32_t* err, int64_t* out_ids, float* out_d,
                       const FlaggedRows& flagged, cudaStream_t st) {
  int grid = (int)((nq + 7) / 8);
  if (grid > 152 * 32) grid = 152 * 32;
  if (KP == 32)
    k_rerank_knn<32><<<grid, 256, 0, st>>>(Q, nq, X, n, dpad, metric, cand, thr, k, qnorms, norm_max, tile_u, err,
                                           out_ids, out_d, flagged);
  else if (KP == 64)
    k_rerank_knn<64><<<grid, 256, 0, st>>>(Q, nq, X, n, dpad, metric, cand, thr, k, qnorms, norm_max, tile_u, err,
                                           out_ids, out_d, flagged);
  else
    k_rerank_knn<128><<<grid, 256, 0, st>>>(Q, nq, X, n, dpad, metric, cand, thr, k, qnorms, norm_max, tile_u, err,
                                            out_ids, out_d, flagged);
}

// ------------------------------------------ rows the pool did not settle

__global__ void __launch_bounds__(256) k_gather_flagged(FlaggedRows f, int64_t max_rows, int64_t row0, int32_t causal,
                                                        int32_t skip_self, int64_t nb, const uint4* __restrict__ hi,
                                                        const uint4* __restrict__ lo, const float* __restrict__ norms,
                                                        int32_t quads, uint4* __restrict__ hi_out,
                                                        uint4* __restrict__ lo_out, float* __restrict__ norms_out,
                                                        int32_t* __restrict__ lim, int32_t* __restrict__ self) {
  const int lane = threadIdx.x & 31;
  const int64_t nf = min((int64_t)*f.count, max_rows);
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < nf;
       i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t r = f.rows[i];
    for (int c = lane; c < quads; c += 32) {
      hi_out[i * quads + c] = __ldg(hi + r * quads + c);
      lo_out[i * quads + c] = __ldg(lo + r * quads + c);
    }
    if (lane == 0) {
      norms_out[i] = norms[r];
      lim[i] = (int32_t)(causal ? row0 + r : nb);
      self[i] = skip_self ? (int32_t)r : -1;
    }
  }
}

void launch_gather_flagged(const FlaggedRows& f, int64_t max_rows, int64_t row0, bool causal, bool skip_self,
                           int64_t nb, const void* hi, const void* lo, const float* norms, int32_t dk, void* hi_out,
                           void* lo_out, float* norms_out, int32_t* lim, int32_t* self, cudaStream_t st) {
  int grid = (int)((max_rows + 7) / 8);
  if (grid > 152 * 8) grid = 152 * 8;
  k_gather_flagged<<<grid, 256, 0, st>>>(f, max_rows, row0, causal ? 1 : 0, skip_self ? 1 : 0, nb,
                                         static_cast<const uint4*>(hi), static_cast<const uint4*>(lo), norms, dk / 8,
                                         static_cast<uint4*>(hi_out), static_cast<uint4*>(lo_out), norms_out, lim,
                                         self);
}

// One warp per flagged row: its collected columns' exact distances into a
// sorted list.  `row` gives the column's row in X, `to_key` its key index.
template <int R, class RowOf, class KeyOf>
__device__ __forceinline__ bool rerank_collected(const float* __restrict__ a, const float* __restrict__ X, int64_t i,
                                                 int32_t ns, const uint32_t* __restrict__ cols,
                                                 const int32_t* __restrict__ ncols, int32_t cap, int32_t dpad,
                                                 int32_t metric, float thr, RowOf row_of, KeyOf key_of,
                                                 uint64_t (&v)[R]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = kEmpty;
  const int64_t seg0 = (i / kTileRows) * ns * kTileRows + i % kTileRows;
  bool over = isinf(thr);  // no bound: nothing says that the columns are all there
  for (int s = lane; s < ns; s += 32) over |= ncols[seg0 + (int64_t)s * kTileRows] > cap;
  if (__any_sync(0xffffffffu, over)) return false;
  for (int s = 0; s < ns; ++s) {
    const int64_t seg = seg0 + (int64_t)s * kTileRows;
    const int c = ncols[seg];
    for (int b = 0; b < c; b += 32) {
      const int cnt = min(32, c - b);
      const uint32_t col = lane < cnt ? cols[seg * cap + b + lane] : 0u;
      const int64_t key = lane < cnt ? (int64_t)key_of(col) : 0;
      const int64_t row = lane < cnt ? (int64_t)row_of(key) : 0;
      const float dv = warp_exact_dist32(a, X, row, cnt, dpad, metric);
      merge_sorted32(v, warp_sort_asc(lane < cnt ? pack(dv, (uint32_t)key) : kEmpty));
    }
  }
  return true;
}

__global__ void __launch_bounds__(256) k_rerank_collected_fwd(const float* __restrict__ xw,
                                                              const int32_t* __restrict__ ids, FlaggedRows f,
                                                              int64_t max_rows, int64_t row0, int32_t dpad,
                                                              int32_t metric, const int32_t* __restrict__ inv,
                                                              int64_t nb, unsigned grid,
                                                              const uint32_t* __restrict__ cols,
                                                              const int32_t* __restrict__ ncols, int32_t cap,
                                                              int32_t M, int32_t* __restrict__ fwd,
                                                              float* __restrict__ fwd_d, int32_t* __restrict__ over,
                                                              const int32_t* __restrict__ err) {
  const int64_t nf = min((int64_t)*f.count, max_rows);
  if (nf <= 0) return;
  const int32_t ns = collect_splits(grid, nf, nb);
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < nf;
       i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t r = f.rows[i];
    const int64_t j = inv ? (int64_t)inv[r] : row0 + r;
    uint64_t v[1];  // M <= 32
    const bool ok = *err == 0 && rerank_collected(
                                     xw + (ids ? (int64_t)ids[j] : j) * dpad, xw, i, ns, cols, ncols, cap, dpad, metric,
                                     f.thr[i], [&](int64_t pos) { return ids ? (int64_t)ids[pos] : pos; },
                                     [&](uint32_t c) { return inv ? (uint32_t)inv[c] : c; }, v);
    if (ok)
      write_fwd(v, j, M, fwd, fwd_d);
    else if ((threadIdx.x & 31) == 0)
      over[1 + atomicAdd(over, 1)] = (int32_t)(row0 + r);
  }
}

void launch_rerank_collected_fwd(const float* xw, const int32_t* ids, const FlaggedRows& f, int64_t max_rows,
                                 int64_t row0, int32_t dpad, int32_t metric, const int32_t* inv, int64_t nb,
                                 unsigned grid, const uint32_t* cols, const int32_t* ncols, int32_t cap, int32_t M,
                                 int32_t* fwd, float* fwd_d, int32_t* over, const int32_t* err, cudaStream_t st) {
  int g = (int)((max_rows + 7) / 8);
  if (g > 152 * 16) g = 152 * 16;
  k_rerank_collected_fwd<<<g, 256, 0, st>>>(xw, ids, f, max_rows, row0, dpad, metric, inv, nb, grid, cols, ncols, cap,
                                            M, fwd, fwd_d, over, err);
}

__global__ void __launch_bounds__(256) k_rerank_collected_knn(const float* __restrict__ Q, const float* __restrict__ X,
                                                              FlaggedRows f, int64_t max_rows, int32_t dpad,
                                                              int32_t metric, int64_t nb, unsigned grid,
                                                              const uint32_t* __restrict__ cols,
                                                              const int32_t* __restrict__ ncols, int32_t cap,
                                                              int32_t k, int64_t* __restrict__ out_ids,
                                                              float* __restrict__ out_d, int32_t* __restrict__ over,
                                                              const int32_t* __restrict__ err) {
  const int64_t nf = min((int64_t)*f.count, max_rows);
  if (nf <= 0) return;
  const int32_t ns = collect_splits(grid, nf, nb);
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < nf;
       i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t q = f.rows[i];
    uint64_t v[4];  // k <= 112
    const bool ok = *err == 0 &&
                    rerank_collected(
                        Q + q * dpad, X, i, ns, cols, ncols, cap, dpad, metric, f.thr[i], [](int64_t c) { return c; },
                        [](uint32_t c) { return c; }, v) &&
                    list_key(v, k - 1) != kEmpty;
    if (ok)
      write_knn(v, q, k, metric, out_ids, out_d);
    else if ((threadIdx.x & 31) == 0)
      over[1 + atomicAdd(over, 1)] = (int32_t)q;
  }
}

void launch_rerank_collected_knn(const float* Q, const float* X, const FlaggedRows& f, int64_t max_rows, int32_t dpad,
                                 int32_t metric, int64_t nb, unsigned grid, const uint32_t* cols,
                                 const int32_t* ncols, int32_t cap, int32_t k, int64_t* out_ids, float* out_d,
                                 int32_t* over, const int32_t* err, cudaStream_t st) {
  int g = (int)((max_rows + 7) / 8);
  if (g > 152 * 16) g = 152 * 16;
  k_rerank_collected_knn<<<g, 256, 0, st>>>(Q, X, f, max_rows, dpad, metric, nb, grid, cols, ncols, cap, k, out_ids,
                                            out_d, over, err);
}

// Exact forward lists of flagged rows, batched: a block takes RT flagged
// rows (kept in shared memory) and streams every candidate column once for
// all of them, so the columns are read once per RT rows instead of once per
// row.  Each distance is formed exactly as warp_exact_dist32 forms it (lane
// l sums the squared differences of elements l, l+32, ... in order with
// FMA, then the xor butterfly over the 32 lanes), so a flagged row gets the
// list the certified path would give it.  Column validity: mode 0 (causal,
// NSW) columns before the row in insertion order, mode 1 (kNN) all other
// columns.  inv maps insertion ranks to layer positions (nullptr: the
// identity, as for points appended by an insertion).  KD = dpad / 32 when dpad <= 128 (the loads of CPG columns are
// issued together), else 0 (any dpad, one column at a time, read once).
template <int KM, int RT, int KD>
__global__ void __launch_bounds__(256, 2) k_exact_rows(const float* __restrict__ xw, const int32_t* __restrict__ ids,
                                                       int64_t s, int32_t dpad, int32_t metric,
                                                       const int32_t* __restrict__ inv, int32_t mode,
                                                       const int32_t* __restrict__ rows, int32_t nrows, int32_t M,
                                                       int32_t* __restrict__ fwd, float* __restrict__ fwd_d) {
  constexpr int CPG = KD > 0 ? 4 : 1;  // columns whose loads are in flight together
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* qrows = reinterpret_cast<float*>(smem_raw);                   // RT x dpad
  uint64_t* merged = reinterpret_cast<uint64_t*>(qrows + RT * dpad);  // warps x RT x KM
  __shared__ int64_t rank_of[RT];
  const int lane = threadIdx.x & 31;
  const int w = threadIdx.x >> 5;
  const int warps = blockDim.x >> 5;
  const int64_t t0 = (int64_t)blockIdx.x * RT;
  for (int i = 0; i < RT; ++i) {
    const int64_t r = t0 + i < nrows ? (int64_t)rows[t0 + i] : -1;
    if (threadIdx.x == 0) rank_of[i] = r;
    if (r >= 0) {
      const int64_t j = inv ? (int64_t)inv[r] : r;
      const float* src = xw + (ids ? (int64_t)ids[j] : j) * dpad;
      for (int k = threadIdx.x; k < dpad; k += blockDim.x) qrows[i * dpad + k] = src[k];
    }
  }
  __syncthreads();
  int64_t rr[RT];
  int64_t cend = 0;
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    rr[i] = rank_of[i];
    if (rr[i] >= 0) cend = max(cend, mode == 0 ? rr[i] : s);
  }
  WarpList<KM> lists[RT];
#pragma unroll
  for (int i = 0; i < RT; ++i) lists[i].clear();
  const int kd = KD > 0 ? KD : dpad / 32;

  for (int64_t c0 = (int64_t)w * 32; c0 < cend; c0 += (int64_t)warps * 32) {
    // this chunk's 32 columns: lane cc owns column c0 + cc
    const int64_t mycol = c0 + lane;
    int32_t myq = -1;
    const float* myrow = xw;
    if (mycol < cend) {
      myq = inv ? inv[mycol] : (int32_t)mycol;
      myrow = xw + (int64_t)(ids ? ids[myq] : myq) * dpad;
    }
    float dist[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) dist[i] = 0.f;
    const int ncols = (int)min((int64_t)32, cend - c0);
    for (int cc = 0; cc < ncols; cc += CPG) {
      if constexpr (KD > 0) {
        float v[CPG][KD];
#pragma unroll
        for (int g = 0; g < CPG; ++g) {
          const float* p = reinterpret_cast<const float*>(
              __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(myrow), (cc + g) & 31));
          const bool ok = cc + g < ncols;
#pragma unroll
          for (int k = 0; k < KD; ++k) v[g][k] = ok ? __ldg(p + lane + 32 * k) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          float q[KD];
#pragma unroll
          for (int k = 0; k < KD; ++k) q[k] = qrows[i * dpad + lane + 32 * k];
#pragma unroll
          for (int g = 0; g < CPG; ++g) {
            float acc = 0.f;
#pragma unroll
            for (int k = 0; k < KD; ++k) {
              const float t = q[k] - v[g][k];
              acc = fmaf(t, t, acc);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == cc + g) dist[i] = acc;
          }
        }
      } else {
        // any width: the column is read once, 8 elements per lane at a time,
        // into every row's running sum (same element order per row)
        const float* p = reinterpret_cast<const float*>(
            __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(myrow), cc & 31));
        float acc[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) acc[i] = 0.f;
        for (int k0 = 0; k0 < kd; k0 += 8) {
          float v[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) v[t] = k0 + t < kd ? __ldg(p + lane + 32 * (k0 + t)) : 0.f;
#pragma unroll
          for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int t = 0; t < 8; ++t)
              if (k0 + t < kd) {
                const float u = qrows[i * dpad + lane + 32 * (k0 + t)] - v[t];
                acc[i] = fmaf(u, u, acc[i]);
              }
        }
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          float r = acc[i];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
          if (lane == cc) dist[i] = r;
        }
      }
    }
    // lane cc holds column c0 + cc's distance to every row of the tile
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const bool valid = mycol < cend && rr[i] >= 0 && (mode == 0 ? mycol < rr[i] : mycol != rr[i]);
      const float dv = metric == HENN_ANGULAR ? 0.5f * dist[i] : dist[i];
      const uint64_t key = valid ? pack(dv, (uint32_t)myq) : kEmpty;
      unsigned m = __ballot_sync(0xffffffffu, key < lists[i].worst());
      while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const uint64_t k2 = shfl64(key, src);
        if (k2 < lists[i].worst()) lists[i].insert(k2);
      }
    }
  }
  // merge the warps' lists row by row
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int q = 0; q < KM / 32; ++q) merged[((int64_t)w * RT + i) * KM + q * 32 + lane] = lists[i].v[q];
  __syncthreads();
  for (int i = w; i < RT; i += warps) {
    if (rank_of[i] < 0) continue;
    WarpList<KM> all;
    all.clear();
    for (int o = 0; o < warps; ++o)
      for (int c = 0; c < KM; ++c) {
        const uint64_t key = merged[((int64_t)o * RT + i) * KM + c];
        if (key < all.worst()) all.insert(key);
      }
    const int64_t j = inv ? (int64_t)inv[rank_of[i]] : rank_of[i];
#pragma unroll
    for (int q = 0; q < KM / 32; ++q) {
      const int g = q * 32 + lane;
      if (g < M) {
        const uint64_t key = all.v[q];
        fwd[j * M + g] = key == kEmpty ? -1 : (int32_t)key_index(key);
        fwd_d[j * M + g] = key == kEmpty ? __int_as_float(0x7f800000) : key_dist(key);
      }
    }
  }
}

template <int KM, int KD>
static void launch_exact_rows_t(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, int32_t metric,
                                const int32_t* inv, int32_t mode, const int32_t* rows, int32_t nrows, int32_t M,
                                int32_t* fwd, float* fwd_d, cudaStream_t st) {
  constexpr int RT = 8;
  const int threads = 256;
  const size_t smem = (size_t)RT * dpad * sizeof(float) + (size_t)(threads / 32) * RT * KM * sizeof(uint64_t);
  auto kern = k_exact_rows<KM, RT, KD>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int grid = (int)((nrows + RT - 1) / RT);
  kern<<<grid, threads, smem, st>>>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d);
}

void launch_exact_rows(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, int32_t metric, const int32_t* inv,
                       int32_t mode, const int32_t* rows, int32_t nrows, int32_t M, int32_t* fwd, float* fwd_d,
                       cudaStream_t st) {
  if (nrows <= 0) return;
  const int kd = dpad / 32;
  if (M <= 32) {
    if (kd == 1) return launch_exact_rows_t<32, 1>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d, st);
    if (kd == 2) return launch_exact_rows_t<32, 2>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d, st);
    if (kd == 3) return launch_exact_rows_t<32, 3>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d, st);
    if (kd == 4) return launch_exact_rows_t<32, 4>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d, st);
    return launch_exact_rows_t<32, 0>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d, st);
  }
  if (kd == 4) return launch_exact_rows_t<64, 4>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d, st);
  return launch_exact_rows_t<64, 0>(xw, ids, s, dpad, metric, inv, mode, rows, nrows, M, fwd, fwd_d, st);
}

// Exact k-NN by a scan of all columns, for calls too small for the tiles and
// for queries whose candidate lists and collected columns prove nothing.  An
// item is 32 queries, four per warp, and one of sweep_runs runs of columns; a
// block copies 32 KB of columns at a time to shared memory (double-buffered;
// columns follow each other, so a chunk is one piece) and each warp forms the
// differences of 8 columns and its 4 queries in registers, lane l the
// elements l, l + 32, ..., summed over the lanes as warp_exact_dist32 does:
// the same bits.  Bound by issue and by shared memory (a load of a column's 32
// elements serves 4 queries): 10,000 queries x 100,000 x 128 all swept 18 ms;
// a warp per query reading the columns from L2 took 62 ms.  KD = dpad / 32 up
// to 4 (the queries in registers), else 0 (in shared memory).
// rowsel / count (nullable): the queries rowsel[0 .. *count - 1] only.  List i
// of run s (KP keys, ascending) is lists[(s * rows + i) * KP ..].
constexpr int kSweepBytes = 32768;  // of columns per buffer

// acc += (a - x, b - x) squared, each step rounded as a - x and fmaf round it
__device__ __forceinline__ void add_sq_diff2(float2& acc, float a, float b, float x) {
  asm("{\n\t.reg .b64 q, xx, t, s;\n\t"
      "mov.b64 q, {%2, %3};\n\t"
      "mov.b64 xx, {%4, %4};\n\t"
      "mov.b64 s, {%0, %1};\n\t"
      "sub.rn.f32x2 t, q, xx;\n\t"
      "fma.rn.f32x2 s, t, t, s;\n\t"
      "mov.b64 {%0, %1}, s;\n\t}"
      : "+f"(acc.x), "+f"(acc.y)
      : "f"(a), "f"(b), "f"(x));
}

template <int KP, int KD>
__global__ void __launch_bounds__(256) k_sweep_knn(const float* __restrict__ Q, int64_t nq, const float* __restrict__ X,
                                                  int64_t n, int32_t dpad, int32_t metric,
                                                  const int32_t* __restrict__ rowsel,
                                                  const int32_t* __restrict__ count, uint64_t* __restrict__ lists) {
  constexpr int QW = kSweepRows / 8;  // queries per warp
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* buf = reinterpret_cast<float*>(smem_raw);  // 2 x kSweepBytes, then the queries (KD = 0)
  float* qsm = buf + 2 * (kSweepBytes / 4);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t rows = count ? min(nq, (int64_t)*count) : nq;
  if (rows <= 0) return;
  const int kd = KD > 0 ? KD : dpad / 32;
  // columns per chunk: as many 32s as the buffer holds, or 16 or 8 of wide rows
  const int cb = kd <= 8 ? 256 / kd / 32 * 32 : (kd <= 16 ? 16 : 8);
  const int64_t blocks = (rows + kSweepRows - 1) / kSweepRows;
  const int32_t runs = sweep_runs(gridDim.x, rows, n);
  const int64_t tiles = (n + 31) / 32, per = (tiles + runs - 1) / runs;  // of 32 columns
  for (int64_t item = blockIdx.x; item < blocks * runs; item += gridDim.x) {
    const int64_t s = item / blocks, i0 = (item - s * blocks) * kSweepRows + w * QW;
    const int64_t c_end = min(n, (s + 1) * per * 32);
    const int64_t c_first = s * per * 32;
    const int64_t chunks = c_end > c_first ? (c_end - c_first + cb - 1) / cb : 0;
    auto fetch = [&](int64_t ch) {  // columns c_first + ch * cb .. into buffer ch & 1
      const int64_t c = c_first + ch * cb;
      const int words = (int)min((int64_t)cb, c_end - c) * dpad;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(buf + (ch & 1) * (kSweepBytes / 4));
      for (int e = 4 * threadIdx.x; e < words; e += 4 * 256)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 4 * e), "l"(X + c * dpad + e) : "memory");
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    __syncthreads();  // the last item's buffers are read
    if (chunks > 0) fetch(0);
    float qr[QW][KD > 0 ? KD : 1];
#pragma unroll
    for (int r = 0; r < QW; ++r) {
      // past the last query: the last one again (its list is not written)
      const int64_t i = min(i0 + r, rows - 1);
      const float* q = Q + (rowsel ? (int64_t)rowsel[i] : i) * dpad;
      if constexpr (KD > 0) {
#pragma unroll
        for (int k = 0; k < KD; ++k) qr[r][k] = __ldg(q + 32 * k + lane);
      } else {
        for (int k = 0; k < kd; ++k) qsm[(w * QW + r) * dpad + 32 * k + lane] = __ldg(q + 32 * k + lane);
      }
    }
    uint64_t v[QW][KP / 32];
    float dist[QW];  // lane: of column 8 (lane & 3) + (lane >> 2) of the 32
#pragma unroll
    for (int r = 0; r < QW; ++r) {
      dist[r] = 0.f;
#pragma unroll
      for (int g = 0; g < KP / 32; ++g) v[r][g] = kEmpty;
    }
    for (int64_t ch = 0; ch < chunks; ++ch) {
      if (ch + 1 < chunks) {
        fetch(ch + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
      const int64_t c0 = c_first + ch * cb;
      const int have = (int)min((int64_t)cb, c_end - c0);
      const float* cols = buf + (ch & 1) * (kSweepBytes / 4) + lane;
#pragma unroll 1
      for (int g = 0; 8 * g < have && i0 < rows; ++g) {
        float2 acc[QW / 2][8];  // queries 2 p and 2 p + 1
#pragma unroll
        for (int p = 0; p < QW / 2; ++p)
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[p][i] = make_float2(0.f, 0.f);
        auto step = [&](int k, const float (&q)[QW]) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float x = cols[(8 * g + i) * dpad + 32 * k];  // past the last column: not used
#pragma unroll
            for (int p = 0; p < QW / 2; ++p) add_sq_diff2(acc[p][i], q[2 * p], q[2 * p + 1], x);
          }
        };
        if constexpr (KD > 0) {
#pragma unroll
          for (int k = 0; k < KD; ++k) {
            float q[QW];
#pragma unroll
            for (int r = 0; r < QW; ++r) q[r] = qr[r][k];
            step(k, q);
          }
        } else {
#pragma unroll 2
          for (int k = 0; k < kd; ++k) {
            float q[QW];
#pragma unroll
            for (int r = 0; r < QW; ++r) q[r] = qsm[(w * QW + r) * dpad + 32 * k + lane];
            step(k, q);
          }
        }
        // these 8 are columns 8 * at .. of their 32
        const int64_t c8 = c0 / 8 + g;
        const int at = (int)(c8 & 3);
#pragma unroll
        for (int r = 0; r < QW; ++r) {
          float sum[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) sum[i] = r & 1 ? acc[r / 2][i].y : acc[r / 2][i].x;
#pragma unroll
          for (int o = 16; o >= 4; o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < o / 4; ++i) {
              const float keep = up ? sum[i + o / 4] : sum[i];
              const float send = up ? sum[i] : sum[i + o / 4];
              sum[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          }
          sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], 2);
          sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], 1);
          if ((lane & 3) == at) dist[r] = sum[0];
        }
        if (at == 3 || 8 * (c8 + 1) >= c_end) {  // the 32 are complete
          const int64_t col = (c8 - at) * 8 + 8 * (lane & 3) + (lane >> 2);
#pragma unroll
          for (int r = 0; r < QW; ++r) {
            const float dv = metric == HENN_ANGULAR ? 0.5f * dist[r] : dist[r];
            const uint64_t key = col < c_end ? pack(dv, (uint32_t)col) : kEmpty;
            if (__any_sync(0xffffffffu, key < shfl64(v[r][KP / 32 - 1], 31))) merge_sorted32(v[r], warp_sort_asc(key));
          }
        }
      }
      __syncthreads();  // the buffer is read before the copy after next
    }
#pragma unroll
    for (int r = 0; r < QW; ++r)
      if (i0 + r < rows)  // warp-uniform
#pragma unroll
        for (int g = 0; g < KP / 32; ++g) lists[(s * rows + i0 + r) * KP + 32 * g + lane] = v[r][g];
  }
}

// the runs' lists of one query into its k results
template <int KP>
__global__ void __launch_bounds__(256) k_sweep_results(const uint64_t* __restrict__ lists, int64_t nq, int64_t n,
                                                      int32_t metric, int32_t k, unsigned sweep_grid,
                                                      const int32_t* __restrict__ rowsel,
                                                      const int32_t* __restrict__ count,
                                                      int64_t* __restrict__ out_ids, float* __restrict__ out_d) {
  const int lane = threadIdx.x & 31;
  const int64_t rows = count ? min(nq, (int64_t)*count) : nq;
  if (rows <= 0) return;
  const int32_t runs = sweep_runs(sweep_grid, rows, n);
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < rows;
       i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    uint64_t v[KP / 32];
#pragma unroll
    for (int r = 0; r < KP / 32; ++r) v[r] = kEmpty;
    for (int32_t s = 0; s < runs; ++s)
#pragma unroll
      for (int r = 0; r < KP / 32; ++r) merge_sorted32(v, __ldg(lists + ((int64_t)s * rows + i) * KP + 32 * r + lane));
    write_knn(v, rowsel ? (int64_t)rowsel[i] : i, k, metric, out_ids, out_d);
  }
}

unsigned sweep_grid() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return 1;
  return (unsigned)(2 * sms);
}

void launch_sweep_knn(const float* Q, int64_t nq, const float* X, int64_t n, int32_t dpad, int32_t metric, int32_t k,
                     unsigned grid, uint64_t* lists, const int32_t* rowsel, const int32_t* count, int64_t* out_ids,
                     float* out_d, cudaStream_t st) {
  int g = (int)((nq + 7) / 8);
  if (g > 152 * 16) g = 152 * 16;
  const size_t smem = 2 * kSweepBytes + (dpad > 128 ? sizeof(float) * kSweepRows * (size_t)dpad : 0);
  auto both = [&](auto scan, auto results) {
    cudaFuncSetAttribute(scan, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    scan<<<grid, 256, smem, st>>>(Q, nq, X, n, dpad, metric, rowsel, count, lists);
    results<<<g, 256, 0, st>>>(lists, nq, n, metric, k, grid, rowsel, count, out_ids, out_d);
  };
  auto width = [&](auto pool) {
    constexpr int KP = decltype(pool)::value;
    switch (dpad / 32) {
      case 1: both(k_sweep_knn<KP, 1>, k_sweep_results<KP>); break;
      case 2: both(k_sweep_knn<KP, 2>, k_sweep_results<KP>); break;
      case 3: both(k_sweep_knn<KP, 3>, k_sweep_results<KP>); break;
      case 4: both(k_sweep_knn<KP, 4>, k_sweep_results<KP>); break;
      default: both(k_sweep_knn<KP, 0>, k_sweep_results<KP>); break;
    }
  };
  switch (sweep_pool(k)) {
    case 32: width(std::integral_constant<int, 32>()); break;
    case 64: width(std::integral_constant<int, 64>()); break;
    default: width(std::integral_constant<int, 128>()); break;
  }
}

// max of non-negative floats (bit patterns order like the values)
__global__ void k_max_nonneg(const float* __restrict__ v, int64_t n, float* __restrict__ out) {
  float m = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = fmaxf(m, v[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int*>(out), __float_as_int(m));
}

void launch_max_nonneg(const float* v, int64_t n, float* out, cudaStream_t st) {
  cudaMemsetAsync(out, 0, sizeof(float), st);
  k_max_nonneg<<<152 * 2, 256, 0, st>>>(v, n, out);
}

}  // namespace henn
