// kernels.cuh -- launch interfaces between the host orchestration
// (henn_abi.cu) and the kernels of libhenn.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace henn {

constexpr int kMaxD = 1024;

enum RingStatus : int32_t { kRingPass = 1, kRingFail = 2, kRingAmbiguous = 3 };

struct LayerSampleArgs {
  uint64_t base;   // derive(derive(derive(seed, SAMP), layer), attempt)
  int64_t s;       // size of the previous layer
  int64_t t;       // number of draws
  uint8_t* flags;  // s bytes, zeroed by the caller
};

// layers.cu
void launch_sample(const LayerSampleArgs& a, cudaStream_t st);
int64_t scan_tiles(int64_t s);
void launch_compact(const uint8_t* flags, int64_t s, const int32_t* prev_ids, int64_t* tile_buf,
                    int64_t* d_total, int32_t* out_pos, int32_t* out_ids, cudaStream_t st);
void launch_offsets(const int32_t* counts, int64_t s, int64_t* tile_buf, int64_t* out_offsets,
                    cudaStream_t st);
void launch_ring_params(uint64_t bc, uint64_t bs, int32_t r, int64_t s, int64_t span, int32_t* centre,
                        int64_t* start, cudaStream_t st);
// D: r rows of ring_ld(s) floats (16-byte aligned), the distances of ring
// centre q to the layer's s points in row q
int64_t ring_ld(int64_t s);
void launch_ring_dist(const float* x32, int32_t dpad, const int32_t* prev_ids, int64_t s,
                      const int32_t* centre, int32_t r, int32_t metric, const float* inv_norm, float* D,
                      cudaStream_t st);
// Alg. 3 halving: m steps over positions 0..s-1; the survivors (ascending)
// land in pos and their global ids in ids; returns their count.  tmp holds
// ceil(s/2) entries.
int64_t launch_halving(uint64_t seed, int32_t layer, int64_t s, int32_t m, const int32_t* prev_ids, int32_t* tmp,
                       int32_t* pos, int32_t* ids, cudaStream_t st);
void launch_ring_select_decide(const float* D, int64_t s, const int64_t* start, int64_t w, int32_t r,
                               const int32_t* net_pos, const int64_t* nnet_dev, double er, double ea, float* lo,
                               float* hi, int32_t* status, cudaStream_t st);
void launch_ring_recheck(const float* x32, int32_t d, int32_t dpad, const int32_t* prev_ids, int64_t s,
                         int64_t centre_pos, int64_t a0, int64_t w, int32_t metric, const int32_t* net_pos,
                         int64_t nnet, double* D64, double* bounds, int32_t* status, int32_t q,
                         cudaStream_t st);

// prep.cu: vector copies and per-layer preparation
void launch_pad_copy(const float* X, int64_t n, int32_t d, int32_t dpad, float* x32, cudaStream_t st);
void launch_inv_norms(const float* x32, int64_t n, int32_t dpad, float* inv_norm, cudaStream_t st);
void launch_normalise(const float* x32, const float* inv_norm, int64_t n, int32_t dpad, float* xn,
                      cudaStream_t st);
// mean over the rows listed in ids (or rows 0..s-1): partial buffer of
// mean_chunks(s) * dpad floats (16-byte aligned, as are the rows)
int64_t mean_chunks(int64_t s);
void launch_layer_mean(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, float* partial,
                       float* mean, cudaStream_t st);
// insertion order: rank[j] = perm(j), inv[rank] = j; xo[rank] = xw[ids[j]] - mean; norms
void launch_order_gather(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, uint64_t seed,
                         int32_t layer, int32_t graph, const float* mean, int32_t* inv, float* xo,
                         float* norms, cudaStream_t st);
// The operand of the tensor-core tiles in one pass: row j of the layer minus
// its mean at rank perm(j) (identity: j), as BF16 planes hi = bf16(x), lo =
// bf16(x - hi), dk wide, with its squared norm; inv (nullable) as above;
// *norm_max the largest norm (NaN if one is)
void launch_order_split(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, uint64_t seed, int32_t layer,
                        bool identity, const float* mean, int32_t dk, void* hi, void* lo, int32_t* inv, float* norms,
                        float* norm_max, cudaStream_t st);
void launch_gather_rows32(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, float* out,
                          cudaStream_t st);
void launch_quantize(const float* x, int64_t n, int32_t d, int32_t dpad_in, int32_t dpad_out,
                     int32_t storage, void* out, float* scales, cudaStream_t st);

// knn.cu: tiles (approximate distances) + running top-KP per row
//   mode 0: causal (column c valid iff c < row), A == B
//   mode 1: all other rows (c != row), A == B
//   mode 2: rows of A against all rows of B
void launch_tile_topk_simt(const float* A, const float* An, int64_t na, const float* B, const float* Bn,
                           int64_t nb, int32_t dpad, int32_t mode, int32_t KP, int32_t splits,
                           uint64_t* out, cudaStream_t st);
// lists of 32 keys per row and split (splits x rows x 32) -> the 32 smallest
void launch_merge_splits(const uint64_t* in, int64_t rows, int32_t splits, uint64_t* out, cudaStream_t st);
// Sorted lists of 32 keys per row and split (splits x rows x 32, with their
// bounds thr_in) -> the KP (32, 64 or 128) smallest of each row, and a bound
// on what they leave out: every column of the row that is not among them has
// a tile distance of at least thr[row] (+inf: every column that the lists
// were offered is there).
void launch_merge_lists(const uint64_t* in, const float* thr_in, int64_t rows, int32_t splits, int32_t KP,
                        uint64_t* out, float* thr, cudaStream_t st);
// knn_tc.cu: the same tiles on tcgen05 tensor cores (split BF16, lists of
// KP = 32, dpad <= 1024) from BF16 planes of rows and columns, dk =
// roundup(dpad, 64) wide
bool tc_tiles_supported(int32_t dpad, int32_t KP);
// CTAs per row block, each with its own lists, for na rows against nb columns
int32_t tile_list_splits(int64_t na, int64_t nb, bool causal);
// modes 0 - 2; out: splits x na x 32 keys, each list sorted: the row's 16
// nearest columns of two halves of the split's columns (dk > 128: its 32
// nearest of the split); thr (splits x na):
// every other column of the split has a tile distance of at least this (+inf:
// there is none); lim (nullable): row r takes columns 0 .. lim[r] - 1 only
cudaError_t launch_tile_lists_tc(const void* a_hi, const void* a_lo, const float* a_norms, int64_t na,
                                 const void* b_hi, const void* b_lo, const float* b_norms, int64_t nb, int32_t dk,
                                 int32_t mode, const int32_t* lim, int32_t splits, uint64_t* out, float* thr,
                                 int32_t* err, cudaStream_t st);
// Every column of a row whose tile distance is at or under the row's
// threshold.  The number of rows is *count (device, at most max_rows); the
// grid's CTAs are shared out over the 128-row blocks there are
// (collect_splits); CTA b of a block writes row r's columns, at most cap of
// them, at cols + (b * 128 + r) * cap and their number (over cap: some were
// dropped) to ncols[b * 128 + r].
constexpr int kTileRows = 128, kTileCols = 256;
__host__ __device__ inline int32_t collect_splits(unsigned grid, int64_t rows, int64_t nb) {
  const int64_t blocks = (rows + kTileRows - 1) / kTileRows;
  const int64_t most = (nb + 2 * kTileCols - 1) / (2 * kTileCols);  // at least two tiles each
  const int64_t k = (int64_t)grid / blocks;
  return (int32_t)(k < 1 ? 1 : (k > most ? most : k));
}
unsigned tile_collect_grid(int64_t max_rows);
cudaError_t launch_tile_collect_tc(const void* a_hi, const void* a_lo, const float* a_norms, int64_t max_rows,
                                   const void* b_hi, const void* b_lo, const float* b_norms, int64_t nb, int32_t dk,
                                   const int32_t* lim, const int32_t* self, const float* thr, const int32_t* count,
                                   unsigned grid, uint32_t* cols, int32_t* ncols, int32_t cap, int32_t* err,
                                   cudaStream_t st);
// FP32 rows (dpad wide) -> BF16 planes hi = bf16(x), lo = bf16(x - hi), dk wide (zero padded)
void launch_split_bf16(const float* x, int64_t s, int32_t dpad, int32_t dk, void* hi, void* lo, cudaStream_t st);
// mode 2 on tensor cores from pre-split planes: na rows (queries) against nb
// columns (a layer's points), out = na x 32 keys (distance, column); with
// out_d (mode 3) every distance instead, as a 16-bit order-preserving key
// (the distance's float bits 30..15: rounded down to 8 mantissa bits), na
// rows of ldo keys (ldo a multiple of 64, >= nb, out_d 128-byte aligned;
// the key of +inf past column nb)
// b_maps: the four tensor maps of make_column_maps, 128 bytes each;
// tile_n: columns per tile, 128 or 256 (0 = 256), the same results
// out_cmin (mode 3, nullable): each row's minimum over every 32-column chunk,
// as the lower end of its key's bucket, rows of ldc floats (ldc a multiple
// of 8 covering every tile, 16-byte aligned)
cudaError_t launch_tile_cross_tc(const void* a_hi, const void* a_lo, const float* a_norms, int64_t na,
                                 const void* b_maps, const float* b_norms, int64_t nb, int32_t dk, uint64_t* out,
                                 uint16_t* out_d, int64_t ldo, float* out_cmin, int64_t ldc, int32_t* err,
                                 int32_t tile_n, cudaStream_t st);
// Tensor maps of the column operand (hi, lo planes of nb rows, dk wide) for
// launch_tile_cross_tc -- hi and lo for tiles of 256 columns, then for 128 --
// written to maps (4 x 128 bytes); false if not encodable.
bool make_column_maps(const void* b_hi, const void* b_lo, int64_t nb, int32_t dk, void* maps);
// Rows that a candidate list could not settle: their number, the rows, and
// for each the tile distance that every column of its answer lies under.
struct FlaggedRows {
  int32_t* count;
  int32_t* rows;
  float* thr;
};
// exact FP32 rerank of layer candidates -> forward lists (layer-local ids).
// Row r is layer position inv[r], or row0 + r with inv == nullptr (columns
// are then positions too).  thr: the pools' bounds (nullptr: a full pool's
// last key).  nb: the columns; a row may take those before row0 + r (causal)
// or all but itself.  inserted: rows whose pool lacks columns at distances
// that overflow are flagged too (a build's lists leave such columns out).
void launch_rerank_fwd(const float* xw, const int32_t* ids, int64_t nr, int64_t row0, int32_t dpad, int32_t metric,
                       const int32_t* inv, const uint64_t* cand, const float* thr, int64_t nb, bool causal, bool inserted,
                       int32_t KP, int32_t M, const float* norms, const float* norm_max, double tile_u, int32_t* fwd, float* fwd_d,
                       const FlaggedRows& flagged, cudaStream_t st);
// The flagged rows' BF16 planes and norms, compact; lim[i]: causal the row's
// own rank row0 + r, else nb; self[i]: r with skip_self, else -1.
void launch_gather_flagged(const FlaggedRows& f, int64_t max_rows, int64_t row0, bool causal, bool skip_self,
                           int64_t nb, const void* hi, const void* lo, const float* norms, int32_t dk, void* hi_out,
                           void* lo_out, float* norms_out, int32_t* lim, int32_t* self, cudaStream_t st);
// exact FP32 rerank of collected columns -> forward lists of the flagged
// rows; rows with more than cap columns in one CTA or without a bound (or any,
// with *err set)
// go to over (over[0]: their number, then the rows, plus row0)
void launch_rerank_collected_fwd(const float* xw, const int32_t* ids, const FlaggedRows& f, int64_t max_rows,
                                 int64_t row0, int32_t dpad, int32_t metric, const int32_t* inv, int64_t nb,
                                 unsigned grid, const uint32_t* cols, const int32_t* ncols, int32_t cap, int32_t M,
                                 int32_t* fwd, float* fwd_d, int32_t* over, const int32_t* err, cudaStream_t st);
// the same for queries (rows of Q): k results (int64 ids, reported distances)
void launch_rerank_collected_knn(const float* Q, const float* X, const FlaggedRows& f, int64_t max_rows, int32_t dpad,
                                 int32_t metric, int64_t nb, unsigned grid, const uint32_t* cols,
                                 const int32_t* ncols, int32_t cap, int32_t k, int64_t* out_ids, float* out_d,
                                 int32_t* over, const int32_t* err, cudaStream_t st);
// queries' merged tile lists -> k results, and the queries whose list does
// not prove them (thr: launch_merge_lists; err: the tile launch's flag)
void launch_rerank_knn(const float* Q, int64_t nq, const float* X, int64_t n, int32_t dpad, int32_t metric,
                       const uint64_t* cand, const float* thr, int32_t KP, int32_t k, const float* qnorms,
                       const float* norm_max, double tile_u, const int32_t* err, int64_t* out_ids, float* out_d,
                       const FlaggedRows& flagged, cudaStream_t st);
// exact recompute of the forward list of uncertified rows
void launch_exact_rows(const float* xw, const int32_t* ids, int64_t s, int32_t dpad, int32_t metric,
                       const int32_t* inv, int32_t mode, const int32_t* rows, int32_t nrows, int32_t M,
                       int32_t* fwd, float* fwd_d, cudaStream_t st);
// Exact k results by a scan of all n columns (rowsel / count, nullable: of
// the queries rowsel[0 .. *count - 1] only, their number on the device).
// Each block of kSweepRows queries has sweep_runs runs of columns (at least 128
// columns each), shared out over sweep_grid() CTAs; lists: sweep_lists(grid, nq, n)
// lists of sweep_pool(k) keys.
constexpr int kSweepRows = 32;
constexpr int kSweepMaxRuns = 128;
constexpr unsigned kSweepItems = 8;  // per CTA, unless the blocks alone are more
// Runs per block: one wave of the CTAs while there are few blocks, else the
// number of runs with the least time over all waves (10,000 queries are 313
// blocks: one run each would leave the second wave of 304 CTAs empty).
__host__ __device__ inline int32_t sweep_runs(unsigned grid, int64_t rows, int64_t n) {
  const unsigned blocks = (unsigned)((rows + kSweepRows - 1) / kSweepRows);
  const unsigned parts = (unsigned)((n + 127) / 128);
  const unsigned most = parts < (unsigned)kSweepMaxRuns ? parts : (unsigned)kSweepMaxRuns;
  unsigned pick = 1;
  if (blocks * 16 <= grid) {
    pick = grid / blocks;
  } else {
    unsigned best = ~0u;
    for (unsigned k = 1; k <= 16 && (k == 1 || blocks * k <= kSweepItems * grid); ++k) {
      const unsigned waves = (blocks * k + grid - 1) / grid;
      const unsigned cost = waves * ((parts + k - 1) / k + 1);
      if (cost < best) {
        best = cost;
        pick = k;
      }
    }
  }
  return (int32_t)(pick < most ? pick : most);
}
// for any number of rows up to nq
inline size_t sweep_lists(unsigned grid, int64_t nq, int64_t n) {
  const int64_t blocks = (nq + kSweepRows - 1) / kSweepRows, parts = (n + 127) / 128;
  const int64_t most = blocks * (parts < kSweepMaxRuns ? parts : kSweepMaxRuns);
  const int64_t runs = (int64_t)kSweepItems * grid < most ? (int64_t)kSweepItems * grid : most;
  return (size_t)kSweepRows * (size_t)(blocks > runs ? blocks : runs);
}
inline int32_t sweep_pool(int32_t k) { return k <= 32 ? 32 : (k <= 64 ? 64 : 128); }
unsigned sweep_grid();
void launch_sweep_knn(const float* Q, int64_t nq, const float* X, int64_t n, int32_t dpad, int32_t metric, int32_t k,
                     unsigned grid, uint64_t* lists, const int32_t* rowsel, const int32_t* count, int64_t* out_ids,
                     float* out_d, cudaStream_t st);
void launch_max_nonneg(const float* v, int64_t n, float* out, cudaStream_t st);

// graph.cu: edge rule
void launch_rev_count(const int32_t* fwd, int64_t s, int32_t M, int32_t* cnt, cudaStream_t st);
void launch_rev_fill(const int32_t* fwd, const float* fwd_d, int64_t s, int32_t M, const int64_t* off,
                     int32_t* fill, uint64_t* rev, cudaStream_t st);
void launch_select_adj(const int32_t* fwd, const float* fwd_d, int64_t s, int32_t M, const int64_t* off,
                       const uint64_t* rev, int32_t graph, int32_t* adj, cudaStream_t st);

}  // namespace henn
