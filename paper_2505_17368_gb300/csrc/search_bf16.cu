// search_bf16.cu -- the search, serving and probe kernels over BF16 rows.
#define HENN_SEARCH_ROWS
#include "search.cu"

namespace henn {

cudaError_t launch_search_bf16(const SearchArgs& a, int warps, int grid, size_t smem, int64_t beside,
                               cudaStream_t st) {
  return launch_vt<__nv_bfloat16>(a, warps, grid, smem, beside, st);
}

cudaError_t launch_serve_bf16(const ServeArgs& a, int warps, int grid, size_t smem, cudaStream_t st) {
  return launch_serve_vt<__nv_bfloat16>(a, warps, grid, smem, st);
}

cudaError_t launch_probe_bf16(const GreedyProbeArgs& a, cudaStream_t st) { return launch_probe_vt<__nv_bfloat16>(a, st); }

}  // namespace henn
