// search_fp8.cu -- the search, serving and probe kernels over FP8 E4M3 rows.
#define HENN_SEARCH_ROWS
#include "search.cu"

namespace henn {

cudaError_t launch_search_fp8(const SearchArgs& a, int warps, int grid, size_t smem, int64_t beside,
                               cudaStream_t st) {
  return launch_vt<__nv_fp8_e4m3>(a, warps, grid, smem, beside, st);
}

cudaError_t launch_serve_fp8(const ServeArgs& a, int warps, int grid, size_t smem, cudaStream_t st) {
  return launch_serve_vt<__nv_fp8_e4m3>(a, warps, grid, smem, st);
}

cudaError_t launch_probe_fp8(const GreedyProbeArgs& a, cudaStream_t st) { return launch_probe_vt<__nv_fp8_e4m3>(a, st); }

}  // namespace henn
