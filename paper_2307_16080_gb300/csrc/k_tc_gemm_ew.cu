// k_tc_gemm_ew.cu -- the tcgen05 GEMM variants whose elementwise program runs
// in registers (tc_gemm.cuh, EW): a translation unit of its own, because the
// inlined operations take as long to compile as every other variant.
#include "tc_gemm.cuh"

namespace nk {

uint32_t tc_ew_read_and_clear_errors() { return read_and_clear_err(); }

nk_status tc_gemm_ew_launch(const TcParams& p, const nk_schedule& s, int kind, bool ep8, int grid, int smem,
                            cudaStream_t st) {
  return ep8 ? launch_single<true, true>(p, s, kind, 1, grid, smem, st)
             : launch_single<true, false>(p, s, kind, 1, grid, smem, st);
}

}  // namespace nk
