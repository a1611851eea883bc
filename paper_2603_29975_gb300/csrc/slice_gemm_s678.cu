// Compile-time slice counts 6 to 8 of the slice-pair GEMM (one of several translation units, so that
// the instances build in parallel).
#include "slice_gemm.cuh"

namespace ozk {

void launch_slice_gemm_s678(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, int grid, size_t smem,
                            cudaStream_t st) {
  if (p.S == 6) launch_instance<64, 6, false>(ta, tb, p, grid, smem, st);
  else if (p.S == 7 && p.ksplit > 1) launch_instance<64, 7, true>(ta, tb, p, grid, smem, st);
  else if (p.S == 7) launch_instance<64, 7, false>(ta, tb, p, grid, smem, st);
  else launch_instance<64, 8, false>(ta, tb, p, grid, smem, st);
}

}  // namespace ozk
