// Compile-time slice counts 3 to 5 of the slice-pair GEMM (one of several translation units, so that
// the instances build in parallel).
#include "slice_gemm.cuh"

namespace ozk {

void launch_slice_gemm_s345(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, int grid, size_t smem,
                            cudaStream_t st) {
  if (p.S == 3) launch_instance<64, 3, false>(ta, tb, p, grid, smem, st);
  else if (p.S == 4) launch_instance<64, 4, false>(ta, tb, p, grid, smem, st);
  else launch_instance<64, 5, false>(ta, tb, p, grid, smem, st);
}

}  // namespace ozk
