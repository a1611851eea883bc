// Compile-time slice counts 9 and 10 of the slice-pair GEMM (one of several translation units, so that
// the instances build in parallel).
#include "slice_gemm.cuh"

namespace ozk {

void launch_slice_gemm_s910(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, int grid, size_t smem,
                            cudaStream_t st) {
  if (p.S == 9) launch_instance<32, 9, false>(ta, tb, p, grid, smem, st);
  else launch_instance<32, 10, false>(ta, tb, p, grid, smem, st);
}

}  // namespace ozk
