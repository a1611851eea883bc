// Launchers of the slice-pair GEMM (kernel: slice_gemm.cuh) and its small helpers: the finishing
// kernel of a split K and the tile prefix sums of a batch.  The run-time instances of the kernel are
// compiled here, the compile-time slice counts in slice_gemm_s345.cu, slice_gemm_s678.cu and
// slice_gemm_s910.cu.
#include <algorithm>

#include "slice_gemm.cuh"

namespace ozk {

static size_t gemm_smem_bytes(int S, int BN, int nstage) {
  const size_t stage = static_cast<size_t>(S) * (GEMM_BM + BN) * 32;
  const size_t ring = GEMM_TILE_SLOTS * (BN == 64 ? sizeof(TileInfo<64>) : sizeof(TileInfo<32>));
  return 1024 + nstage * stage + ring + (2 * nstage + 20 + 2 * GEMM_TILE_SLOTS) * 8 + 16;
}

int gemm_stages(int S, int BN) {
  int n = 6;
  while (n > 0 && gemm_smem_bytes(S, BN, n) > GEMM_SMEM_MAX) --n;
  return n;
}

static int num_sms() {
  static const int n = [] {                       // initialised once, thread-safe
    int dev = 0, c = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
    return c > 0 ? c : 1;
  }();
  return n;
}

int gpu_sm_count() { return num_sms(); }

void launch_slice_gemm(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p0, int BN,
                       int max_m, int max_n, int batch, cudaStream_t st) {
  GemmParams p = p0;
  p.ntx = (2 * max_n + BN - 1) / BN;
  p.nty = (max_m + GEMM_BM - 1) / GEMM_BM;
  p.batch = batch;
  const int ky = std::min(p.box_m / GEMM_BM, p.nty), kx = std::min((2 * p.box_n) / BN, p.ntx);
  p.tpp = p.ntx * p.nty - kx * ky;
  // with exact enumeration the tile count is on the device: one persistent CTA per SM
  const long long ntiles = static_cast<long long>(p.tpp) * batch * std::max(1, p.ksplit);
  const int grid = static_cast<int>(std::min<long long>(ntiles, num_sms()));
  const size_t smem = gemm_smem_bytes(p.S, BN, p.nstage);
  // the compile-time instances hold only the fast epilogues (no integer group dumps, sums in 64 bits)
  const bool tri = !p.fullset && !p.diag_pairs && !p.wide && p.mode != EPI_GROUPS && p.mode != EPI_RESIDUES;
  const bool ks = p.ksplit > 1;
  // 23 to 63 bits (S = 3..8): compact instances of one schedule and epilogue each.  Split K has an
  // instance of its own at S = 7 only, the precision of the accuracy study's products; at S = 3..6 and 8
  // it takes the run-time instance, which was not compared with more instances
  if (tri && BN == 32 && (p.S == 9 || p.S == 10)) {
    launch_slice_gemm_s910(ta, tb, p, grid, smem, st);
  } else if (tri && BN == 64 && p.S >= 3 && p.S <= 8 && (!ks || p.S == 7)) {
    if (p.S <= 5) launch_slice_gemm_s345(ta, tb, p, grid, smem, st);
    else launch_slice_gemm_s678(ta, tb, p, grid, smem, st);
  } else if (BN == 64) {
    if (ks) launch_instance<64, 0, true>(ta, tb, p, grid, smem, st);
    else launch_instance<64, 0, false>(ta, tb, p, grid, smem, st);
  } else {
    launch_instance<32, 0, false>(ta, tb, p, grid, smem, st);
  }
  record_launch();
}

// Split K of a single problem: output (row, complex column jc) is the sum over the units of
// their exact 64-bit halves (H, L) of the real and imaginary stacked columns 2 jc, 2 jc + 1 (the
// integer sums are split between the units, so their sum is the sum the one-unit epilogue
// forms), rounded once by the same routine and combined with C in the slice GEMM's modes.
template <int G>
__global__ void __launch_bounds__(256) finish_split_kernel(const __grid_constant__ GemmParams p) {
  constexpr int NH = G < 4 ? G : 4;
  constexpr int NL = G - NH;
  constexpr int S8 = 8 * NL;
  grid_dependency_wait();
  const int m = p.m1, n = p.n1, n2 = 2 * n;
  const long long total = static_cast<long long>(m) * n;
  for (long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; idx < total;
       idx += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int row = static_cast<int>(idx % m), jc = static_cast<int>(idx / m);
    long long Hr = 0, Lr = 0, Hi = 0, Li = 0;
    for (int sp = 0; sp < p.ksplit; ++sp) {
      const longlong2 a = p.part[(static_cast<long long>(sp) * n2 + 2 * jc) * m + row];
      const longlong2 b = p.part[(static_cast<long long>(sp) * n2 + 2 * jc + 1) * m + row];
      Hr += a.x; Lr += a.y; Hi += b.x; Li += b.y;
    }
    const int E = p.e[row] + p.base_exp + p.f[jc];
    const uint32_t ehi = round_ehi<S8>(E, false);
    double zr, zi;
    if (exponent_near(E)) {
      zr = round_hl<S8>(Hr, Lr, ehi);
      zi = round_hl<S8>(Hi, Li, ehi);
    } else {
      zr = round_far(Hr, Lr, S8, E);
      zi = round_far(Hi, Li, S8, E);
    }
    double2* dst = p.C1 + row + static_cast<long long>(jc) * p.ldc1;
    if (p.mode == EPI_STORE) {
      if (p.unit_alpha) *dst = make_double2(zr, zi);
      else *dst = make_double2(p.ar * zr - p.ai * zi, p.ar * zi + p.ai * zr);
    } else if (p.mode == EPI_LU) {
      const double2 cv = *dst;
      *dst = make_double2(cv.x - zr, cv.y - zi);
    } else {
      const double2 cv = *dst;
      const double xr = p.ar * zr - p.ai * zi, xi = p.ar * zi + p.ai * zr;
      const double yr = p.br * cv.x - p.bi * cv.y, yi = p.br * cv.y + p.bi * cv.x;
      *dst = make_double2(xr + yr, xi + yi);
    }
  }
}

void launch_finish_split(const GemmParams& p, cudaStream_t st) {
  const long long total = static_cast<long long>(p.m1) * p.n1;
  const unsigned blocks = static_cast<unsigned>(std::min<long long>((total + 255) / 256, 8L * num_sms()));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1] = {pdl_attribute(st)};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  switch (p.ngroups) {
    case 1: cudaLaunchKernelEx(&cfg, finish_split_kernel<1>, p); break;
    case 2: cudaLaunchKernelEx(&cfg, finish_split_kernel<2>, p); break;
    case 3: cudaLaunchKernelEx(&cfg, finish_split_kernel<3>, p); break;
    case 4: cudaLaunchKernelEx(&cfg, finish_split_kernel<4>, p); break;
    case 5: cudaLaunchKernelEx(&cfg, finish_split_kernel<5>, p); break;
    case 6: cudaLaunchKernelEx(&cfg, finish_split_kernel<6>, p); break;
    case 7: cudaLaunchKernelEx(&cfg, finish_split_kernel<7>, p); break;
    default: cudaLaunchKernelEx(&cfg, finish_split_kernel<8>, p); break;
  }
  record_launch();
}

// Tile counts of the problems of a batched GEMM (each over its own grid, tiles wholly inside
// its skip box left out) and their exclusive prefix sums: one CTA, chunks of 1024 problems.
__global__ void __launch_bounds__(1024) tile_prefix_kernel(const int* m, const int* n, const int* skm, const int* skn,
                                                           int batch, int BN, int* out) {
  grid_dependency_wait();
  __shared__ int part[1024];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < batch; base += 1024) {
    const int z = base + static_cast<int>(threadIdx.x);
    int c = 0;
    if (z < batch && m[z] > 0 && n[z] > 0) {
      const BoxTiles bt = box_tiles(m[z], 2 * n[z], skm ? skm[z] : 0, skn ? skn[z] : 0, BN);
      c = bt.ku * bt.xu + bt.nl * bt.ntx;
    }
    part[threadIdx.x] = c;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {          // inclusive scan (Hillis-Steele)
      const int v = threadIdx.x >= static_cast<unsigned>(off) ? part[threadIdx.x - off] : 0;
      __syncthreads();
      part[threadIdx.x] += v;
      __syncthreads();
    }
    if (z < batch) out[z] = carry + part[threadIdx.x] - c;
    __syncthreads();
    if (threadIdx.x == 1023) carry += part[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[batch] = carry;
}

void launch_tile_prefix(const GemmParams& p, int BN, int batch, int* out, cudaStream_t st) {
  launch_pdl(tile_prefix_kernel, 1, 1024, st, p.m, p.n, p.skm, p.skn, batch, BN, out);
  record_launch();
}

}  // namespace ozk
