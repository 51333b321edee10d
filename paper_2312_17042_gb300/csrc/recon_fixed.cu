// recon_fixed.cu -- instantiations of the FP64 path's reconstruction (conserved variables).
#include "recon_fixed.cuh"

namespace cteno {
namespace {

template <int D, int R, int SCHEME>
cudaError_t launch_fixed(const KArgs &a, int threads, cudaStream_t s) {
  using S = TileShape<D, R, 8>;
  threads = std::min(threads, 128);  // the kernel's block: 4 warps at most
  const int64_t cells = (int64_t)(threads / 32) * S::CPW;
  const unsigned grid = (unsigned)((a.N + cells - 1) / cells);
  const size_t smem = S::PHI_BYTES + 16 + (size_t)(threads / 32) * S::WARP_BYTES;
  auto kern = recon_fixed_kernel<D, R, SCHEME>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  launch_stage_kernel(kern, grid, threads, smem, s, a);
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_recon_fixed(int dim, int degree, int scheme, const KArgs &a, int threads, cudaStream_t s) {
#define CTENO_FIXED(D, R) \
  return scheme ? launch_fixed<D, R, 1>(a, threads, s) : launch_fixed<D, R, 0>(a, threads, s)
  if (dim == 2 && degree == 2) CTENO_FIXED(2, 2);
  if (dim == 2 && degree == 3) CTENO_FIXED(2, 3);
  if (dim == 2 && degree == 4) CTENO_FIXED(2, 4);
  if (dim == 2 && degree == 5) CTENO_FIXED(2, 5);
  if (dim == 2 && degree == 6) CTENO_FIXED(2, 6);
  if (dim == 3 && degree == 2) CTENO_FIXED(3, 2);
  if (dim == 3 && degree == 3) CTENO_FIXED(3, 3);
#undef CTENO_FIXED
  return cudaErrorInvalidValue;
}

}  // namespace cteno
