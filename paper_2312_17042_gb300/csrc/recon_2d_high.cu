// recon_2d_high.cu -- instantiations of the reconstruction of central degrees 4 to 6 (2D).
#include "recon_high.cuh"

namespace cteno {

namespace {
template <int R, int SCHEME>
cudaError_t launch_high_stream(const KArgs &a, int threads, cudaStream_t s) {
  using S = TileShape<2, R, 4>;
  threads = std::min(threads, 128);  // the kernel's block: 4 warps at most
  const int64_t cells = (int64_t)(threads / 32) * S::CPW;
  const size_t smem = (size_t)(threads / 32) * S::WARP_BYTES;
  auto kern = recon_high_stream_kernel<R, SCHEME>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  launch_stage_kernel(kern, (unsigned)((a.N + cells - 1) / cells), threads, smem, s, a);
  return cudaSuccess;
}
}  // namespace

// Conserved variables on the mixed path; the characteristic reconstruction on both (conserved variables in
// FP64: recon_fixed.cu).
cudaError_t launch_recon_2d_high(int degree, int fp32, int scheme, const KArgs &a, int block, cudaStream_t s) {
  int threads = block - kLaneSchedule;
  if (!a.characteristic) {
    if (!fp32) return cudaErrorInvalidValue;
    if (block >= kHighOcc) threads = block - kHighOcc;
    if (threads < 32 || threads > 256 || threads % 32) return cudaErrorInvalidValue;
#define CTENO_HIGH(R) \
  if (degree == R) return scheme ? launch_high_stream<R, 1>(a, threads, s) : launch_high_stream<R, 0>(a, threads, s)
    CTENO_HIGH(4);
    CTENO_HIGH(5);
    CTENO_HIGH(6);
#undef CTENO_HIGH
    return cudaErrorInvalidValue;
  }
  if (threads < 32 || threads > 256 || threads % 32) return cudaErrorInvalidValue;
  const int64_t cells_per_block = (int64_t)(threads / 32) * 8;
  const unsigned grid = (unsigned)((a.N + cells_per_block - 1) / cells_per_block);
#define CTENO_HIGH(R, T, SC) launch_stage_kernel(recon_high_kernel<R, T, SC>, grid, threads, 0, s, a)
  if (degree == 4 && fp32 && scheme == 0) CTENO_HIGH(4, float, 0);
  if (degree == 4 && fp32 && scheme == 1) CTENO_HIGH(4, float, 1);
  if (degree == 5 && fp32 && scheme == 0) CTENO_HIGH(5, float, 0);
  if (degree == 5 && fp32 && scheme == 1) CTENO_HIGH(5, float, 1);
  if (degree == 6 && fp32 && scheme == 0) CTENO_HIGH(6, float, 0);
  if (degree == 6 && fp32 && scheme == 1) CTENO_HIGH(6, float, 1);
  if (degree == 4 && !fp32 && scheme == 0) CTENO_HIGH(4, double, 0);
  if (degree == 4 && !fp32 && scheme == 1) CTENO_HIGH(4, double, 1);
  if (degree == 5 && !fp32 && scheme == 0) CTENO_HIGH(5, double, 0);
  if (degree == 5 && !fp32 && scheme == 1) CTENO_HIGH(5, double, 1);
  if (degree == 6 && !fp32 && scheme == 0) CTENO_HIGH(6, double, 0);
  if (degree == 6 && !fp32 && scheme == 1) CTENO_HIGH(6, double, 1);
#undef CTENO_HIGH
  return cudaSuccess;
}

cudaError_t upload_recon_tables_2d_high(int degree, const Tables &t, cudaStream_t s) {
  if (degree == 4) return upload_high_tables<4>(t, s);
  if (degree == 5) return upload_high_tables<5>(t, s);
  if (degree == 6) return upload_high_tables<6>(t, s);
  return cudaErrorInvalidValue;
}

}  // namespace cteno
