// gf_inst_loop.cu -- the one-kernel sweep loop of small handles with many units (FP32-12 and
// FP32-18).
#include "gf_loop.cuh"

namespace gf {

namespace {
constexpr int kMaxDev = 64;
int g_loop_grid[kMaxDev];  // blocks that fit the device together (every instance's minimum)

const void* loop_kernel(int storage, int nd) {
  if (storage == GF_FP32_12) return nd == 4 ? (const void*)k_loop<GF_FP32_12, 4> : (const void*)k_loop<GF_FP32_12, 3>;
  return nd == 4 ? (const void*)k_loop<GF_FP32_18, 4> : (const void*)k_loop<GF_FP32_18, 3>;
}
}  // namespace

// The grid that a cooperative launch may use (outside any stream capture).
cudaError_t prepare_loop() {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= kMaxDev) return cudaErrorInvalidDevice;
  if (g_loop_grid[dev] > 0) return cudaSuccess;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  int least = 1 << 30;
  for (int st : {GF_FP32_12, GF_FP32_18})
    for (int nd : {3, 4}) {
      int per_sm = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, loop_kernel(st, nd), kLoopThreads, 0);
      if (e != cudaSuccess) return e;
      if (per_sm < least) least = per_sm;
    }
  g_loop_grid[dev] = least * sms;
  return cudaSuccess;
}

cudaError_t launch_loop(int storage, int nd, LoopArgs a, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const int most = dev < kMaxDev ? g_loop_grid[dev] : 0;
  if (most <= 0) return cudaErrorInvalidConfiguration;
  const int grid = a.n_tiles < most ? a.n_tiles : most;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(loop_kernel(storage, nd), dim3(grid), dim3(kLoopThreads), args, 0, s);
}

}  // namespace gf
