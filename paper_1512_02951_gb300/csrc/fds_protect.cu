// Dispatch of protect, and the export of the float32 coefficients before rounding (diagnostics).
#include "fds_aux.h"
#include "fds_warp.cuh"

namespace fds {

constexpr int kDctThreads = 128;

// One thread per channel-block, through protect's own row and column passes; the four rational
// positions are exact / 8.
__global__ void __launch_bounds__(kDctThreads) dct_export_kernel(const uint8_t* __restrict__ px, int width, long long ncb,
                                                                 float* __restrict__ out) {
  const long long cb = (long long)blockIdx.x * kDctThreads + threadIdx.x;
  if (cb >= ncb) return;
  const int b = (int)(cb / 3), c = (int)(cb - 3ll * b);
  const uint8_t* blk = px + block_offset(width, b);
  const uint64_t pitch = 3ull * (uint64_t)width;
  float2 P[8][4];
#pragma unroll
  for (int y = 0; y < 8; ++y) {
    const uint2* rp = reinterpret_cast<const uint2*>(blk + y * pitch);
    row_pass(__ldg(rp), __ldg(rp + 1), __ldg(rp + 2), c, P[y]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float2 col[8];
    column_pass(P, j, col);
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        float val = l ? col[u].y : col[u].x;
        if (j == 0 && (u == 0 || u == 4)) val = (u == 0 && l == 0 ? val + 8192.0f : val) * 0.125f;
        out[64 * cb + 8 * u + pair_col(j, l)] = val;
      }
  }
}

// k is uniform over the launch when a.k >= 0; a.k < 0 (batches of mixed k) reads k per tile;
// a.pack (11 or 8: packed streams) is for one image
cudaError_t launch_protect(const TileArgs& a, cudaStream_t s, bool debug, int sms, int per_sm) {
  if (debug) {
    const long long ncb = 3ll * a.nblocks, grid = (ncb + kDctThreads - 1) / kDctThreads;
    if (grid > 0) dct_export_kernel<<<(unsigned)grid, kDctThreads, 0, s>>>(a.pixels_in, a.width, ncb, a.dbg_coefs);
    return cudaGetLastError();
  }
  return a.images ? launch_protect_plan(a, s, sms, per_sm) : launch_protect_warp(a, s, sms);
}

}  // namespace fds
