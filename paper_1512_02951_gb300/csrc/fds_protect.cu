// Dispatch of protect, and the export of the float32 coefficients before rounding (diagnostics).
#include "fds_aux.h"
#include "fds_tile.cuh"

namespace fds {

constexpr int kDctThreads = 128;

// One thread per channel-block, with the operations of the protect kernels: rows from the pixel
// bytes, then columns (0 and 4 from exact integers); the four rational positions are exact / 8.
__global__ void __launch_bounds__(kDctThreads) dct_export_kernel(const uint8_t* __restrict__ px, int width, long long ncb,
                                                                 float* __restrict__ out) {
  const long long cb = (long long)blockIdx.x * kDctThreads + threadIdx.x;
  if (cb >= ncb) return;
  const int b = (int)(cb / 3), c = (int)(cb - 3ll * b);
  const uint8_t* blk = px + block_offset(width, b);
  const uint64_t pitch = 3ull * (uint64_t)width;
  float F[8][8];
#pragma unroll
  for (int y = 0; y < 8; ++y) {
    const uint2* rp = reinterpret_cast<const uint2*>(blk + y * pitch);
    const uint2 w01 = __ldg(rp), w23 = __ldg(rp + 1), w45 = __ldg(rp + 2);
    const uint32_t r[7] = {w01.x, w01.y, w23.x, w23.y, w45.x, w45.y, 0u};
    float X[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int byte = 3 * x;
      const uint32_t w = __funnelshift_r(r[byte >> 2], r[(byte >> 2) + 1], 8 * c);
      X[x] = __int_as_float(__byte_perm(w, 0x4B000000u, 0x7440u | (byte & 3)));
    }
    dct8_row_bytes(X, F[y]);
  }
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    float col[8];
#pragma unroll
    for (int y = 0; y < 8; ++y) col[y] = F[y][v];
    if (v == 0 || v == 4)
      dct8<true, true>(col);
    else
      dct8<false, false>(col);
#pragma unroll
    for (int u = 0; u < 8; ++u) F[u][v] = col[u];
  }
#pragma unroll
  for (int u = 0; u < 8; ++u)
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      float val = F[u][v];
      if (u == 0 && v == 0)
        val = (val + 8192.0f) * 0.125f;
      else if ((u == 0 || u == 4) && (v == 0 || v == 4))
        val *= 0.125f;
      out[64 * cb + 8 * u + v] = val;
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
