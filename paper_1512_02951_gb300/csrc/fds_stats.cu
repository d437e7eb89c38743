// Statistics of an RGB image used to judge a protected image (Sect. 6.6): the histogram of
// every channel (Sect. 6.6.1) and, for the correlation coefficient of adjacent pixels
// (Sect. 6.6.2), exact integer sums over every pair of a pixel and its right, lower and
// lower-right neighbour: n, sum x, sum y, sum x^2, sum y^2, sum x y per direction and channel.
//
// One launch after the clear.  A warp takes a strip of 128 pixels and walks down a segment of its
// rows, each lane four pixels wide, so that a row is loaded once (and one row more per segment):
// the four pixels and their right neighbours are split by channel into packed bytes, and the three
// neighbour products of a channel are one 4-way byte dot product each with the row before.  The
// histogram is one shared-memory reduction per byte into counts of the lane's own (bank = lane, so
// a warp's 32 never conflict).  A level's counts lie 256 bytes apart, so one byte permute forms the
// address of a reduction.  Sum p and sum p^2 come from the histogram at the end.  What a
// direction's sums of x, y, x^2, y^2 lack of the totals are the first and last rows and columns,
// which four CTAs of their own add up; the CTA that finishes last writes the 54 sums.
//
// Four rows' loads are in flight per warp; what bounds it is their latency (4096 x 4096: 13.5 M warp
// instructions, the ALU 37 % busy, 32.9 us cold under ncu and about 28 us after the image has been
// written, against 7.5 us for the 50 MB).  A row's loads at a time took 37 us; the kernel before
// (pixel rows staged in shared memory, a byte at a time, three launches with the clears) took 114
// us and 85 M warp instructions.
#include "fds_tile.cuh"
#include "fds_aux.h"

namespace fds {

constexpr int kStatThreads = 1024;
constexpr int kStatWarps = kStatThreads / 32;
constexpr int kLanePx = 4, kStripPx = 32 * kLanePx;
constexpr int kStatRows = 8192;                   // rows of a segment at most: 32-bit product sums
// counts at fixed shared-window addresses (the dynamic area starts at or below kHistWin): level v
// of channels 0 and 1, lane L at kHistWin + 256 v + 128 c + 4 L, channel 2 64 KB on
constexpr int kHistWin = 2048;
constexpr int kHistEnd = kHistWin + 2 * 65536;
__device__ __forceinline__ constexpr uint32_t hist_off(int c) { return c == 2 ? 65536u : 128u * (uint32_t)c; }
constexpr int kBorderCtas = 4;                    // first row, last row, first column, last column

// work[]: 9 product sums [direction][channel], then 24 border sums [border][channel][p, p^2],
// then the count of finished CTAs (the pair sums' own memory until the last CTA writes them)
constexpr int kWorkBorder = 9, kWorkDone = 33;

struct StatRow {
  uint32_t p[3], r[3];   // per channel: four pixels, and the pixels to their right, as bytes
};

// the five aligned words around the 15 bytes at p (all in the image)
__device__ __forceinline__ void load_words(const uint8_t* __restrict__ p, uint32_t (&w)[5]) {
  const uint32_t* q = reinterpret_cast<const uint32_t*>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3);
#pragma unroll
  for (int i = 0; i < 5; ++i) w[i] = __ldg(q + i);
}
// the 15 bytes (and one more) out of those words
__device__ __forceinline__ void align_words(const uint8_t* p, const uint32_t (&w)[5], uint32_t (&b)[4]) {
  const uint32_t sh = 8u * (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3);
#pragma unroll
  for (int i = 0; i < 4; ++i) b[i] = __funnelshift_r(w[i], w[i + 1], sh);
}
// or byte by byte; left = bytes to the row's end
__device__ __forceinline__ void load_bytes(const uint8_t* __restrict__ p, int left, uint32_t (&b)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) b[i] = 0;
#pragma unroll 1
  for (int i = 0; i < min(15, left); ++i) {
    const uint32_t v = (uint32_t)p[i] << (8 * (i & 3));
    b[0] |= i >> 2 == 0 ? v : 0u;
    b[1] |= i >> 2 == 1 ? v : 0u;
    b[2] |= i >> 2 == 2 ? v : 0u;
    b[3] |= i >> 2 == 3 ? v : 0u;
  }
}
// four pixels and their right neighbours by channel (EDGE: zero outside the image)
template <bool EDGE>
__device__ __forceinline__ StatRow split_row(const uint32_t (&b)[4], uint32_t mask_p, uint32_t mask_r) {
  StatRow s;
  s.p[0] = __byte_perm(__byte_perm(b[0], b[1], 0x0630u), b[2], 0x5210u);   // bytes 0, 3, 6, 9
  s.p[1] = __byte_perm(__byte_perm(b[0], b[1], 0x0741u), b[2], 0x6210u);   // bytes 1, 4, 7, 10
  s.p[2] = __byte_perm(__byte_perm(b[0], b[1], 0x0052u), b[2], 0x7410u);   // bytes 2, 5, 8, 11
#pragma unroll
  for (int c = 0; c < 3; ++c) s.r[c] = __byte_perm(s.p[c], b[3], 0x4321u + ((uint32_t)c << 12));
  if (EDGE) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s.p[c] &= mask_p;
      s.r[c] &= mask_r;
    }
  }
  return s;
}

// one lane's walk down rows y0 .. y1 - 1 at column x (EDGE: the strip reaches the last column)
template <bool EDGE>
__device__ __forceinline__ void stat_walk(const uint8_t* __restrict__ img, int width, int height, int x, int y0, int y1,
                                          uint32_t lane4, uint32_t (&s)[9]) {
  const long long w3 = 3ll * width, total = w3 * height;
  const int np = EDGE ? min(kLanePx, width - x) : kLanePx, nr = EDGE ? min(kLanePx, width - 1 - x) : kLanePx;
  const uint32_t mask_p = np == 4 ? 0xffffffffu : (1u << (8 * np)) - 1u;
  const uint32_t mask_r = nr == 4 ? 0xffffffffu : (1u << (8 * nr)) - 1u;
  const int left = 3 * min(5, width - x);
  // rows whose 20-byte window around the lane's bytes lies in the image
  const int f0 = x > 0 ? 0 : (int)((3 + w3 - 1) / w3);
  const long long room = total - 20 - 3ll * x;
  const int f1 = room < 0 ? 0 : (int)min((long long)height, room / w3 + 1);
  const uint8_t* p = img + w3 * y0 + 3ll * x;
  auto row = [&](const uint8_t* q, int y) {
    uint32_t b[4];
    if (y >= f0 && y < f1) {
      uint32_t w[5];
      load_words(q, w);
      align_words(q, w, b);
    } else {
      load_bytes(q, left, b);
    }
    return split_row<EDGE>(b, mask_p, mask_r);
  };
  auto add = [&](const StatRow& cur, const StatRow& nxt) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s[c] = __dp4a(cur.p[c], cur.r[c], s[c]);
      s[3 + c] = __dp4a(cur.p[c], nxt.p[c], s[3 + c]);
      s[6 + c] = __dp4a(cur.p[c], nxt.r[c], s[6 + c]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (!EDGE || j < np)
          asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(__byte_perm(cur.p[c], lane4, 0x5504u | ((uint32_t)j << 4)) +
                                                           ((uint32_t)kHistWin + hist_off(c)))
                       : "memory");
    }
  };
  StatRow cur = row(p, y0);
  int y = y0;
  // four rows' loads in flight at a time
  const int yv = min(min(y1, height - 1), f1 - 1) - 3;
  if (y0 + 1 >= f0)
#pragma unroll 1
    for (; y < yv; y += 4) {
      uint32_t w[4][5];
#pragma unroll
      for (int i = 0; i < 4; ++i) load_words(p + (i + 1) * w3, w[i]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        p += w3;
        uint32_t b[4];
        align_words(p, w[i], b);
        const StatRow nxt = split_row<EDGE>(b, mask_p, mask_r);
        add(cur, nxt);
        cur = nxt;
      }
    }
#pragma unroll 1
  for (; y < y1; ++y) {
    p += w3;
    StatRow nxt{};
    if (y + 1 < height) nxt = row(p, y + 1);
    add(cur, nxt);
    cur = nxt;
  }
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
  for (int m = 16; m; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

__global__ void __launch_bounds__(kStatThreads, 1) image_stats_kernel(const uint8_t* __restrict__ img, int width,
                                                                      int height, int nseg, int seg_rows, int warps,
                                                                      unsigned long long* hist, long long* sums,
                                                                      unsigned long long* counters) {
  extern __shared__ __align__(16) uint8_t smem_stat[];
  __shared__ unsigned long long sh_sum[9];
  __shared__ int sh_last;
  unsigned long long* work = reinterpret_cast<unsigned long long*>(sums);
  const int t = threadIdx.x, lane = t & 31;
  const long long total = 3ll * width * height;
  const uint32_t win0 = smem_u32(smem_stat);
  if (win0 > (uint32_t)kHistWin) {   // see the launcher
    if (t == 0 && blockIdx.x == 0 && counters) atomicAdd(&counters[2], 1ull);
    return;
  }
  if ((int)blockIdx.x < kBorderCtas) {
    const int d = blockIdx.x;
    const int n = d < 2 ? width : height;
    const long long step = d < 2 ? 3 : 3ll * width;
    const uint8_t* p0 = img + (d == 1 ? total - 3ll * width : (d == 3 ? 3ll * (width - 1) : 0));
    unsigned long long s[6] = {0, 0, 0, 0, 0, 0};
    for (int i = t; i < n; i += kStatThreads)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const uint32_t p = p0[step * i + c];
        s[2 * c] += p;
        s[2 * c + 1] += p * p;
      }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const unsigned long long v = warp_sum(s[j]);
      if (lane == 0 && v) atomicAdd(&work[kWorkBorder + 6 * d + j], v);
    }
  } else {
    uint8_t* const hist_s = smem_stat + (kHistWin - win0);
    for (int i = t; i < 2 * 65536 / 16; i += kStatThreads) reinterpret_cast<uint4*>(hist_s)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (t < 9) sh_sum[t] = 0;
    __syncthreads();
    const int strips = (width + kStripPx - 1) / kStripPx;
    const long long items = (long long)strips * nseg;
    const long long ctas = gridDim.x - kBorderCtas;
    for (long long item = (t >> 5) < warps ? (blockIdx.x - kBorderCtas) * (long long)warps + (t >> 5) : items; item < items;
         item += ctas * warps) {
      const int seg = (int)(item / strips), strip = (int)(item - (long long)seg * strips);
      const int x = strip * kStripPx + lane * kLanePx;
      const int y0 = seg * seg_rows, y1 = min(height, y0 + seg_rows);
      uint32_t s[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
      if (strip * kStripPx + kStripPx < width)
        stat_walk<false>(img, width, height, x, y0, y1, 4u * lane, s);
      else if (x < width)
        stat_walk<true>(img, width, height, x, y0, y1, 4u * lane, s);
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        const unsigned long long v = warp_sum(s[j]);
        if (lane == 0 && v) atomicAdd(&sh_sum[j], v);
      }
    }
    __syncthreads();
    for (int b = t >> 5; b < 768; b += kStatWarps) {
      const uint32_t n = __reduce_add_sync(0xffffffffu, *reinterpret_cast<const uint32_t*>(hist_s + 256 * (b & 255) + hist_off(b >> 8) + 4 * lane));
      if (lane == 0 && n) atomicAdd(&hist[b], (unsigned long long)n);
    }
    if (t < 9 && sh_sum[t]) atomicAdd(&work[t], sh_sum[t]);
  }
  // the last CTA to finish writes the 54 pair sums [direction][channel][6]
  __threadfence();
  __syncthreads();
  if (t == 0) sh_last = atomicAdd(&work[kWorkDone], 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!sh_last || t >= 96) return;
  __threadfence();
  const int c = t >> 5;
  unsigned long long s1 = 0, s2 = 0;
  for (int v = lane; v < 256; v += 32) {
    const unsigned long long n = __ldcg(&hist[256 * c + v]);
    s1 += n * v;
    s2 += n * (unsigned long long)(v * v);
  }
  const long long S1 = (long long)warp_sum(s1), S2 = (long long)warp_sum(s2);
  auto w = [&](int i) { return (long long)__ldcg(&work[i]); };
  auto border = [&](int d, int j) { return w(kWorkBorder + 6 * d + 2 * c + j); };
  const long long FR1 = border(0, 0), FR2 = border(0, 1), LR1 = border(1, 0), LR2 = border(1, 1);
  const long long FC1 = border(2, 0), FC2 = border(2, 1), LC1 = border(3, 0), LC2 = border(3, 1);
  const long long right = w(c), down = w(3 + c), diag = w(6 + c);
  const long long p00 = img[c], pll = img[total - 3 + c];
  asm volatile("bar.sync 1, 96;" ::: "memory");   // the three warps have read the work area
  if (lane == 0) {
    const long long W = width, H = height;
    long long* o = sums + 6 * c;                   // direction stride 18
    o[0] = (W - 1) * H;                            // right
    o[1] = S1 - LC1;
    o[2] = S1 - FC1;
    o[3] = S2 - LC2;
    o[4] = S2 - FC2;
    o[5] = right;
    o[18] = W * (H - 1);                           // down
    o[19] = S1 - LR1;
    o[20] = S1 - FR1;
    o[21] = S2 - LR2;
    o[22] = S2 - FR2;
    o[23] = down;
    o[36] = (W - 1) * (H - 1);                     // down-right
    o[37] = S1 - LR1 - LC1 + pll;
    o[38] = S1 - FR1 - FC1 + p00;
    o[39] = S2 - LR2 - LC2 + pll * pll;
    o[40] = S2 - FR2 - FC2 + p00 * p00;
    o[41] = diag;
  }
}

__global__ void __launch_bounds__(768) stats_clear_kernel(unsigned long long* hist, long long* sums) {
  hist[threadIdx.x] = 0;
  if (threadIdx.x < 54) sums[threadIdx.x] = 0;
}

cudaError_t launch_image_stats(const uint8_t* img, int width, int height, unsigned long long* hist, long long* sums,
                               cudaStream_t s, int sms, unsigned long long* counters) {
  static bool attr[kMaxAttrDevices];
  static bool window_ok[kMaxAttrDevices];
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
  if (!window_ok[dev]) {
    if ((e = smem_window_start_ok(image_stats_kernel, (uint32_t)kHistWin)) != cudaSuccess) return e;
    window_ok[dev] = true;
  }
  e = smem_attr_once(image_stats_kernel, kHistEnd, attr);
  if (e != cudaSuccess) return e;
  // segments: one strip segment for each warp, of at least eight rows; one CTA per SM with the
  // border CTAs (a second wave would double the time)
  const int main_ctas = sms > 2 * kBorderCtas ? sms - kBorderCtas : sms;
  const long long strips = (width + kStripPx - 1) / kStripPx;
  long long nseg = (long long)main_ctas * kStatWarps / strips;
  const long long lo = ((long long)height + kStatRows - 1) / kStatRows, hi = ((long long)height + 7) / 8;
  nseg = nseg < lo ? lo : (nseg > hi ? hi : nseg);
  const int seg_rows = (int)((height + nseg - 1) / nseg);
  nseg = ((long long)height + seg_rows - 1) / seg_rows;
  // few items (up to about 640 x 480) are spread over the SMs: a CTA's 32 warps would take turns at its
  // counts (320 x 240: 22.0 -> 18.5 us); more of them share a CTA's clearing and its final sums (1600 x
  // 1200 spread out: 26.6 us against 24.2)
  const long long items = strips * nseg;
  const long long ctas = items <= 4ll * main_ctas ? (items < main_ctas ? items : main_ctas) : (items + kStatWarps - 1) / kStatWarps;
  const int grid = (int)(ctas < main_ctas ? ctas : main_ctas);
  const long long per = (items + grid - 1) / grid;
  stats_clear_kernel<<<1, 768, 0, s>>>(hist, sums);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  image_stats_kernel<<<grid + kBorderCtas, kStatThreads, kHistEnd, s>>>(
      img, width, height, (int)nseg, seg_rows, (int)(per < kStatWarps ? per : kStatWarps), hist, sums, counters);
  return cudaGetLastError();
}

}  // namespace fds
