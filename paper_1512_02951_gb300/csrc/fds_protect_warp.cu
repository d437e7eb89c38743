// Fused protect kernel in its warp form (Sect. 6.3.1, Fig. 6): 8x8 DCT-II per channel, int16
// rounding, zigzag fragmentation, AES-128-CTR of the confidential fragment, of one image.
//
// A subtile is 32 consecutive channel-blocks (cb = 3 * block + channel), one per lane; its public
// and private parts are 64 (63 - k) and 64 (k + 1) bytes, whole 16-byte units.  Each warp works
// on subtiles of its own with its own shared-memory area, and no barrier joins the warps after
// the AES table is filled.  What bounds it is the issue of instructions, not memory (4096 x 4096,
// k = 5: 41.5 M warp instructions = 33 us of issue slots against 22.6 us for the 151 MB), so the
// warps have to keep issuing.  The form before it, groups of six warps that met at three named
// barriers per 192 channel-blocks, spent its time at those barriers: 4.5 of the six warps had
// AES blocks to do, and issue activity was 57 %; here it is 72 %.  Per subtile:
//   1. its pixels are in the warp's buffer (bulk copies that complete on the warp's mbarrier);
//      row butterflies; the buffer is free, so the next subtile's pixels start loading
//   2. column butterflies by pairs of columns, rounded and written as int16 to the staging area;
//      a pair of columns in which some lane has a value within the error guard of a
//      half-integer (one three-input maximum per two values, one vote) marks those values
//   3. marked values are decided exactly, four at a time (decide_ties), in place
//   4. the public part leaves (bulk store); the private parts of several subtiles are collected
//      until their keystream blocks fill whole warps (k = 5: 24 blocks each, four subtiles fill
//      three), encrypted, and leave
// Counter blocks that share all but their last byte share the first AES round and most of the
// second (aes_window): 133 table lookups a block instead of 160.
// Measured on 4096 x 4096, k = 5: 72.3 -> 53.5 us; 3240 x 2592, k = 9: 55.9 -> 37.2 us (before:
// the grouped form; its 8-byte pixel loads and 240 AES blocks on 192 threads cost the latter
// more).  16 warps of 128 registers; 20 of 96 measured 53.6 and 39.6 us, with spills.  Pixels two
// subtiles ahead, or loaded with cp.async through L1, measured slower (59 / 64 us against 51 and
// 53 us with exact decisions left out): the shared memory taken leaves L1 too small for them.
#include "fds_aux.h"
#include "fds_warp.cuh"

namespace fds {

// one pixel row of a subtile: at most 12 blocks, in at most two segments that each start and end
// on 16-byte boundaries
constexpr int kWPixPitch = 320;
constexpr int kWPixBytes = 8 * kWPixPitch;
constexpr int kWStageBytes = 5248;                // public part, then the private parts of kAcc subtiles
constexpr int kWPix = 0;
constexpr int kWStage = kWPix + kWPixBytes;
constexpr int kWList = kWStage + kWStageBytes;    // the staged private parts' subtiles
constexpr int kWBar = kWList + 4 * 8;             // mbarrier of the pixel loads
constexpr int kWArea = (kWBar + 8 + 31) & ~31;
constexpr int kWWinBytes = 20 * kWins + 16;       // and the CTA's subtile counter
constexpr int kBelow = ((int)kTpairWin - 1024) / kWArea;    // areas below the pair table
constexpr int kWLow = (int)kTpairWin - kBelow * kWArea;     // window address of the first
constexpr int kAbove = kWarps > kBelow ? kWarps - kBelow : 0;
constexpr int kWWin = (int)kTpairWin + kTpairBytes + kAbove * kWArea;
constexpr int kWEnd = kWWin + kWWinBytes;
static_assert(kWEnd <= 227 * 1024, "protect (warp form) shared memory");

// subtiles whose private parts are encrypted together: the fewest lanes left idle in the last
// round of 32 keystream blocks, as far as the staging area holds them
__host__ __device__ constexpr int acc_tiles(int k) {
  int best = 1, bn = 4 * (k + 1), bp = (bn + 31) / 32;
  for (int g = 2; g <= 8; ++g) {
    if ((63 - k) * 64 + g * (k + 1) * 64 > kWStageBytes) break;
    const int n = g * 4 * (k + 1), p = (n + 31) / 32;
    if (n * bp > bn * p) {
      best = g;
      bn = n;
      bp = p;
    }
  }
  return best;
}

// Where a lane's channel-block lies in the pixel buffer: byte offsets of its block in even and
// odd pixel rows, plus the channel
struct PixAt {
  uint32_t even, odd, c;
};

// The pixels of the subtile of n channel-blocks at lane position p into the warp's pixel buffer.
// BULK: one bulk copy per pixel row and run of blocks (a subtile lies in at most two block rows:
// bx_count >= 12), each widened to 16-byte boundaries inside the image (its base is 16-byte
// aligned and it is a multiple of 64 bytes long); lanes 0..7 copy the first run, 8..15 the second.
// Else 8-byte pieces: lane's piece c of its block in 8 rows, then the pieces of the two boundary
// blocks that other subtiles' lanes own.
template <bool BULK>
__device__ __forceinline__ PixAt load_subtile(const uint8_t* img, uint64_t pitch, uint32_t bx_count, const CbPos& p,
                                              uint32_t n, int lane, uint32_t pix, uint64_t* bar) {
  const uint32_t c0 = __shfl_sync(0xffffffffu, p.c, 0);
  PixAt at;
  at.c = p.c;
  if constexpr (BULK) {
    const uint32_t bx0 = __shfl_sync(0xffffffffu, p.bx, 0), by0 = __shfl_sync(0xffffffffu, p.by, 0);
    const uint32_t nblk = (c0 + n + 2) / 3;                       // blocks the subtile touches
    const uint32_t m0 = min(nblk, bx_count - bx0);    // in the first block row
    const uint32_t odd = (uint32_t)pitch & 8u;                    // skew change from row to row
    const uint32_t sk0 = (24u * bx0) & 8u;                        // skew of even rows, first run
    const uint32_t seg1 = (24u * m0 + 8u + 15u) & ~15u;           // where the second run starts
    // 8 * pitch is a multiple of 64, so a block row's even rows have the same skew
    {
      const bool second = lane >= 8;
      const uint32_t y = lane & 7;
      const uint32_t m = second ? nblk - m0 : m0;
      const uint32_t bx = second ? 0u : bx0, by = by0 + (second ? 1u : 0u);
      const uint64_t off = ((uint64_t)by * 8 + y) * pitch + 24ull * bx;
      const uint64_t lo = off & ~15ull, hi = (off + 24ull * m + 15) & ~15ull;
      const bool on = lane < 16 && m > 0;
      const uint32_t bytes = on ? (uint32_t)(hi - lo) : 0u;
      const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
      if (lane == 0) mbar_expect_tx(bar, total);
      __syncwarp();
      if (on)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                         pix + y * kWPixPitch + (second ? seg1 : 0u)),
                     "l"(img + lo), "r"(bytes), "r"(smem_u32(bar))
                     : "memory");
    }
    const bool in1 = p.by != by0;
    const uint32_t base = in1 ? seg1 + 24u * p.bx : 24u * (p.bx - bx0), sk = in1 ? 0u : sk0;
    at.even = base + sk;
    at.odd = base + (sk ^ odd);
  } else {
    const uint64_t off = (uint64_t)p.by * (8 * pitch) + 24ull * p.bx;
    const uint8_t* src = img + off + 8 * p.c;
    const uint32_t dst = pix + 8 * (c0 + lane);
    if ((uint32_t)lane < n) {
#pragma unroll
      for (int y = 0; y < 8; ++y) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst + y * kWPixPitch), "l"(src) : "memory");
        src += pitch;
      }
    }
    const uint32_t e1 = n == 32 ? (c0 == 0 ? 1u : (c0 == 1 ? 0u : 2u)) : 0u;
    const uint32_t y = lane >> 2, sl = lane & 3;
    const bool head = sl < c0;
    const uint64_t eoff = __shfl_sync(0xffffffffu, off, head ? 0 : 31);
    if (sl < c0 + e1) {
      const uint32_t q = head ? sl : sl - c0 + (3 - e1);            // piece of the block
      const uint32_t j = head ? sl : c0 + 32 + (sl - c0);           // its place in the row
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(pix + y * kWPixPitch + 8 * j),
                   "l"(img + eoff + y * pitch + 8 * q)
                   : "memory");
    }
    cp_async_commit();
    at.even = at.odd = 8 * (c0 + lane - p.c);
  }
  return at;
}

// AES-128-CTR over the first `total` keystream blocks of staged private parts (subtiles list[0 ..],
// nb = 4 (k + 1) blocks each); wc: the constants of the windows from wbase on
__device__ __forceinline__ void ctr_warp(const TileArgs& a, uint8_t* buf, const uint32_t* list, uint32_t total, uint32_t nb,
                                         const uint32_t* wc, uint64_t wbase, int lane) {
  const PairLanes lc = pair_lanes();
#pragma unroll 1
  for (uint32_t i = lane; i < total; i += 32) {
    const uint32_t j = i / nb;
    const uint64_t b = (a.iv_lo & 255u) + (uint64_t)list[j] * nb + (i - j * nb);   // from the IV's window
    const uint32_t* src = wc + 5 * (uint32_t)((b >> 8) - wbase);
    const uint32_t w[5] = {src[0], src[1], src[2], src[3], src[4]};
    uint32_t s[4];
    aes_from_window(w, (uint32_t)b & 255u, a.rk, lc, s);
    uint4* p = reinterpret_cast<uint4*>(buf + 16 * i);
    uint4 d = *p;
    if (a.plain_out) {
      const uint64_t at = 16 * ((uint64_t)list[j] * nb + (i - j * nb));
      if (at < 6ull * (uint32_t)a.nblocks * (nb >> 2)) *reinterpret_cast<uint4*>(a.plain_out + at) = d;
    }
    d.x ^= s[0];
    d.y ^= s[1];
    d.z ^= s[2];
    d.w ^= s[3];
    *p = d;
  }
}

// `bytes` staged bytes to global memory by one lane: a bulk store and a tail of 2-byte stores
__device__ __forceinline__ void store_run(uint8_t* dst, const uint8_t* src, int bytes) {
  if (bytes >> 4) bulk_store(dst, src, (uint32_t)(bytes & ~15));
  bulk_commit();
  for (int j = bytes & ~15; j < bytes; j += 2)
    *reinterpret_cast<uint16_t*>(dst + j) = *reinterpret_cast<const uint16_t*>(src + j);
}

// Row butterflies of a lane's channel-block from its pixel buffer; returns their error weight
__device__ __forceinline__ float transform_rows(const uint8_t* px_even, const uint8_t* px_odd, uint32_t c, float2 (&P)[8][4]) {
  float V = 0.0f;
#pragma unroll
  for (int y = 0; y < 8; ++y) {
    const uint2* rp = reinterpret_cast<const uint2*>((y & 1 ? px_odd : px_even) + y * kWPixPitch);
    V += row_pass(rp[0], rp[1], rp[2], c, P[y]);
  }
  return V;
}

// Column butterflies, rounding and staging of a lane's channel-block (z = 0 .. k at priv_cb, the
// rest at pub_cb); bit 8 u + v of mhi:mlo marks a value within the error guard of a half-integer
// (none where the lane is not live)
__device__ __forceinline__ void stage_columns(const float2 (&P)[8][4], float V, int k, bool live, int16_t* pub_cb,
                                              int16_t* priv_cb, uint32_t& mlo, uint32_t& mhi) {
  auto put = [&](int u, int v, uint32_t q) {
    const int z = zigzag_of(u, v);
    if (z <= k)
      priv_cb[z] = (int16_t)q;
    else
      pub_cb[z - k - 1] = (int16_t)q;
  };
  mlo = mhi = 0;
  float thr = 1.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {          // a pair of columns: transformed, rounded and staged
    float2 col[8];
    const float W = column_pass(P, j, col);
    if (j == 0 && live) thr = 0.5f - fminf(fmaf(V, kGuardV, fmaf(W, kGuardW, kGuardU)), kGuardFwd);
    float big = 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if ((u == 0 || u == 4) && j == 0) {
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const int v = pair_col(0, l);
          const int T = __float_as_int((l ? col[u].y : col[u].x) + kMagic) - kMagicBits;  // 8 F, exact
          put(u, v, (uint32_t)((u == 0 && v == 0) ? ((T + 4) >> 3) + 1024 : (T + 4 - (T < 0 ? 1 : 0)) >> 3));
        }
        col[u] = make_float2(0.0f, 0.0f);
      } else {
        const float2 yv = add2(col[u], make_float2(kMagic, kMagic));
        col[u] = sub2(col[u], add2(yv, make_float2(-kMagic, -kMagic)));
        put(u, pair_col(j, 0), __float_as_uint(yv.x));   // low 16 bits: the int16 result
        put(u, pair_col(j, 1), __float_as_uint(yv.y));
        big = fmaxf(fmaxf(big, fabsf(col[u].x)), fabsf(col[u].y));
      }
    }
    if (__any_sync(0xffffffffu, big > thr)) {   // rare: a near tie in these columns
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const int v = pair_col(j, l);
          if (fabsf(l ? col[u].y : col[u].x) > thr) {
            if (8 * u + v < 32)
              mlo |= 1u << (8 * u + v);
            else
              mhi |= 1u << (8 * u + v - 32);
          }
        }
    }
  }
}

constexpr int kTieFrac = 46;
// Where kSideBySide lanes or more have marked values, each decides one of its own in turn, until fewer
// have any left; returns the lane's, and those too near a boundary for fixed point.  blk, pub_cb, priv_cb:
// the lane's own.  Two pixel rows at a time (all eight held spilled); a function of its own, because
// inside the kernel its code slowed down what runs without it (batch of 1000 images, k = 0: 863 us
// against 782).  Below eight lanes two turns at most do (tie block: turns alone 117 us, with it 39.5).
constexpr int kSideBySide = 8;
__device__ __noinline__ uint64_t decide_side_by_side(const uint8_t* blk, uint64_t pitch, uint32_t c, int k, uint32_t mlo,
                                                     uint32_t mhi, int16_t* pub_cb, int16_t* priv_cb, const uint32_t* table) {
  uint32_t hlo = 0, hhi = 0;               // too near a boundary: by a group after all
  do {
    if (mlo | mhi) {
      const int pos = mlo ? __ffs(mlo) - 1 : __ffs(mhi) + 31;
      const uint8_t* row = blk;
      int n[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
      for (int g = 0; g < 4; ++g) {
        const uint4* t4 = reinterpret_cast<const uint4*>(table + pos * 128) + g;
        uint32_t P[4];
        pixel_row_global(row, c, P[0], P[1]);
        pixel_row_global(row + pitch, c, P[2], P[3]);
        row += 2 * pitch;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint4 w = __ldg(t4 + 4 * j);
          n[j] = dp4a_us(P[1], w.y, dp4a_us(P[0], w.x, n[j]));
          n[j] = dp4a_us(P[3], w.w, dp4a_us(P[2], w.z, n[j]));
        }
      }
      bool sure;
      const int q = round_lane<kTieFrac>(n, sure), z = c_zigzag.z[pos];
      *(z <= k ? priv_cb + z : pub_cb + (z - k - 1)) = (int16_t)q;
      const uint32_t lo = mlo & -mlo, hi = mlo ? 0u : mhi & -mhi;
      mlo ^= lo;
      mhi ^= hi;
      if (!sure) hlo |= lo, hhi |= hi;
    }
  } while (__popc(__ballot_sync(0xffffffffu, (mlo | mhi) != 0)) >= kSideBySide);
  return (uint64_t)(mhi | hhi) << 32 | (mlo | hlo);
}

// The marked values of a subtile, decided exactly (take_ties) and staged.  block(): the lane's own
// block in the image; pub0, priv0: the first lane's place in the staging area; table: a.cfwd, whose
// row of a position holds eight words a coordinate pair: a lane takes a pixel row and its two words.
// |n_j| <= 2 . 64 . 255 and so is their sum, so 46 fraction bits fit.
template <typename Block>
__device__ __forceinline__ void decide_ties(Block block, uint64_t pitch, uint32_t c, int k, uint32_t mlo, uint32_t mhi,
                                            int16_t* pub0, int16_t* priv0, const uint32_t* table, int lane, int& nties,
                                            int& esc, bool& fail) {
  uint32_t who = __ballot_sync(0xffffffffu, (mlo | mhi) != 0);
  if (__builtin_expect(who == 0, 1)) return;
  // read here, so that what depends on it is not kept through the subtiles without near ties
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
  nties += (int)__reduce_add_sync(0xffffffffu, (uint32_t)(__popc(mlo) + __popc(mhi)));
  const unsigned long long blk = reinterpret_cast<unsigned long long>(block());
  const long long cos_l = group_cos<kTieFrac>(lane);
  const int l = lane & 7;
  if (__popc(who) >= kSideBySide) {
    const uint64_t left = decide_side_by_side(reinterpret_cast<const uint8_t*>(blk), pitch, c, k, mlo, mhi,
                                              pub0 + lane * (63 - k), priv0 + lane * (k + 1), table);
    mlo = (uint32_t)left;
    mhi = (uint32_t)(left >> 32);
    who = __ballot_sync(0xffffffffu, left != 0);
  }
  while (who) {
    const TieTurn t = take_ties(who, mlo, mhi, lane);
    const uint8_t* row = reinterpret_cast<const uint8_t*>(__shfl_sync(0xffffffffu, blk, t.src)) + l * pitch;
    const uint32_t sc = __shfl_sync(0xffffffffu, c, t.src);
    int n[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (t.on) {
      const uint2* w2 = reinterpret_cast<const uint2*>(table + t.pos * 128) + l;
      uint32_t lo, hi;
      pixel_row_global(row, sc, lo, hi);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint2 w = __ldg(w2 + 8 * j);
        n[j] = dp4a_us(hi, w.y, dp4a_us(lo, w.x, 0));
      }
    }
    const int q = round_group<kTieFrac, 1 << 15>(group_sum(n, lane), cos_l, t.on, lane, esc, fail);
    if (t.on && l == 0) {
      const int z = c_zigzag.z[t.pos];
      *(z <= k ? priv0 + t.src * (k + 1) + z : pub0 + t.src * (63 - k) + (z - k - 1)) = (int16_t)q;
    }
    who = __ballot_sync(0xffffffffu, (mlo | mhi) != 0);
  }
}

// ---- packed storage (Sect. 6.4.3, Table 5): after a subtile's ties are decided its staged
// coefficients are packed, the public part in place and out at once, the private parts of a few
// subtiles side by side until they are encrypted.  The packing itself is the cost (11 bits: 60.9 M
// warp instructions for 4096 x 4096, k = 5, against 41.5 M for int16): 78 us a launch, 104 us in
// the grouped form, 101 us before private words were built per channel-block and fields were
// placed by multiply-adds.

// field code of AC value v in W bits: sign-magnitude; 8-bit storage saturates the magnitude, in 11
// bits none is too large (|AC| <= 255 sum |basis| / 2 <= 1020)
template <int W>
__device__ __forceinline__ uint32_t ac_code(int v) {
  const int s = v >> 31;
  int mag = (v ^ s) - s;
  if (W < 11) mag = min(mag, (1 << (W - 1)) - 1);
  // a zero has no sign: s is 0 there
  return ((uint32_t)s & (1u << (W - 1))) | (uint32_t)mag;
}
// w |= c << b for a field that does not overlap what w holds: a multiply-add, off the ALU
__device__ __forceinline__ uint32_t put_bits(uint32_t w, uint32_t c, int b) { return c * (1u << b) + w; }

// bytes of a full subtile's packed public and private part (multiples of 4, so that a subtile's
// part of either stream starts on a word of it)
template <int W>
__device__ __forceinline__ uint32_t pack_pub_bytes(int k) {
  return 4u * (uint32_t)((63 - k) * W);
}
template <int W>
__host__ __device__ constexpr uint32_t pack_priv_bytes(int k) {
  return 4u * (uint32_t)(kDcBits + k * W);
}
// packed private parts encrypted together: as many as leave the fewest lanes idle in the rounds of
// 32 keystream blocks (a run of n parts overlaps at most 16-byte blocks of its bytes and one more),
// as far as the area behind the int16 coefficients holds them; 0: none, packed in place
constexpr int kPackAcc = kWStageBytes - kWCb * 128;
template <int W>
__host__ __device__ constexpr int pack_acc_tiles(int k) {
  const int per = (int)pack_priv_bytes<W>(k);
  int best = 0, bn = 0, bp = 1;
  for (int g = 1; g <= 8 && g * per <= kPackAcc; ++g) {
    const int n = g * per, p = (n / 16 + 1 + 31) / 32;
    if (!best || n * bp > bn * p) {
      best = g;
      bn = n;
      bp = p;
    }
  }
  return best;
}

// Pack the staged int16 public coefficients of n channel-blocks in place: fields f (int16 at
// pub + f) in groups of 32; group g fills words [W g, W g + W).  Each round reads its inputs into
// registers before it writes, and the words it writes lie below what later rounds read (32 fields
// are 64 bytes as int16, at most 44 packed).
template <int W>
__device__ __forceinline__ void pack_public(int16_t* pub, int n, int npub, int lane) {
  const int nf = n * npub, ngroups = (nf + 31) >> 5;
  uint32_t* const pubw = reinterpret_cast<uint32_t*>(pub);
#pragma unroll 1
  for (int r0 = 0; r0 < ngroups; r0 += 32) {
    const int g = r0 + lane;
    uint32_t pw[W];
#pragma unroll
    for (int j = 0; j < W; ++j) pw[j] = 0;
    if (g < ngroups) {
      const int f0 = 32 * g;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        // fields past the last one are zero padding (the area behind them is readable)
        const uint4 x = reinterpret_cast<const uint4*>(pub + f0)[q];
        const uint32_t u[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const int i = 8 * q + m;
          int v = (int)(u[m >> 1] << (m & 1 ? 0 : 16)) >> 16;
          if (f0 + i >= nf) v = 0;
          const uint32_t c = ac_code<W>(v);
          const int b = W * i;
          pw[b >> 5] = put_bits(pw[b >> 5], c, b & 31);
          if ((b & 31) + W > 32) pw[(b >> 5) + 1] |= c >> (32 - (b & 31));
        }
      }
    }
    __syncwarp();
    if (g < ngroups) {
#pragma unroll
      for (int j = 0; j < W; ++j) pubw[W * g + j] = pw[j];
    }
    __syncwarp();
  }
}

// Pack the staged int16 private coefficients of n channel-blocks to dst (their own place, or the
// area behind them): word j gathers the fields overlapping bits [32 j, 32 j + 32); a channel-block
// takes 11 + k W bits.  In place, a round's words lie below what later rounds read (a word holds
// at least 2.9 fields, which took 5.8 bytes).
template <int W>
__device__ __forceinline__ void pack_private(const int16_t* priv, uint32_t* dst, int n, int k, int lane) {
  const int period = kDcBits + k * W, pbits = n * period, nwords = (pbits + 31) >> 5;
#pragma unroll 1
  for (int r0 = 0; r0 < nwords; r0 += 32) {
    const int g = r0 + lane;
    uint32_t vw = 0;
    if (g < nwords) {
      const int bit = 32 * g, end = min(bit + 32, pbits);
      int cb = bit / period;
      const int r = bit - cb * period;
      int z = r < kDcBits ? 0 : 1 + (r - kDcBits) / W;
      int pos = cb * period + (z == 0 ? 0 : kDcBits + (z - 1) * W);
      while (pos < end) {
        const int v = priv[cb * (k + 1) + z];
        const uint32_t c = z == 0 ? ((uint32_t)v & 0x7ffu) : ac_code<W>(v);
        const int sh = pos - bit;   // in (-11, 32)
        vw |= sh >= 0 ? c << sh : c >> (-sh);
        pos += z == 0 ? kDcBits : W;
        if (++z > k) {
          z = 0;
          ++cb;
        }
      }
    }
    __syncwarp();
    if (g < nwords) dst[g] = vw;
    __syncwarp();
  }
}

// The same for a k known here, to an area of its own: a lane's channel-block as words, shifted to
// its place and merged in (pack_private took a third of the packing's instructions at k = 5)
template <int K, int W>
__device__ __forceinline__ void pack_private_k(const int16_t* priv, uint32_t* dst, int n, int lane) {
  constexpr int kPeriod = kDcBits + K * W, kWords = (kPeriod + 31) / 32;
#pragma unroll 1
  for (int i = lane; i < kPeriod; i += 32) dst[i] = 0;       // 32 channel-blocks: kPeriod words
  uint32_t w[kWords + 1];
#pragma unroll
  for (int i = 0; i <= kWords; ++i) w[i] = 0;
#pragma unroll
  for (int z = 0; z <= K; ++z) {
    const int v = priv[lane * (K + 1) + z];
    const uint32_t c = z == 0 ? ((uint32_t)v & 0x7ffu) : ac_code<W>(v);
    const int b = z == 0 ? 0 : kDcBits + (z - 1) * W, fw = z == 0 ? kDcBits : W;
    w[b >> 5] = put_bits(w[b >> 5], c, b & 31);
    if ((b & 31) + fw > 32) w[(b >> 5) + 1] |= c >> (32 - (b & 31));
  }
  __syncwarp();
  if (lane < n) {
    const int at = lane * kPeriod, sh = at & 31;
    uint32_t* const q = dst + (at >> 5);
#pragma unroll
    for (int i = 0; i <= kWords; ++i) {
      const uint32_t x = __funnelshift_l(i > 0 ? w[i - 1] : 0u, w[i], sh);   // w[kWords] holds no bits
      if (x) atomicOr(q + i, x);
    }
  }
  __syncwarp();
}

// AES-128-CTR over the packed bytes [off, off + bytes) of the private stream at w (off a multiple
// of 4): a lane per keystream block they overlap; a block that two warps' parts share is generated
// by both, each XORing its own words
__device__ __forceinline__ void ctr_packed(const TileArgs& a, uint32_t* w, uint64_t off, int bytes, int lane) {
  const PairLanes lc = pair_lanes();
  const uint64_t b0 = off >> 4;
  const int nblk = (int)(((off + (uint64_t)bytes + 15) >> 4) - b0);
  const int nw = (bytes + 3) >> 2, skew = (int)((off & 15) >> 2);
#pragma unroll 1
  for (int i = lane; i < nblk; i += 32) {
    uint32_t s[4];
    ctr_block(a.iv_hi, a.iv_lo, b0 + i, s);
    aes128_encrypt_pair(s, a.rk, lc);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int wi = 4 * i + m - skew;
      if (wi >= 0 && wi < nw) w[wi] ^= s[m];
    }
  }
}

// packed bytes to a stream by the whole warp, as wide as the destination is aligned
__device__ __forceinline__ void store_packed(uint8_t* dst, const uint8_t* src, int bytes, int lane) {
  const uintptr_t al = reinterpret_cast<uintptr_t>(dst);
  if ((al & 7) == 0) {
    for (int i = lane; i < (bytes >> 3); i += 32) reinterpret_cast<uint2*>(dst)[i] = reinterpret_cast<const uint2*>(src)[i];
    if (lane < (bytes & 7)) dst[(bytes & ~7) + lane] = src[(bytes & ~7) + lane];
  } else if ((al & 3) == 0) {
    for (int i = lane; i < (bytes >> 2); i += 32)
      reinterpret_cast<uint32_t*>(dst)[i] = reinterpret_cast<const uint32_t*>(src)[i];
    if (lane < (bytes & 3)) dst[(bytes & ~3) + lane] = src[(bytes & ~3) + lane];
  } else {
    for (int i = lane; i < bytes; i += 32) dst[i] = src[i];
  }
}

// PACK: 0 = int16 fragments; 11 or 8 = packed streams
template <int K, bool BULK, int PACK = 0>
__global__ void __launch_bounds__(kWarps * 32, 1) protect_warp_kernel(const __grid_constant__ TileArgs a) {
  extern __shared__ __align__(128) uint8_t smem_cta[];
  const uint32_t win0 = smem_u32(smem_cta);
  if (win0 > (uint32_t)kWLow) {   // see the launcher
    if (threadIdx.x == 0 && a.counters) atomicAdd(&a.counters[2], 1ull);
    return;
  }
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  uint8_t* area = smem_cta + ((warp < kBelow ? (uint32_t)(kWLow + warp * kWArea)
                                             : kTpairWin + kTpairBytes + (uint32_t)(warp - kBelow) * kWArea) -
                              win0);
  const uint32_t pix = smem_u32(area + kWPix);
  uint8_t* stage = area + kWStage;
  uint64_t* bar = reinterpret_cast<uint64_t*>(area + kWBar);
  uint32_t* list = reinterpret_cast<uint32_t*>(area + kWList);
  uint32_t* wins = reinterpret_cast<uint32_t*>(smem_cta + (kWWin - win0));
  uint32_t* next = wins + 5 * kWins;
  const int k = K >= 0 ? K : a.k;
  const int npub = 63 - k;
  const uint32_t nb = 4u * (uint32_t)(k + 1);       // keystream blocks per subtile
  const uint32_t ncb = 3u * (uint32_t)a.nblocks, nsub = (ncb + 31u) >> 5;
  const int act = a.groups;       // working warps of each CTA
  // the CTA's subtiles [s0, s1): taken one by one by its warps (dynamic), which evens out the
  // last round of a small image, or, where their counter windows are more than the table holds,
  // a run for each warp
  const uint32_t s0 = (uint32_t)((uint64_t)nsub * blockIdx.x / gridDim.x);
  const uint32_t s1 = (uint32_t)((uint64_t)nsub * (blockIdx.x + 1) / gridDim.x);
  const uint32_t iv8 = (uint32_t)a.iv_lo & 255u;
  uint64_t wbase = (iv8 + (uint64_t)s0 * nb) >> 8;
  const uint64_t wlast = (iv8 + (uint64_t)s1 * nb - 1) >> 8;
  const bool dynamic = PACK == 0 && wlast - wbase < kWins;
  uint32_t t = s1, tend = s1;
  if (warp < act) {
    t = dynamic ? s0 + warp : s0 + (uint32_t)((uint64_t)(s1 - s0) * warp / act);
    if (!dynamic) tend = s0 + (uint32_t)((uint64_t)(s1 - s0) * (warp + 1) / act);
  }
  const uint64_t pitch = 3ull * (uint64_t)a.width;
  if (BULK && lane == 0) {
    mbar_init(bar);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  PixAt at{};
  Loads ld;
  auto load = [&](uint32_t s) {
    at = load_subtile<BULK>(a.pixels_in, pitch, (uint32_t)a.bx_count, cb_pos(a, 32u * s + lane), min(32u, ncb - 32u * s), lane,
                            pix, bar);
    if (BULK) ld.issued(0);
  };
  if (t < tend) load(t);
  if (threadIdx.x == 0) *next = s0 + act;
  fill_pair_table(smem_cta + (kTpairWin - win0), a.T, (int)threadIdx.x, kWarps * 32);
  __syncthreads();
  if (PACK == 0 && !a.plain_private) {
    if (dynamic) {
      const int i = (int)threadIdx.x;
      if ((uint32_t)(i & ~31) <= wlast - wbase) put_window(a, wbase + i, (uint32_t)i <= wlast - wbase ? i : -1, wins);
      __syncthreads();
    } else {
      wins += 10 * warp;
      wbase = ~0ull - 1;
    }
  }

  constexpr int kG = K >= 0 ? acc_tiles(K >= 0 ? K : 0) : 0;
  const int G = K >= 0 ? kG : a.run_tiles;           // subtiles between two AES phases
  int esc = 0, nties = 0;
  bool fail = false, lost = false;         // exact_round failed; a load did not arrive in time
  int acc = 0;
  int16_t* const pubst = reinterpret_cast<int16_t*>(stage);
  uint8_t* const privst = stage + kWCb * 2 * npub;

  while (t < tend) {
    uint32_t tn = t + 1;                   // the warp's next subtile
    if (dynamic) {
      if (lane == 0) tn = atomicAdd(next, 1u);
      tn = __shfl_sync(0xffffffffu, tn, 0);
    }
    const uint32_t n = min(32u, ncb - 32u * t);
    if constexpr (BULK) {
      if (!load_wait(ld, bar, 0)) {        // gave up: nothing more is written
        lost = true;
        break;
      }
    } else {
      cp_async_wait_all();
      __syncwarp();
    }
    const uint32_t c = at.c;
    const uint8_t* px_even = area + kWPix + at.even;
    const uint8_t* px_odd = area + kWPix + at.odd;
    float2 P[8][4];
    const float V = transform_rows(px_even, px_odd, c, P);
    __syncwarp();                          // the pixel buffer is read: the next subtile's load starts
    if (tn < tend) load(tn);
    bulk_wait_read_all();                  // the staging area may be written again
    __syncwarp();
    int16_t* pub_cb = pubst + lane * npub;
    int16_t* priv_cb = reinterpret_cast<int16_t*>(privst) + ((PACK ? 0 : acc * kWCb) + lane) * (k + 1);
    uint32_t mlo, mhi;
    stage_columns(P, V, k, (uint32_t)lane < n, pub_cb, priv_cb, mlo, mhi);
    decide_ties(
        [&] {
          const CbPos p = cb_pos(a, 32u * t + lane);
          return a.pixels_in + (uint64_t)p.by * (8 * pitch) + 24ull * p.bx;
        },
        pitch, c, k, mlo, mhi, pubst, priv_cb - lane * (k + 1), a.cfwd, lane, nties, esc, fail);
    if constexpr (PACK != 0) {
      constexpr int kPW = PACK ? PACK : 8;
      __syncwarp();                        // every staged coefficient is final
      pack_public<kPW>(pubst, (int)n, npub, lane);
      store_packed(reinterpret_cast<uint8_t*>(a.pub_out) + (uint64_t)t * pack_pub_bytes<kPW>(k), stage,
                   ((int)n * npub * kPW + 7) >> 3, lane);
      const uint32_t per = pack_priv_bytes<kPW>(k);
      const int GP = K >= 0 ? pack_acc_tiles<kPW>(K >= 0 ? K : 0) : a.run_tiles;
      uint8_t* const pst = GP ? stage + kWCb * 128 : privst;
      if constexpr (K >= 0 && pack_acc_tiles<kPW>(K >= 0 ? K : 0) > 0)
        pack_private_k<K, kPW>(reinterpret_cast<const int16_t*>(privst), reinterpret_cast<uint32_t*>(pst + acc * per), (int)n,
                               lane);
      else
        pack_private<kPW>(reinterpret_cast<const int16_t*>(privst), reinterpret_cast<uint32_t*>(pst + acc * per), (int)n, k,
                          lane);
      ++acc;
      if (acc >= GP || tn >= tend) {
        const uint64_t off = (uint64_t)(t + 1 - acc) * per;
        const int bytes = (acc - 1) * (int)per + (((int)n * (kDcBits + k * kPW) + 7) >> 3);
        ctr_packed(a, reinterpret_cast<uint32_t*>(pst), off, bytes, lane);
        __syncwarp();
        store_packed(a.priv_out + off, pst, bytes, lane);
        acc = 0;
      }
      __syncwarp();                        // the staging area may be written again
      t = tn;
      continue;
    }
    fence_proxy_async();                   // staged coefficients, before the bulk store
    __syncwarp();
    if (lane == 0) store_run(reinterpret_cast<uint8_t*>(a.pub_out) + (uint64_t)t * (64u * npub), stage, (int)n * 2 * npub);
    if (lane == 0) list[acc] = t;
    ++acc;
    if (acc == G || tn >= tend) {
      __syncwarp();
      if (!a.plain_private) {
        if (!dynamic) {                    // a run of subtiles: at most two windows
          const uint64_t q = (iv8 + (uint64_t)(t + 1 - acc) * nb) >> 8;
          if (q < wbase || ((iv8 + (uint64_t)(t + 1) * nb - 1) >> 8) > wbase + 1) {
            wbase = q;
            put_window(a, q + (lane & 1), lane < 2 ? lane : -1, wins);
            __syncwarp();
          }
        }
        // the image's last, short subtile, if it is among them, was claimed last
        ctr_warp(a, privst, list, (acc - 1) * nb + ((n * 2 * (k + 1) + 15) >> 4), nb, wins, wbase, lane);
        fence_proxy_async();
        __syncwarp();
      }
      if (lane < acc) {
        const uint32_t tj = list[lane];
        store_run(a.priv_out + (uint64_t)tj * (64u * (k + 1)), privst + lane * (64 * (k + 1)),
                  (int)min(32u, ncb - 32u * tj) * 2 * (k + 1));
      }
      acc = 0;
    }
    t = tn;
  }
  if (BULK && lost) load_drain(ld, bar, 1);
  bulk_wait_all();
  if (lane == 0) {
    if (a.counters) {
      if (nties) atomicAdd(&a.counters[0], (unsigned long long)nties);
      if (esc) atomicAdd(&a.counters[1], (unsigned long long)esc);
      if (fail || lost) atomicAdd(&a.counters[2], 1ull);
    }
  }
}

// ---- batches ---------------------------------------------------------------------------------

constexpr int kPSlot = kWBar + 8;                 // two slots after the single-image area
constexpr int kPWins = kPSlot + 2 * (int)sizeof(PlanSlot);   // the warp's two windows
constexpr int kPArea = (kPWins + 40 + 31) & ~31;
constexpr int kPBelow = ((int)kTpairWin - 1024) / kPArea;
constexpr int kPLow = (int)kTpairWin - kPBelow * kPArea;
constexpr int kPAbove = kWarps > kPBelow ? kWarps - kPBelow : 0;
constexpr int kPTail = (int)kTpairWin + kTpairBytes + kPAbove * kPArea;   // counter
constexpr int kPEnd = kPTail + 16;
static_assert(kPEnd <= 227 * 1024 && kPSlot % 8 == 0, "protect (batches) shared memory");

// acc_tiles(k), at most a tile
struct AccTable {
  uint8_t n[64];
};
constexpr AccTable make_acc_table() {
  AccTable t{};
  for (int k = 0; k < 64; ++k) t.n[k] = (uint8_t)(acc_tiles(k) < kTileSubs ? acc_tiles(k) : kTileSubs);
  return t;
}
static __constant__ AccTable c_acc = make_acc_table();

// Protect of a batch: every tile of 64 blocks of every image, six subtiles a tile.  A CTA has a
// run of the batch's tiles, taken by its warps as PlanClaim says; or (a.dispenser) every warp takes
// tiles from one counter.  Bound by issue, as one image: 1000 images (2.97 GB in and out), k = 0,
// 1210 -> 786 us (24 warps of 80 registers per SM, which spilled and met at three barriers a tile, before).
template <int K>
__global__ void __launch_bounds__(kWarps * 32, 1) protect_plan_kernel(const __grid_constant__ TileArgs a) {
  extern __shared__ __align__(128) uint8_t smem_cta[];
  const uint32_t win0 = smem_u32(smem_cta);
  if (win0 > (uint32_t)kPLow) {   // see the launcher
    if (threadIdx.x == 0 && a.counters) atomicAdd(&a.counters[2], 1ull);
    return;
  }
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  uint8_t* area = smem_cta + ((warp < kPBelow ? (uint32_t)(kPLow + warp * kPArea)
                                              : kTpairWin + kTpairBytes + (uint32_t)(warp - kPBelow) * kPArea) -
                              win0);
  const uint32_t pix = smem_u32(area + kWPix);
  uint8_t* const stage = area + kWStage;
  uint64_t* const bar = reinterpret_cast<uint64_t*>(area + kWBar);
  PlanSlot* const slots = reinterpret_cast<PlanSlot*>(area + kPSlot);
  uint32_t* const wins = reinterpret_cast<uint32_t*>(area + kPWins);
  uint32_t* const next = reinterpret_cast<uint32_t*>(smem_cta + (kPTail - win0));
  const int act = a.groups;
  PairFill<kWarps * 32> fill;
  fill.load(a.T, (int)threadIdx.x);
  PlanClaim claim(a, act);
  PlanKeys keys;
  Loads ld;
  // subtile t of slot s starts loading; bulk: by bulk copies (they complete on the mbarrier)
  auto load = [&](const PlanSlot* s, uint32_t t, bool& bulk) {
    const uint32_t cb = 32u * t + lane, b = cb / 3, bxc = s->bx_count;
    CbPos p;
    p.c = cb - 3 * b;
    p.by = b / bxc;
    p.bx = b - p.by * bxc;
    const uint64_t pitch = 3ull * s->width;
    const uint32_t n = min(32u, s->ncb - 32u * t);
    bulk = bxc >= 12 && (reinterpret_cast<uintptr_t>(s->px) & 15) == 0;
    if (bulk) ld.issued(0);
    return bulk ? load_subtile<true>(s->px, pitch, bxc, p, n, lane, pix, bar)
                : load_subtile<false>(s->px, pitch, bxc, p, n, lane, pix, bar);
  };

  if (lane == 0) {
    mbar_init(bar);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    slots[0].image = slots[1].image = ~0u;
  }
  if (threadIdx.x == 0) *next = (uint32_t)act;
  __syncthreads();                         // a first claim may go on to the counter
  int esc = 0, nties = 0;
  bool fail = false, lost = false, bulk = false;
  uint32_t t = 0, end = 0, tn, endn;
  PlanSlot *s = slots, *sn = slots + 1;
  PixAt at{};
  if (warp < act) {                        // the first run starts loading before the tables are filled
    claim(a, act, next, s, s, c_acc.n, warp, lane, t, end, keys);
    if (t < end) at = load(s, t, bulk);
  }
  fill.store(smem_cta + (kTpairWin - win0), (int)threadIdx.x);
  put_keys(s, keys, lane);
  __syncthreads();
  if (warp >= act) return;

  while (t < end && !lost) {
    claim(a, act, next, sn, s, c_acc.n, warp, lane, tn, endn, keys);
    put_keys(sn, keys, lane);
    const int k = K >= 0 ? K : s->k, npub = 63 - k;
    const int G = s->acc;
    uint8_t* const privst = stage + kWCb * 2 * npub;
    const uint64_t pitch = 3ull * s->width;
    int acc = 0;
    for (; t < end; ++t) {
      const uint32_t n = min(32u, s->ncb - 32u * t);
      if (bulk) {
        if (!load_wait(ld, bar, 0)) {      // gave up: nothing more is written
          lost = true;
          break;
        }
      } else {
        cp_async_wait_all();
      }
      __syncwarp();
      const uint32_t c = at.c;
      float2 P[8][4];
      const float V = transform_rows(area + kWPix + at.even, area + kWPix + at.odd, c, P);
      // cp.async wrote the buffer through the generic proxy; a bulk copy may write it next
      if (!bulk) fence_proxy_async();
      __syncwarp();                        // the pixel buffer is read: the next subtile's load starts
      if (t + 1 < end)
        at = load(s, t + 1, bulk);
      else if (tn < endn)
        at = load(sn, tn, bulk);
      bulk_wait_read_all();                // the staging area may be written again
      __syncwarp();
      int16_t* const pub_cb = reinterpret_cast<int16_t*>(stage) + lane * npub;
      int16_t* const priv_cb = reinterpret_cast<int16_t*>(privst) + (acc * kWCb + lane) * (k + 1);
      uint32_t mlo, mhi;
      stage_columns(P, V, k, (uint32_t)lane < n, pub_cb, priv_cb, mlo, mhi);
      decide_ties(
          [&] {
            const uint32_t b = (32u * t + lane) / 3, by = b / s->bx_count;
            return s->px + (uint64_t)by * (8 * pitch) + 24ull * (b - by * s->bx_count);
          },
          pitch, c, k, mlo, mhi, reinterpret_cast<int16_t*>(stage), priv_cb - lane * (k + 1), a.cfwd, lane, nties, esc, fail);
      fence_proxy_async();                 // staged coefficients, before the bulk store
      __syncwarp();
      if (lane == 0) store_run(s->pub + (uint64_t)t * (64u * npub), stage, (int)n * 2 * npub);
      ++acc;
      if (acc == G || t + 1 == end) {
        const uint32_t ta = t + 1 - acc;
        const int bytes = ((acc - 1) * 32 + (int)n) * 2 * (k + 1);
        ctr_plan(privst, (bytes + 15) >> 4, (uint64_t)ta * (uint32_t)(4 * (k + 1)), s, wins, lane);
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) store_run(s->priv + (uint64_t)ta * (64u * (k + 1)), privst, bytes);
        acc = 0;
      }
    }
    PlanSlot* const x = s;
    s = sn;
    sn = x;
    t = tn;
    end = endn;
  }
  if (lost) load_drain(ld, bar, 1);
  bulk_wait_all();
  if (lane == 0 && a.counters) {
    if (nties) atomicAdd(&a.counters[0], (unsigned long long)nties);
    if (esc) atomicAdd(&a.counters[1], (unsigned long long)esc);
    if (fail || lost) atomicAdd(&a.counters[2], 1ull);
  }
}

template <int K, bool BULK, int PACK = 0>
static cudaError_t launch_w(const TileArgs& a, cudaStream_t s, int sms) {
  static bool attr[kMaxAttrDevices];
  static bool window_ok[kMaxAttrDevices];
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
  if (!window_ok[dev]) {
    if ((e = smem_window_start_ok(protect_warp_kernel<K, BULK, PACK>, (uint32_t)kWLow)) != cudaSuccess) return e;
    window_ok[dev] = true;
  }
  e = smem_attr_once(protect_warp_kernel<K, BULK, PACK>, kWEnd, attr);
  if (e != cudaSuccess) return e;
  TileArgs b = a;
  const long long nsub = (3ll * a.nblocks + 31) / 32;
  const int grid = (int)(nsub < sms ? nsub : sms);
  const long long per = (nsub + grid - 1) / (grid ? grid : 1);
  b.groups = PACK ? working_warps(per) : (int)(per < kWarps ? per : kWarps);
  bx_division(b);
  b.run_tiles = PACK == 11 ? pack_acc_tiles<11>(a.k) : (PACK == 8 ? pack_acc_tiles<8>(a.k) : acc_tiles(a.k));
  if (grid > 0) protect_warp_kernel<K, BULK, PACK><<<grid, kWarps * 32, kWEnd, s>>>(b);
  return cudaGetLastError();
}

// per_sm: a quarter of the CTA's warps each (1 .. 3; else all)
template <int K>
static cudaError_t launch_plan(const TileArgs& a, cudaStream_t s, int sms, int per_sm) {
  static bool attr[kMaxAttrDevices];
  static bool window_ok[kMaxAttrDevices];
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
  if (!window_ok[dev]) {
    if ((e = smem_window_start_ok(protect_plan_kernel<K>, (uint32_t)kPLow)) != cudaSuccess) return e;
    window_ok[dev] = true;
  }
  e = smem_attr_once(protect_plan_kernel<K>, kPEnd, attr);
  if (e != cudaSuccess) return e;
  TileArgs b = a;
  b.groups = per_sm >= 1 && per_sm < 4 ? per_sm * kWarps / 4 : kWarps;
  const int grid = a.total_tiles < sms ? a.total_tiles : sms;
  if (grid > 0) protect_plan_kernel<K><<<grid, kWarps * 32, kPEnd, s>>>(b);
  return cudaGetLastError();
}

cudaError_t launch_protect_plan(const TileArgs& a, cudaStream_t s, int sms, int per_sm) {
  if (!a.images || a.pack || a.plain_private) return cudaErrorInvalidValue;
  if (a.k == 0) return launch_plan<0>(a, s, sms, per_sm);
  if (a.k == 5) return launch_plan<5>(a, s, sms, per_sm);
  return launch_plan<-1>(a, s, sms, per_sm);
}

cudaError_t launch_protect_warp(const TileArgs& a, cudaStream_t s, int sms) {
  if (a.images || a.k < 0 || a.k > 63 || (a.pack && a.pack != 11 && a.pack != 8)) return cudaErrorInvalidValue;
  // bulk copies of whole row runs need 16-byte aligned pixels and subtiles of at most two block
  // rows
  const bool bulk = a.bx_count >= 12 && ((uintptr_t)a.pixels_in & 15) == 0;
  if (a.pack == 11) return !bulk ? launch_w<-1, false, 11>(a, s, sms)
                                 : (a.k == 5 ? launch_w<5, true, 11>(a, s, sms) : launch_w<-1, true, 11>(a, s, sms));
  if (a.pack == 8) return !bulk ? launch_w<-1, false, 8>(a, s, sms)
                                : (a.k == 5 ? launch_w<5, true, 8>(a, s, sms) : launch_w<-1, true, 8>(a, s, sms));
  if (bulk) {
    if (a.k == 0) return launch_w<0, true>(a, s, sms);
    if (a.k == 5) return launch_w<5, true>(a, s, sms);
    return launch_w<-1, true>(a, s, sms);
  }
  return launch_w<-1, false>(a, s, sms);
}

}  // namespace fds
