// Fused restore kernel in its warp form (defragmentation, Sect. 3.2, Fig. 3): CTR decryption of
// the confidential fragment, merge by zigzag position, inverse 8x8 DCT, round half away from zero
// (exact), clamp to [0, 255], of one image, of packed fragments and of a batch; and the public-image
// form (Sect. 6.5.1).
//
// As in the warp form of protect, each warp works on subtiles of 32 channel-blocks of its own,
// with no barrier between warps after the AES table is filled.  It is bound by the issue of
// instructions (4096 x 4096, k = 5: 45.5 M warp instructions = 36.2 us of issue slots against
// 22.6 us for the 151 MB); two CTAs of six warps that met at three barriers per 192
// channel-blocks issued in 61 % of the cycles, sixteen independent warps in 71 %.  Per subtile:
//   1. its public part has arrived (bulk copy on the warp's mbarrier); two columns at a time the
//      coefficients are gathered, converted and transformed (the loads of the next two stay
//      behind: with all 64 in flight the kernel spilled 200 bytes and took 78 us); the buffer is
//      free, so the next subtile's public part starts loading
//   2. row butterflies, round and clamp, bytes into the warp's pixel buffer; a row in which some
//      lane has a value within the error guard of a half-integer marks those values
//   3. marked values are decided exactly, four at a time (decide_pixels): public coefficients from
//      global memory, private ones from the decrypted buffer
//   4. the ten whole blocks go out as 8-byte pieces, each lane its block's piece c; the two
//      channel-blocks of a block shared with a neighbouring subtile as bytes
// Private parts come in runs of subtiles whose keystream blocks fill whole warps (k = 5: four
// subtiles, 96 blocks), one run ahead, and are decrypted in place.  The last two or so subtiles a
// warp are claimed one by one, so that a CTA's warps end together.
// Measured on 4096 x 4096: k = 5 79.0 -> 60.4 us; the public-image form 66.6 -> 45.4 us.  Testing a row for values outside [0, 255] and
// clamping only then (96 instructions a subtile less) measured no faster: 60.6 us.
#include "fds_aux.h"
#include "fds_warp.cuh"

namespace fds {

constexpr int kRPitch = 12 * 24;                  // one pixel row of a subtile: at most 12 blocks
constexpr int kRPix = 0;
constexpr int kRFrag = kRPix + 8 * kRPitch;       // public part, then the private parts of a run of
constexpr int kRFragBytes = 6784;                 // subtiles, twice where that fits
constexpr int kRBar = kRFrag + kRFragBytes;       // mbarriers: public, private (two)
constexpr int kRSlot = kRBar + 3 * 8;             // what a warp looks at once per run (WarpSlot)
constexpr int kRArea = (kRSlot + 32 + 31) & ~31;
constexpr int kRWinBytes = 20 * kWins + 16;       // windows, subtile counter
constexpr int kRBelow = ((int)kTpairWin - 1024) / kRArea;
constexpr int kRLow = (int)kTpairWin - kRBelow * kRArea;
constexpr int kRAbove = kWarps > kRBelow ? kWarps - kRBelow : 0;
constexpr int kRWin = (int)kTpairWin + kTpairBytes + kRAbove * kRArea;
constexpr int kREnd = kRWin + kRWinBytes;
static_assert(kREnd <= 227 * 1024, "restore (warp form) shared memory");

// subtiles whose private parts are loaded and decrypted together (the fewest idle lanes), and
// whether two such runs fit
__host__ __device__ constexpr int run_tiles(int k) {
  int best = 1, bn = 4 * (k + 1), bp = (bn + 31) / 32;
  for (int g = 2; g <= 8; ++g) {
    if ((63 - k) * 64 + 2 * g * (k + 1) * 64 > kRFragBytes) break;
    const int n = g * 4 * (k + 1), p = (n + 31) / 32;
    if (n * bp > bn * p) {
      best = g;
      bn = n;
      bp = p;
    }
  }
  return best;
}
__host__ __device__ constexpr bool run_twice(int k) { return (63 - k) * 64 + 2 * run_tiles(k) * (k + 1) * 64 <= kRFragBytes; }

// bytes of a fragment part to shared memory: a bulk copy completing on bar (lane 0 announces it),
// and a tail of 2-byte copies (only behind the last, short subtile of an image: where another
// image's part follows in the buffer, the lanes fence their stores before the next bulk copy)
__device__ __forceinline__ void load_part(uint8_t* dst, const uint8_t* src, int bytes, int lane, uint64_t* bar) {
  const int b16 = bytes & ~15;
  if (lane == 0) {
    mbar_expect_tx(bar, (uint32_t)b16);
    if (b16) bulk_load(dst, src, (uint32_t)b16, bar);
  }
  const int j = b16 + 2 * lane;
  if (j < bytes) *reinterpret_cast<uint16_t*>(dst + j) = *reinterpret_cast<const uint16_t*>(src + j);
}

// per-warp state that is not worth registers: counts, own subtiles still to claim, first window
struct WarpSlot {
  int ties, esc, fail;
  uint32_t rt, rend, pad;
  uint64_t wbase;
};
static_assert(sizeof(WarpSlot) == 32, "WarpSlot");

// The coefficients of a lane's channel-block (z = 0 .. k at priv_cb, the rest at pub_cb) to
// floats, two columns at a time through the column butterflies; returns sum |F|
template <bool PUBIMG>
__device__ __forceinline__ float gather_columns(const int16_t* pub_cb, const int16_t* priv_cb, int k, float2 (&G2)[8][4]) {
  float l1 = 0.0f;  // sum |F|, exact (integers below 2^24)
#pragma unroll
  for (int j = 0; j < 4; ++j) {        // two columns: gathered and transformed
    float2 col[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int z0 = zigzag_of(u, 2 * j), z1 = zigzag_of(u, 2 * j + 1);
      const int q0 = z0 <= k ? (PUBIMG ? (z0 == 0 ? 1024 : 0) : priv_cb[z0]) : pub_cb[z0 - k - 1];
      const int q1 = z1 <= k ? (PUBIMG ? 0 : priv_cb[z1]) : pub_cb[z1 - k - 1];
      col[u] = add2(make_float2(__int_as_float(kMagicBits + q0), __int_as_float(kMagicBits + q1)),
                    make_float2(-kMagic, -kMagic));
      l1 += fabsf(col[u].x);
      l1 += fabsf(col[u].y);
    }
    idct8_2(col);
#pragma unroll
    for (int y = 0; y < 8; ++y) G2[y][j] = col[y];
    if (j < 3) asm volatile("" ::: "memory");   // the next columns' loads stay behind
  }
  return l1;
}

// Row butterflies, rounding and clamping; bytes into the pixel buffer at out; bit 8 y + x of
// mhi:mlo marks a value within the error guard of a half-integer (none where the lane is not live)
__device__ __forceinline__ void emit_rows(const float2 (&G2)[8][4], float l1, bool live, uint8_t* out, uint32_t& mlo,
                                          uint32_t& mhi) {
  const float thr = live ? 0.5f - l1 * kGuardInvScale : 1.0f;
  mlo = mhi = 0;
#pragma unroll
  for (int y = 0; y < 8; ++y) {
    float row[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      row[2 * j] = G2[y][j].x;
      row[2 * j + 1] = G2[y][j].y;
    }
    idct8(row);
    float2 r[4];
    float big = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 pc = make_float2(fminf(fmaxf(row[2 * j], 0.0f), 255.0f), fminf(fmaxf(row[2 * j + 1], 0.0f), 255.0f));
      const float2 yv = add2(pc, make_float2(kMagic, kMagic));
      r[j] = sub2(pc, add2(yv, make_float2(-kMagic, -kMagic)));
      big = fmaxf(fmaxf(big, fabsf(r[j].x)), fabsf(r[j].y));
      out[y * kRPitch + 6 * j] = (uint8_t)__float_as_uint(yv.x);
      out[y * kRPitch + 6 * j + 3] = (uint8_t)__float_as_uint(yv.y);
    }
    if (__any_sync(0xffffffffu, big > thr)) {   // rare: a near tie in this row
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int l = 0; l < 2; ++l)
          if (fabsf(l ? r[j].y : r[j].x) > thr) {
            if (8 * y + 2 * j + l < 32)
              mlo |= 1u << (8 * y + 2 * j + l);
            else
              mhi |= 1u << (8 * y + 2 * j + l - 32);
          }
    }
  }
}

// A coefficient of a channel-block by zigzag index
template <bool PUBIMG, bool STAGED>
__device__ __forceinline__ int coefficient(const int16_t* pub, const int16_t* priv, int k, int z) {
  return z <= k ? (PUBIMG ? (z == 0 ? 1024 : 0) : priv[z]) : (STAGED ? pub[z - k - 1] : __ldg(pub + z - k - 1));
}
__device__ __forceinline__ void put_pixel(uint8_t* block, int pos, int p) {
  block[(pos >> 3) * kRPitch + 3 * (pos & 7)] = (uint8_t)(p < 0 ? 0 : (p > 255 ? 255 : p));
}

// Of the channel-blocks with kBlockTies marked pixels or more (flat ones, a half level off, have 64),
// the whole warp decides 32 at a time, a pixel a lane, and passes over coefficients that are zero;
// returns what the lane has left, and the pixels too near a boundary for fixed point.  Arguments as of
// decide_pixels; at: the lane's block in the pixel buffer.  Turns alone took 1316 us for DC-only blocks
// (119 with this).  From 6 or 8 marked pixels on it was slower where blocks are not sparse: public image
// of random rectangles 24.6 -> 26.5 and 27.1 us.  A function of its own: inside the kernel it slowed down
// what runs without it (batch of 300 images of mixed k, 599 us against 585).
constexpr int kPixFrac = 40;
constexpr int kBlockTies = 16;
template <bool PUBIMG, bool STAGED>
__device__ __noinline__ uint64_t decide_blocks(uint32_t mlo, uint32_t mhi, const int16_t* pub_g, const int16_t* priv0, int k,
                                               const uint32_t* table, uint8_t* pix, uint32_t at) {
  const int lane = (int)(threadIdx.x & 31);
  for (uint32_t many = __ballot_sync(0xffffffffu, __popc(mlo) + __popc(mhi) >= kBlockTies); many; many &= many - 1) {
    const int src = __ffs(many) - 1;
    const uint32_t to = __shfl_sync(0xffffffffu, at, src);
    const int16_t* pub = pub_g + src * (63 - k);
    const int16_t* priv = priv0 + src * (k + 1);
    const uint32_t Q = __byte_perm((uint32_t)coefficient<PUBIMG, STAGED>(pub, priv, k, 2 * lane),
                                   (uint32_t)coefficient<PUBIMG, STAGED>(pub, priv, k, 2 * lane + 1), 0x5410u);
    const uint32_t used = __ballot_sync(0xffffffffu, Q != 0);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const bool on = (__shfl_sync(0xffffffffu, h ? mhi : mlo, src) >> lane) & 1u;
      int n[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      for (uint32_t m = used; m;) {        // four coefficients at a time
        const int t = (__ffs(m) - 1) >> 1;
        m &= ~(3u << (2 * t));
        const uint32_t q0 = __shfl_sync(0xffffffffu, Q, 2 * t), q1 = __shfl_sync(0xffffffffu, Q, 2 * t + 1);
        const uint32_t* w = table + 64 * 128 + 512 * t + 32 * h + lane;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t x = __ldg(w + 64 * j);
          n[j] = dp2a_hi(q1, x, dp2a_lo(q0, x, n[j]));
        }
      }
      bool sure;
      const int p = round_lane<kPixFrac>(n, sure);
      if (on) put_pixel(pix + to, 32 * h + lane, p);
      const uint32_t left = __ballot_sync(0xffffffffu, on && !sure);
      if (lane == src) (h ? mhi : mlo) = left;
    }
  }
  return (uint64_t)mhi << 32 | mlo;
}

// The marked pixels of a subtile, decided exactly (take_ties) and written to the pixel buffer pix, where
// out is the lane's own block and channel.  pub_g: the subtile's public coefficients in global memory,
// or STAGED in shared memory; priv0: the first lane's (decrypted) private ones; table: a.cinv, whose
// row of a position holds a word for four coefficients in zigzag order: a lane takes eight of them.
// int16 coefficients of any value make the sum of the |n_j| at most 2^22, so 40 fraction bits fit.
template <bool PUBIMG, bool STAGED = false>
__device__ __forceinline__ void decide_pixels(uint32_t mlo, uint32_t mhi, const int16_t* pub_g, const int16_t* priv0, int k,
                                              const uint32_t* table, int lane, WarpSlot* slot, uint8_t* pix,
                                              const uint8_t* out) {
  uint32_t who = __ballot_sync(0xffffffffu, (mlo | mhi) != 0);
  if (__builtin_expect(who == 0, 1)) return;
  // read here, so that what depends on it is not kept through the subtiles without near ties
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
  int esc = 0;
  bool fail = false;
  const int nties = (int)__reduce_add_sync(0xffffffffu, (uint32_t)(__popc(mlo) + __popc(mhi)));
  const uint32_t at = (uint32_t)(out - pix);
  const long long cos_l = group_cos<kPixFrac>(lane);
  const int l = lane & 7;
  if (__any_sync(0xffffffffu, __popc(mlo) + __popc(mhi) >= kBlockTies)) {
    const uint64_t left = decide_blocks<PUBIMG, STAGED>(mlo, mhi, pub_g, priv0, k, table, pix, at);
    mlo = (uint32_t)left;
    mhi = (uint32_t)(left >> 32);
    who = __ballot_sync(0xffffffffu, left != 0);
  }
  while (who) {
    const TieTurn t = take_ties(who, mlo, mhi, lane);
    const uint32_t to = __shfl_sync(0xffffffffu, at, t.src);
    int n[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (t.on) {
      const uint2* w2 = reinterpret_cast<const uint2*>(table + t.pos * 128) + l;
      const int16_t* pub = pub_g + t.src * (63 - k);
      const int16_t* priv = priv0 + t.src * (k + 1);
      uint32_t Q[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int q[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) q[h] = coefficient<PUBIMG, STAGED>(pub, priv, k, 8 * l + 2 * i + h);
        Q[i] = __byte_perm((uint32_t)q[0], (uint32_t)q[1], 0x5410u);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint2 w = __ldg(w2 + 8 * j);
        n[j] = dp2a_hi(Q[3], w.y, dp2a_lo(Q[2], w.y, dp2a_hi(Q[1], w.x, dp2a_lo(Q[0], w.x, 0))));
      }
    }
    const int p = round_group<kPixFrac, 1 << 22>(group_sum(n, lane), cos_l, t.on, lane, esc, fail);
    if (t.on && l == 0) put_pixel(pix + to, t.pos, p);
    who = __ballot_sync(0xffffffffu, (mlo | mhi) != 0);
  }
  if (lane == 0) {
    slot->ties += nties;
    if (esc | fail) slot->esc += esc, slot->fail |= fail;
  }
}

// The pixel buffer of a subtile of n channel-blocks to the image; at: the lane's place in it
__device__ __forceinline__ void store_pixels(uint8_t* img, uint64_t pitch, const CbPos& at, uint32_t c0, int n, int lane,
                                             const uint8_t* pix) {
  // whole blocks: lane's 8-byte piece c of its block in 8 rows; a block shared with the next
  // or previous subtile: its channels' bytes
  uint8_t* const blk = img + ((uint64_t)at.by * (8 * pitch) + 24ull * at.bx);
  const int b0l = lane - (int)at.c;
  const bool whole = b0l >= 0 && b0l + 2 < n;
  if (whole) {
    uint8_t* dst = blk + 8 * at.c;
    const uint8_t* src = pix + 8 * (c0 + lane);
#pragma unroll
    for (int y = 0; y < 8; ++y) {
      *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src + y * kRPitch);
      dst += pitch;
    }
  }
  for (uint32_t who = __ballot_sync(0xffffffffu, !whole && lane < n); who; who &= who - 1) {
    const int src = __ffs(who) - 1;
    const uint32_t sc = __shfl_sync(0xffffffffu, at.c, src);
    uint8_t* const sb = reinterpret_cast<uint8_t*>(__shfl_sync(0xffffffffu, (unsigned long long)blk, src));
    const uint8_t* sp = pix + 8 * (c0 + src - sc) + sc;
    const int x3 = 3 * (lane & 7), y0 = lane >> 3;
    sb[y0 * pitch + x3 + sc] = sp[y0 * kRPitch + x3];
    sb[(y0 + 4) * pitch + x3 + sc] = sp[(y0 + 4) * kRPitch + x3];
  }
}

template <int K, bool PUBIMG>
__global__ void __launch_bounds__(kWarps * 32, 1) restore_warp_kernel(const __grid_constant__ TileArgs a) {
  extern __shared__ __align__(128) uint8_t smem_cta[];
  const uint32_t win0 = smem_u32(smem_cta);
  if (win0 > (uint32_t)kRLow) {   // see the launcher
    if (threadIdx.x == 0 && a.counters) atomicAdd(&a.counters[2], 1ull);
    return;
  }
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  uint8_t* area = smem_cta + ((warp < kRBelow ? (uint32_t)(kRLow + warp * kRArea)
                                              : kTpairWin + kTpairBytes + (uint32_t)(warp - kRBelow) * kRArea) -
                              win0);
  uint8_t* const pix = area + kRPix;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(area + kRBar);
  uint32_t* wins = reinterpret_cast<uint32_t*>(smem_cta + (kRWin - win0));
  uint32_t* const next = wins + 5 * kWins;
  const int k = K >= 0 ? K : a.k;
  const int npub = 63 - k;
  const uint32_t nb = 4u * (uint32_t)(k + 1);       // keystream blocks per subtile
  const int G = K >= 0 ? run_tiles(K >= 0 ? K : 0) : a.run_tiles & 15;
  const bool twice = K >= 0 ? run_twice(K >= 0 ? K : 0) : (a.run_tiles & 16) != 0;
  const bool cipher = !PUBIMG && !a.plain_private;
  uint8_t* const pubst = area + kRFrag;
  uint8_t* const privst = pubst + kWCb * 2 * npub;
  const int priv_half = twice ? G * 64 * (k + 1) : 0;
  const uint32_t ncb = 3u * (uint32_t)a.nblocks, nsub = (ncb + 31u) >> 5;
  const int act = a.groups;       // working warps of each CTA
  const uint32_t s0 = (uint32_t)((uint64_t)nsub * blockIdx.x / gridDim.x);
  const uint32_t s1 = (uint32_t)((uint64_t)nsub * (blockIdx.x + 1) / gridDim.x);
  const uint32_t iv8 = (uint32_t)a.iv_lo & 255u;
  uint64_t wbase = (iv8 + (uint64_t)s0 * nb) >> 8;
  const uint64_t wlast = (iv8 + (uint64_t)s1 * nb - 1) >> 8;
  const bool table = wlast - wbase < kWins;         // the CTA's windows fit the table
  // the CTA's subtiles: the first ones as runs of G for each warp in turn, the last (about two a
  // warp) one by one to whichever warp is free
  const uint32_t per = (s1 - s0) / (uint32_t)act;
  const uint32_t own = per > 2 ? (per - 2) / G * G : 0;
  const uint32_t sfree = s0 + own * act;
  WarpSlot* const slot = reinterpret_cast<WarpSlot*>(area + kRSlot);
  if (lane == 0) {
    slot->ties = slot->esc = slot->fail = 0;
    slot->rt = s0 + own * (uint32_t)warp;
    slot->rend = slot->rt + own;
  }
  // claim the next run: its first subtile and length (start >= s1: none left)
  auto claim = [&](int& cnt) -> uint32_t {
    uint32_t t = 0;
    if (lane == 0) {
      t = slot->rt;
      if (t < slot->rend)
        slot->rt = t + G;
      else
        t = atomicAdd(next, 1u) | 0x80000000u;
    }
    t = __shfl_sync(0xffffffffu, t, 0);
    cnt = t >> 31 ? 1 : G;
    return t & 0x7fffffffu;
  };
  auto nof = [&](uint32_t t) { return (int)min(32u, ncb - 32u * t); };
  Loads ld;                                // barrier 0: public, 1 and 2: the private buffers
  auto load_pub = [&](uint32_t t) {
    load_part(pubst, reinterpret_cast<const uint8_t*>(a.pub_in) + (uint64_t)t * (64u * npub), nof(t) * 2 * npub, lane, bars);
    ld.issued(0);
  };
  auto load_priv = [&](uint32_t t, int cnt, int half) {
    load_part(privst + half * priv_half, a.priv_in + (uint64_t)t * (64u * (k + 1)),
              ((cnt - 1) * 32 + nof(t + cnt - 1)) * 2 * (k + 1), lane, bars + 1 + half);
    ld.issued(1 + half);
  };

  if (lane == 0) {
    mbar_init(bars);
    mbar_init(bars + 1);
    mbar_init(bars + 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the warp's first run (without the shared counter) starts loading before the tables are filled
  int cnt = 0, cnt_n = 0, half = 0;
  uint32_t run = s1, run_n = s1;
  __syncwarp();
  if (warp < act) {
    if (own)
      run = claim(cnt);
    else
      run = s0 + warp, cnt = 1;
    if (run < s1) {
      load_pub(run);
      if (!PUBIMG) load_priv(run, cnt, 0);
    }
  }
  if (threadIdx.x == 0) *next = own ? sfree : s0 + act;
  if (cipher) fill_pair_table(smem_cta + (kTpairWin - win0), a.T, (int)threadIdx.x, kWarps * 32);
  __syncthreads();
  if (cipher) {
    if (table) {
      const int i = (int)threadIdx.x;
      if ((uint32_t)(i & ~31) <= wlast - wbase) put_window(a, wbase + i, (uint32_t)i <= wlast - wbase ? i : -1, wins);
      __syncthreads();
    } else {
      wins += 10 * warp;
      wbase = ~0ull - 1;
    }
    if (lane == 0) slot->wbase = wbase;
    __syncwarp();
  }
  bool lost = false;
  while (run < s1) {
    run_n = claim(cnt_n);
    if (!PUBIMG) {
      if (twice && run_n < s1) {
        fence_proxy_async();               // the buffer was decrypted in place
        __syncwarp();
        load_priv(run_n, cnt_n, half ^ 1);
      }
      if (!load_wait(ld, bars, 1 + half)) {
        lost = true;
        break;
      }
      __syncwarp();
      if (cipher) {
        uint8_t* const buf = privst + half * priv_half;
        const uint32_t total = (uint32_t)(((cnt - 1) * 32 + nof(run + cnt - 1)) * 2 * (k + 1) + 15) >> 4;
        const uint64_t b0 = iv8 + (uint64_t)run * nb;     // from the IV's window
        uint64_t wbase = slot->wbase;
        if (!table && ((b0 >> 8) < wbase || ((b0 + total - 1) >> 8) > wbase + 1)) {
          wbase = b0 >> 8;
          __syncwarp();
          put_window(a, wbase + (lane & 1), lane < 2 ? lane : -1, wins);
          if (lane == 0) slot->wbase = wbase;
          __syncwarp();
        }
        const PairLanes lc = pair_lanes();
#pragma unroll 1
        for (uint32_t i = lane; i < total; i += 32) {
          const uint64_t b = b0 + i;
          const uint32_t* src = wins + 5 * (uint32_t)((b >> 8) - wbase);
          const uint32_t w[5] = {src[0], src[1], src[2], src[3], src[4]};
          uint32_t s[4];
          aes_from_window(w, (uint32_t)b & 255u, a.rk, lc, s);
          uint4* p = reinterpret_cast<uint4*>(buf + 16 * i);
          uint4 d = *p;
          d.x ^= s[0];
          d.y ^= s[1];
          d.z ^= s[2];
          d.w ^= s[3];
          *p = d;
        }
      }
    }
#pragma unroll 1
    for (int ti = 0; ti < cnt; ++ti) {
      const uint32_t t = run + ti;
      const int n = nof(t);
      const CbPos at = cb_pos(a, 32u * t + lane);
      if (!load_wait(ld, bars, 0)) {       // gave up: nothing more is written
        lost = true;
        break;
      }
      __syncwarp();
      const int16_t* pub_cb = reinterpret_cast<const int16_t*>(pubst) + lane * npub;
      const int16_t* priv_cb = reinterpret_cast<const int16_t*>(privst + half * priv_half) + (ti * kWCb + lane) * (k + 1);
      float2 G2[8][4];
      const float l1 = gather_columns<PUBIMG>(pub_cb, priv_cb, k, G2);
      __syncwarp();                        // the public part is read: the next one starts loading
      {
        const uint32_t tn = ti + 1 < cnt ? t + 1 : run_n;
        if (tn < s1) load_pub(tn);
      }
      const uint32_t c0 = __shfl_sync(0xffffffffu, at.c, 0);
      uint8_t* const out = pix + 8 * (c0 + lane - at.c) + at.c;
      uint32_t mlo, mhi;
      emit_rows(G2, l1, lane < n, out, mlo, mhi);
      decide_pixels<PUBIMG>(mlo, mhi, a.pub_in + (uint64_t)(32u * t) * npub, priv_cb - lane * (k + 1), k, a.cinv, lane, slot, pix,
                            out);
      if (!PUBIMG && !twice) fence_proxy_async();
      __syncwarp();                        // the pixel rows are complete
      if (!PUBIMG && !twice && ti + 1 == cnt && run_n < s1) load_priv(run_n, cnt_n, 0);
      store_pixels(a.pixels_out, 3ull * (uint64_t)a.width, at, c0, n, lane, pix);
      __syncwarp();                        // the pixel buffer may be written again
    }
    if (lost) break;
    run = run_n;
    cnt = cnt_n;
    if (twice) half ^= 1;
  }
  if (lost) load_drain(ld, bars, 3);
  if (lane == 0 && a.counters) {
    if (slot->ties) atomicAdd(&a.counters[0], (unsigned long long)slot->ties);
    if (slot->esc) atomicAdd(&a.counters[1], (unsigned long long)slot->esc);
    if (slot->fail || lost) atomicAdd(&a.counters[2], 1ull);
  }
}

// ---- packed storage (Sect. 6.4.3) ----------------------------------------------------------------

// A subtile's packed parts land as they lie in the streams (4-byte granular: widened to 16-byte
// boundaries for a bulk copy), the private ones of a run of subtiles at a time, and are unpacked
// into an int16 staging area, which the transform and the exact decisions read; a landing area is
// free, and loads again, as soon as it is unpacked.  Bound by issue (4096 x 4096, k = 5: 56.4 M warp
// instructions, issued in 69 % of the cycles): 104 -> 76 us (11 and 8 bits).
constexpr int kUPix = 0;
constexpr int kUStage = kUPix + 8 * kRPitch;      // int16 coefficients of a subtile
constexpr int kULand = kUStage + kWCb * 128;      // public landing, private landing
constexpr int kULandBytes = 3632;
constexpr int kUBar = kULand + kULandBytes;
constexpr int kUSlot = kUBar + 16;                // mbarriers: public, private
constexpr int kUArea = (kUSlot + 32 + 31) & ~31;
constexpr int kUBelow = ((int)kTpairWin - 1024) / kUArea;
constexpr int kULow = (int)kTpairWin - kUBelow * kUArea;
constexpr int kUAbove = kWarps > kUBelow ? kWarps - kUBelow : 0;
constexpr int kUTail = (int)kTpairWin + kTpairBytes + kUAbove * kUArea;
constexpr int kUEnd = kUTail;
static_assert(kUEnd <= 227 * 1024 && kUSlot % 8 == 0, "packed restore shared memory");

template <int W>
__host__ __device__ constexpr int land_pub_bytes(int k) { return (4 * (63 - k) * W + 31) & ~15; }   // + 12 of skew
template <int W>
__host__ __device__ constexpr int run_tiles_packed(int k) {
  const int per = 4 * (kDcBits + k * W);
  int best = 1, bn = per, bp = (per / 16 + 2 + 31) / 32;
  for (int g = 2; g <= 8 && land_pub_bytes<W>(k) + g * per + 28 <= kULandBytes; ++g) {
    const int n = g * per, p = (n / 16 + 2 + 31) / 32;
    if (n * bp > bn * p) {
      best = g;
      bn = n;
      bp = p;
    }
  }
  return best;
}

// bytes [off, off + bytes) of a stream of `total` bytes (off a multiple of 4, the stream 8-byte
// aligned) to the 16-byte aligned dst, whose first byte stands for the 16-byte boundary at or below
// the first one; returns the distance from there.  Where the widened copy would leave the stream,
// the lanes copy words and bytes (by_lanes: fence their stores before the next bulk copy there).
__device__ __forceinline__ uint32_t land_stream(uint8_t* dst, const uint8_t* stream, uint64_t total, uint64_t off, int bytes,
                                                int lane, uint64_t* bar, bool& by_lanes) {
  const uint8_t* src = stream + off;
  const uint32_t skew = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15);
  const uint32_t wide = (skew + (uint32_t)bytes + 15u) & ~15u;
  by_lanes = off < skew || off - skew + wide > total;
  if (!by_lanes) {
    if (lane == 0) {
      mbar_expect_tx(bar, wide);
      if (wide) bulk_load(dst, src - skew, wide, bar);
    }
  } else {
    for (int i = lane; i < (bytes >> 2); i += 32)
      reinterpret_cast<uint32_t*>(dst + skew)[i] = __ldg(reinterpret_cast<const uint32_t*>(src) + i);
    if (lane < (bytes & 3)) dst[skew + (bytes & ~3) + lane] = src[(bytes & ~3) + lane];
    __syncwarp();
    if (lane == 0) mbar_expect_tx(bar, 0u);
  }
  return skew;
}

// sign-magnitude code of W bits -> value
template <int W>
__device__ __forceinline__ int ac_value(uint32_t c) {
  const int mag = (int)(c & ((1u << (W - 1)) - 1u));
  return (c >> (W - 1)) & 1u ? -mag : mag;
}

// n channel-blocks' packed public fields (words at w) -> int16 at pub, 32 fields (W words) a lane
// and round
template <int W>
__device__ __forceinline__ void unpack_public(const uint32_t* w, int16_t* pub, int n, int npub, int lane) {
  const int ngroups = (n * npub + 31) >> 5;
#pragma unroll 1
  for (int g = lane; g < ngroups; g += 32) {
    uint32_t word[W];
#pragma unroll
    for (int j = 0; j < W; ++j) word[j] = w[W * g + j];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t u[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        uint32_t v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int b = W * (8 * q + 2 * m + h);
          const uint32_t c = (b & 31) + W > 32 ? __funnelshift_r(word[b >> 5], word[(b >> 5) + 1], b & 31) : word[b >> 5] >> (b & 31);
          v[h] = (uint32_t)ac_value<W>(c);
        }
        u[m] = __byte_perm(v[0], v[1], 0x5410u);
      }
      reinterpret_cast<uint4*>(pub + 32 * g)[q] = make_uint4(u[0], u[1], u[2], u[3]);   // past the last field: not read
    }
  }
}

// a lane's channel-block cb of a landed private run (words at w) -> its k + 1 int16 at dst
template <int W>
__device__ __forceinline__ void unpack_private(const uint32_t* w, int16_t* dst, int cb, int k) {
  int pos = cb * (kDcBits + k * W);
  dst[0] = (int16_t)(__funnelshift_r(w[pos >> 5], w[(pos >> 5) + 1], pos & 31) & ((1u << kDcBits) - 1u));
  pos += kDcBits;
#pragma unroll 1
  for (int z = 1; z <= k; ++z, pos += W)
    dst[z] = (int16_t)ac_value<W>(__funnelshift_r(w[pos >> 5], w[(pos >> 5) + 1], pos & 31));
}

template <int K, int W>
__global__ void __launch_bounds__(kWarps * 32, 1) restore_packed_kernel(const __grid_constant__ TileArgs a) {
  extern __shared__ __align__(128) uint8_t smem_cta[];
  const uint32_t win0 = smem_u32(smem_cta);
  if (win0 > (uint32_t)kULow) {   // see the launcher
    if (threadIdx.x == 0 && a.counters) atomicAdd(&a.counters[2], 1ull);
    return;
  }
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  uint8_t* area = smem_cta + ((warp < kUBelow ? (uint32_t)(kULow + warp * kUArea)
                                              : kTpairWin + kTpairBytes + (uint32_t)(warp - kUBelow) * kUArea) -
                              win0);
  uint8_t* const pix = area + kUPix;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(area + kUBar);
  WarpSlot* const slot = reinterpret_cast<WarpSlot*>(area + kUSlot);
  const int k = K >= 0 ? K : a.k;
  const int npub = 63 - k, period = kDcBits + k * W;
  const uint32_t pub_per = 4u * (uint32_t)(npub * W), priv_per = 4u * (uint32_t)period;
  const int G = K >= 0 ? run_tiles_packed<W>(K >= 0 ? K : 0) : a.run_tiles;
  uint8_t* const land_pub = area + kULand;
  uint8_t* const land_priv = land_pub + land_pub_bytes<W>(k);
  int16_t* const pubst = reinterpret_cast<int16_t*>(area + kUStage);
  int16_t* const privst = pubst + kWCb * npub;
  const uint32_t ncb = 3u * (uint32_t)a.nblocks, nsub = (ncb + 31u) >> 5;
  const uint64_t pub_total = ((uint64_t)ncb * (uint32_t)(npub * W) + 7) >> 3, priv_total = ((uint64_t)ncb * (uint32_t)period + 7) >> 3;
  const int act = a.groups;       // working warps of each CTA, each with a run of the subtiles
  const uint32_t id = blockIdx.x * act + warp, nw = gridDim.x * act;
  const uint32_t t0 = warp < act ? (uint32_t)((uint64_t)nsub * id / nw) : 0u;
  const uint32_t t1 = warp < act ? (uint32_t)((uint64_t)nsub * (id + 1) / nw) : 0u;
  auto nof = [&](uint32_t t) { return (int)min(32u, ncb - 32u * t); };
  Loads ld;                                // barrier 0: public, 1: private
  bool lanes_pub = false;                  // the public part at hand was landed by the lanes
  auto load_pub = [&](uint32_t t) {
    ld.issued(0);
    return land_stream(land_pub, reinterpret_cast<const uint8_t*>(a.pub_in), pub_total, (uint64_t)t * pub_per,
                       (nof(t) * npub * W + 7) >> 3, lane, bars, lanes_pub);
  };
  auto load_priv = [&](uint32_t t) {
    const int cnt = min(G, (int)(t1 - t));
    bool by_lanes;                         // fenced below in any case
    ld.issued(1);
    return land_stream(land_priv, a.priv_in, priv_total, (uint64_t)t * priv_per,
                       (cnt - 1) * (int)priv_per + ((nof(t + cnt - 1) * period + 7) >> 3), lane, bars + 1, by_lanes);
  };

  if (lane == 0) {
    mbar_init(bars);
    mbar_init(bars + 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    slot->ties = slot->esc = slot->fail = 0;
  }
  __syncwarp();
  uint32_t skew_pub = 0, skew_priv = 0;
  if (t0 < t1) {
    skew_pub = load_pub(t0);
    skew_priv = load_priv(t0);
  }
  fill_pair_table(smem_cta + (kTpairWin - win0), a.T, (int)threadIdx.x, kWarps * 32);
  __syncthreads();

  bool lost = false;
  uint32_t run = t0;                       // the run's first subtile
#pragma unroll 1
  for (uint32_t t = t0; t < t1; ++t) {
    const int n = nof(t);
    if (t == run) {                        // a new run: decrypt its private parts where they landed
      if (!load_wait(ld, bars, 1)) {
        lost = true;
        break;
      }
      __syncwarp();
      const int cnt = min(G, (int)(t1 - t));
      const uint64_t off = (uint64_t)t * priv_per;
      const int nblk = (int)((skew_priv + (cnt - 1) * priv_per + (uint32_t)((nof(t + cnt - 1) * period + 7) >> 3) + 15) >> 4);
      const PairLanes lc = pair_lanes();
#pragma unroll 1
      for (int i = lane; i < nblk; i += 32) {
        uint32_t ks[4];
        ctr_block(a.iv_hi, a.iv_lo, (off >> 4) + i, ks);
        aes128_encrypt_pair(ks, a.rk, lc);
        uint4* p = reinterpret_cast<uint4*>(land_priv + 16 * i);
        uint4 d = *p;
        d.x ^= ks[0];
        d.y ^= ks[1];
        d.z ^= ks[2];
        d.w ^= ks[3];
        *p = d;
      }
      __syncwarp();
    }
    if (!load_wait(ld, bars, 0)) {         // gave up: nothing more is written
      lost = true;
      break;
    }
    __syncwarp();
    unpack_public<W>(reinterpret_cast<const uint32_t*>(land_pub + skew_pub), pubst, n, npub, lane);
    unpack_private<W>(reinterpret_cast<const uint32_t*>(land_priv + skew_priv), privst + lane * (k + 1),
                      (int)(t - run) * kWCb + (lane < n ? lane : 0), k);
    if (t + 1 < t1) {
      const bool last = t + 1 - run == (uint32_t)G;   // of the run: the next one's private parts load too
      // the private parts were decrypted in place, or the public one landed by the lanes' stores
      if (last || lanes_pub) fence_proxy_async();
      __syncwarp();                        // unpacked: the landing areas are free
      skew_pub = load_pub(t + 1);
      if (last) {
        run = t + 1;
        skew_priv = load_priv(run);
      }
    } else {
      __syncwarp();
    }
    const CbPos at = cb_pos(a, 32u * t + lane);
    const int16_t* pub_cb = pubst + lane * npub;
    const int16_t* priv_cb = privst + lane * (k + 1);
    float2 G2[8][4];
    const float l1 = gather_columns<false>(pub_cb, priv_cb, k, G2);
    const uint32_t c0 = __shfl_sync(0xffffffffu, at.c, 0);
    uint8_t* const out = pix + 8 * (c0 + lane - at.c) + at.c;
    uint32_t mlo, mhi;
    emit_rows(G2, l1, lane < n, out, mlo, mhi);
    decide_pixels<false, true>(mlo, mhi, pubst, privst, k, a.cinv, lane, slot, pix, out);
    __syncwarp();                          // the pixel rows are complete
    store_pixels(a.pixels_out, 3ull * (uint64_t)a.width, at, c0, n, lane, pix);
    __syncwarp();                          // the staging area and the pixel buffer may be written again
  }
  if (lost) load_drain(ld, bars, 2);
  if (lane == 0 && a.counters) {
    if (slot->ties) atomicAdd(&a.counters[0], (unsigned long long)slot->ties);
    if (slot->esc) atomicAdd(&a.counters[1], (unsigned long long)slot->esc);
    if (slot->fail || lost) atomicAdd(&a.counters[2], 1ull);
  }
}

template <int K, int W>
static cudaError_t launch_packed(const TileArgs& a, cudaStream_t s, int sms) {
  static bool attr[kMaxAttrDevices];
  static bool window_ok[kMaxAttrDevices];
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
  if (!window_ok[dev]) {
    if ((e = smem_window_start_ok(restore_packed_kernel<K, W>, (uint32_t)kULow)) != cudaSuccess) return e;
    window_ok[dev] = true;
  }
  e = smem_attr_once(restore_packed_kernel<K, W>, kUEnd, attr);
  if (e != cudaSuccess) return e;
  TileArgs b = a;
  const long long nsub = (3ll * a.nblocks + 31) / 32;
  const int grid = (int)(nsub < sms ? nsub : sms);
  b.groups = working_warps((nsub + grid - 1) / (grid ? grid : 1));
  bx_division(b);
  b.run_tiles = run_tiles_packed<W>(a.k);
  if (grid > 0) restore_packed_kernel<K, W><<<grid, kWarps * 32, kUEnd, s>>>(b);
  return cudaGetLastError();
}

// ---- batches ---------------------------------------------------------------------------------

constexpr int kQSlot = (kRSlot + 32 + 7) & ~7;    // two PlanSlots after the single-image area
constexpr int kQWins = kQSlot + 2 * (int)sizeof(PlanSlot);   // the warp's two windows
constexpr int kQArea = (kQWins + 40 + 31) & ~31;
constexpr int kQBelow = ((int)kTpairWin - 1024) / kQArea;
constexpr int kQLow = (int)kTpairWin - kQBelow * kQArea;
constexpr int kQAbove = kWarps > kQBelow ? kWarps - kQBelow : 0;
constexpr int kQTail = (int)kTpairWin + kTpairBytes + kQAbove * kQArea;   // counter
constexpr int kQEnd = kQTail + 16;
static_assert(kQEnd <= 227 * 1024, "restore (batches) shared memory");

// by k: run_tiles (at most a tile), and 16 where two runs fit
struct RunTable {
  uint8_t n[64];
};
constexpr RunTable make_run_table() {
  RunTable t{};
  for (int k = 0; k < 64; ++k)
    t.n[k] = (uint8_t)((run_tiles(k) < kTileSubs ? run_tiles(k) : kTileSubs) | (run_twice(k) ? 16 : 0));
  return t;
}
static __constant__ RunTable c_run = make_run_table();

// Restore of a batch (the tiles as in protect_plan_kernel).  Where the next run is of an image
// with another k, its parts lie elsewhere in the buffers and are loaded only when the run before
// is done.  Bound by issue (241 M warp instructions, issued in 66 % of the cycles: its code is the
// largest, and fetching it the first stall): 300 images (742 MB in and out), k = 5, 445 -> 308 us (two
// CTAs per SM, a tile of six warps each, before).
template <int K>
__global__ void __launch_bounds__(kWarps * 32, 1) restore_plan_kernel(const __grid_constant__ TileArgs a) {
  extern __shared__ __align__(128) uint8_t smem_cta[];
  const uint32_t win0 = smem_u32(smem_cta);
  if (win0 > (uint32_t)kQLow) {   // see the launcher
    if (threadIdx.x == 0 && a.counters) atomicAdd(&a.counters[2], 1ull);
    return;
  }
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  uint8_t* area = smem_cta + ((warp < kQBelow ? (uint32_t)(kQLow + warp * kQArea)
                                              : kTpairWin + kTpairBytes + (uint32_t)(warp - kQBelow) * kQArea) -
                              win0);
  uint8_t* const pix = area + kRPix;
  uint8_t* const frag = area + kRFrag;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(area + kRBar);
  WarpSlot* const slot = reinterpret_cast<WarpSlot*>(area + kRSlot);
  PlanSlot* const slots = reinterpret_cast<PlanSlot*>(area + kQSlot);
  uint32_t* const wins = reinterpret_cast<uint32_t*>(area + kQWins);
  uint32_t* const next = reinterpret_cast<uint32_t*>(smem_cta + (kQTail - win0));
  const int act = a.groups;
  PairFill<kWarps * 32> fill;
  fill.load(a.T, (int)threadIdx.x);
  PlanClaim claim(a, act);
  PlanKeys keys;
  auto nof = [&](const PlanSlot* s, uint32_t t) { return (int)min(32u, s->ncb - 32u * t); };
  Loads ld;                                // barrier 0: public, 1 and 2: the private buffers
  auto load_pub = [&](const PlanSlot* s, uint32_t t) {
    const int npub = 63 - (K >= 0 ? K : s->k);
    ld.issued(0);
    load_part(frag, s->pub + (uint64_t)t * (64u * npub), nof(s, t) * 2 * npub, lane, bars);
  };
  auto load_priv = [&](const PlanSlot* s, uint32_t t, int cnt, int half) {
    const int k = K >= 0 ? K : s->k;
    ld.issued(1 + half);
    load_part(frag + kWCb * 2 * (63 - k) + half * (s->acc & 15) * 64 * (k + 1), s->priv + (uint64_t)t * (64u * (k + 1)),
              ((cnt - 1) * 32 + nof(s, t + cnt - 1)) * 2 * (k + 1), lane, bars + 1 + half);
  };

  if (lane == 0) {
    mbar_init(bars);
    mbar_init(bars + 1);
    mbar_init(bars + 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    slots[0].image = slots[1].image = ~0u;
    slot->ties = slot->esc = slot->fail = 0;
  }
  if (threadIdx.x == 0) *next = (uint32_t)act;
  __syncthreads();                         // a first claim may go on to the counter
  bool lost = false;
  PlanSlot *s = slots, *sx = slots + 1;    // the run's image; the other slot
  uint32_t r = 0, end = 0;                 // the run's first subtile, the end of what was claimed
  int half = 0;
  if (warp < act) {                        // the first run starts loading before the tables are filled
    claim(a, act, next, s, s, c_run.n, warp, lane, r, end, keys);
    if (r < end) {
      load_priv(s, r, min(s->acc & 15, (int)(end - r)), 0);
      load_pub(s, r);
    }
  }
  fill.store(smem_cta + (kTpairWin - win0), (int)threadIdx.x);
  put_keys(s, keys, lane);
  __syncthreads();
  if (warp >= act) return;

  while (r < end && !lost) {
    const int k = K >= 0 ? K : s->k, npub = 63 - k;
    const int G = s->acc & 15, cnt = min(G, (int)(end - r));
    const bool twice = s->acc & 16;
    // the next run: of the same claim, or of a new one
    PlanSlot* n = s;
    uint32_t rn = r + cnt, endn = end;
    if (rn >= end) {
      n = sx;
      claim(a, act, next, n, s, c_run.n, warp, lane, rn, endn, keys);
      put_keys(n, keys, lane);
    }
    const bool have = rn < endn, pipe = have && (K >= 0 || n->k == k);
    const int cntn = have ? min(n->acc & 15, (int)(endn - rn)) : 0;
    uint8_t* const privst = frag + kWCb * 2 * npub + half * G * 64 * (k + 1);
    if (twice && pipe) {
      fence_proxy_async();                 // the buffer was decrypted in place
      __syncwarp();
      load_priv(n, rn, cntn, half ^ 1);
    }
    if (!load_wait(ld, bars, 1 + half)) {
      lost = true;
      break;
    }
    __syncwarp();
    ctr_plan(privst, (((cnt - 1) * 32 + nof(s, r + cnt - 1)) * 2 * (k + 1) + 15) >> 4, (uint64_t)r * (uint32_t)(4 * (k + 1)),
             s, wins, lane);
    __syncwarp();
#pragma unroll 1
    for (int ti = 0; ti < cnt; ++ti) {
      const uint32_t t = r + ti;
      const int m = nof(s, t);
      CbPos at;
      {
        const uint32_t cb = 32u * t + lane, b = cb / 3, bxc = s->bx_count;
        at.c = cb - 3 * b;
        at.by = b / bxc;
        at.bx = b - at.by * bxc;
      }
      if (!load_wait(ld, bars, 0)) {       // gave up: nothing more is written
        lost = true;
        break;
      }
      __syncwarp();
      const int16_t* pub_cb = reinterpret_cast<const int16_t*>(frag) + lane * npub;
      const int16_t* priv_cb = reinterpret_cast<const int16_t*>(privst) + (ti * kWCb + lane) * (k + 1);
      float2 G2[8][4];
      const float l1 = gather_columns<false>(pub_cb, priv_cb, k, G2);
      if (m < kWCb) fence_proxy_async();   // load_part's tail, before the next image's bulk copy
      __syncwarp();                        // the public part is read: the next one starts loading
      if (ti + 1 < cnt)
        load_pub(s, t + 1);
      else if (pipe)
        load_pub(n, rn);
      const uint32_t c0 = __shfl_sync(0xffffffffu, at.c, 0);
      uint8_t* const out = pix + 8 * (c0 + lane - at.c) + at.c;
      uint32_t mlo, mhi;
      emit_rows(G2, l1, lane < m, out, mlo, mhi);
      decide_pixels<false>(mlo, mhi, reinterpret_cast<const int16_t*>(s->pub) + (uint64_t)(32u * t) * npub, priv_cb - lane * (k + 1),
                           k, a.cinv, lane, slot, pix, out);
      if (ti + 1 == cnt && have && !(twice && pipe)) fence_proxy_async();
      __syncwarp();                        // the pixel rows are complete
      if (ti + 1 == cnt && have && !(twice && pipe)) {
        if (!pipe) load_pub(n, rn);
        load_priv(n, rn, cntn, 0);
      }
      store_pixels(s->px, 3ull * s->width, at, c0, m, lane, pix);
      __syncwarp();                        // the pixel buffer may be written again
    }
    if (lost) break;
    half = twice && pipe ? half ^ 1 : 0;
    if (n != s) {
      sx = s;
      s = n;
    }
    r = rn;
    end = endn;
  }
  if (lost) load_drain(ld, bars, 3);
  if (lane == 0 && a.counters) {
    if (slot->ties) atomicAdd(&a.counters[0], (unsigned long long)slot->ties);
    if (slot->esc) atomicAdd(&a.counters[1], (unsigned long long)slot->esc);
    if (slot->fail || lost) atomicAdd(&a.counters[2], 1ull);
  }
}

template <int K, bool PUBIMG>
static cudaError_t launch_w(const TileArgs& a, cudaStream_t s, int sms) {
  static bool attr[kMaxAttrDevices];
  static bool window_ok[kMaxAttrDevices];
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
  if (!window_ok[dev]) {
    if ((e = smem_window_start_ok(restore_warp_kernel<K, PUBIMG>, (uint32_t)kRLow)) != cudaSuccess) return e;
    window_ok[dev] = true;
  }
  e = smem_attr_once(restore_warp_kernel<K, PUBIMG>, kREnd, attr);
  if (e != cudaSuccess) return e;
  TileArgs b = a;
  const long long nsub = (3ll * a.nblocks + 31) / 32;
  const int grid = (int)(nsub < sms ? nsub : sms);
  const long long per = (nsub + grid - 1) / (grid ? grid : 1);
  b.groups = working_warps(per);
  bx_division(b);
  b.run_tiles = run_tiles(a.k) | (run_twice(a.k) ? 16 : 0);
  if (grid > 0) restore_warp_kernel<K, PUBIMG><<<grid, kWarps * 32, kREnd, s>>>(b);
  return cudaGetLastError();
}

// per_sm: half of the CTA's warps (1; else all)
template <int K>
static cudaError_t launch_plan(const TileArgs& a, cudaStream_t s, int sms, int per_sm) {
  static bool attr[kMaxAttrDevices];
  static bool window_ok[kMaxAttrDevices];
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxAttrDevices) return cudaErrorInvalidDevice;
  if (!window_ok[dev]) {
    if ((e = smem_window_start_ok(restore_plan_kernel<K>, (uint32_t)kQLow)) != cudaSuccess) return e;
    window_ok[dev] = true;
  }
  e = smem_attr_once(restore_plan_kernel<K>, kQEnd, attr);
  if (e != cudaSuccess) return e;
  TileArgs b = a;
  b.groups = per_sm == 1 ? kWarps / 2 : kWarps;
  const int grid = a.total_tiles < sms ? a.total_tiles : sms;
  if (grid > 0) restore_plan_kernel<K><<<grid, kWarps * 32, kQEnd, s>>>(b);
  return cudaGetLastError();
}

cudaError_t launch_restore_plan(const TileArgs& a, cudaStream_t s, int sms, int per_sm) {
  if (!a.images || a.pack || a.plain_private || a.public_image) return cudaErrorInvalidValue;
  if (a.k == 0) return launch_plan<0>(a, s, sms, per_sm);
  if (a.k == 5) return launch_plan<5>(a, s, sms, per_sm);
  return launch_plan<-1>(a, s, sms, per_sm);
}

cudaError_t launch_restore_warp(const TileArgs& a, cudaStream_t s, int sms) {
  if (a.images || a.k < 0 || a.k > 63) return cudaErrorInvalidValue;
  if (a.pack) {
    if (a.public_image || a.plain_private) return cudaErrorInvalidValue;
    if (a.pack == 11) return a.k == 5 ? launch_packed<5, 11>(a, s, sms) : launch_packed<-1, 11>(a, s, sms);
    if (a.pack == 8) return a.k == 5 ? launch_packed<5, 8>(a, s, sms) : launch_packed<-1, 8>(a, s, sms);
    return cudaErrorInvalidValue;
  }
  if (a.public_image) return a.k == 5 ? launch_w<5, true>(a, s, sms) : launch_w<-1, true>(a, s, sms);
  if (a.k == 0) return launch_w<0, false>(a, s, sms);
  if (a.k == 5) return launch_w<5, false>(a, s, sms);
  return launch_w<-1, false>(a, s, sms);
}

}  // namespace fds
