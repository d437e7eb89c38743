// What the warp forms of protect and restore share: subtiles of 32 consecutive channel-blocks (one
// per lane), their place in the image, and AES-128-CTR with the first rounds of neighbouring
// counter blocks computed once.
#pragma once
#include "fds_tile.cuh"

namespace fds {

constexpr int kWCb = 32;                          // channel-blocks per subtile, one per lane
constexpr int kWarps = 16;                        // per CTA, one CTA per SM
// AES constants of counter windows, 5 words each: of the whole CTA's range where it has at most
// kWins, else two for each warp
constexpr int kWins = 64;

// One image position of a lane's channel-block: block column, block row, channel
struct CbPos {
  uint32_t bx, by, c;
};

__device__ __forceinline__ CbPos cb_pos(const TileArgs& a, uint32_t cb) {
  CbPos p;
  const uint32_t b = cb / 3;
  p.c = cb - 3 * b;
  p.by = (uint32_t)(((uint64_t)b * a.bx_magic) >> a.bx_shift);   // b / bx_count
  p.bx = b - p.by * (uint32_t)a.bx_count;
  return p;
}

// block / bx_count as a multiply and a shift, exact for block numbers below 2^31: with l the
// smallest integer such that bx_count <= 2^l, the multiplier is off by less than 2^l / bx_count
inline void bx_division(TileArgs& a) {
  int l = 0;
  while ((1ll << l) < a.bx_count) ++l;
  a.bx_shift = 31 + l;
  a.bx_magic = (uint32_t)((1ull << (31 + l)) / (uint64_t)a.bx_count + 1);
}

// AES constants of counter window q (256 counter blocks that differ in the last byte only)
__device__ __forceinline__ void aes_window(uint64_t iv_hi, uint64_t iv_lo, uint64_t q, const uint32_t* rk, PairLanes lc,
                                           uint32_t (&w)[5]) {
  auto r8 = [](uint32_t x) { return __byte_perm(x, x, 0x2103u); };
  uint32_t s[4];
  ctr_block(iv_hi, iv_lo & ~255ull, q << 8, s);
  const uint32_t s0 = s[0] ^ rk[0], s1 = s[1] ^ rk[1], s2 = s[2] ^ rk[2], s3 = s[3] ^ rk[3];
  // round 1: column 0 lacks T3 of the last byte
  const uint32_t n0 = tpair<0>(s0, lc.c0) ^ tpair<2>(s2, lc.c2) ^ rk[4] ^ r8(tpair<1>(s1, lc.c0));
  const uint32_t n1 = tpair<0>(s1, lc.c0) ^ tpair<2>(s3, lc.c2) ^ rk[5] ^ r8(tpair<1>(s2, lc.c0) ^ tpair<3>(s0, lc.c2));
  const uint32_t n2 = tpair<0>(s2, lc.c0) ^ tpair<2>(s0, lc.c2) ^ rk[6] ^ r8(tpair<1>(s3, lc.c0) ^ tpair<3>(s1, lc.c2));
  const uint32_t n3 = tpair<0>(s3, lc.c0) ^ tpair<2>(s1, lc.c2) ^ rk[7] ^ r8(tpair<1>(s0, lc.c0) ^ tpair<3>(s2, lc.c2));
  w[0] = n0;
  // round 2 without the terms of column 0
  w[1] = tpair<2>(n2, lc.c2) ^ rk[8] ^ r8(tpair<1>(n1, lc.c0) ^ tpair<3>(n3, lc.c2));
  w[2] = tpair<0>(n1, lc.c0) ^ tpair<2>(n3, lc.c2) ^ rk[9] ^ r8(tpair<1>(n2, lc.c0));
  w[3] = tpair<0>(n2, lc.c0) ^ rk[10] ^ r8(tpair<1>(n3, lc.c0) ^ tpair<3>(n1, lc.c2));
  w[4] = tpair<0>(n3, lc.c0) ^ tpair<2>(n1, lc.c2) ^ rk[11] ^ r8(tpair<3>(n2, lc.c2));
}

// keystream block whose counter's last byte is x, in the window of constants w
__device__ __forceinline__ void aes_from_window(const uint32_t (&w)[5], uint32_t x, const uint32_t* rk, PairLanes lc,
                                                uint32_t (&s)[4]) {
  auto r8 = [](uint32_t v) { return __byte_perm(v, v, 0x2103u); };
  const uint32_t n0 = w[0] ^ r8(tpair<0>(x ^ (rk[3] >> 24), lc.c2));
  uint32_t s0 = w[1] ^ tpair<0>(n0, lc.c0);
  uint32_t s1 = w[2] ^ r8(tpair<3>(n0, lc.c2));
  uint32_t s2 = w[3] ^ tpair<2>(n0, lc.c2);
  uint32_t s3 = w[4] ^ r8(tpair<1>(n0, lc.c0));
#pragma unroll 1
  for (int r = 3; r < 10; ++r) {
    const uint32_t m0 = tpair<0>(s0, lc.c0) ^ tpair<2>(s2, lc.c2) ^ rk[4 * r] ^ r8(tpair<1>(s1, lc.c0) ^ tpair<3>(s3, lc.c2));
    const uint32_t m1 = tpair<0>(s1, lc.c0) ^ tpair<2>(s3, lc.c2) ^ rk[4 * r + 1] ^ r8(tpair<1>(s2, lc.c0) ^ tpair<3>(s0, lc.c2));
    const uint32_t m2 = tpair<0>(s2, lc.c0) ^ tpair<2>(s0, lc.c2) ^ rk[4 * r + 2] ^ r8(tpair<1>(s3, lc.c0) ^ tpair<3>(s1, lc.c2));
    const uint32_t m3 = tpair<0>(s3, lc.c0) ^ tpair<2>(s1, lc.c2) ^ rk[4 * r + 3] ^ r8(tpair<1>(s0, lc.c0) ^ tpair<3>(s2, lc.c2));
    s0 = m0;
    s1 = m1;
    s2 = m2;
    s3 = m3;
  }
  auto last = [&](uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    const uint32_t lo = __byte_perm(tpair<0>(a, lc.c2), tpair<1>(b, lc.c0), 0x3250u);
    const uint32_t hi = __byte_perm(tpair<2>(c, lc.c0), tpair<3>(d, lc.c2), 0x7210u);
    return __byte_perm(lo, hi, 0x7610u);
  };
  s[0] = last(s0, s1, s2, s3) ^ rk[40];
  s[1] = last(s1, s2, s3, s0) ^ rk[41];
  s[2] = last(s2, s3, s0, s1) ^ rk[42];
  s[3] = last(s3, s0, s1, s2) ^ rk[43];
}

// the constants of window q to wc[5 * slot] (every lane its own; slot < 0: none)
__device__ __forceinline__ void put_window(const TileArgs& a, uint64_t q, int slot, uint32_t* wc) {
  uint32_t w[5];
  aes_window(a.iv_hi, a.iv_lo, q, a.rk, pair_lanes(), w);
  if (slot >= 0) {
#pragma unroll
    for (int i = 0; i < 5; ++i) wc[5 * slot + i] = w[i];
  }
}

}  // namespace fds
