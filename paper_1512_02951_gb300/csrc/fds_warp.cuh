// What the warp forms of protect and restore share: subtiles of 32 consecutive channel-blocks (one
// per lane), their place in the image, and AES-128-CTR with the first rounds of neighbouring
// counter blocks computed once.
#pragma once
#include "fds_loads.h"
#include "fds_tile.cuh"

namespace fds {

constexpr int kWCb = 32;                          // channel-blocks per subtile, one per lane
constexpr int kWarps = 16;                        // per CTA, one CTA per SM
// AES constants of counter windows, 5 words each: of the whole CTA's range where it has at most
// kWins, else two for each warp
constexpr int kWins = 64;

// wait for the copy pending on barrier i of the warp's (the whole warp); false: gave up
__device__ __forceinline__ bool load_wait(Loads& ld, uint64_t* bars, int i) {
  const bool ok = __all_sync(0xffffffffu, mbar_wait(bars + i, ld.parity(i)));
  if (ok) ld.arrived(i);
  return ok;
}
// after giving up: the copies still under way
__device__ __forceinline__ void load_drain(const Loads& ld, uint64_t* bars, int n) {
  ld.drain(n, [&](int i, uint32_t parity) { mbar_wait(bars + i, parity); });
}

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

// Working warps of a CTA for `per` subtiles an SM.  Up to three warps on a scheduler a round takes
// the latency of one subtile, the fourth makes it longer; so twelve warps take less than sixteen where
// they need no more rounds (17 .. 24 and 33 .. 36): restore of 4096 x 512, k = 5, 20 subtiles an SM, 18.4
// -> 17.6 us; packed protect of 20000 x 88, k = 17 (18 an SM), 27.0 -> 25.3, of 2600 x 1400 (36), 8 bits,
// 39.2 -> 33.7.  Evening the rounds out further (two of fourteen for 28) was slower: 31.3 -> 33.1.
inline int working_warps(long long per) {
  if (per <= kWarps) return (int)per;
  return (per + 11) / 12 == (per + kWarps - 1) / kWarps ? 12 : kWarps;
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

// ---- the forward transform of a channel-block, as protect computes it and as the coefficients are
// exported before rounding

// Row butterflies of channel c of one row of a block (24 bytes): outputs as pairs of columns (0, 4),
// (1, 2), (3, 5), (6, 7), so that the column pass runs on two columns per packed f32x2 instruction;
// returns the row's error weight
__device__ __forceinline__ float row_pass(uint2 w01, uint2 w23, uint2 w45, uint32_t c, float2 (&P)[4]) {
  const uint32_t r[7] = {w01.x, w01.y, w23.x, w23.y, w45.x, w45.y, 0u};
  uint32_t w[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) w[i] = __funnelshift_r(r[i], r[i + 1], 8 * c);
  float X[8];
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int byte = 3 * x;
    X[x] = __int_as_float(__byte_perm(w[byte >> 2], 0x4B000000u, 0x7440u | (byte & 3)));
  }
  float fr[8];
  const float weight = dct8_row_bytes_w(X, fr);
  P[0] = make_float2(fr[0], fr[4]);
  P[1] = make_float2(fr[1], fr[2]);
  P[2] = make_float2(fr[3], fr[5]);
  P[3] = make_float2(fr[6], fr[7]);
  return weight;
}
// Column butterflies of pair j (columns 0 and 4, pair 0, start from exact integers and stay unscaled
// at the four rational positions); returns pair 0's error weight
__device__ __forceinline__ float column_pass(const float2 (&P)[8][4], int j, float2 (&col)[8]) {
#pragma unroll
  for (int y = 0; y < 8; ++y) col[y] = P[y][j];
  if (j == 0) return dct8_rat_w2(col);
  dct8_2<false, false>(col);
  return 0.0f;
}

// ---- near ties: the marked values of a subtile (bit pos of a lane's mhi:mlo), decided exactly four at
// a time, each by a group of eight lanes.  Eight times the value is n_0 + sum n_j c(j) (fds_device.cuh);
// a lane takes an eighth of the block and of the coordinate table's row (dot products of packed
// bytes), a transposing sum leaves lane j of the group with n_j, and the eight products with c(j) in
// 64-bit fixed point are summed again.  Where many lanes (protect) or many values of one lane (restore)
// are marked, a lane takes a whole value: a pass of the warp then decides up to 32, for the price of
// two to four turns.  What bounds it is issue where ties are many and the chain of a turn (loads from
// L2, three exchanges, twice) where one block has many.  A whole warp for each value, as before, made
// content with many near ties slow; 2048 x 2048, k = 5, us: protect of black and white noise 57.9 ->
// 33.6, of a slow ramp 81.6 -> 42.9, of a block of four ties repeated 303 -> 39.5; the public image of
// text 48.6 -> 20.0; restore of DC-only blocks half a level off (every pixel a tie, k = 0) 3457 -> 119;
// smooth scenes with ten ties a thousand channel-blocks 21.1 -> 20.8 and 24.3 -> 22.8.

// zigzag index by position 8 u + v
struct ZigzagTable {
  uint8_t z[64];
};
constexpr ZigzagTable make_zigzag_table() {
  ZigzagTable t{};
  for (int i = 0; i < 64; ++i) t.z[i] = (uint8_t)zigzag_of(i >> 3, i & 7);
  return t;
}
static __constant__ ZigzagTable c_zigzag = make_zigzag_table();

// The value that the lane's group takes this turn: of lane src, at pos (on: there is one).  who: the
// lanes that have marked values, which drop those taken: one of each of the first four lanes, or two
// of each of two, or four of one.
struct TieTurn {
  int src, pos;
  bool on;
};
__device__ __forceinline__ void drop_lowest(uint32_t& lo, uint32_t& hi) {
  if (lo)
    lo &= lo - 1;
  else
    hi &= hi - 1;
}
__device__ __forceinline__ TieTurn take_ties(uint32_t who, uint32_t& mlo, uint32_t& mhi, int lane) {
  const int m = __popc(who), g = lane >> 3;
  TieTurn t;
  int skip = 0, taken = 0;                 // of src's values, for the groups before; of the lane's own
  bool on = true;
  if (m > 2) {
    uint32_t w = who;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (i < g) w &= w - 1;
    on = w != 0;
    t.src = (__ffs(w) - 1) & 31;
    taken = __popc(who & ((1u << lane) - 1u)) < 4 ? 1 : 0;
  } else {
    t.src = m == 2 && g & 1 ? 31 - __clz(who) : __ffs(who) - 1;
    skip = m == 2 ? g >> 1 : g;
    taken = m == 2 ? 2 : 4;
  }
  uint32_t lo = __shfl_sync(0xffffffffu, mlo, t.src), hi = __shfl_sync(0xffffffffu, mhi, t.src);
  for (int i = 0; i < skip && (lo | hi); ++i) drop_lowest(lo, hi);
  t.on = on && (lo | hi) != 0;
  t.pos = t.on ? (lo ? __ffs(lo) - 1 : __ffs(hi) + 31) : 0;
  for (int i = 0; i < taken && (mlo | mhi); ++i) drop_lowest(mlo, mhi);
  return t;
}

// the sum over the lane's group of n[l], l the lane's place in it
__device__ __forceinline__ int group_sum(const int (&n)[8], int lane) {
  int a[4], b[2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    a[i] = (lane & 4 ? n[i + 4] : n[i]) + __shfl_xor_sync(0xffffffffu, lane & 4 ? n[i] : n[i + 4], 4);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    b[i] = (lane & 2 ? a[i + 2] : a[i]) + __shfl_xor_sync(0xffffffffu, lane & 2 ? a[i] : a[i + 2], 2);
  return (lane & 1 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, lane & 1 ? b[0] : b[1], 1);
}

// exact_round of the values of the groups that fixed point could not decide, in their first lanes; q:
// the others' results
static __device__ __noinline__ int round_far(int n_l, bool far, int q, int lane, int* esc, bool* fail) {
  int n[9], e = 0;
  bool f = false;
#pragma unroll
  for (int j = 0; j < 8; ++j) n[j] = __shfl_sync(0xffffffffu, n_l, (lane & 24) + j);
  n[8] = 0;
  if (far && (lane & 7) == 0) q = exact_round(n, &e, &f);
  *esc += __popc(__ballot_sync(0xffffffffu, e != 0));
  *fail |= (bool)__any_sync(0xffffffffu, f);
  return q;
}

// c(l) with FRAC fraction bits, l the lane's place in its group
template <int FRAC>
__device__ __forceinline__ long long group_cos(int lane) {
  const int l = lane & 7;
  return l ? c_cos_q62[l - 1] >> (62 - FRAC) : 1ll << FRAC;
}

// A value alone in its lane, all its coordinates at hand: the same in one lane.  sure: decided; else too
// near a boundary for fixed point (left to a group)
template <int FRAC>
__device__ __forceinline__ int round_lane(const int (&n)[8], bool& sure) {
  long long d = ((long long)n[0] + 4) << FRAC;
  int err = 0;
#pragma unroll
  for (int j = 1; j < 8; ++j) {
    d += n[j] * (c_cos_q62[j - 1] >> (62 - FRAC));
    err += abs(n[j]);
  }
  const int q = (int)(d >> (FRAC + 3));
  const long long rem = d & ((8ll << FRAC) - 1);
  sure = err == 0 || (rem > err && rem < (8ll << FRAC) - err);
  return err == 0 && rem == 0 && q <= 0 ? q - 1 : q;
}

// Rounds, half away from zero, the value of the lane's group whose eightfold has the coordinates n_l
// (one a lane; on: there is one); the result is the group's first lane's.  Each c(j) 2^FRAC is within a
// unit, so the sum is within sum |n_j| <= BOUND units.  Nearer than that to a boundary it is a tie if it
// is rational (about half of all near ties of protect: positions whose u and v are 2 or 6), and else
// left to exact_round.
template <int FRAC, int BOUND>
__device__ __forceinline__ int round_group(int n_l, long long cos_l, bool on, int lane, int& esc, bool& fail) {
  const bool rational = ((__ballot_sync(0xffffffffu, (lane & 7) && n_l != 0) >> (lane & 24)) & 0xffu) == 0;
  long long d = n_l * cos_l;
#pragma unroll
  for (int i = 1; i < 8; i <<= 1) d += __shfl_xor_sync(0xffffffffu, d, i);
  d += 4ll << FRAC;                        // d / 2^(FRAC + 3) = the value + 1/2
  int q = (int)(d >> (FRAC + 3));
  const long long rem = d & ((8ll << FRAC) - 1);
  if (rational && rem == 0 && q <= 0) --q;
  const bool far = on && !rational && (rem <= BOUND || rem >= (8ll << FRAC) - BOUND);
  if (__any_sync(0xffffffffu, far)) {
    int e = 0;
    bool f = false;
    q = round_far(n_l, far, q, lane, &e, &f);
    esc += e;
    fail |= f;
  }
  return q;
}

// ---- batches: what a warp knows about the image of a tile it works on (shared memory; two per
// warp, the tile's and the next one's)
struct PlanSlot {
  uint8_t* px;                    // the image's pixels, public and private fragments
  uint8_t* pub;
  uint8_t* priv;
  uint64_t iv_hi, iv_lo, wbase;   // wbase: first counter window of the warp's two, ~0 if none
  uint32_t width, bx_count, ncb, image;
  int32_t k, acc;                 // acc: subtiles between two AES phases
  uint32_t rk[44];
};
static_assert(sizeof(PlanSlot) % 8 == 0, "PlanSlot");
constexpr int kTileSubs = kTileCb / kWCb;         // subtiles of a 64-block tile

// Round keys on their way from global memory into a slot (a lane's two words)
struct PlanKeys {
  uint32_t lo, hi;
  bool due = false;
};
__device__ __forceinline__ void put_keys(PlanSlot* s, PlanKeys& keys, int lane) {
  if (!keys.due) return;
  s->rk[lane] = keys.lo;
  if (lane < 12) s->rk[32 + lane] = keys.hi;
  keys.due = false;
  __syncwarp();
}

// The image of tile g into slot s (the whole warp; acc_of: subtiles between two AES phases by k), but
// for its round keys, which put_keys stores; hint: a slot whose image it often is; returns the tile's
// index in the image
__device__ __forceinline__ int plan_slot(const TileArgs& a, int g, PlanSlot* s, const PlanSlot* hint, const uint8_t* acc_of,
                                         int lane, PlanKeys& keys) {
  uint32_t im = hint->image;
  if (!(im < (uint32_t)a.n_images && __ldg(a.tile_start + im) <= g && g < __ldg(a.tile_start + im + 1))) {
    int lo = 0, hi = a.n_images;                 // tile_start[lo] <= g < tile_start[hi]
    while (hi - lo > 1) {
      const int step = (hi - lo + 31) >> 5, p = min(lo + step * lane, hi);
      const uint32_t le = __ballot_sync(0xffffffffu, __ldg(a.tile_start + p) <= g);
      lo += step * (__popc(le) - 1);
      hi = min(lo + step, hi);
    }
    im = (uint32_t)lo;
  }
  const int local = g - __ldg(a.tile_start + im);
  const bool other = s->image != im;
  __syncwarp();
  if (other) {
    const BatchImage& b = a.images[im];
    const uint32_t* rk = a.round_keys + 44 * b.key_slot;
    keys.lo = __ldg(rk + lane);
    keys.hi = lane < 12 ? __ldg(rk + 32 + lane) : 0u;
    keys.due = true;
    if (lane == 0) {
      s->px = const_cast<uint8_t*>(a.pixels_in ? a.pixels_in : a.pixels_out) + b.pixel_offset;
      s->pub = reinterpret_cast<uint8_t*>(a.pub_in ? const_cast<int16_t*>(a.pub_in) : a.pub_out) + b.public_offset;
      s->priv = (a.priv_in ? const_cast<uint8_t*>(a.priv_in) : a.priv_out) + b.private_offset;
      s->iv_hi = b.iv_hi;
      s->iv_lo = b.iv_lo;
      s->wbase = ~0ull - 1;
      s->width = (uint32_t)b.width;
      s->bx_count = (uint32_t)b.width >> 3;
      s->ncb = 3u * ((uint32_t)b.width >> 3) * ((uint32_t)b.height >> 3);
      s->image = im;
      s->k = b.k;
      s->acc = acc_of[b.k];
    }
  } else if (lane == 0) {
    s->wbase = ~0ull - 1;         // the windows may have been the other slot's
  }
  __syncwarp();
  return local;
}

// The next run of subtiles of one image for a warp: [t, end), none left where t == end.  A CTA's
// tiles are [g0, g1).  As many as give every warp the same number of whole tiles are handed out
// whole, the last 2 act subtiles or so one by one, those between in halves, so that the CTA's warps
// end together: with all but the last whole, 12 tiles a CTA left warps idle for a whole tile (30
// images of mixed k, protect 56.0 -> 49.3 us, restore 61.8 -> 56.5).  A warp's first run is its own,
// so that it starts loading before the CTA's tables are filled; the others come from `next`, which
// starts at act and is set before any claim (a first run may be an empty one).  A CTA with no more
// units than warps has nothing behind the first runs, and does not ask (batches of a few hundred
// tiles, below).  Or (a.dispenser) every warp takes tiles from one counter.
// A call of one round of units is a chain in one warp, about 17,000 cycles long (restore, k = 0, a few
// hundred tiles).  The AES table's entries are on their way from the kernel's start and stored while the
// first run's parts and keys are still coming, and nothing is claimed where nothing is left: restore of
// eight images, k = 0, 14.3 -> 12.3 us and 28.7 -> 26.9 (12.3 and 28.6 before the warp form), protect
// 26.4 -> 24.7 (25.6); of thirty images of mixed k 56.1 -> 55.0 and 48.0 -> 46.7.
struct PlanClaim {
  int g0, g1, whole, halves;
  bool first, more;

  __device__ __forceinline__ PlanClaim(const TileArgs& a, int act) {
    g0 = (int)((int64_t)a.total_tiles * blockIdx.x / gridDim.x);
    g1 = (int)((int64_t)a.total_tiles * (blockIdx.x + 1) / gridDim.x);
    const int rest = max(0, g1 - g0 - (2 * act + kTileSubs - 1) / kTileSubs);
    whole = rest / act * act;
    halves = rest - whole;
    first = true;
    more = a.dispenser != nullptr || whole + 2 * halves + kTileSubs * (g1 - g0 - whole - halves) > act;
  }
  __device__ __forceinline__ void operator()(const TileArgs& a, int act, uint32_t* next, PlanSlot* s, const PlanSlot* hint,
                                             const uint8_t* acc_of, int warp, int lane, uint32_t& t, uint32_t& end,
                                             PlanKeys& keys) {
    while (first || more) {
      uint32_t u = 0;
      if (a.dispenser == nullptr) {
        if (first)
          u = (uint32_t)warp;
        else if (lane == 0)
          u = atomicAdd(next, 1u);
      } else if (first) {
        u = blockIdx.x * act + warp;
      } else if (lane == 0) {
        u = atomicAdd(a.dispenser, 1u) + gridDim.x * act;
      }
      u = __shfl_sync(0xffffffffu, u, 0);
      first = false;
      int g = (int)u, sub = 0, len = kTileSubs;
      if (a.dispenser != nullptr) {
        if (u >= (uint32_t)a.total_tiles) break;
      } else {
        int v = (int)u - whole;
        if (v >= 2 * halves) {
          v -= 2 * halves;
          g = whole + halves + v / kTileSubs;
          sub = v % kTileSubs;
          len = 1;
        } else if (v >= 0) {
          g = whole + (v >> 1);
          len = kTileSubs / 2;
          sub = v & 1 ? len : 0;
        }
        g += g0;
        if (g >= g1) break;
      }
      const int local = plan_slot(a, g, s, hint, acc_of, lane, keys);
      t = (uint32_t)(local * kTileSubs + sub);
      end = min(t + len, (s->ncb + 31u) >> 5);
      if (t < end) return;
    }
    t = end = 0;
  }
};

// AES-128-CTR over nblk keystream blocks at buf, the first being block `first` of the slot's
// image: through the warp's two counter windows (wins) where it has them or where more than two
// rounds of blocks pay for their constants
__device__ __forceinline__ void ctr_plan(uint8_t* buf, int nblk, uint64_t first, PlanSlot* s, uint32_t* wins, int lane) {
  const PairLanes lc = pair_lanes();
  const uint64_t b0 = (s->iv_lo & 255u) + first;               // from the IV's window
  uint64_t wbase = s->wbase;
  bool use = (b0 >> 8) >= wbase && ((b0 + nblk - 1) >> 8) <= wbase + 1;
  if (!use && nblk > 64) {
    wbase = b0 >> 8;
    uint32_t w[5];
    aes_window(s->iv_hi, s->iv_lo, wbase + (lane & 1), s->rk, lc, w);
    __syncwarp();
    if (lane < 2) {
#pragma unroll
      for (int i = 0; i < 5; ++i) wins[5 * lane + i] = w[i];
    }
    if (lane == 0) s->wbase = wbase;
    __syncwarp();
    use = true;
  }
#pragma unroll 1
  for (int i = lane; i < nblk; i += 32) {
    uint32_t ks[4];
    if (use) {
      const uint64_t b = b0 + i;
      const uint32_t* src = wins + ((b >> 8) != wbase ? 5 : 0);
      const uint32_t w[5] = {src[0], src[1], src[2], src[3], src[4]};
      aes_from_window(w, (uint32_t)b & 255u, s->rk, lc, ks);
    } else {
      ctr_block(s->iv_hi, s->iv_lo, first + i, ks);
      aes128_encrypt_pair(ks, s->rk, lc);
    }
    uint4* p = reinterpret_cast<uint4*>(buf + 16 * i);
    uint4 d = *p;
    d.x ^= ks[0];
    d.y ^= ks[1];
    d.z ^= ks[2];
    d.w ^= ks[3];
    *p = d;
  }
}

}  // namespace fds
