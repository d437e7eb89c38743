// Restore of one image with the inverse transform on tensor cores, and the dispatch of restore (its
// float32 forms: fds_restore_warp.cu): CTR decryption of the confidential fragment, merge with the
// public fragment by zigzag position, inverse 8x8 DCT, round half away from zero (exact), clamp to
// [0, 255].
//
// Persistent CTAs over the image's tiles, b, b + gridDim.x, ..; per tile (see fds_tile.cuh):
//   A. the tile's fragments are in shared memory, already decrypted; the next tile's start
//      loading (one bulk copy per fragment range, or cp.async pieces)
//   1. the coefficients as the MMAs' f16 operand, the accumulators back from TMEM (or, per
//      channel-block, float32 inverse butterflies, columns then rows); round + clamp, bytes into
//      the interleaved pixel tile; values within the error guard of a half-integer are queued
//   B. 2. queued pixels are re-decided exactly (integer coordinates in Z[cos(pi/16)]) by the
//      last threads while the first ones decrypt the next tile's private range in place
//      (AES-128-CTR)
//   C. 3. the pixel tile goes to global memory: one bulk (TMA engine) store per pixel row when
//      the tile's rows are contiguous and 16-byte aligned, else 8-byte stores.  The pixel tile
//      is double-buffered so the bulk stores overlap the next tile.
#include "fds_mma.cuh"

namespace fds {

constexpr int kSmemCoef = 0;                                 // 2 fragment staging areas
constexpr int kSmemPix = kSmemCoef + 2 * kCoefBytes;         // 2 pixel tiles
constexpr int kSmemQueue = kSmemPix + 2 * kPixBytes;
constexpr int kSmemSlot = kSmemQueue + 4 * kQueueCap;        // 3 tile slots (ring)
constexpr int kSlotBytes = (sizeof(TileSlot) + 15) & ~15;
constexpr int kSmemBar = kSmemSlot + 3 * kSlotBytes;         // 2 mbarriers (staging areas)
constexpr int kSmemMisc = kSmemBar + 16;
constexpr int kSmemBytes = kSmemMisc + 32;
// the AES table T0 replicated per lane (32 KB; conflict-free lookups) after the rest
constexpr int kSmemTrep = kSmemBytes;
constexpr int kSmemBytesRep = kSmemTrep + 4 * kTrepWords;
// tensor-core inverse (TC): after the rest, on a 1024-byte boundary, the A operand (256 rows
// of 64 f16 coefficients: the tile's 192 channel-blocks as two MMA row blocks of 128) and the
// B operand (the inverse basis, three f16 limbs x 64 pixels), an mbarrier and the TMEM address
constexpr int kTcA = 256 * 128;
constexpr int kSmemBytesTc = kSmemBytesRep + 1024 + kTcA + kMmaInvBytes + 16;
constexpr int kTcCols = 2 * 192;                       // accumulator columns: 2 row blocks x 3 limbs x 64
static_assert(kTcCols <= 512, "TMEM columns");
constexpr uint32_t kTcInvIdesc = idesc_f16(192, false);
// guard of the TC inverse, per channel-block with S = sum |q|: S 2^-24 + 2^-22 (the host
// proves, when it builds the limb table, that split remainder plus combining roundings stay
// below S 2^-24, and refuses otherwise; 2^-22 covers the roundings of the guard itself)
constexpr float kTcInvGuardS = 1.0f / 16777216.0f;
constexpr float kTcInvGuard0 = 1.0f / 4194304.0f;

// gather the 64 int16 coefficients of tile channel-block cb in zigzag order, two per word
__device__ __forceinline__ void gather_coefs(const int16_t* pubst, const int16_t* privst, int cb,
                                             int k, uint32_t (&Q)[32]) {
  const uint16_t* pu = reinterpret_cast<const uint16_t*>(pubst) + cb * (63 - k) - (k + 1);
  const uint16_t* pv = reinterpret_cast<const uint16_t*>(privst) + cb * (k + 1);
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const uint32_t lo = 2 * i <= k ? pv[2 * i] : pu[2 * i];
    const uint32_t hi = 2 * i + 1 <= k ? pv[2 * i + 1] : pu[2 * i + 1];
    Q[i] = lo | (hi << 16);
  }
}

// True if both fragment ranges of the tile are whole 16-byte units (then each arrives as one
// bulk copy completing on an mbarrier; else as 16-byte cp.async pieces)
__device__ __forceinline__ bool frag_bulk(const TileSlot* sl) {
  const int k = sl->k, nb = sl->nb;
  return ((nb * 6 * (63 - k)) & 15) == 0 && ((nb * 6 * (k + 1)) & 15) == 0;
}
// Load the public and private ranges of slot sl's tile into staging area st (all threads call
// it; thread 0 issues the bulk copies)
__device__ __forceinline__ void load_fragments(const TileSlot* sl, uint8_t* st, uint64_t* bar) {
  const int t = threadIdx.x;
  const int k = sl->k, npub = 63 - k, nb = sl->nb;
  const int pub_bytes = nb * 6 * npub, priv_bytes = nb * 6 * (k + 1);
  const uint8_t* psrc = sl->pub_in + (uint64_t)sl->local * kTileBlocks * 6ull * npub;
  const uint8_t* vsrc = sl->priv_in + (uint64_t)sl->local * kTileBlocks * 6ull * (k + 1);
  uint8_t* vdst = st + kTileCb * 2 * npub;
  if (frag_bulk(sl)) {
    if (t == 0) {
      mbar_expect_tx(bar, (uint32_t)(pub_bytes + priv_bytes));
      if (pub_bytes) bulk_load(st, psrc, (uint32_t)pub_bytes, bar);
      if (priv_bytes) bulk_load(vdst, vsrc, (uint32_t)priv_bytes, bar);
    }
    return;
  }
  const int p16 = pub_bytes >> 4, v16 = priv_bytes >> 4;
  for (int i = t; i < p16 + v16; i += kThreads) {
    if (i < p16)
      cp_async16(st + 16 * i, psrc + 16 * i);
    else
      cp_async16(vdst + 16 * (i - p16), vsrc + 16 * (i - p16));
  }
  for (int j = (p16 << 4) + 2 * t; j < pub_bytes; j += 2 * kThreads)
    *reinterpret_cast<uint16_t*>(st + j) = *reinterpret_cast<const uint16_t*>(psrc + j);
  for (int j = (v16 << 4) + 2 * t; j < priv_bytes; j += 2 * kThreads)
    *reinterpret_cast<uint16_t*>(vdst + j) = *reinterpret_cast<const uint16_t*>(vsrc + j);
  cp_async_commit();
}
// Wait until this thread may read what load_fragments loaded (a barrier must follow);
// phase: the next phase of bar; lost counts bulk loads that did not complete in time
__device__ __forceinline__ void wait_fragments(const TileSlot* sl, uint64_t* bar, uint32_t& phase, int& lost) {
  if (frag_bulk(sl)) {
    if (!mbar_wait(bar, phase)) ++lost;
    phase ^= 1u;
  } else {
    cp_async_wait_all();
  }
}

// CTR decryption of the private range of slot sl's tile, in staging area st (int16 storage)
__device__ __forceinline__ void decrypt_fragments(const TileSlot* sl, const uint32_t* rk, uint8_t* st, const uint32_t* Trep) {
  const int k = sl->k;
  const uint64_t first = ((uint64_t)sl->local * kTileBlocks * 6ull * (uint64_t)(k + 1)) >> 4;
  ctr_tile_rep(st + kTileCb * 2 * (63 - k), sl->nb * 6 * (k + 1), first, sl, rk, Trep, (int)threadIdx.x);
}

// The inverse transform as tcgen05 MMAs (one image, int16 storage; a.tc_b = the inverse basis
// table); a tile holding a coefficient of magnitude 2048 or more takes the float32 butterflies
// instead.  Round keys are read from the kernel parameters.
template <int K>
__global__ void __launch_bounds__(kThreads, 1) restore_tc_kernel(const __grid_constant__ TileArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  uint32_t* Ts = reinterpret_cast<uint32_t*>(smem + kSmemTrep);   // T0 replicated per lane
  uint32_t* queue = reinterpret_cast<uint32_t*>(smem + kSmemQueue);
  // misc: [0] queue size, [1] queued total, [2] escalations, [3] failures, [4..5] schedule
  int* misc = reinterpret_cast<int*>(smem + kSmemMisc);
  const int t = threadIdx.x;
  const int ntiles = (a.nblocks + kTileBlocks - 1) / kTileBlocks;
  if ((int)blockIdx.x >= ntiles) return;
  auto slot = [&](int i) { return reinterpret_cast<TileSlot*>(smem + kSmemSlot + i * kSlotBytes); };
  auto stage = [&](int i) { return smem + kSmemCoef + i * kCoefBytes; };

  for (int i = t; i < kTrepWords; i += kThreads) Ts[i] = __ldg(a.T + (i >> 5));
  if (t < 4) misc[t] = 0;
  if (t == 0) {
    misc[6] = 0;                         // TC: a tensor-core wait gave up
    misc[4] = blockIdx.x;
    misc[5] = blockIdx.x + gridDim.x;
  }
  if (t < kTileBlocks) fill_slot(a, blockIdx.x, slot(0), t);
  __syncthreads();
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kSmemBar);
  uint32_t phase[2] = {0u, 0u};
  int lost = 0;
  // TC: operands, MMA barrier, TMEM (kTcCols columns rounded up to 512)
  uint8_t* const tcbase =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem + kSmemBytesRep) + 1023) & ~(uintptr_t)1023);
  uint8_t* const tA = tcbase;
  uint8_t* const tB = tcbase + kTcA;
  uint64_t* const tbar = reinterpret_cast<uint64_t*>(tcbase + kTcA + kMmaInvBytes);
  uint32_t* const tslot = reinterpret_cast<uint32_t*>(tcbase + kTcA + kMmaInvBytes + 8);
  {
    for (int i = t; i < kMmaInvBytes / 16; i += kThreads) reinterpret_cast<uint4*>(tB)[i] = a.tc_b[i];
    for (int i = t; i < 64 * 128 / 16; i += kThreads)    // A rows 192..255 (never a channel-block)
      reinterpret_cast<uint4*>(tA + 192 * 128)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (t < 32) tmem_alloc<512>(tslot);
    fence_proxy_async();
  }
  if (t == 0) {
    mbar_init(bars);
    mbar_init(bars + 1);
    mbar_init(tbar);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  load_fragments(slot(0), stage(0), bars);
  wait_fragments(slot(0), bars, phase[0], lost);
  __syncthreads();
  decrypt_fragments(slot(0), a.rk, stage(0), Ts);
  int esc = 0;
  bool fail = false;
  // a fragment load that did not complete in time leaves its tile's pixels unwritten (the
  // failure counter records it): cur_lost for the tile being transformed, lost counts them all
  int cur_lost = lost;
  uint32_t tmem = 0, tphase = 0;
  {
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    tmem = *tslot;
  }
  for (int it = 0;; ++it) {
    const int buf = it & 1;
    const int cur = misc[4 + buf], nxt = misc[4 + (buf ^ 1)];
    if (cur >= ntiles) break;
    const TileSlot* sl = slot(it % 3);
    if (nxt < ntiles && t < kTileBlocks) fill_slot(a, nxt, slot((it + 1) % 3), t);
    uint8_t* pix = smem + kSmemPix + buf * kPixBytes;
    if (t == 0) {
      misc[0] = 0;
      // the stores of two tiles ago have read pix (each tile commits one bulk group)
      asm volatile("cp.async.bulk.wait_group.read 1;\n" ::: "memory");
    }
    __syncthreads();                                                       // A
    if (t == 0) misc[4 + buf] = nxt < ntiles ? (int)(blockIdx.x + (it + 2) * gridDim.x) : ntiles;
    if (nxt < ntiles) {
      load_fragments(slot((it + 1) % 3), stage(buf ^ 1), bars + (buf ^ 1));
    }
    const int k = K >= 0 ? K : sl->k;
    const int npub = 63 - k;
    const int nb = sl->nb;
    const int16_t* pubst = reinterpret_cast<const int16_t*>(stage(buf));
    const int16_t* privst = reinterpret_cast<const int16_t*>(stage(buf) + kTileCb * 2 * npub);
    const int cb = t, b = t / 3, c = t - 3 * (t / 3);
    uint8_t* out = pix + b * 24 + c;
    uint32_t mlo = 0, mhi = 0;
    // one row of restored values: clamp, round, mark the values within the guard of a
    // half-integer, bytes into the interleaved pixel tile
    auto emit_row = [&](int y, const float (&row)[8], float thr) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 pc = make_float2(fminf(fmaxf(row[2 * j], 0.0f), 255.0f), fminf(fmaxf(row[2 * j + 1], 0.0f), 255.0f));
        const float2 yv = add2(pc, make_float2(kMagic, kMagic));
        const float2 r = sub2(pc, add2(yv, make_float2(-kMagic, -kMagic)));
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const int x = 2 * j + l;
          if (fabsf(l ? r.y : r.x) > thr) {
            if (8 * y + x < 32)
              mlo |= 1u << (8 * y + x);
            else
              mhi |= 1u << (8 * y + x - 32);
          }
          out[y * kRowBytes + 3 * x] = (uint8_t)__float_as_uint(l ? yv.y : yv.x);
        }
      }
    };
    bool tc_done = false;
    {
      // A row t: the channel-block's 64 coefficients in zigzag order (the K order of the
      // basis table), as f16 -- exact for |q| < 2048; S = sum |q| sizes the guard
      int S = 0;
      bool big = false;
      if (b < nb) {
        const int16_t* pub_cb = pubst + cb * npub;
        const int16_t* priv_cb = privst + cb * (k + 1);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          uint32_t w[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int z0 = 8 * j + 2 * m, z1 = z0 + 1;
            const int q0 = z0 <= k ? priv_cb[z0] : pub_cb[z0 - k - 1];
            const int q1 = z1 <= k ? priv_cb[z1] : pub_cb[z1 - k - 1];
            const int m0 = q0 < 0 ? -q0 : q0, m1 = q1 < 0 ? -q1 : q1;
            S += m0 + m1;
            big |= (m0 | m1) >= 2048;
            const __half2 h = __floats2half2_rn((float)q0, (float)q1);
            w[m] = *reinterpret_cast<const uint32_t*>(&h);
          }
          *reinterpret_cast<uint4*>(tA + sw128_offset(t, j)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      fence_proxy_async();
      if (!__syncthreads_or(big || misc[6] != 0)) {                           // A2
        if (t == 0) {
          tc_fence_after_sync();
          const uint32_t a0 = smem_u32(tA), b0 = smem_u32(tB);
#pragma unroll
          for (int rb = 0; rb < 2; ++rb)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              mma_f16(tmem + 192u * rb, sw128_kmajor_desc(a0 + rb * 128 * 128) + 2 * ks, sw128_kmajor_desc(b0) + 2 * ks,
                      kTcInvIdesc, ks > 0 ? 1u : 0u);
          mma_commit(tbar);
        }
        const bool ok = __all_sync(0xffffffffu, mbar_wait(tbar, tphase));
        tphase ^= 1u;
        tc_fence_after_sync();
        if (!ok) {                               // the tile's pixels stay unwritten; later
          ++cur_lost;                            // tiles take the float32 path
          ++lost;
          if ((t & 31) == 0) misc[6] = 1;
        }
        // this warp's TMEM lanes: row block t / 128, lanes 32 (warp % 4) ..
        const int warp = t >> 5;
        const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (warp >= 4 ? 192u : 0u);
        const float thr = 0.5f - fmaf((float)S, kTcInvGuardS, kTcInvGuard0);
#pragma unroll
        for (int h = 0; h < 4; ++h) {          // pixel rows 2h and 2h + 1
          uint32_t d0[16], d1[16], d2[16];
          tmem_ld16(tl + 16 * h, d0);
          tmem_ld16(tl + 64 + 16 * h, d1);
          tmem_ld16(tl + 128 + 16 * h, d2);
          tmem_ld_wait();
          if (ok && b < nb) {
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
              float row[8];
#pragma unroll
              for (int x = 0; x < 8; ++x) {
                const int i = 8 * rr + x;
                row[x] = fmaf(fmaf(__uint_as_float(d2[i]), 1.0f / 256.0f, __uint_as_float(d1[i])), 1.0f / 256.0f,
                              __uint_as_float(d0[i])) * (1.0f / 512.0f);
              }
              emit_row(2 * h + rr, row, thr);
            }
          }
        }
        tc_fence_before_sync();
        tc_done = true;
      }
    }
    if (!tc_done && b < nb) {
      const int16_t* pub_cb = pubst + cb * npub;
      const int16_t* priv_cb = privst + cb * (k + 1);
      // coefficients as pairs of adjacent columns: the column pass runs on two columns per
      // packed f32x2 instruction
      float2 G[8][4];
      float l1 = 0.0f;  // sum |F|, exact (integers below 2^24)
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int z0 = zigzag_of(u, 2 * j), z1 = zigzag_of(u, 2 * j + 1);
          const int q0 = z0 <= k ? priv_cb[z0] : pub_cb[z0 - k - 1];
          const int q1 = z1 <= k ? priv_cb[z1] : pub_cb[z1 - k - 1];
          G[u][j] = add2(make_float2(__int_as_float(kMagicBits + q0), __int_as_float(kMagicBits + q1)),
                         make_float2(-kMagic, -kMagic));
          l1 += fabsf(G[u][j].x);
          l1 += fabsf(G[u][j].y);
        }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float2 col[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) col[u] = G[u][j];
        idct8_2(col);
#pragma unroll
        for (int y = 0; y < 8; ++y) G[y][j] = col[y];
      }
      const float thr = 0.5f - l1 * kGuardInvScale;
#pragma unroll
      for (int y = 0; y < 8; ++y) {
        float row[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          row[2 * j] = G[y][j].x;
          row[2 * j + 1] = G[y][j].y;
        }
        idct8(row);
        emit_row(y, row, thr);
      }
    }
    if (b < nb) {
      uint64_t mask = ((uint64_t)mhi << 32) | mlo;
      while (mask) {
        const int pos = __ffsll((long long)mask) - 1;
        mask &= mask - 1;
        const int idx = atomicAdd(&misc[0], 1);
        if (idx < kQueueCap) {
          queue[idx] = ((uint32_t)cb << 8) | (uint32_t)pos;
        } else {  // queue full: decide here
          uint32_t Q[32];
          int n[9];
          gather_coefs(pubst, privst, cb, k, Q);
          coords_inv(Q, pos, a.cinv, n);
          const int p = exact_round(n, &esc, &fail);
          out[(pos >> 3) * kRowBytes + 3 * (pos & 7)] = (uint8_t)(p < 0 ? 0 : (p > 255 ? 255 : p));
        }
      }
    }
    const int lost_before_next = lost;
    if (nxt < ntiles) {
      wait_fragments(slot((it + 1) % 3), bars + (buf ^ 1), phase[buf ^ 1], lost);
    }
    __syncthreads();                                                       // B
    {
      // queued pixels (from the last thread down) re-decided exactly while the first threads
      // decrypt the next tile's private range
      const int nq = min(misc[0], kQueueCap);
      for (int i = kThreads - 1 - t; i < nq; i += kThreads) {
        const uint32_t e = queue[i];
        const int ecb = (int)(e >> 8), pos = (int)(e & 255);
        const int eb = ecb / 3, ec = ecb - 3 * eb;
        uint32_t Q[32];
        int n[9];
        gather_coefs(pubst, privst, ecb, k, Q);
        coords_inv(Q, pos, a.cinv, n);
        const int p = exact_round(n, &esc, &fail);
        pix[(pos >> 3) * kRowBytes + eb * 24 + 3 * (pos & 7) + ec] = (uint8_t)(p < 0 ? 0 : (p > 255 ? 255 : p));
      }
      if (t == 0) misc[1] += misc[0];
    }
    if (nxt < ntiles) decrypt_fragments(slot((it + 1) % 3), a.rk, stage(buf ^ 1), Ts);
    fence_proxy_async();                                  // pixel writes before the bulk stores
    const bool skip = __syncthreads_or(cur_lost != 0);                     // C
    cur_lost = lost - lost_before_next;                   // the next tile's fragments
    if (skip) {
      if (t == 0) bulk_commit();                 // an empty group keeps one group per tile
    } else {
      // the pixel tile to global memory: one bulk (TMA engine) store per pixel row when the
      // tile's blocks are contiguous and 16-byte aligned in every row, else 8-byte stores
      const uint64_t w3 = (uint64_t)sl->width * 3ull;
      uint8_t* row0 = sl->px_out + sl->blk[0];
      if (sl->px_out16) {
        if (t == 0) {
#pragma unroll 1
          for (int y = 0; y < 8; ++y) bulk_store(row0 + y * w3, pix + y * kRowBytes, (uint32_t)(nb * 24));
          bulk_commit();
        }
      } else {
        if (t == 0) bulk_commit();               // an empty group keeps one group per tile
        for (int i = t; i < 8 * kTileBlocks * 3; i += kThreads) {
          const int y = i / (kTileBlocks * 3), rem = i - y * (kTileBlocks * 3);
          const int bb = rem / 3, q = rem - 3 * bb;
          if (bb < nb)
            *reinterpret_cast<uint2*>(sl->px_out + sl->blk[bb] + y * w3 + 8 * q) =
                *reinterpret_cast<const uint2*>(pix + y * kRowBytes + bb * 24 + 8 * q);
        }
      }
    }
  }
  if (esc) atomicAdd(&misc[2], esc);
  if (fail || lost) atomicAdd(&misc[3], 1);
  tc_fence_before_sync();
  __syncthreads();
  {
    tc_fence_after_sync();
    if (t < 32) tmem_dealloc<512>(tmem);
  }
  if (t == 0) bulk_wait_all();
  if (t == 0 && a.counters) {
    if (misc[1]) atomicAdd(&a.counters[0], (unsigned long long)misc[1]);
    if (misc[2]) atomicAdd(&a.counters[1], (unsigned long long)misc[2]);
    if (misc[3]) atomicAdd(&a.counters[2], (unsigned long long)misc[3]);
  }
}

template <int K>
static cudaError_t launch_k(const TileArgs& a, cudaStream_t s, int sms) {
  static bool attr[kMaxAttrDevices];
  cudaError_t e = smem_attr_once(restore_tc_kernel<K>, kSmemBytesTc, attr);
  if (e != cudaSuccess) return e;
  const int ntiles = total_tiles(a);
  const int grid = ntiles < sms ? ntiles : sms;
  if (grid > 0) restore_tc_kernel<K><<<grid, kThreads, kSmemBytesTc, s>>>(a);
  return cudaGetLastError();
}

// the tensor-core inverse form (one image, int16 storage; a.tc_b = the inverse basis table),
// one CTA per SM (the operands and TMEM take what a second CTA would need)
cudaError_t launch_restore_tc(const TileArgs& a, cudaStream_t s, int sms) {
  if (a.images || a.k < 0 || a.public_image || a.pack || a.plain_private || !a.tc_b) return cudaErrorInvalidValue;
  if (a.k == 0) return launch_k<0>(a, s, sms);
  if (a.k == 5) return launch_k<5>(a, s, sms);
  return launch_k<-1>(a, s, sms);
}

// k is uniform over the launch when a.k >= 0; a.k < 0 (batches of mixed k) reads k per tile
cudaError_t launch_restore(const TileArgs& a, cudaStream_t s, int sms, int per_sm) {
  return a.images ? launch_restore_plan(a, s, sms, per_sm) : launch_restore_warp(a, s, sms);
}

}  // namespace fds
