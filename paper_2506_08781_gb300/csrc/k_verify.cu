// Verification kernels: epoch seeds, hashing and scalar aggregation, point decoding and sums,
// window tables and the final cofactored check.
#include "common.cuh"
#include "compact.cuh"
#include "stage.h"

namespace poslo {

template <int INST>
__global__ void k_epoch_seeds(const DsNode* __restrict__ ds, int nds, uint64_t e0, uint64_t ne,
                              uint32_t* __restrict__ x0_out, uint32_t* __restrict__ status) {
  AesCtx c{};
  if constexpr (INST == kInstAes) {
    __shared__ AesShared sh;
    aes_tables_init(sh);
    c = aes_ctx(&sh);
  }
  const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= ne) return;
  const uint64_t target = e0 + k;
  // pop from the top of the stack until a node covers leaf `target`
  int top = nds - 1;
  bool ok = top >= 0;
  if (ok) {
    const DsNode& n = ds[top];
    ok = target < (((uint64_t)n.i + 1) << n.d);
  }
  while (ok && target < ((uint64_t)ds[top].i << ds[top].d)) {
    --top;
    ok = top >= 0;
  }
  uint32_t x[4] = {0, 0, 0, 0};
  if (ok) {
    const DsNode n = ds[top];
    x[0] = n.seed[0]; x[1] = n.seed[1]; x[2] = n.seed[2]; x[3] = n.seed[3];
    const uint64_t off = target - ((uint64_t)n.i << n.d);
    for (int j = (int)n.d - 1; j >= 0; --j) {
      uint32_t y[4];
      prf_node_i<INST>(c, x, (uint32_t)(off >> j) & 1u, y);
      x[0] = y[0]; x[1] = y[1]; x[2] = y[2]; x[3] = y[3];
    }
  } else {
    atomicOr(status, kErrSeed);
  }
  uint4* o = reinterpret_cast<uint4*>(x0_out) + k;
  *o = make_uint4(x[0], x[1], x[2], x[3]);
}

// Entries are processed in tiles of kHashTile by groups of kHashThreads threads; inside a tile
// they are reordered by their number of compressions (a counting sort in shared memory), so
// the lanes of a warp run the same number.  A thread's second entry comes from the other end of
// the order, so that the warps of a group carry like amounts of work.  Per entry, one loop
// drives every SHA-256 compression (the PRF block, the message blocks, and the weight block in
// weighted mode) through a single inlined copy of the compression function.
constexpr int kHashClasses = 32;   // one per lane: the prefix sums are a warp scan
constexpr int kHashPer = kHashTile / kHashThreads;
static_assert(kHashPer == 2, "a thread takes one entry from each end of the order");

// Barrier of one group of kHashThreads threads (the whole block when it is one group).
template <int GROUPS>
__device__ __forceinline__ void group_sync(int g) {
  if constexpr (GROUPS == 1) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(kHashThreads) : "memory");
}

// z_t = SHA-256("POSLO-Z" || verifier_seed || le64(t)): the single padded block.
__device__ __forceinline__ void weight_block(const uint32_t zpre[10], uint64_t zi, uint32_t w[16]) {
  const uint32_t lo = (uint32_t)zi, hi = (uint32_t)(zi >> 32);
#pragma unroll
  for (int q = 0; q < 9; ++q) w[q] = zpre[q];
  w[9] = zpre[9] | (lo & 0xffu);
  w[10] = ((lo >> 8) & 0xffu) << 24 | ((lo >> 16) & 0xffu) << 16 | ((lo >> 24) & 0xffu) << 8 | (hi & 0xffu);
  w[11] = ((hi >> 8) & 0xffu) << 24 | ((hi >> 16) & 0xffu) << 16 | ((hi >> 24) & 0xffu) << 8 | 0x80u;
  w[12] = 0; w[13] = 0; w[14] = 0; w[15] = 47 * 8;
}

// The verifier's weights alone: z_t for entries first .. first + n - 1 (one SHA-256 block
// each), so that the MSM's counting sort need not wait for the message hashing.
__global__ void k_weights(const ZPre zp, uint64_t n, uint64_t first, uint32_t* z_out) {
  uint32_t pre[10];
#pragma unroll
  for (int q = 0; q < 10; ++q) pre[q] = zp.w[q];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    uint32_t w[16], st[8];
    weight_block(pre, first + t, w);
    sha256_init(st);
    sha256_compress(st, w);
    reinterpret_cast<uint4*>(z_out)[t] =
        make_uint4(bswap32(st[0]), bswap32(st[1]), bswap32(st[2]), bswap32(st[3]) & 0x7fffffffu);
  }
}

// ---- message bytes of a tile (SHA-256) ----
// The entries of a tile lie back to back in memory, so the block copies them to shared memory
// with 16-byte loads in order and the lanes pick their words there (read directly, each of a
// warp's loads touches 32 lines), and a last block's tail words come from a column of shared
// memory instead of selects: 2^20 x U[32, 256] bytes 422 -> 375 us, weighted 464 -> 407 us, 16
// bytes 184 -> 170 us.  Tiles of more than kStageMax bytes (and malformed ones) are read
// directly.  The copy keeps the bytes' alignment modulo 16 and reads no 4-byte word without a
// message byte in it (stage.h).
constexpr uint32_t kStageBytes = 40960;              // with the rest below 48 KiB: four blocks per SM
constexpr uint32_t kStageMax = kStageBytes - 16 - 112;   // a last block is read up to 112 bytes past its message
constexpr int kTailRows = 6;                         // x || 0x80 shifted into place (5 words), a zero word

__device__ __forceinline__ void stage_tile(uint32_t* stage, const uint8_t* src, uint32_t total) {
  const uint32_t a0 = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15u);
  const uint8_t* s16 = src - a0;
  const uint32_t hi = stage_granule_hi(a0, total);
  for (uint32_t i = stage_granule_lo(a0) + threadIdx.x; i < hi; i += blockDim.x)
    reinterpret_cast<uint4*>(stage)[i] = __ldg(reinterpret_cast<const uint4*>(s16) + i);
  uint32_t w;
  if (threadIdx.x < 8 && stage_end_word(a0, total, threadIdx.x, w))
    stage[w] = __ldg(reinterpret_cast<const uint32_t*>(s16) + w);
}

// The 16 words of the block at word offset ob of the padded stream m || x || 0x80 || 0..: message
// words below a4 = L / 4 (from shared memory, or directly at most up to word kmax), then the
// lane's column of tail words.
template <bool STAGED>
__device__ __forceinline__ void message_block(uint32_t w[16], const uint32_t* m, int32_t kmax, uint32_t sel,
                                              uint32_t ob, uint32_t a4, const uint32_t* tail) {
  auto ld = [&](uint32_t i) -> uint32_t {
    if (STAGED) return m[i];
    return (int32_t)i <= kmax ? __ldg(m + i) : 0u;
  };
  uint32_t v = ld(ob);
  if (ob + 16 <= a4) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const uint32_t nx = ld(ob + q + 1);
      w[q] = __byte_perm(v, nx, sel);
      v = nx;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const uint32_t nx = ld(ob + q + 1);
      const uint32_t t = tail[min(ob + q - a4, (uint32_t)kTailRows - 1) * kHashThreads];   // (wraps to the zero row below a4)
      w[q] = ob + q < a4 ? __byte_perm(v, nx, sel) : t;
      v = nx;
    }
  }
}

// MINB: resident blocks per SM the kernel is compiled for.  GROUPS: groups per block, each with
// its own tiles and partial; more than one where the block's tables fill most of an SM's shared
// memory (POSLO+), so that the groups share them.
template <int INST, int MINB, int GROUPS>
__global__ void __launch_bounds__(kHashThreads * GROUPS, MINB) k_hash(const HashArgs a) {
  AesWide c{};
  if constexpr (INST == kInstAes) c = aes_wide_init();
  static_assert(INST == kInstAes || GROUPS == 1, "one tile buffer per block");
  __shared__ __align__(16) uint32_t stage[INST == kInstAes ? 4 : kStageBytes / 4];
  __shared__ uint32_t tails[INST == kInstAes ? 1 : kTailRows * kHashThreads];
  acc13 acc_e, acc_s;
  acc_zero(acc_e);
  acc_zero(acc_s);
  uint32_t bad = 0;
  __shared__ uint16_t s_order_[GROUPS][kHashTile];
  __shared__ uint32_t s_cnt_[GROUPS][kHashClasses], s_off_[GROUPS][kHashClasses];
  const int g = GROUPS == 1 ? 0 : (int)(threadIdx.x / kHashThreads);
  const uint32_t tid = threadIdx.x % kHashThreads;
  const uint32_t group = blockIdx.x * a.steps.block_step + g * a.steps.group_step;
  uint16_t* s_order = s_order_[g];
  uint32_t *s_cnt = s_cnt_[g], *s_off = s_off_[g];
  uint32_t* tail = tails + (INST == kInstAes ? 0 : tid);
  if constexpr (INST == kInstSha) tail[(kTailRows - 1) * kHashThreads] = 0;
  const uint64_t ntiles = (a.n + kHashTile - 1) / kHashTile;
  for (uint64_t tile = group; tile < ntiles && group < a.ngroups; tile += a.ngroups) {
    const uint64_t base = tile * kHashTile;
    const uint64_t rem = a.n - base;
    const uint32_t m = rem < (uint64_t)kHashTile ? (uint32_t)rem : (uint32_t)kHashTile;
    if (tid < kHashClasses) s_cnt[tid] = 0;
    group_sync<GROUPS>(g);
    uint32_t cls[kHashPer], pos[kHashPer];
    bool malformed = false;
#pragma unroll
    for (int r = 0; r < kHashPer; ++r) {
      const uint32_t k = tid + r * kHashThreads;
      if (k < m) {
        const uint64_t lo = a.offs[base + k], hi = a.offs[base + k + 1];
        if (hi < lo || lo < a.base_off || hi - lo > 0xffffffffull) {
          atomicOr(a.status, kErrInput);
          malformed = true;
        }
        const uint64_t L = hi >= lo ? hi - lo : 0;
        const uint64_t nblk = INST == kInstAes ? (L + 32) >> 4 : (L + 88) >> 6;
        cls[r] = nblk < (uint64_t)(kHashClasses - 1) ? (uint32_t)nblk : (uint32_t)(kHashClasses - 1);
        pos[r] = atomicAdd(&s_cnt[cls[r]], 1u);
      }
    }
    bool staged = false;
    uint32_t stage_off = 0;   // buffer offset of the tile's first byte, less its offset: see below
    uint64_t b0 = 0;
    if constexpr (INST == kInstSha) {
      const bool any = __syncthreads_or(malformed) != 0;
      b0 = a.offs[base];
      const uint64_t total = a.offs[base + m] - b0;   // non-decreasing offsets unless any
      staged = !any && total <= kStageMax;
      if (staged) {
        const uint8_t* src = a.msgs + (b0 - a.base_off);
        stage_off = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15u);
        stage_tile(stage, src, (uint32_t)total);
      }
    } else {
      group_sync<GROUPS>(g);
    }
    if (tid < kHashClasses) {   // one warp: exclusive prefix sums of the class counts
      const uint32_t own = s_cnt[tid];
      uint32_t incl = own;
#pragma unroll
      for (int o = 1; o < kHashClasses; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)tid >= o) incl += v;
      }
      s_off[tid] = incl - own;
    }
    group_sync<GROUPS>(g);
#pragma unroll
    for (int r = 0; r < kHashPer; ++r) {
      const uint32_t k = tid + r * kHashThreads;
      if (k < m) s_order[s_off[cls[r]] + pos[r]] = (uint16_t)k;
    }
    group_sync<GROUPS>(g);
#pragma unroll 1
    for (int r = 0; r < kHashPer; ++r) {
      if (tid + r * kHashThreads >= m) continue;
      const uint64_t t = base + s_order[r == 0 ? tid : m - 1 - tid];
      uint64_t gi, i, j, seed_idx, zi;
      if (a.n_seg) {
        const uint32_t d = segment_of(a.seg_start, a.n_seg, t);
        gi = a.seg_first[d] + (t - a.seg_start[d]);
        const uint32_t n2 = a.seg_n2[d];
        i = gi / n2;
        j = gi - i * n2;
        seed_idx = a.seg_seed_off[d] + (i - a.seg_e0[d]);
        zi = t;
      } else {
        gi = a.first_index + t;
        if (a.n2_log2 != 0xffffffffu) {
          i = gi >> a.n2_log2;
          j = gi & ((1ull << a.n2_log2) - 1);
        } else {
          i = gi / a.n2;
          j = gi - i * a.n2;
        }
        seed_idx = i - a.e0;
        zi = gi;
      }
      const uint4 xs = __ldg(reinterpret_cast<const uint4*>(a.seeds) + seed_idx);
      const uint64_t o0 = a.offs[t] - a.base_off, o1 = a.offs[t + 1] - a.base_off;
      // malformed offsets (flagged above) hash as empty messages and never read memory
      const uint32_t L = (o1 >= o0 && o1 - o0 <= 0xffffffffull && a.offs[t] >= a.base_off) ? (uint32_t)(o1 - o0) : 0u;
      uint32_t st[8], dig[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      if constexpr (INST == kInstAes) {
        // x_t = MMO-AES-128 PRF, e_t from MDC-2-AES-128 over m || x_t, then z_t by SHA-256
        const uint32_t x0[4] = {xs.x, xs.y, xs.z, xs.w};
        uint32_t x[4];
        prf_entry_aes(c, x0, (uint32_t)j, x);
        mdc2_stream(c, entry_stream(a.msgs + o0, L, x), dig);
        if (a.weighted && !a.z_in) {
          uint32_t w[16];
          weight_block(a.zpre, zi, w);
          sha256_init(st);
          sha256_compress(st, w);
        }
      } else {
        // padded stream of m || x (x is known after the PRF block): the message's aligned words,
        // their realignment, and the message bytes past its last whole word
        const uint8_t* mp = a.msgs + o0;
        const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(mp) & 3u);
        const uint32_t sel = (sh + 3) | ((sh + 2) << 4) | ((sh + 1) << 8) | (sh << 12);
        const uint32_t a4 = L >> 2, odd = L & 3u;
        const int32_t kmax = L > 0 ? (int32_t)((L + sh - 1) >> 2) : -1;   // last word with a message byte
        const uint32_t* mw = staged ? stage + ((stage_off + (uint32_t)(a.offs[t] - b0)) >> 2)
                                    : reinterpret_cast<const uint32_t*>(mp - sh);
        uint32_t part = 0;
        if (odd) {
          uint32_t lo, hi;
          if (staged) {
            lo = mw[a4];
            hi = mw[a4 + 1];
          } else {
            lo = __ldg(mw + a4);
            hi = (int32_t)a4 + 1 <= kmax ? __ldg(mw + a4 + 1) : 0u;
          }
          part = __byte_perm(lo, hi, sel) & (0xffffffffu << (32 - 8 * odd));
        }
        const uint32_t total = L + 16;
        const uint32_t nb = (total + 9 + 63) >> 6;
        const uint32_t iters = 1 + nb + (a.weighted && !a.z_in ? 1u : 0u);
        sha256_init(st);
#pragma unroll 1
        for (uint32_t it = 0; it < iters; ++it) {
          uint32_t w[16];
          if (it == 0) {
            // PRF_0(x_0[i] || le32(j)): x0 || le32(j) || 0x00 || 0x80 ... || bitlen(21 bytes)
            w[0] = xs.x; w[1] = xs.y; w[2] = xs.z; w[3] = xs.w;
            w[4] = bswap32((uint32_t)j);
            w[5] = 0x00800000u;
#pragma unroll
            for (int q = 6; q < 15; ++q) w[q] = 0;
            w[15] = 21 * 8;
          } else if (it <= nb) {
            const uint32_t ob = (it - 1) << 4;
            if (staged) message_block<true>(w, mw, kmax, sel, ob, a4, tail);
            else message_block<false>(w, mw, kmax, sel, ob, a4, tail);
            if (it == nb) {
              w[14] |= total >> 29;
              w[15] |= total << 3;
            }
          } else {
            weight_block(a.zpre, zi, w);
          }
          sha256_compress(st, w);
          if (it == 0) {
            // x = first 16 bytes of the PRF digest, then 0x80, behind the message's last bytes
            const uint32_t sr = 8u * odd;
            tail[0] = __funnelshift_r(st[0], 0u, sr) | part;
            tail[1 * kHashThreads] = __funnelshift_r(st[1], st[0], sr);
            tail[2 * kHashThreads] = __funnelshift_r(st[2], st[1], sr);
            tail[3 * kHashThreads] = __funnelshift_r(st[3], st[2], sr);
            tail[4 * kHashThreads] = __funnelshift_r(0x80000000u, st[3], sr);
            sha256_init(st);
          } else if (it == nb) {
#pragma unroll
            for (int q = 0; q < 8; ++q) dig[q] = bswap32(st[q]);
            sha256_init(st);
          }
        }
      }
      const sc e = sc_reduce256(dig);
      if (a.e_out) {
        uint4* eo = reinterpret_cast<uint4*>(a.e_out + 32 * t);
        eo[0] = make_uint4(e.v[0], e.v[1], e.v[2], e.v[3]);
        eo[1] = make_uint4(e.v[4], e.v[5], e.v[6], e.v[7]);
      }
      uint32_t s[8];
      if (a.s) {
        const uint4* sp = reinterpret_cast<const uint4*>(a.s + 32 * t);
        const uint4 s0 = __ldg(sp), s1 = __ldg(sp + 1);
        s[0] = s0.x; s[1] = s0.y; s[2] = s0.z; s[3] = s0.w; s[4] = s1.x; s[5] = s1.y; s[6] = s1.z; s[7] = s1.w;
        const bool canon = sc_is_canonical(s);
        bad += canon ? 0u : 1u;
        if (a.sbad_out) a.sbad_out[t] = canon ? 0 : 1;
      }
      if (a.weighted) {
        // z_t: the first 16 digest bytes as a little-endian integer, bit 127 cleared
        uint32_t z[4];
        if (a.z_in) {
          const uint4 zz = __ldg(reinterpret_cast<const uint4*>(a.z_in) + t);
          z[0] = zz.x; z[1] = zz.y; z[2] = zz.z; z[3] = zz.w;
        } else {
          z[0] = bswap32(st[0]); z[1] = bswap32(st[1]); z[2] = bswap32(st[2]); z[3] = bswap32(st[3]) & 0x7fffffffu;
        }
        if (a.z_out) reinterpret_cast<uint4*>(a.z_out)[t] = make_uint4(z[0], z[1], z[2], z[3]);
        uint32_t pr[12];
        mul_4x8(pr, z, e.v);
        acc_add<12>(acc_e, pr);
        if (a.s) {
          mul_4x8(pr, z, s);
          acc_add<12>(acc_s, pr);
        }
      } else {
        acc_add<8>(acc_e, e.v);
        if (a.s) acc_add<8>(acc_s, s);
      }
    }
    group_sync<GROUPS>(g);
  }
  // reduction of the group's limb values as 64-bit sums
  __shared__ unsigned long long red_[GROUPS][kHashThreads / 32][kPartialWords];
  unsigned long long (*red)[kPartialWords] = red_[g];
  const int lane = threadIdx.x & 31, warp = tid >> 5;
#pragma unroll
  for (int k = 0; k < kPartialWords; ++k) {
    unsigned long long v = k < 13 ? acc_e.v[k] : (k < 26 ? acc_s.v[k - 13] : bad);
    warp_sum_u64(v);
    if (lane == 0) red[warp][k] = v;
  }
  group_sync<GROUPS>(g);
  if (tid < kPartialWords && group < a.ngroups) {
    unsigned long long v = 0;
    for (int w = 0; w < kHashThreads / 32; ++w) v += red[w][tid];
    a.partial[(uint64_t)group * kPartialWords + tid] = v;
  }
}

// Strict decoding of R_t, its affine form for the MSM and its decode flag, and its addition
// into the thread's unit sum (32 words at acc).
__device__ __forceinline__ void decode_one(const PointArgs& a, uint64_t t, uint32_t* acc, uint32_t& bad) {
  const uint4* rp = reinterpret_cast<const uint4*>(a.R + 32 * t);
  const uint4 r0 = __ldg(rp), r1 = __ldg(rp + 1);
  const uint32_t b[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
  ge P;
  const bool ok = ge_decode(b, P);
  bad += ok ? 0u : 1u;
  if (a.bad_out) a.bad_out[t] = ok ? 0 : 1;
  const fe t2d = fe_mul(P.T, fe_d2());
  if (a.pts_out) {
    uint4* dst = reinterpret_cast<uint4*>(a.pts_out + (size_t)kPtsWords * t);
    dst[0] = make_uint4(P.X.v[0], P.X.v[1], P.X.v[2], P.X.v[3]);
    dst[1] = make_uint4(P.X.v[4], P.X.v[5], P.X.v[6], P.X.v[7]);
    dst[2] = make_uint4(P.Y.v[0], P.Y.v[1], P.Y.v[2], P.Y.v[3]);
    dst[3] = make_uint4(P.Y.v[4], P.Y.v[5], P.Y.v[6], P.Y.v[7]);
    dst[4] = make_uint4(t2d.v[0], t2d.v[1], t2d.v[2], t2d.v[3]);
    dst[5] = make_uint4(t2d.v[4], t2d.v[5], t2d.v[6], t2d.v[7]);
  }
  if (ok && !(a.skip && a.skip[t])) ge_store16(acc, ge_madd(ge_load16(acc), P.X, P.Y, t2d));
}

// Every R_t: blocks take chunks of kPointChunk points from a shared counter, so a block that
// starts late (its SM busy with the hashing beside it) simply takes fewer chunks; then the
// block's unit sum and decode-failure count.
//
// Bound by the IMAD pipe (255 squarings and 28 products a point: 1.38 ms for 2^20 points with
// every wide product at 4 cycles).  What a thread does not need during the squarings stays out
// of its registers: its unit sum in its row of shared memory, the exponent chain's factors in
// local memory.  104 registers instead of 146 let four blocks share an SM instead of three:
// Distill of 2^20 entries 3.56 -> 3.47 ms.  Five blocks (94 registers) took 3.48 ms, six (80,
// with the curve equation's terms spilt) 3.49 ms and 7 us more on a batch of 60.
__global__ void __launch_bounds__(kPointThreads, kPointBlocksPerSm) k_points(const PointArgs a) {
  __shared__ __align__(16) uint32_t sp[kPointThreads][32];
  uint32_t* const acc = sp[threadIdx.x];
  ge_store16(acc, ge_identity());
  uint32_t bad = 0;
  __shared__ uint64_t s_base;
  for (;;) {
    if (threadIdx.x == 0) s_base = (uint64_t)atomicAdd(a.work, 1u) * kPointChunk;
    __syncthreads();
    const uint64_t base = s_base;
    __syncthreads();
    if (base >= a.count) break;
    const uint64_t end = min(base + kPointChunk, a.count);
    for (uint64_t t = base + threadIdx.x; t < end; t += blockDim.x) decode_one(a, t, acc, bad);
  }
  // the block's sum by quads (a few us less at the end of a small launch than one lane per
  // addition), over as many points as the block can hold
  __shared__ uint32_t sbad;
  if (threadIdx.x == 0) sbad = 0;
  __syncthreads();
  if (bad) atomicAdd(&sbad, bad);
  compact::quad_tree(sp, a.count < 1 ? 1 : a.count < kPointThreads ? (int)a.count : kPointThreads);
  if (threadIdx.x < 32) a.partial[(uint64_t)blockIdx.x * kPointPartialWords + threadIdx.x] = sp[0][threadIdx.x];
  if (threadIdx.x == 0) a.partial[(uint64_t)blockIdx.x * kPointPartialWords + 32] = sbad;
}

// Fixed-window tables table[w][d-1] = d 16^w P (w = 0..63, d = 1..8) of n keys, in two
// launches.  k_table_chain: one quad of lanes per key walks P, 16P, ..., 16^63 P with
// quad-cooperative doublings (252 of them, at a quarter of a doubling's dependent
// multiplications each) and writes each 16^w P as table[w][0].  k_table_fill: one quad per
// (key, window) forms d 16^w P for d = 2..8 by quad additions.  Entries are stored in cached
// form.  The key of
// index k is the encoding enc + 8 k, the decoded point pts + kPtsWords * list[k] (affine
// x, y; k itself without a list), or G (use_base).  An encoding that does not decode gives
// the identity's table and sets bad_out[k] (when given) or the kErrKey status bit.
__global__ void __launch_bounds__(128) k_table_chain(const uint32_t* __restrict__ enc,
                                                     const uint32_t* __restrict__ pts,
                                                     const uint32_t* __restrict__ list, uint32_t n,
                                                     uint32_t* __restrict__ tables, uint32_t* const* dst,
                                                     uint32_t* __restrict__ status, int use_base,
                                                     uint8_t* __restrict__ bad_out) {
  const uint32_t quad = ((uint32_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const uint32_t k = quad < n ? quad : n - 1;   // surplus quads repeat the last key, unwritten
  const bool writer = quad < n;
  ge P;
  if (use_base) {
    P = ge_base();
  } else if (pts) {
    fe t2d;
    pts_load(pts + (size_t)kPtsWords * (list ? list[k] : k), P.X, P.Y, t2d);
    P.Z = fe_one();
    P.T = fe_mul(P.X, P.Y);
  } else {
    uint32_t b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) b[i] = enc[8 * (size_t)k + i];
    const bool ok = ge_decode(b, P);
    if (!ok) P = ge_identity();
    if (writer && quad_lane() == 0) {
      if (bad_out) bad_out[k] = ok ? 0 : 1;   // the caller reports which key failed
      else if (!ok) atomicOr(status, kErrKey);
    }
  }
  uint32_t* table = dst ? dst[k] : tables + (size_t)k * kTableWords;
  fe Q = qp_spread(P);
  // every lane runs every quad operation (full-mask shuffles)
#pragma unroll 1
  for (int w = 0; w < kTableWindows; ++w) {
    const fe c = qp_cached(Q);
    if (writer) qp_store(table + (size_t)w * kTableDigits * 32, c);
    if (w + 1 < kTableWindows) {
#pragma unroll 1
      for (int i = 0; i < 4; ++i) Q = qp_dbl(Q);
    }
  }
}

__global__ void __launch_bounds__(128) k_table_fill(uint32_t n, uint32_t* __restrict__ tables, uint32_t* const* dst) {
  const uint64_t total = (uint64_t)n * kTableWindows;
  const uint64_t quad = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const uint64_t q = quad < total ? quad : total - 1;
  const bool writer = quad < total;
  const uint64_t key = q / kTableWindows;
  uint32_t* row = (dst ? dst[key] : tables + key * kTableWords) + (q % kTableWindows) * kTableDigits * 32;
  const fe Pw = qp_load(row);
  fe acc = qp_from_cached(Pw);
#pragma unroll 1
  for (int d = 2; d <= kTableDigits; ++d) {
    acc = qp_add_cached(acc, Pw);
    const fe c = qp_cached(acc);
    if (writer) qp_store(row + (d - 1) * 32, c);
  }
}

// The final check in two halves, so that the expensive one overlaps the MSM:
// k_final_prep (side stream, after hashing and the window table of Y) reduces the scalar
// partials to e and s and evaluates [e]Y + [s]G from the two window tables (128 terms
// summed by a shared-memory tree); k_final_check (after the MSM) only forms
// [8](R - ([e]Y + [s]G)) and tests it for the identity.
constexpr int kPrepThreads = 128;
__global__ void __launch_bounds__(128) k_final_prep(const PrepArgs a) {
  __shared__ unsigned long long sums[kPartialWords];
  __shared__ int8_t dig_e[64], dig_s[64];
  __shared__ __align__(16) uint32_t pts_[kPrepThreads][32];
  __shared__ uint32_t bad_flag;
  const int tid = threadIdx.x;
  if (tid < kPartialWords) sums[tid] = 0;
  __syncthreads();
  constexpr int kLanesPerWord = kPrepThreads / kPartialWords;   // blocks split over lanes per word
  if (tid < kLanesPerWord * kPartialWords) {
    const int w = tid % kPartialWords, lane = tid / kPartialWords;
    unsigned long long v = 0;
    for (uint32_t b = lane; b < a.nhash; b += kLanesPerWord) v += a.hash_partial[(size_t)b * kPartialWords + w];
    atomicAdd(&sums[w], v);
  }
  __syncthreads();
  if (tid == 0) {
    const sc e = limb_sums_to_scalar(sums);
    sc s;
    uint32_t bf = sums[26] != 0 ? 1u : 0u;
    if (a.s_given) {
#pragma unroll
      for (int k = 0; k < 8; ++k)
        s.v[k] = a.s_given[4 * k] | (a.s_given[4 * k + 1] << 8) | (a.s_given[4 * k + 2] << 16) |
                 ((uint32_t)a.s_given[4 * k + 3] << 24);
      if (!sc_is_canonical(s.v)) bf = 1;
    } else {
      s = limb_sums_to_scalar(sums + 13);
    }
    recode4(e.v, dig_e);
    recode4(s.v, dig_s);
    bad_flag = bf;
  }
  __syncthreads();
  const ge term = tid < 64 ? table_pick(a.tableY, tid, dig_e[tid]) : table_pick(a.tableG, tid - 64, dig_s[tid - 64]);
  ge_store(pts_[tid], term);
  static_assert(kPrepThreads == 128 && kWindowThreads == 128, "one table term per thread");
  compact::quad_tree(pts_, 128);
  if (tid < 32) a.prep[tid] = pts_[0][tid];
  if (tid == 0) a.prep[32] = bad_flag;
}

// Per-window weighted check, scalar side.  With z_t = sum_w d_{t,w} 2^(c w) in the MSM's
// signed window digits, window w of the batch equation is
//   sum_t d_{t,w} R_t = [E_w] Y + [S_w] G,  E_w = sum_t d_{t,w} e_t,  S_w = sum_t d_{t,w} s_t (mod q).
// k_window_sums: grid (x, windows), blockIdx.y = w; each thread recodes the weights of its
// entries up to window w and adds |d| x, with x = e_t (s_t) for a positive digit and q - x for
// a negative one, into exact 416-bit accumulators; per block 13 limb sums of E_w and 13 of
// S_w (26 u64 at partial[(w * gridDim.x + blockIdx.x) * 26]).
__global__ void __launch_bounds__(kWindowThreads) k_window_sums(const uint8_t* e, const uint8_t* s, const uint32_t* z,
                                                                const uint64_t* idx, uint64_t n, MsmPlan pl,
                                                                unsigned long long* partial) {
  const int w = blockIdx.y;
  acc13 ae, as;
  acc_zero(ae);
  acc_zero(as);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint64_t t = idx ? idx[i] : i;   // all entries, or the n listed ones
    bool neg;
    const uint32_t d = weight_digit(z, t, w, pl.c, neg);
    if (d) add_window_terms(ae, as, e + 32 * t, s + 32 * t, d, neg);
  }
  __shared__ unsigned long long red[kWindowThreads / 32][26];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 26; ++k) {
    unsigned long long v = k < 13 ? ae.v[k] : as.v[k - 13];
    warp_sum_u64(v);
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < 26) {
    unsigned long long v = 0;
    for (int i = 0; i < kWindowThreads / 32; ++i) v += red[i][threadIdx.x];
    partial[((size_t)w * gridDim.x + blockIdx.x) * 26 + threadIdx.x] = v;
  }
}

// One block per window: E_w and S_w from the partials of k_window_sums (minus those of `less`,
// when given: the sums over a few entries left out), then
// P_w = [E_w] Y + [S_w] G from the two window tables (128 terms, shared-memory tree) into
// Pw[w] (32 words).  Block 0 also writes the malformed-s flag of the hashing partials to *bad.
__global__ void __launch_bounds__(kWindowThreads) k_window_prep(const unsigned long long* partial, uint32_t nblocks,
                                                                const unsigned long long* less, uint32_t nless,
                                                                const unsigned long long* hash_partial, uint32_t nhash,
                                                                const uint32_t* tableY, const uint32_t* tableG,
                                                                uint32_t* Pw, uint32_t* bad) {
  __shared__ unsigned long long sums[2][26];
  __shared__ int8_t dig_e[64], dig_s[64];
  __shared__ __align__(16) uint32_t pts_[kWindowThreads][32];
  const int w = blockIdx.x, tid = threadIdx.x;
  if (tid < 52) sums[tid / 26][tid % 26] = 0;
  __syncthreads();
  // word k of every block's partial, the blocks split over four lanes per word
  for (int h = 0; h < 2; ++h) {
    const unsigned long long* src = h ? less : partial;
    const uint32_t nb = h ? nless : nblocks;
    if (src && tid < 4 * 26) {
      unsigned long long v = 0;
      for (uint32_t b = tid / 26; b < nb; b += 4) v += src[((size_t)w * nb + b) * 26 + tid % 26];
      atomicAdd(&sums[h][tid % 26], v);
    }
  }
  if (w == 0 && hash_partial && tid >= 32 && tid < 64) {
    unsigned long long v = 0;
    for (uint32_t b = tid - 32; b < nhash; b += 32) v += hash_partial[(size_t)b * kPartialWords + 26];
    warp_sum_u64(v);
    if (tid == 32) *bad = v != 0 ? 1u : 0u;
  }
  __syncthreads();
  if (tid < 64 && (tid & 31) == 0) {   // E_w by one warp, S_w by another
    const int o = tid ? 13 : 0;
    sc x = limb_sums_to_scalar(sums[0] + o);
    if (less) x = sc_sub(x, limb_sums_to_scalar(sums[1] + o));
    recode4(x.v, tid ? dig_s : dig_e);
  }
  __syncthreads();
  const ge term = tid < 64 ? table_pick(tableY, tid, dig_e[tid]) : table_pick(tableG, tid - 64, dig_s[tid - 64]);
  ge_store(pts_[tid], term);
  compact::quad_tree(pts_, 128);
  if (tid < 32) Pw[32 * w + tid] = pts_[0][tid];
}

// One warp (quad operations: every lane takes part).
__global__ void k_final_check(const uint32_t* prep, const uint32_t* R, const uint32_t* point_bad,
                              const uint32_t* status, uint8_t* accept) {
  if (blockIdx.x != 0) return;
  const bool eq = compact::quad_equal(R, prep);
  const bool ok = eq && prep[32] == 0 && !(point_bad && *point_bad) && (*status & kErrKey) == 0;
  if (threadIdx.x == 0) accept[0] = ok ? 1 : 0;
}

// Host launchers (kernel templates are launched from the translation unit that defines them).
void launch_epoch_seeds(int inst, unsigned grid, unsigned block, cudaStream_t st, const DsNode* ds, int nds,
                        uint64_t e0, uint64_t ne, uint32_t* x0_out, uint32_t* status) {
  if (inst == kInstAes) k_epoch_seeds<kInstAes><<<grid, block, 0, st>>>(ds, nds, e0, ne, x0_out, status);
  else k_epoch_seeds<kInstSha><<<grid, block, 0, st>>>(ds, nds, e0, ne, x0_out, status);
}

// POSLO+ blocks hold the 128 KiB of tables, one block per SM: four groups (512 threads, all the
// registers) when the hashing has the SMs to itself, two beside the decoding.  With one, two and
// four groups beside it, ms: AVer of 2^20 entries 3.00, 2.64, 2.53 and of 40,000 0.251, 0.231,
// 0.234; Distill 4.34, 3.84, 3.82 and 0.435, 0.420, 0.421; weighted shard records 4.20, 3.65, 3.69.
constexpr int kAesGroupsAlone = 4, kAesGroupsBeside = 2;

unsigned hash_groups(int inst, int sm_count, uint64_t n) {
  return hash_groups_of(n, (uint32_t)sm_count * (inst == kInstAes ? kAesGroupsAlone : kHashBlocksPerSm));
}

cudaError_t hash_kernels_init() {
  const cudaError_t e = cudaFuncSetAttribute(k_hash<kInstAes, 1, kAesGroupsAlone>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAesWideBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_hash<kInstAes, 2, kAesGroupsBeside>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kAesWideBytes);
}

void launch_hash(int inst, unsigned groups, int sm_count, cudaStream_t st, HashArgs a, HashPlace place) {
  const uint32_t per = inst != kInstAes ? 1 : place == kHashAlone ? kAesGroupsAlone : kAesGroupsBeside;
  const uint32_t blocks = hash_blocks(groups, per, place == kHashApart ? 0 : sm_count);
  a.ngroups = groups;
  a.steps = hash_steps(groups, blocks, per);
  if (inst != kInstAes)
    k_hash<kInstSha, kHashBlocksPerSm, 1><<<blocks, kHashThreads, 0, st>>>(a);
  else if (place == kHashAlone)
    k_hash<kInstAes, 1, kAesGroupsAlone><<<blocks, kHashThreads * kAesGroupsAlone, kAesWideBytes, st>>>(a);
  else
    k_hash<kInstAes, 2, kAesGroupsBeside><<<blocks, kHashThreads * kAesGroupsBeside, kAesWideBytes, st>>>(a);
}

void launch_points(unsigned grid, cudaStream_t st, const PointArgs& a) {
  k_points<<<grid, kPointThreads, 0, st>>>(a);
}

}  // namespace poslo
