// Distill / SeBVer at entry granularity (Fig. 3b semantics, Sec. 4.3): find every entry that
// fails its own check by recursively re-verifying subset aggregates on the device.
//
// The subsets are the nodes of a segment tree over the entries: node (l, k) aggregates
// entries [k 2^l, (k+1) 2^l) as (sum R_t, sum e_t mod q, sum s_t mod q).  A node is checked
// with the paper's aggregate equation [8](R - eY - sG) = O; the descendants of failing nodes
// (one or several levels down) are checked next, down to single entries.  Unit sums can hide a pair of invalid
// entries whose errors cancel, so the host confirms the rest of the batch with the weighted
// check afterwards and falls back to per-entry checks of everything when that fails.
#include "common.cuh"
#include "compact.cuh"

namespace poslo {

__device__ __forceinline__ bool flagged(const uint8_t* a, const uint8_t* b, uint64_t t) {
  return (a && a[t]) || (b && b[t]);
}

__device__ __forceinline__ sc sc_load(const uint8_t* p) {
  const uint4* q = reinterpret_cast<const uint4*>(p);
  const uint4 a = q[0], b = q[1];
  sc r;
  r.v[0] = a.x; r.v[1] = a.y; r.v[2] = a.z; r.v[3] = a.w; r.v[4] = b.x; r.v[5] = b.y; r.v[6] = b.z; r.v[7] = b.w;
  return r;
}

__device__ __forceinline__ void sc_store(uint8_t* p, const sc& r) {
  uint4* q = reinterpret_cast<uint4*>(p);
  q[0] = make_uint4(r.v[0], r.v[1], r.v[2], r.v[3]);
  q[1] = make_uint4(r.v[4], r.v[5], r.v[6], r.v[7]);
}

__device__ __forceinline__ sc sc_zero() {
  sc r;
#pragma unroll
  for (int k = 0; k < 8; ++k) r.v[k] = 0;
  return r;
}

// Leaf t as (point, e, s); flagged or padding leaves are (O, 0, 0).
__device__ __forceinline__ void leaf(const TreeArgs& a, uint64_t t, ge& P, sc& e, sc& s) {
  if (t >= a.n || flagged(a.skip1, a.skip2, t)) {
    P = ge_identity();
    e = sc_zero();
    s = sc_zero();
    return;
  }
  fe t2d;
  pts_load(a.pts + (size_t)kPtsWords * t, P.X, P.Y, t2d);
  P.Z = fe_one();
  P.T = fe_mul(P.X, P.Y);
  e = sc_load(a.e + 32 * t);
  s = sc_load(a.s + 32 * t);
}

// Level 1 of the tree from the leaves.
__global__ void __launch_bounds__(128) k_tree_leaves(const TreeArgs a) {
  const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.M / 2) return;
  ge P0, P1;
  sc e0, e1, s0, s1;
  leaf(a, 2 * k, P0, e0, s0);
  leaf(a, 2 * k + 1, P1, e1, s1);
  ge_store16(a.tree_pts + 32 * k, ge_add(P0, P1));
  sc_store(a.tree_e + 32 * k, sc_add(e0, e1));
  sc_store(a.tree_s + 32 * k, sc_add(s0, s1));
}

// Level l+1 from level l: node k = child 2k + child 2k+1.
__global__ void __launch_bounds__(128) k_tree_level(const TreeArgs a, uint64_t in_off, uint64_t out_off,
                                                    uint64_t count) {
  const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const uint64_t c0 = in_off + 2 * k, c1 = c0 + 1, o = out_off + k;
  ge_store16(a.tree_pts + 32 * o, ge_add(ge_load16(a.tree_pts + 32 * c0), ge_load16(a.tree_pts + 32 * c1)));
  sc_store(a.tree_e + 32 * o, sc_add(sc_load(a.tree_e + 32 * c0), sc_load(a.tree_e + 32 * c1)));
  sc_store(a.tree_s + 32 * o, sc_add(sc_load(a.tree_s + 32 * c0), sc_load(a.tree_s + 32 * c1)));
}

// The checks of one pass: w = 0 .. total - 1, LANES lanes each (check_lanes).  Check w is of
// descendant (w mod 2^j) of failing node fail_in[w >> j], at level tl.  The loop runs the same
// number of times for all lanes of a warp (the checks shuffle across the warp); a group past
// the end repeats a node and records nothing.
template <int LANES>
__device__ __forceinline__ void bisect_pass(const TreeArgs& a, const uint64_t* fail_in, uint64_t total, int j, int tl,
                                            const uint32_t* tY, const uint32_t* tG, uint64_t* fail_out,
                                            unsigned long long* cnt_out, uint8_t* invalid) {
  constexpr int kPerWarp = 32 / LANES;
  const uint64_t mask = (1ull << j) - 1;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t grp = (threadIdx.x & 31) / LANES;
#pragma unroll 1
  for (uint64_t w0 = kPerWarp * warp; w0 < total; w0 += kPerWarp * nwarps) {
    const uint64_t w = w0 + grp;
    bool live = w < total;
    const uint64_t wc = live ? w : total - 1;
    const uint64_t k = (fail_in[wc >> j] << j) | (wc & mask);
    fe minus_P;
    const uint8_t *e, *s;
    if (tl > 0) {
      const uint64_t node = a.M - (a.M >> (tl - 1)) + k;   // levels 1 .. tl-1 hold M/2 + ... + M/2^(tl-1) nodes
      minus_P = qp_minus_extended(a.tree_pts + 32 * node);
      e = a.tree_e + 32 * node;
      s = a.tree_s + 32 * node;
    } else {
      // malformed entries are flagged already; padding leaves hold nothing
      live = live && k < a.n && !flagged(a.skip1, a.skip2, k);
      const uint64_t t = k < a.n ? k : a.n - 1;
      minus_P = qp_minus_affine(a.pts + (size_t)kPtsWords * t);
      e = a.e + 32 * t;
      s = a.s + 32 * t;
    }
    const bool ok = check_lanes<LANES>(e, s, minus_P, tY, tG);
    if (live && !ok && (threadIdx.x & (LANES - 1)) == 0) {
      if (tl > 0) fail_out[atomicAdd(cnt_out, 1ull)] = k;
      else invalid[k] = 1;
    }
  }
}

// One step of the descent, several levels at a time.  The step reads the failing nodes of
// level l (state.fail[s % 3], count state.cnt[s % 3], level state.level[s % 2]) and checks
// their descendants j levels further down, j from bisect_depth: with few failing nodes a step
// jumps many levels, with many it descends one.  Failing descendants go to the next list
// (state.fail[(s+1) % 3]); at level 0 the descendants are entries, checked on their own, and
// failing ones are marked invalid.  Each step also clears the counter the step after it will
// fill, and block 0 publishes the level it reached; a step that starts at level 0 (done)
// returns at once, so the host issues as many steps as there can be without reading anything
// back.  Checking the descendants of a failing node directly, instead of its children first,
// only adds checks of nodes whose ancestors failed: every entry that fails its own check is
// still found, and entries are flagged only by their own check.
//
// A step takes about 40 us for 1,300 checks and 75 for 4,200 (the chains of point additions; as
// many lanes per check as the grid has for their number keep them short).
__global__ void __launch_bounds__(128, POSLO_BISECT_MINB) k_bisect_step(const TreeArgs a, BisectState st, int step,
                                                     uint64_t slots, const uint32_t* tY, const uint32_t* tG,
                                                     uint8_t* invalid) {
  const int l = st.level[step & 1];
  const uint64_t* fail_in = st.fail[step % 3];
  uint64_t* fail_out = st.fail[(step + 1) % 3];
  unsigned long long* cnt_out = reinterpret_cast<unsigned long long*>(st.cnt + (step + 1) % 3);
  if (blockIdx.x == 0 && threadIdx.x == 0) st.cnt[(step + 2) % 3] = 0;
  if (l <= 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) st.level[(step + 1) & 1] = l;
    return;
  }
  const uint64_t F = st.cnt[step % 3];
  const int j = bisect_depth(F, l, slots);
  const int tl = l - j;
  if (blockIdx.x == 0 && threadIdx.x == 0) st.level[(step + 1) & 1] = tl;
  const uint64_t total = F << j, threads = (uint64_t)gridDim.x * blockDim.x;
  if (total == 0) return;
  if (32 * total <= threads) bisect_pass<32>(a, fail_in, total, j, tl, tY, tG, fail_out, cnt_out, invalid);
  else if (16 * total <= threads) bisect_pass<16>(a, fail_in, total, j, tl, tY, tG, fail_out, cnt_out, invalid);
  else bisect_pass<8>(a, fail_in, total, j, tl, tY, tG, fail_out, cnt_out, invalid);
}

// Confirmation of a few flagged entries, point side: F_w = sum of d_{t,w} R_t over the flagged
// entries idx[0 .. cnt) whose point decodes, d_{t,w} the MSM's signed digit of window w
// (blockIdx.y).  One quad per (entry, window): |d| R by double-and-add over c bits (the same
// steps for every quad), negated for a negative digit; per block a partial sum (decode
// partial format).  Latency-bound: c doublings and additions, about 30 us, instead of an MSM over
// the flagged entries whose windows Horner's rule then joins (280 us).
__global__ void __launch_bounds__(128) k_flagged_windows(const uint32_t* pts, const uint32_t* z, const uint8_t* badR,
                                                         const uint64_t* idx, uint64_t cnt, MsmPlan pl,
                                                         uint32_t* partial) {
  const int w = blockIdx.y;
  const uint32_t quad = threadIdx.x >> 2, nq = blockDim.x >> 2;
  fe sum = qp_identity();
  // block-uniform trip count (quad operations need every lane)
  for (uint64_t i0 = (uint64_t)blockIdx.x * nq; i0 < cnt; i0 += (uint64_t)gridDim.x * nq) {
    const uint64_t i = i0 + quad;
    const uint64_t t = idx[i < cnt ? i : cnt - 1];
    bool neg;
    uint32_t d = weight_digit(z, t, w, pl.c, neg);
    if (i >= cnt || (badR && badR[t])) d = 0;
    // +-R_t in cached form
    fe P = qp_minus_affine(pts + (size_t)kPtsWords * t);
    P = fe_select(qp_neg_cached(P), P, neg);
    fe acc = qp_identity();
#pragma unroll 1
    for (int bit = pl.c - 1; bit >= 0; --bit) {
      acc = qp_dbl(acc);
      acc = fe_select(acc, qp_add_cached(acc, P), ((d >> bit) & 1u) != 0);
    }
    sum = qp_add(sum, acc);
  }
  __shared__ __align__(16) uint32_t sp[32][32];
  qp_store(sp[quad], sum);
  compact::quad_tree(sp, 32);
  const size_t o = ((size_t)w * gridDim.x + blockIdx.x) * kPointPartialWords;
  if (threadIdx.x < 32) partial[o + threadIdx.x] = sp[0][threadIdx.x];
  if (threadIdx.x == 0) partial[o + 32] = 0;
}

// Confirmation of a few flagged entries: for every window w
//   [8](W_w - F_w - P_w) = O
// with W_w the whole batch's window sum (left by k_msm_window_check), F_w the flagged entries'
// and P_w = [E'_w] Y + [S'_w] G over the others (k_window_prep).  One warp, a quad per window;
// the windows together imply the check with the full weights.
__global__ void __launch_bounds__(32) k_confirm_windows(const uint32_t* W, const uint32_t* F, const uint32_t* Pw,
                                                        int windows, uint8_t* accept) {
  const int lane = threadIdx.x & 31, quad = lane >> 2;
  bool ok = true;
#pragma unroll 1
  for (int r0 = 0; r0 < windows; r0 += 8) {
    const int w = r0 + quad, wc = w < windows ? w : windows - 1;
    const fe d = qp_add(qp_load(W + 32 * (size_t)wc), qp_neg(qp_load(F + 32 * (size_t)wc)));
    const bool eq = qp_is_torsion(qp_add(d, qp_neg(qp_load(Pw + 32 * (size_t)wc))));
    if (w < windows) ok = ok && eq;
  }
  const bool all = __all_sync(0xffffffffu, ok);
  if (lane == 0) *accept = all ? 1 : 0;
}

// The flagged entries' rows for the MSM of the confirmation: decoded point (kPtsWords words),
// weight z_t (4 words) and "point did not decode" (the MSM leaves those out), at the local
// indices idx[0 .. cnt).
__global__ void k_gather_flagged(const uint32_t* pts, const uint32_t* z, const uint8_t* badR, const uint64_t* idx,
                                 uint64_t cnt, uint32_t* gp, uint32_t* gz, uint8_t* gs) {
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= cnt) return;
  const uint64_t k = idx[t];
  const uint4* src = reinterpret_cast<const uint4*>(pts + (size_t)kPtsWords * k);
  uint4* dst = reinterpret_cast<uint4*>(gp + (size_t)kPtsWords * t);
#pragma unroll
  for (int i = 0; i < kPtsWords / 4; ++i) dst[i] = src[i];
  reinterpret_cast<uint4*>(gz)[t] = reinterpret_cast<const uint4*>(z)[k];
  gs[t] = badR ? badR[k] : 0;
}

// ccd^v's point: the batch's unit sum of its decodable R_t (unit, 32 words) minus the flagged
// entries' decodable R_t (local indices idx[0 .. *nf_dev), the count left in device memory by
// the compaction), encoded to enc_out (32 bytes).  One block: the flagged points are few next
// to the batch.
__global__ void __launch_bounds__(256) k_ccd_points(const uint32_t* pts, const uint8_t* badR, const uint64_t* idx,
                                                    const uint64_t* nf_dev, const uint32_t* unit, uint8_t* enc_out) {
  __shared__ __align__(16) uint32_t sp[256][32];
  ge acc = ge_identity();
  const uint64_t nf = *nf_dev;
  for (uint64_t i = threadIdx.x; i < nf; i += blockDim.x) {
    const uint64_t t = idx[i];
    if (badR && badR[t]) continue;
    fe x, y, t2d;
    pts_load(pts + (size_t)kPtsWords * t, x, y, t2d);
    acc = ge_madd(acc, x, y, t2d);
  }
  ge_store(sp[threadIdx.x], acc);
  // once per call: compact (out-of-line) point operations, the code being fetched cold
  compact::quad_tree(sp, nf < 1 ? 1 : nf < 256 ? (int)nf : 256);
  if (threadIdx.x < 32) {
    const fe v = qp_add(qp_load(unit), qp_neg(qp_load(sp[0])));
    __syncwarp();
    if (threadIdx.x < 4) qp_store(sp[0], v);
    __syncwarp();
    if (threadIdx.x == 0) {
      uint32_t w[8];
      compact::encode(ge_load(sp[0]), w);
      for (int k = 0; k < 8; ++k) {
        enc_out[4 * k] = (uint8_t)w[k]; enc_out[4 * k + 1] = (uint8_t)(w[k] >> 8);
        enc_out[4 * k + 2] = (uint8_t)(w[k] >> 16); enc_out[4 * k + 3] = (uint8_t)(w[k] >> 24);
      }
    }
  }
}

// out = a - b (b = nullptr: out = a), extended points of 32 words.
__global__ void k_point_diff(const uint32_t* a, const uint32_t* b, uint32_t* out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  ge_store(out, b ? ge_sub(ge_load(a), ge_load(b)) : ge_load(a));
}

// Weighted scalar sums sum z_t e_t, sum z_t s_t over the entries not flagged (same partial
// layout as k_hash).
__global__ void __launch_bounds__(kHashThreads) k_weighted_sums(const uint8_t* e, const uint8_t* s, const uint32_t* z,
                                                               const uint8_t* skip1, const uint8_t* skip2, uint64_t n,
                                                               unsigned long long* partial) {
  acc13 acc_e, acc_s;
  acc_zero(acc_e);
  acc_zero(acc_s);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    if (flagged(skip1, skip2, t)) continue;
    const uint4 zz = __ldg(reinterpret_cast<const uint4*>(z) + t);
    const uint32_t zw[4] = {zz.x, zz.y, zz.z, zz.w};
    const sc ev = sc_load(e + 32 * t), sv = sc_load(s + 32 * t);
    uint32_t p[12];
    mul_4x8(p, zw, ev.v);
    acc_add<12>(acc_e, p);
    mul_4x8(p, zw, sv.v);
    acc_add<12>(acc_s, p);
  }
  __shared__ unsigned long long red[kHashThreads / 32][kPartialWords];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kPartialWords; ++k) {
    unsigned long long v = k < 13 ? acc_e.v[k] : (k < 26 ? acc_s.v[k - 13] : 0ull);
    warp_sum_u64(v);
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < kPartialWords) {
    unsigned long long v = 0;
    for (int w = 0; w < kHashThreads / 32; ++w) v += red[w][threadIdx.x];
    partial[(uint64_t)blockIdx.x * kPartialWords + threadIdx.x] = v;
  }
}

// out[t] = a[t] | b[t] | c[t] (NULL arrays count as zero).
__global__ void k_flags_or(const uint8_t* a, const uint8_t* b, const uint8_t* c, uint64_t n, uint8_t* out) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride)
    out[t] = (uint8_t)(((a && a[t]) || (b && b[t]) || (c && c[t])) ? 1 : 0);
}

}  // namespace poslo
