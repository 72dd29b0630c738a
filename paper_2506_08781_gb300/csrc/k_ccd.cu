// POSLO-C distillation and selective batch verification (Fig. 3b): per-epoch sums of e,
// grouped sums of scalars and points (ccd^v, the umbrellas ccd^u, SeBVer's V and U sums).  The
// independent cofactored checks [8](R_k - e_k Y - s_k G) = O (the per-epoch C.AVer of Distill
// and the checks of SeBVer) are the entry checks of k_check.cu.
#include "common.cuh"
#include "compact.cuh"

namespace poslo {

// out[g] = sum of the 32-byte scalars x[g G .. (g+1) G) not flagged in skip, mod q.
// One block per group; each thread keeps 64-bit limb sums, reduced once per group.
__global__ void __launch_bounds__(kCcdThreads) k_scalar_group_sums(const uint8_t* x, uint64_t G, uint64_t n,
                                                                   const uint8_t* skip, uint32_t* out) {
  const uint64_t g = blockIdx.x;
  acc13 a;
  acc_zero(a);
  const uint64_t lo = g * G, hi = min(lo + G, n);
  for (uint64_t t = lo + threadIdx.x; t < hi; t += blockDim.x) {
    if (skip && skip[t]) continue;
    uint32_t v[8];
    const uint4* p = reinterpret_cast<const uint4*>(x + 32 * t);
    const uint4 v0 = p[0], v1 = p[1];
    v[0] = v0.x; v[1] = v0.y; v[2] = v0.z; v[3] = v0.w; v[4] = v1.x; v[5] = v1.y; v[6] = v1.z; v[7] = v1.w;
    acc_add<8>(a, v);
  }
  __shared__ unsigned long long red[kCcdThreads / 32][13];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < 13; ++k) {
    unsigned long long v = a.v[k];
    warp_sum_u64(v);
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long sums[13];
    for (int k = 0; k < 13; ++k) {
      unsigned long long v = 0;
      for (int w = 0; w < kCcdThreads / 32; ++w) v += red[w][k];
      sums[k] = v;
    }
    const sc r = limb_sums_to_scalar(sums);
    for (int k = 0; k < 8; ++k) out[8 * g + k] = r.v[k];
  }
}

// enc[g] = encoding of the sum of the decoded points pts[g G .. (g+1) G) that are neither
// flagged in skip nor undecodable (bad), and (given partial) the sum itself in the decoding's
// partial format (kPointPartialWords, bad count 0), so that the sum over all groups needs no second pass over
// the points.  One block of T threads per group: latency-bound, G / T additions of a lane, a
// tree by quads and one inversion (64 groups of 64 points: 74 -> 35 us; all 4,096 points in one
// block before: 177 us).
template <int T>
__global__ void __launch_bounds__(T) k_point_group_sums(const uint32_t* pts, const uint8_t* bad, uint64_t G,
                                                        uint64_t n, const uint8_t* skip, uint8_t* enc,
                                                        uint32_t* partial) {
  const uint64_t g = blockIdx.x;
  ge acc = ge_identity();
  const uint64_t lo = g * G, hi = min(lo + G, n);
  for (uint64_t t = lo + threadIdx.x; t < hi; t += T) {
    if ((skip && skip[t]) || (bad && bad[t])) continue;
    fe x, y, t2d;
    pts_load(pts + (size_t)kPtsWords * t, x, y, t2d);
    acc = ge_madd(acc, x, y, t2d);
  }
  __shared__ __align__(16) uint32_t sp[T][32];
  ge_store(sp[threadIdx.x], acc);
  compact::quad_tree(sp, G < T ? (int)G : T);
  if (partial && threadIdx.x < 32) partial[kPointPartialWords * g + threadIdx.x] = sp[0][threadIdx.x];
  if (threadIdx.x == 0) {
    if (partial) partial[kPointPartialWords * g + 32] = 0;
    uint32_t b[8];
    compact::encode(ge_load(sp[0]), b);
    for (int k = 0; k < 8; ++k) reinterpret_cast<uint32_t*>(enc + 32 * g)[k] = b[k];
  }
}

void launch_point_group_sums(unsigned groups, cudaStream_t st, const uint32_t* pts, const uint8_t* bad, uint64_t G,
                             uint64_t n, const uint8_t* skip, uint8_t* enc, uint32_t* partial) {
  if (G > 128) k_point_group_sums<256><<<groups, 256, 0, st>>>(pts, bad, G, n, skip, enc, partial);
  else k_point_group_sums<128><<<groups, 128, 0, st>>>(pts, bad, G, n, skip, enc, partial);
}

// bad[k] = 1 when s_k is not canonical (the checks' other malformed input).
__global__ void k_noncanonical(const uint8_t* s, uint64_t n, uint8_t* bad) {
  const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const uint4* sp = reinterpret_cast<const uint4*>(s + 32 * k);
  const uint4 s0 = sp[0], s1 = sp[1];
  const uint32_t v[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
  bad[k] = sc_is_canonical(v) ? 0 : 1;
}

// dst[k] = src[idx[k]] for 32-byte records.
__global__ void k_gather32(const uint8_t* src, const uint64_t* idx, uint64_t n, uint8_t* dst) {
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * n) return;
  const uint64_t k = t >> 1, half = t & 1;
  reinterpret_cast<uint4*>(dst + 32 * k)[half] = reinterpret_cast<const uint4*>(src + 32 * idx[k])[half];
}

// ok[k] = 1 - flag[k]: the bits b_i from the invalid flags.
__global__ void k_flip(const uint8_t* flag, uint64_t n, uint8_t* ok) {
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) ok[t] = flag[t] ? 0 : 1;
}

}  // namespace poslo
