// Point arithmetic for the single-block kernels that run once per call (the combined check of
// shard records, the finishing steps): their instructions are fetched from a cold instruction
// cache on every launch, so inlined copies of the field multiplication at every call site
// (tens of kilobytes of straight-line code) cost more than the arithmetic.  The same formulas
// as ge25519.cuh, built from one out-of-line copy of each field operation.
#pragma once
#include "ge25519.cuh"

namespace poslo {
namespace compact {

static __device__ __noinline__ fe mul(const fe& a, const fe& b) { return fe_mul(a, b); }
static __device__ __noinline__ fe sq(const fe& a) { return fe_sq(a); }
static __device__ __noinline__ fe canon(const fe& a) { return fe_canon(a); }

// Unified addition (add-2008-hwcd-3, a = -1, k = 2d), as ge_add.
static __device__ __noinline__ ge add(const ge& p, const ge& q) {
  const fe A = mul(fe_sub(p.Y, p.X), fe_sub(q.Y, q.X));
  const fe B = mul(fe_add(p.Y, p.X), fe_add(q.Y, q.X));
  const fe C = mul(mul(p.T, fe_d2()), q.T);
  const fe Zp = mul(p.Z, q.Z);
  const fe D = fe_add(Zp, Zp);
  const fe E = fe_sub(B, A), F = fe_sub(D, C), G = fe_add(D, C), H = fe_add(B, A);
  ge r;
  r.X = mul(E, F);
  r.Y = mul(G, H);
  r.Z = mul(F, G);
  r.T = mul(E, H);
  return r;
}

// The compressed encoding (y with the parity of x in bit 255), as ge_encode.
static __device__ __noinline__ void encode(const ge& p, uint32_t b[8]) {
  const fe zi = fe_inv(p.Z);
  const fe x = canon(mul(p.X, zi));
  const fe y = canon(mul(p.Y, zi));
#pragma unroll
  for (int i = 0; i < 8; ++i) b[i] = y.v[i];
  b[7] |= (x.v[0] & 1u) << 31;
}

// The sum of the n points sp[0 .. n) (32 words each, 16-byte aligned shared memory, n >= 1) into
// sp[0] by the block's quads, one addition per pair and level: about 2,000 cycles a level where
// one lane's addition takes 6,000.  Every thread of the block calls it (full-mask shuffles,
// barriers inside; blockDim.x a multiple of 32); the caller has stored the points.
static __device__ __noinline__ void quad_tree(uint32_t (*sp)[32], int n) {
  const int quad = threadIdx.x >> 2, nq = blockDim.x >> 2;
  __syncthreads();
#pragma unroll 1
  while (n > 1) {
    const int half = (n + 1) >> 1, pairs = n - half;   // sp[k] += sp[k + half]
#pragma unroll 1
    for (int k0 = 0; k0 < pairs; k0 += nq) {
      const int k = k0 + quad, c = k < pairs ? k : pairs - 1;   // surplus quads repeat the last pair, unwritten
      const fe sum = qp_add(qp_load(sp[c]), qp_load(sp[c + half]));
      __syncthreads();
      if (k < pairs) qp_store(sp[k], sum);
    }
    __syncthreads();
    n = half;
  }
}

// [8](a - b) = O for two points of 32 words, by the quads of one warp (every lane calls it).
static __device__ __noinline__ bool quad_equal(const uint32_t* a, const uint32_t* b) {
  return qp_is_torsion(qp_add(qp_load(a), qp_neg(qp_load(b))));
}

}  // namespace compact
}  // namespace poslo
