// edwards25519 group operations: -x^2 + y^2 = 1 + d x^2 y^2 over F_p, extended coordinates
// (X:Y:Z:T) with x = X/Z, y = Y/Z, xy = T/Z (Hisil, Wong, Carter, Dawson, "Twisted Edwards
// curves revisited", ASIACRYPT 2008).  The paper writes its group multiplicatively
// (alpha^x mod p, products of commitments); here alpha^x is [x]G and a product is a sum.
#pragma once
#include "fe25519.cuh"
#include "sc25519.cuh"

namespace poslo {

struct ge { fe X, Y, Z, T; };

__device__ __forceinline__ ge ge_identity() {
  ge r; r.X = fe_zero(); r.Y = fe_one(); r.Z = fe_one(); r.T = fe_zero(); return r;
}

// Base point G: y = 4/5, x even (RFC 8032 Sec. 5.1).
__device__ __forceinline__ ge ge_base() {
  ge r;
  r.X = fe_const(0x8f25d51au, 0xc9562d60u, 0x9525a7b2u, 0x692cc760u, 0xfdd6dc5cu, 0xc0a4e231u, 0xcd6e53feu, 0x216936d3u);
  r.Y = fe_const(0x66666658u, 0x66666666u, 0x66666666u, 0x66666666u, 0x66666666u, 0x66666666u, 0x66666666u, 0x66666666u);
  r.Z = fe_one();
  r.T = fe_const(0xa5b7dda3u, 0x6dde8ab3u, 0x775152f5u, 0x20f09f80u, 0x64abe37du, 0x66ea4e8eu, 0xd78b7665u, 0x67875f0fu);
  return r;
}

// Unified addition (add-2008-hwcd-3 with a = -1, k = 2d): complete on this curve because d
// is not a square in F_p.  9M.
__device__ __forceinline__ ge ge_add(const ge& p, const ge& q) {
  const fe A = fe_mul(fe_sub(p.Y, p.X), fe_sub(q.Y, q.X));
  const fe B = fe_mul(fe_add(p.Y, p.X), fe_add(q.Y, q.X));
  const fe C = fe_mul(fe_mul(p.T, fe_d2()), q.T);
  const fe Zp = fe_mul(p.Z, q.Z);
  const fe D = fe_add(Zp, Zp);
  const fe E = fe_sub(B, A), F = fe_sub(D, C), G = fe_add(D, C), H = fe_add(B, A);
  ge r;
  r.X = fe_mul(E, F); r.Y = fe_mul(G, H); r.Z = fe_mul(F, G); r.T = fe_mul(E, H);
  return r;
}

// Doubling (dbl-2008-hwcd with a = -1).  4M + 4S; T of the input is not used.
__device__ __forceinline__ ge ge_dbl(const ge& p) {
  const fe A = fe_sq(p.X);
  const fe B = fe_sq(p.Y);
  const fe Z2 = fe_sq(p.Z);
  const fe C = fe_add(Z2, Z2);
  const fe E = fe_sub(fe_sub(fe_sq(fe_add(p.X, p.Y)), A), B);
  const fe G = fe_sub(B, A);          // D + B with D = -A
  const fe F = fe_sub(G, C);
  const fe H = fe_neg(fe_add(A, B));  // D - B
  ge r;
  r.X = fe_mul(E, F); r.Y = fe_mul(G, H); r.Z = fe_mul(F, G); r.T = fe_mul(E, H);
  return r;
}

__device__ __forceinline__ ge ge_neg(const ge& p) {
  ge r = p; r.X = fe_neg(p.X); r.T = fe_neg(p.T); return r;
}

__device__ __forceinline__ ge ge_sub(const ge& p, const ge& q) { return ge_add(p, ge_neg(q)); }

__device__ __forceinline__ ge ge_select(const ge& a, const ge& b, bool pick_b) {
  ge r;
  r.X = fe_select(a.X, b.X, pick_b); r.Y = fe_select(a.Y, b.Y, pick_b);
  r.Z = fe_select(a.Z, b.Z, pick_b); r.T = fe_select(a.T, b.T, pick_b);
  return r;
}

// P = O  <=>  X = 0 and Y = Z.
__device__ __forceinline__ bool ge_is_identity(const ge& p) { return fe_is_zero(p.X) && fe_eq(p.Y, p.Z); }

__device__ __forceinline__ ge ge_mul_cofactor(const ge& p) { return ge_dbl(ge_dbl(ge_dbl(p))); }

// Strict decoding of a 32-byte compressed point (RFC 8032 Sec. 5.1.3): reject y >= p,
// reject when (y^2 - 1)/(d y^2 + 1) has no square root, reject x = 0 with the sign bit set.
// The root of u/v is u v^3 (u v^7)^((p-5)/8), corrected by sqrt(-1) when needed.
__device__ __forceinline__ bool ge_decode(const uint32_t b[8], ge& out) {
  fe y;
#pragma unroll
  for (int i = 0; i < 8; ++i) y.v[i] = b[i];
  const uint32_t sign = b[7] >> 31;
  y.v[7] &= 0x7fffffffu;
  // y < p  <=>  canon(y) == y
  const fe yc = fe_canon(y);
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 8; ++i) ok &= (yc.v[i] == y.v[i]);
  const fe y2 = fe_sq(y);
  const fe u = fe_sub(y2, fe_one());
  const fe v = fe_add(fe_mul(fe_d(), y2), fe_one());
  const fe v3 = fe_mul(fe_sq(v), v);
  const fe v7 = fe_mul(fe_sq(v3), v);
  fe x = fe_mul(fe_mul(u, v3), fe_pow_p58(fe_mul(u, v7)));
  const fe vx2 = fe_mul(v, fe_sq(x));
  const bool root = fe_eq(vx2, u);
  const bool root_neg = fe_eq(vx2, fe_neg(u));
  x = fe_select(x, fe_mul(x, fe_sqrtm1()), !root && root_neg);
  ok &= (root || root_neg);
  x = fe_canon(x);
  bool xzero = true;
#pragma unroll
  for (int i = 0; i < 8; ++i) xzero &= (x.v[i] == 0);
  ok &= !(xzero && sign);
  x = fe_select(x, fe_neg(x), (x.v[0] & 1u) != sign);
  out.X = x;
  out.Y = y;
  out.Z = fe_one();
  out.T = fe_mul(x, y);
  return ok;
}

// Compressed encoding: y with the parity of x in bit 255.
__device__ __forceinline__ void ge_encode(const ge& p, uint32_t b[8]) {
  const fe zi = fe_inv(p.Z);
  const fe x = fe_canon(fe_mul(p.X, zi));
  const fe y = fe_canon(fe_mul(p.Y, zi));
#pragma unroll
  for (int i = 0; i < 8; ++i) b[i] = y.v[i];
  b[7] |= (x.v[0] & 1u) << 31;
}

// Mixed addition with an affine point given as (x, y, t2d = 2d x y): the "precomputed"
// form of the unified addition, 7M (Hisil et al. 2008, Sec. 3.1 with Z2 = 1).
__device__ __forceinline__ ge ge_madd(const ge& p, const fe& x, const fe& y, const fe& t2d) {
  const fe A = fe_mul(fe_sub(p.Y, p.X), fe_sub(y, x));
  const fe B = fe_mul(fe_add(p.Y, p.X), fe_add(y, x));
  const fe C = fe_mul(p.T, t2d);
  const fe D = fe_add(p.Z, p.Z);
  const fe E = fe_sub(B, A), F = fe_sub(D, C), G = fe_add(D, C), H = fe_add(B, A);
  ge r;
  r.X = fe_mul(E, F); r.Y = fe_mul(G, H); r.Z = fe_mul(F, G); r.T = fe_mul(E, H);
  return r;
}

// ge_madd of P or of -P = (-x, y, -t2d): negation swaps y - x with y + x and negates t2d.
__device__ __forceinline__ ge ge_madd_signed(const ge& p, const fe& x, const fe& y, const fe& t2d, bool neg) {
  const fe ym = fe_sub(y, x), yp = fe_add(y, x);
  const fe A = fe_mul(fe_sub(p.Y, p.X), fe_select(ym, yp, neg));
  const fe B = fe_mul(fe_add(p.Y, p.X), fe_select(yp, ym, neg));
  const fe C = fe_mul(p.T, fe_select(t2d, fe_neg(t2d), neg));
  const fe D = fe_add(p.Z, p.Z);
  const fe E = fe_sub(B, A), F = fe_sub(D, C), G = fe_add(D, C), H = fe_add(B, A);
  ge r;
  r.X = fe_mul(E, F); r.Y = fe_mul(G, H); r.Z = fe_mul(F, G); r.T = fe_mul(E, H);
  return r;
}

// P + Q for Q given as (Y-X, Y+X, 2Z, 2dT) ("cached" form, the window tables' entries): 8M.
__device__ __forceinline__ ge ge_add_cached(const ge& p, const fe& ymx, const fe& ypx, const fe& z2, const fe& t2d) {
  const fe A = fe_mul(fe_sub(p.Y, p.X), ymx);
  const fe B = fe_mul(fe_add(p.Y, p.X), ypx);
  const fe C = fe_mul(p.T, t2d);
  const fe D = fe_mul(p.Z, z2);
  const fe E = fe_sub(B, A), F = fe_sub(D, C), G = fe_add(D, C), H = fe_add(B, A);
  ge r;
  r.X = fe_mul(E, F); r.Y = fe_mul(G, H); r.Z = fe_mul(F, G); r.T = fe_mul(E, H);
  return r;
}

// ---- points spread over a quad --------------------------------------------------------
// Four consecutive lanes of a warp (a quad) hold one point: lane q has coordinate q of
// (X, Y, Z, T), one field element.  An addition of a cached point is two rounds of one product
// per lane with three exchanges between them (32 word shuffles, two additions a lane), a
// doubling a squaring and a product.  Where every lane held the whole point and repeated the
// additions, an addition took three rounds, 64 shuffles and nine additions a lane (about 760
// instructions against 450) and four times the registers.  Every lane of the warp must take
// part (full-mask shuffles); each quad works on its own point.
__device__ __forceinline__ int quad_lane() { return threadIdx.x & 3; }

// The element held by lane `src` of the own quad.
__device__ __forceinline__ fe fe_quad(const fe& a, int src) {
  const int lane = (threadIdx.x & 28) | src;
  fe r;
#pragma unroll
  for (int i = 0; i < 8; ++i) r.v[i] = __shfl_sync(0xffffffffu, a.v[i], lane);
  return r;
}

__device__ __forceinline__ fe fe_shfl_xor(const fe& a, int mask) {
  fe r;
#pragma unroll
  for (int i = 0; i < 8; ++i) r.v[i] = __shfl_xor_sync(0xffffffffu, a.v[i], mask);
  return r;
}

__device__ __forceinline__ fe fe_small(uint32_t k) { fe r = fe_zero(); r.v[0] = k; return r; }

__device__ __forceinline__ fe qp_identity() {
  const int q = quad_lane();
  return fe_small(q == 1 || q == 2 ? 1u : 0u);
}

// Coordinate q of a point of 32 words (16-byte aligned), and back.
__device__ __forceinline__ fe qp_load(const uint32_t* p) {
  const uint4* s = reinterpret_cast<const uint4*>(p + 8 * quad_lane());
  const uint4 a = s[0], b = s[1];
  return fe_const(a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w);
}

__device__ __forceinline__ void qp_store(uint32_t* p, const fe& v) {
  uint4* d = reinterpret_cast<uint4*>(p + 8 * quad_lane());
  d[0] = make_uint4(v.v[0], v.v[1], v.v[2], v.v[3]);
  d[1] = make_uint4(v.v[4], v.v[5], v.v[6], v.v[7]);
}

// The own coordinate of a point that every lane of the quad holds whole.
__device__ __forceinline__ fe qp_spread(const ge& p) {
  const int q = quad_lane();
  fe r = fe_select(p.X, p.Y, q == 1);
  r = fe_select(r, p.Z, q == 2);
  return fe_select(r, p.T, q == 3);
}

// (X, Y, Z, T) -> (Y-X, Y+X, Z, T)
__device__ __forceinline__ fe qp_prepare(const fe& v) {
  const int q = quad_lane();
  const fe s = fe_addsub(fe_shfl_xor(v, 1), v, q == 0);
  return fe_select(s, v, q >= 2);
}

// The cached form (Y-X, Y+X, 2Z, 2dT).
__device__ __forceinline__ fe qp_cached(const fe& v) {
  const int q = quad_lane();
  const fe k = fe_select(fe_small(q == 2 ? 2u : 1u), fe_d2(), q == 3);
  return fe_mul(qp_prepare(v), k);
}

// A point from its cached form: (2X, 2Y, 2Z, 2T).
__device__ __forceinline__ fe qp_from_cached(const fe& c) {
  const int q = quad_lane();
  const fe s = fe_select(fe_addsub(fe_shfl_xor(c, 1), c, q == 0), c, q >= 2);
  return fe_mul(s, fe_select(fe_one(), fe_dinv(), q == 3));
}

// Negation: of a point (X, T), and of a cached form (the first two exchanged, the last negated).
__device__ __forceinline__ fe qp_neg(const fe& v) {
  const int q = quad_lane();
  return fe_select(v, fe_neg(v), q == 0 || q == 3);
}

__device__ __forceinline__ fe qp_neg_cached(const fe& c) {
  const int q = quad_lane();
  const fe o = fe_shfl_xor(c, 1);
  return fe_select(fe_select(c, o, q < 2), fe_neg(c), q == 3);
}

// a + b, b in cached form.  Lanes: A B D C, then E H G F, then E F, G H, F G, E H.
__device__ __forceinline__ fe qp_add_cached(const fe& a, const fe& c) {
  const int q = quad_lane();
  const fe m = fe_mul(qp_prepare(a), c);
  const fe v = fe_addsub(fe_shfl_xor(m, 1), m, q == 0 || q == 3);
  const fe u = fe_quad(v, q == 3 ? 1 : q), w = fe_quad(v, q == 3 ? 0 : q == 1 ? 2 : 3);
  return fe_mul(u, w);
}

__device__ __forceinline__ fe qp_add(const fe& a, const fe& b) { return qp_add_cached(a, qp_cached(b)); }

// 2a.  Lanes: A = X^2, B = Y^2, ZZ, S = (X+Y)^2, then G = B-A, -H = A+B, -F = 2ZZ-G, E = S-(A+B); the
// products of these are the doubled point with all four coordinates negated.
__device__ __forceinline__ fe qp_dbl(const fe& a) {
  const int q = quad_lane();
  const fe in = fe_select(a, fe_add(fe_quad(a, 0), fe_quad(a, 1)), q == 3);
  const fe s = fe_sq(in);
  const fe t = fe_addsub(fe_shfl_xor(s, 1), s, q == 0);            // lanes 0, 1: G, A+B
  const fe b = fe_select(s, fe_add(s, s), q == 2);
  const fe v = fe_select(fe_sub(b, fe_quad(t, q == 2 ? 0 : 1)), t, q < 2);
  const fe u = fe_quad(v, q == 0 ? 3 : q), w = fe_quad(v, q == 0 ? 2 : q == 3 ? 1 : 0);
  return fe_mul(u, w);
}

// X = 0 and Y = Z; the same answer in every lane of the quad.
__device__ __forceinline__ bool qp_is_identity(const fe& a) {
  const int q = quad_lane();
  const bool z = fe_is_zero(fe_select(a, fe_sub(a, fe_quad(a, 2)), q == 1));
  const uint32_t votes = __ballot_sync(0xffffffffu, z || q >= 2) >> (threadIdx.x & 28);
  return (votes & 15u) == 15u;
}

// [8]a = O.
__device__ __forceinline__ bool qp_is_torsion(fe a) {
#pragma unroll 1
  for (int i = 0; i < 3; ++i) a = qp_dbl(a);
  return qp_is_identity(a);
}

// Signed 4-bit recoding of a scalar below 2^253: 64 digits in [-8, 8), sum d_i 16^i = k.
__device__ __forceinline__ int sc_digit4(const uint32_t k[8], int w, int& carry) {
  int d = (int)((k[w >> 3] >> ((w & 7) * 4)) & 15u) + carry;
  carry = d >= 8 ? 1 : 0;
  return d - (carry << 4);
}

// Plain left-to-right double-and-add [k]P for a scalar of `bits` bits (used off the hot
// path: key generation, table construction, single-entry checks in tests).
__device__ __forceinline__ ge ge_scalarmult(const uint32_t k[8], const ge& P, int bits) {
  ge acc = ge_identity();
  for (int i = bits - 1; i >= 0; --i) {
    acc = ge_dbl(acc);
    const bool bit = (k[i >> 5] >> (i & 31)) & 1u;
    const ge s = ge_add(acc, P);
    acc = ge_select(acc, s, bit);
  }
  return acc;
}

}  // namespace poslo
