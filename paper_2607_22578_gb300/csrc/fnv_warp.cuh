// FNV-1a-64 of one row by a whole warp, for batches whose time is the latency
// of one row's serial chain.
//
// FNV-1a looks serial, but only the low octet l of the state is: a round is
//   h' = p * (h + (x - l)),   x = l xor b,
// so with every l known the state is a sum of products, and l itself goes by
//   l' = x * 0xb3 mod 256,
// where bit j of l' is bit j of x, xor bits that depend on lower bits of x
// alone (0xb3 is odd).  So for all octets at once, bit j of l is an exclusive
// prefix xor once the lower bits are known: eight prefix xors, each over the
// 32 octets a lane holds (bit i of a word = octet i) and over the lanes by a
// ballot.  Then every lane knows the low octet l_s its 32 octets start from
// and runs the plain rounds from the state l_s; with F their result the state
// after them is F + p^32 (h_s - l_s), and the lanes' parts add up with powers
// of p.

#pragma once

#include "fnv.cuh"

namespace hs {
namespace fnv {

struct Powers {
  uint64_t lane[32];           // p^(32 (31 - i)): rounds after lane i's octets
  uint64_t unpad[256];         // p^(-4 t): undoes t zero tokens
  uint64_t p32, p1024;
};
constexpr uint64_t power(uint64_t base, int n) {
  uint64_t r = 1;
  for (int i = 0; i < n; ++i) r *= base;
  return r;
}
constexpr uint64_t inverse_prime() {
  uint64_t inv = kPrime;                       // x = inv solves x * prime = 1 (mod 8)
  for (int i = 0; i < 5; ++i) inv *= 2 - kPrime * inv;   // Newton: the exact bits double
  return inv;
}
constexpr Powers make_powers() {
  Powers w{};
  w.p32 = power(kPrime, 32);
  w.lane[31] = 1;
  for (int i = 30; i >= 0; --i) w.lane[i] = w.lane[i + 1] * w.p32;
  w.p1024 = w.lane[0] * w.p32;
  const uint64_t i4 = power(inverse_prime(), 4);
  w.unpad[0] = 1;
  for (int t = 1; t < 256; ++t) w.unpad[t] = w.unpad[t - 1] * i4;
  return w;
}
static_assert(make_powers().unpad[1] * power(kPrime, 4) == 1, "inverse of the prime");
static __device__ const Powers kPowers = make_powers();

// 8x8 bit transpose in each of the four octet columns of u[0..7]: bit k of
// octet b of u[j] becomes bit j of octet b of u[k].
__device__ __forceinline__ void transpose_bits(uint32_t (&u)[8]) {
#pragma unroll
  for (int d = 4; d > 0; d >>= 1) {
    const uint32_t m = d == 4 ? 0x0f0f0f0fu : d == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (!(k & d)) {
        const uint32_t t = ((u[k] >> d) ^ u[k + d]) & m;
        u[k + d] ^= t;
        u[k] ^= t << d;
      }
  }
}

__device__ __forceinline__ uint32_t maj(uint32_t a, uint32_t b, uint32_t c) {
  return (a & b) | (c & (a | b));
}

// Low octet of the state before this lane's 32 octets w[0..7] (little-endian
// words), given the state before the warp's 1024.
__device__ __forceinline__ uint32_t start_octet(const uint32_t (&w)[8], uint32_t h_lo,
                                                uint32_t lt_mask) {
  // u[k] octet b = octet 8 b + k of the lane; transposed, u[j] = bit j of each
  uint32_t u[8];
#pragma unroll
  for (int o = 0; o < 2; ++o) {                // even tokens, odd tokens
    const uint32_t a01 = __byte_perm(w[o], w[o + 2], 0x5140), b01 = __byte_perm(w[o + 4], w[o + 6], 0x5140);
    const uint32_t a23 = __byte_perm(w[o], w[o + 2], 0x7362), b23 = __byte_perm(w[o + 4], w[o + 6], 0x7362);
    u[4 * o] = __byte_perm(a01, b01, 0x5410);
    u[4 * o + 1] = __byte_perm(a01, b01, 0x7632);
    u[4 * o + 2] = __byte_perm(a23, b23, 0x5410);
    u[4 * o + 3] = __byte_perm(a23, b23, 0x7632);
  }
  transpose_bits(u);
  uint32_t x[8], start = 0;
  // bit j of every x, given c = the bits of x * 0xb3 above x itself
  auto bit = [&](int j, uint32_t c) {
    const uint32_t d = u[j] ^ c;
    uint32_t pre = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) pre ^= pre << o;
    const unsigned odd = __ballot_sync(0xffffffffu, (pre >> 31) != 0u);
    const uint32_t in = (__popc(odd & lt_mask) ^ (h_lo >> j)) & 1u;
    start |= in << j;
    x[j] = u[j] ^ (pre << 1) ^ (0u - in);
  };
  // x * 0xb3 = x + 2x + 16x + 32x + 128x, column by column with its carries
  bit(0, 0u);
  bit(1, x[0]);
  const uint32_t k1 = x[1] & x[0];
  bit(2, x[1] ^ k1);
  const uint32_t k2 = maj(x[2], x[1], k1);
  bit(3, x[2] ^ k2);
  const uint32_t k3 = maj(x[3], x[2], k2);
  bit(4, x[3] ^ x[0] ^ k3);
  const uint32_t s4 = x[4] ^ x[3] ^ k3, c1 = maj(x[4], x[3], k3), c2 = s4 & x[0];
  const uint32_t t5 = x[0] ^ c1 ^ c2;
  bit(5, x[4] ^ x[1] ^ t5);
  const uint32_t s5 = x[5] ^ x[4] ^ x[1], ca = maj(x[5], x[4], x[1]), cb = maj(x[0], c1, c2);
  const uint32_t cc = s5 & t5, t6 = x[1] ^ ca ^ cb;
  bit(6, x[5] ^ x[2] ^ t6 ^ cc);
  const uint32_t s6 = x[6] ^ x[5] ^ x[2];
  bit(7, x[6] ^ x[3] ^ x[2] ^ x[0] ^ maj(x[6], x[5], x[2]) ^ maj(x[1], ca, cb) ^ maj(s6, t6, cc));
  return start;
}

// Sum of v over the warp, mod 2^64, in every lane.
__device__ __forceinline__ uint64_t warp_sum(uint64_t v) {
  const uint32_t lo = (uint32_t)v;
  const uint32_t a = __reduce_add_sync(0xffffffffu, lo & 0xffffu);
  const uint32_t b = __reduce_add_sync(0xffffffffu, lo >> 16);
  const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 32));
  return ((uint64_t)c << 32) + ((uint64_t)b << 16) + a;
}

// The hash of a row of L tokens from state h, by a whole warp (every lane gets
// it).  VEC: the row is 16-byte aligned and its last piece may be read whole.
template <bool VEC>
__device__ __forceinline__ uint64_t hash_row_warp(const uint32_t* __restrict__ row, int32_t L,
                                                  uint64_t h) {
  constexpr int kBlock = 256;                  // tokens: eight per lane
  const int lane = threadIdx.x & 31;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint64_t weight = kPowers.lane[lane], p32 = kPowers.p32, p1024 = kPowers.p1024;
  uint32_t nxt[8];
  auto load = [&](int64_t t0) {                // this lane's tokens of the block at t0
    const int64_t t = t0 + lane * 8;
#pragma unroll
    for (int q = 0; q < 8; q += 4) {
      if (VEC) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (t + q < L) v = __ldg(reinterpret_cast<const uint4*>(row + t + q));
        nxt[q] = v.x;
        nxt[q + 1] = t + q + 1 < L ? v.y : 0u;
        nxt[q + 2] = t + q + 2 < L ? v.z : 0u;
        nxt[q + 3] = t + q + 3 < L ? v.w : 0u;
      } else {
#pragma unroll
        for (int i = q; i < q + 4; ++i) nxt[i] = t + i < L ? __ldg(row + t + i) : 0u;
      }
    }
  };
  load(0);
  for (int64_t t0 = 0; t0 < L; t0 += kBlock) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = nxt[i];
    if (t0 + kBlock < L) load(t0 + kBlock);
    const uint32_t ls = start_octet(w, (uint32_t)h, lt_mask);
    uint32_t lo = ls, hi = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) hash_word_full(lo, hi, w[i]);
    const uint64_t part = (((uint64_t)hi << 32) | lo) - p32 * ls;
    h = p1024 * h + warp_sum(weight * part);
  }
  const int32_t pad = (kBlock - (L % kBlock)) % kBlock;
  return h * kPowers.unpad[pad];
}

}  // namespace fnv
}  // namespace hs
