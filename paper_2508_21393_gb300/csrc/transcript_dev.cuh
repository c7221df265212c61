// Device transcript with the message blocks built in registers.
//
// Same transcript as transcript.cuh (start, absorb, counter-mode squeeze),
// specialised for the messages the device hashes: the state S is kept as
// the eight big-endian digest words, which are also the first eight message
// words of the next hash, so no byte buffer is needed.  The byte after S is
// the label; field elements follow as little-endian limbs, one byte out of
// word alignment, so message word 8 + i is (limb[i-1].byte3, limb[i].byte0,
// limb[i].byte1, limb[i].byte2) with the label standing in for byte 3 of
// limb[-1].  Every block is a fixed-index register array (no local memory).
#pragma once
#include <stdint.h>

#include "fr.cuh"
#include "sha256.cuh"
#include "transcript.cuh"

namespace vl {

__device__ __forceinline__ uint32_t bswap32(uint32_t x) { return __byte_perm(x, 0, 0x0123); }
__device__ __forceinline__ uint32_t rotr_dev(uint32_t x, int n) { return __funnelshift_r(x, x, n); }

struct ShaState {
  uint32_t h[8];
};
struct ShaBlock {
  uint32_t w[16];
};

// Word i + 16 of the message schedule from the latest 16 (word i among them).
__device__ __forceinline__ uint32_t sha_next(const ShaBlock& m, int i) {
  const uint32_t x = m.w[(i + 1) & 15], y = m.w[(i + 14) & 15];
  return m.w[i & 15] + (rotr_dev(x, 7) ^ rotr_dev(x, 18) ^ (x >> 3)) + m.w[(i + 9) & 15] +
         (rotr_dev(y, 17) ^ rotr_dev(y, 19) ^ (y >> 10));
}

// The round constants for indices that are not known at compile time.
static __constant__ uint32_t sha_kc[64] = {VL_SHA_K};

// One SHA-256 compression, kept out of line (one copy per kernel module) and as
// loops over 16 rounds: the transcript is a serial chain of compressions, and
// straight-line code for 64 rounds (or a copy at every call site) does not stay in
// the instruction cache.  h + K + W is formed off the e-chain, Ch and Maj use their
// two-operation forms.
static __device__ __noinline__ ShaState sha256_block_ni(ShaState st, ShaBlock m) {
  uint32_t a = st.h[0], b = st.h[1], c = st.h[2], d = st.h[3], e = st.h[4], f = st.h[5], g = st.h[6],
           h = st.h[7];
  auto round = [&](uint32_t kw) {
    const uint32_t hkw = h + kw;
    const uint32_t s1 = rotr_dev(e, 6) ^ rotr_dev(e, 11) ^ rotr_dev(e, 25);
    const uint32_t ch = g ^ (e & (f ^ g));
    const uint32_t t1 = hkw + ch + s1;
    const uint32_t s0 = rotr_dev(a, 2) ^ rotr_dev(a, 13) ^ rotr_dev(a, 22);
    const uint32_t mj = (a & b) | (c & (a | b));
    h = g; g = f; f = e; e = d + t1; d = c; c = b; b = a; a = t1 + (s0 + mj);
  };
#pragma unroll
  for (int i = 0; i < 16; i++) round(sha_k(i) + m.w[i]);
#pragma unroll 1
  for (int q = 16; q < 64; q += 16) {
#pragma unroll
    for (int i = 0; i < 16; i++) {
      m.w[i] = sha_next(m, i);
      round(sha_kc[q + i] + m.w[i]);
    }
  }
  st.h[0] += a; st.h[1] += b; st.h[2] += c; st.h[3] += d;
  st.h[4] += e; st.h[5] += f; st.h[6] += g; st.h[7] += h;
  return st;
}

__device__ __forceinline__ void sha256_iv(uint32_t st[8]) {
  st[0] = 0x6a09e667u; st[1] = 0xbb67ae85u; st[2] = 0x3c6ef372u; st[3] = 0xa54ff53au;
  st[4] = 0x510e527fu; st[5] = 0x9b05688cu; st[6] = 0x1f83d9abu; st[7] = 0x5be0cd19u;
}

// One compression split over two warps: the schedule warp makes the words
// 16..63 with their round constants added (wk, shared memory), announcing each
// 16 of them on named barriers bar, bar + 1, bar + 2 (64 threads: it arrives,
// the other warp waits); the round warp runs the rounds.  A lone warp is bound
// by its issue rate (22 instructions per round, measured 1.65 us per
// compression); without the schedule a round has 14 (1.12 us).
__device__ __forceinline__ void named_sync(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
static __device__ __noinline__ void sha_sched_ni(ShaBlock m, uint32_t* wk, int bar) {
#pragma unroll 1
  for (int q = 16; q < 64; q += 16) {
#pragma unroll
    for (int i = 0; i < 16; i++) {
      m.w[i] = sha_next(m, i);
      if ((i & 3) == 3)
        *reinterpret_cast<uint4*>(wk + q + i - 3) =
            make_uint4(m.w[i - 3] + sha_kc[q + i - 3], m.w[i - 2] + sha_kc[q + i - 2],
                       m.w[i - 1] + sha_kc[q + i - 1], m.w[i] + sha_kc[q + i]);
    }
    named_arrive(bar + (q >> 4) - 1, 64);
  }
}
// The rounds as a loop over 16: its body fits the instruction cache beside what
// the other warps run (unrolled over 64, the first compression after other code
// took 2700 to 3400 cycles against 2050 for the next: 7B step 2.03 -> 2.00 ms, 128
// batched claims 762 -> 742 us).
static __device__ __noinline__ ShaState sha_rounds_ni(ShaState st, ShaBlock m, const uint32_t* wk, int bar) {
  uint32_t a = st.h[0], b = st.h[1], c = st.h[2], d = st.h[3], e = st.h[4], f = st.h[5], g = st.h[6], h = st.h[7];
#pragma unroll
  for (int i = 0; i < 16; i++) m.w[i] += sha_k(i);
#pragma unroll 1
  for (int q = 0; q < 4; q++) {
    if (q > 0) {
      named_sync(bar + q - 1, 64);
#pragma unroll
      for (int p = 0; p < 4; p++) {
        const uint4 v = *reinterpret_cast<const uint4*>(wk + 16 * q + 4 * p);
        m.w[4 * p] = v.x, m.w[4 * p + 1] = v.y, m.w[4 * p + 2] = v.z, m.w[4 * p + 3] = v.w;
      }
    }
#pragma unroll
    for (int i = 0; i < 16; i++) {
      const uint32_t hkw = h + m.w[i];
      const uint32_t s1 = rotr_dev(e, 6) ^ rotr_dev(e, 11) ^ rotr_dev(e, 25);
      const uint32_t ch = g ^ (e & (f ^ g));
      const uint32_t t1 = hkw + ch + s1;
      const uint32_t s0 = rotr_dev(a, 2) ^ rotr_dev(a, 13) ^ rotr_dev(a, 22);
      const uint32_t mj = (a & b) | (c & (a | b));
      h = g; g = f; f = e; e = d + t1; d = c; c = b; b = a; a = t1 + (s0 + mj);
    }
  }
  st.h[0] += a; st.h[1] += b; st.h[2] += c; st.h[3] += d;
  st.h[4] += e; st.h[5] += f; st.h[6] += g; st.h[7] += h;
  return st;
}
__device__ __forceinline__ ShaState sha_iv_state() {
  ShaState s;
  sha256_iv(s.h);
  return s;
}
// 16 message words from 16-byte aligned memory.
__device__ __forceinline__ ShaBlock sha_load(const uint32_t* m) {
  ShaBlock b;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const uint4 v = reinterpret_cast<const uint4*>(m)[q];
    b.w[4 * q] = v.x, b.w[4 * q + 1] = v.y, b.w[4 * q + 2] = v.z, b.w[4 * q + 3] = v.w;
  }
  return b;
}

// One compression of a 16-word block into the chaining value st.
__device__ __forceinline__ void sha256_block(uint32_t st[8], const uint32_t blk[16]) {
  ShaState s;
  ShaBlock m;
#pragma unroll
  for (int i = 0; i < 8; i++) s.h[i] = st[i];
#pragma unroll
  for (int i = 0; i < 16; i++) m.w[i] = blk[i];
  s = sha256_block_ni(s, m);
#pragma unroll
  for (int i = 0; i < 8; i++) st[i] = s.h[i];
}


// S <- SHA256(S || label || x_0 || ... || x_{N-1}) for N canonical field elements.
// Message length 33 + 32N bytes; each 16-word block is built just before
// its compression (all indices are compile-time constants).
template <int N>
__device__ __forceinline__ void dev_absorb_fr(uint32_t S[8], uint32_t label, const Fr (&x)[N]) {
  constexpr int LEN = 33 + 32 * N;
  constexpr int NB = (LEN + 9 + 63) / 64;
  uint32_t st[8];
  sha256_iv(st);
#pragma unroll
  for (int b = 0; b < NB; b++) {
    uint32_t m[16];
#pragma unroll
    for (int i = 0; i < 16; i++) {
      const int gi = 16 * b + i;  // word index in the padded message
      uint32_t w = 0;
      if (gi < 8) {
        w = S[gi];
      } else if (gi < 8 + 8 * N) {
        const int q = gi - 8;
        const uint32_t cur = x[q / 8].v[q % 8];
        // the label sits where byte 3 of a previous limb would
        const uint32_t prev = q == 0 ? (label << 24) : x[(q - 1) / 8].v[(q - 1) % 8];
        w = __byte_perm(cur, prev, 0x7012);
      } else if (gi == 8 + 8 * N) {
        w = (x[N - 1].v[7] & 0xff000000u) | 0x00800000u;  // last data byte, then the 0x80 pad byte
      }
      if (gi == 16 * NB - 1) w = (uint32_t)LEN * 8u;
      m[i] = w;
    }
    sha256_block(st, m);
  }
#pragma unroll
  for (int i = 0; i < 8; i++) S[i] = st[i];
}

// One-block messages of a squeeze, from the state S before the squeeze:
//   kind 0/1: challenge t, half `kind`:  S || label || t u32le || kind   (38 bytes)
//   kind 2  : closing state update:      S || label || count u32le       (37 bytes)
// Returns the digest in out[8] (big-endian words).
__device__ __forceinline__ void squeeze_words(const uint32_t S[8], uint32_t label, uint32_t t_or_count, int kind,
                                              uint32_t (&m)[16]) {
#pragma unroll
  for (int i = 0; i < 8; i++) m[i] = S[i];
  const uint32_t v = t_or_count;
  // bytes 32..: label, v.b0, v.b1, v.b2 | v.b3, then (kind byte, 0x80) or 0x80
  m[8] = (label << 24) | ((v & 0xffu) << 16) | (((v >> 8) & 0xffu) << 8) | ((v >> 16) & 0xffu);
  if (kind == 2) {
    m[9] = ((v >> 24) << 24) | 0x00800000u;
    m[15] = 37u * 8u;
  } else {
    m[9] = ((v >> 24) << 24) | ((uint32_t)kind << 16) | 0x00008000u;
    m[15] = 38u * 8u;
  }
#pragma unroll
  for (int i = 10; i < 15; i++) m[i] = 0;
}
__device__ __forceinline__ void dev_squeeze_block(const uint32_t S[8], uint32_t label, uint32_t t_or_count, int kind,
                                                  uint32_t out[8]) {
  uint32_t m[16];
  squeeze_words(S, label, t_or_count, kind, m);
  sha256_iv(out);
  sha256_block(out, m);
}

// A 32-byte digest (big-endian words) read as a little-endian 256-bit integer.
__device__ __forceinline__ Fr digest_le(const uint32_t d[8]) {
  Fr x;
#pragma unroll
  for (int i = 0; i < 8; i++) x.v[i] = __byte_perm(d[i], 0, 0x0123);
  return x;
}

// SHA256(tag byte || Y_0 || ... || Y_{N-1}) for big-endian words Y, one thread.
template <int N>
__device__ __forceinline__ void dev_hash_tagged(uint32_t tag, const uint32_t (&Y)[N], uint32_t (&out)[8]) {
  constexpr int LEN = 1 + 4 * N;
  constexpr int NB = (LEN + 9 + 63) / 64;
  sha256_iv(out);
#pragma unroll
  for (int b = 0; b < NB; b++) {
    uint32_t m[16];
#pragma unroll
    for (int i = 0; i < 16; i++) {
      const int gi = 16 * b + i;
      uint32_t w = 0;
      if (gi < N) w = __funnelshift_r(Y[gi < N ? gi : 0], gi == 0 ? tag : Y[gi > 0 && gi < N ? gi - 1 : 0], 8);
      else if (gi == N) w = (Y[N - 1] << 24) | 0x00800000u;
      if (gi == 16 * NB - 1) w = (uint32_t)LEN * 8u;
      m[i] = w;
    }
    sha256_block(out, m);
  }
}

// S <- SHA256(S || label || Y_0 || ... || Y_{N-1}) for big-endian words Y, one thread.
template <int N>
__device__ __forceinline__ void dev_absorb_words(uint32_t (&S)[8], uint32_t label, const uint32_t (&Y)[N]) {
  constexpr int LEN = 33 + 4 * N;
  constexpr int NB = (LEN + 9 + 63) / 64;
  uint32_t st[8];
  sha256_iv(st);
#pragma unroll
  for (int b = 0; b < NB; b++) {
    uint32_t m[16];
#pragma unroll
    for (int i = 0; i < 16; i++) {
      const int gi = 16 * b + i, q = gi - 8;
      uint32_t w = 0;
      if (gi < 8) w = S[gi < 8 ? gi : 0];
      else if (q < N) w = __funnelshift_r(Y[q >= 0 && q < N ? q : 0], q == 0 ? label : Y[q > 0 && q < N ? q - 1 : 0], 8);
      else if (q == N) w = (Y[N - 1] << 24) | 0x00800000u;
      if (gi == 16 * NB - 1) w = (uint32_t)LEN * 8u;
      m[i] = w;
    }
    sha256_block(st, m);
  }
#pragma unroll
  for (int i = 0; i < 8; i++) S[i] = st[i];
}


// A message whose layout is known only at run time (transcript starts, long
// absorbs): the lanes of one warp write its bytes to shared memory, then
// every lane runs the compressions on the same words (one warp instruction
// either way), so the digest ends in every lane's registers.  One thread feeding
// a byte-wise hash with its buffer in local memory took several times as long:
// with both sides' eq factors formed from small tables, a lone 64 x 128 x 64
// proof went from 278 to 256 us, the 256 update proofs of a 7B step from 382 to
// 303 us and four chained 7B projections from 1014 to 787 us.
// `buf`: 16-byte aligned shared memory of at least 64 ceil((bytes + 9) / 64).
struct WarpMsg {
  uint8_t* buf;
  int len;
  __device__ explicit WarpMsg(void* shared) : buf(static_cast<uint8_t*>(shared)), len(0) {}
  __device__ void bytes(const void* src, int n) {
    for (int i = threadIdx.x & 31; i < n; i += 32) buf[len + i] = static_cast<const uint8_t*>(src)[i];
    len += n;
  }
  __device__ void byte(uint32_t x) {
    if ((threadIdx.x & 31) == 0) buf[len] = (uint8_t)x;
    len += 1;
  }
  __device__ void u32le(uint32_t x) {
    const int lane = threadIdx.x & 31;
    if (lane < 4) buf[len + lane] = (uint8_t)(x >> (8 * lane));
    len += 4;
  }
  __device__ void u64le(uint64_t x) {
    u32le((uint32_t)x);
    u32le((uint32_t)(x >> 32));
  }
  // a transcript state (eight big-endian words, in memory)
  __device__ void state(const uint32_t* S) {
    const int lane = threadIdx.x & 31;
    buf[len + lane] = (uint8_t)(S[lane >> 2] >> (24 - 8 * (lane & 3)));
    len += 32;
  }
  // Padding and length; the number of bytes then (whole blocks).
  __device__ int pad() {
    const int end = (len + 9 + 63) / 64 * 64;
    for (int i = len + (int)(threadIdx.x & 31); i < end; i += 32)
      buf[i] = i == len ? 0x80 : i >= end - 4 ? (uint8_t)((uint32_t)(len * 8) >> (8 * (end - 1 - i))) : 0;
    __syncwarp();
    return end;
  }
  // Block b of the padded message.
  __device__ ShaBlock block(int b) const {
    ShaBlock m;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint4 v = reinterpret_cast<const uint4*>(buf + 64 * b)[q];
      m.w[4 * q] = bswap32(v.x), m.w[4 * q + 1] = bswap32(v.y), m.w[4 * q + 2] = bswap32(v.z), m.w[4 * q + 3] = bswap32(v.w);
    }
    return m;
  }
  // The digest (big-endian words); the buffer may be reused afterwards.
  __device__ void hash(uint32_t (&out)[8]) {
    const int n = pad() / 64;
    sha256_iv(out);
    for (int b = 0; b < n; b++) {
      const ShaBlock m = block(b);
      sha256_block(out, m.w);
    }
    __syncwarp();
  }
};
// Lane 0 stores a digest that every lane holds.
__device__ __forceinline__ void store_digest(uint32_t* dst, const uint32_t (&d)[8]) {
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int i = 0; i < 8; i++) dst[i] = d[i];
  }
}
// The same as 32 bytes (16-byte aligned).
__device__ __forceinline__ void store_digest_bytes(uint8_t* dst, const uint32_t (&d)[8]) {
#pragma unroll
  for (int i = 0; i < 8; i++) reinterpret_cast<uint32_t*>(dst)[i] = bswap32(d[i]);
}

}  // namespace vl
