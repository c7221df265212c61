// Prologue of each proof: transcript start, the squeezes of u (d0 row
// challenges) and v (d2 column challenges), and the eq tables
//   E_u[i] = eq(u, bits(i)),  E_v[j] = eq(v, bits(j))
// of Eq. eq:MLE (Sec. II-B), written only for the real (unpadded) indices.
//
// eq(x, bits(i)) = prod_t (x_t if b_t else 1 - x_t), b_1 the MSB.  Split the d
// variables into a high block (first d - s) and a low block (last s): then
// E[i] = E_hi[i >> s] . E_lo[i mod 2^s], each factor table small enough for
// shared memory, and every output entry costs one Montgomery product.
// E_hi is kept in Montgomery form, E_lo in double-Montgomery form, so the
// product lands in double-Montgomery form (x.R^2), the weight format the
// int16 fold needs.  The kernel also writes 2^15 . sum_i E[i] (Montgomery),
// the correction for the +2^15 offset that the int16 fold applies.
#pragma once
#include "common.cuh"
#include "reduce.cuh"
#include "transcript.cuh"
#include "fr_dev.cuh"
#include "transcript_dev.cuh"

namespace vl {

static constexpr int MAX_VARS = 16;      // log2 of VL_MAX_REDUCE
static constexpr int MAX_HALF = 1 << 8;  // 2^(MAX_VARS / 2)

// Two fp16 values from bytes of w selected by `sel` (0x64bb is 1024 + bb).
__device__ __forceinline__ uint32_t pro_bytes_f16x2(uint32_t w, uint32_t sel) {
  const uint32_t v = __byte_perm(w, 0x64646464u, sel);
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0x64006400u));
  return r;
}

// Entry i of the tensor-core weight table: the 32 bytes of e as fp16 values,
// at row i % 64 of its 4 KB chunk (MN-major core matrices: [i / 8 % 8][byte
// group][i % 8][8 bytes]).
__device__ __forceinline__ void store_w8(uint32_t* w8, int i, const Fr& e) {
  uint4* chunk = reinterpret_cast<uint4*>(w8) + (size_t)(i >> 6) * 256;
  const int kk = i & 63;
#pragma unroll
  for (int g = 0; g < 4; g++) {
    const uint32_t a = e.v[2 * g], b = e.v[2 * g + 1];
    chunk[(kk >> 3) * 32 + g * 8 + (kk & 7)] = make_uint4(pro_bytes_f16x2(a, 0x4140), pro_bytes_f16x2(a, 0x4342),
                                                          pro_bytes_f16x2(b, 0x4140), pro_bytes_f16x2(b, 0x4342));
  }
}

__device__ static Fr build_eq(const Fr* x, int d, int size, int tabs, Fr* out, uint32_t* out_soa, int pitch,
                              uint32_t* w8, Fr* lo, Fr* hi, Fr* red) {
  const int tid = threadIdx.x;
  const int s = (d + 1) >> 1;          // low-block variables
  const int dh = d - s;                // high-block variables
  const int nlo = 1 << s;
  const int nhi = (size + nlo - 1) >> s;
  for (int j = tid; j < nlo; j += blockDim.x) {
    Fr acc = fr_r2();  // 1 in double-Montgomery form
    for (int t = 0; t < s; t++) {
      const Fr& xt = x[dh + t];
      int b = (j >> (s - 1 - t)) & 1;
      acc = mont_mul_ni(acc, b ? xt : fr_sub(fr_r1(), xt));
    }
    lo[j] = acc;
  }
  for (int j = tid; j < nhi; j += blockDim.x) {
    Fr acc = fr_r1();  // 1 in Montgomery form
    for (int t = 0; t < dh; t++) {
      const Fr& xt = x[t];
      int b = (j >> (dh - 1 - t)) & 1;
      acc = mont_mul_ni(acc, b ? xt : fr_sub(fr_r1(), xt));
    }
    hi[j] = acc;
  }
  __syncthreads();
  Fr sum[1] = {fr_zero()};
  for (int i = tid; i < size; i += blockDim.x) {
    Fr e = mont_mul_ni(hi[i >> s], lo[i & (nlo - 1)]);
    if (tabs & TAB_LIMBS) {
      out[i] = e;
#pragma unroll
      for (int l = 0; l < 8; l++) out_soa[l * pitch + i] = e.v[l];
    }
    if (tabs & TAB_BYTES) store_w8(w8, i, e);
    sum[0] = fr_add(sum[0], e);
  }
  if (tabs & TAB_BYTES) {
    const int end = (size + 127) & ~127;  // whole 128-entry stages of the tensor-core fold
    for (int i = size + tid; i < end; i += blockDim.x) store_w8(w8, i, fr_zero());
  }
  block_sum_fr<1>(sum, red);
  // sum = sum_i E_i . R^2; one Montgomery product with the plain integer 2^15
  // gives 2^15 . sum_i E_i . R.
  return mont_mul_ni(sum[0], fr_small(1u << 15));
}

// The challenge halves of a squeeze: thread i of n = 2 count (whole warps from a
// multiple of 32 on; lanes past n may take part) holds half i & 1 of challenge
// i >> 1 as a digest; even threads write the challenges (Montgomery) to x:
// challenge i = (lo + hi . 2^256) mod r in Montgomery form = REDC(lo . R^2) +
// REDC(hi . R^3) by two lanes at once, then one addition.
__device__ __forceinline__ void squeeze_store(const uint32_t (&d)[8], int i, int n, Fr* x) {
  const Fr part = mont_mul_ni(digest_le(d), (i & 1) ? fr_r3() : fr_r2());
  const Fr other = shfl_xor_fr(part, 1);
  if (i < n && !(i & 1)) x[i >> 1] = fr_add(part, other);
}

// Squeeze `count` challenges with `label` from the state Sw (big-endian
// words): thread 2t + h hashes half h of challenge t, thread 2 count the
// closing update.  Writes the challenges (Montgomery) to x and the new state
// to Sn.  Block-wide (one barrier).
__device__ static void squeeze_dev(const uint32_t* Sw, uint32_t label, int count, Fr* x, uint32_t* Sn) {
  const int tid = threadIdx.x;
  if ((tid & ~31) <= 2 * count) {
    uint32_t st[8], d[8];
#pragma unroll
    for (int i = 0; i < 8; i++) st[i] = Sw[i];
    const bool half = tid < 2 * count;
    dev_squeeze_block(st, label, (uint32_t)(half ? tid >> 1 : count), half ? tid & 1 : 2, d);
    if (tid == 2 * count) {
#pragma unroll
      for (int i = 0; i < 8; i++) Sn[i] = d[i];
    }
    squeeze_store(d, tid, 2 * count, x);
  }
  __syncthreads();
}

// Two squeezes in a row, na challenges x with label la, then nb challenges y with
// lb (at most 31 each): the threads of the second, from thread 64 on, each form
// the state between the two for themselves, so the chain is two compressions
// and one product.  Block-wide (at least 128 threads, one barrier).
__device__ static void squeeze2_dev(const uint32_t* Sw, uint32_t la, int na, Fr* x, uint32_t lb, int nb, Fr* y,
                                    uint32_t* Sn) {
  const int tid = threadIdx.x, i = tid & 63;
  const bool second = tid >= 64;
  if (tid < 128 && (i & ~31) <= 2 * (second ? nb : na)) {
    uint32_t st[8], d[8];
#pragma unroll
    for (int q = 0; q < 8; q++) st[q] = Sw[q];
    if (second) {
      dev_squeeze_block(st, la, (uint32_t)na, 2, d);
#pragma unroll
      for (int q = 0; q < 8; q++) st[q] = d[q];
    }
    const int n = second ? nb : na;
    const bool half = i < 2 * n;
    dev_squeeze_block(st, second ? lb : la, (uint32_t)(half ? i >> 1 : n), half ? i & 1 : 2, d);
    if (second && i == 2 * n) {
#pragma unroll
      for (int q = 0; q < 8; q++) Sn[q] = d[q];
    }
    squeeze_store(d, i, 2 * n, second ? y : x);
  }
  __syncthreads();
}

// Transcript start and the squeezes of u, v into shared memory, or, for a
// proof with a given point, the given start state and point; the state after
// them goes to P.scr->state.  Block-wide (at least 128 threads); S0: 24 words;
// msg: START_SCRATCH bytes of scratch.  JOIN, the shorter chain for a block with
// an SM's issue slots to itself: warp 0 runs the rounds of the start's three
// blocks, warps 1 to 3 a schedule each, and both squeezes run at once.  Else
// the fewer instructions: one warp hashes, one squeeze after the other.
static constexpr int START_SCRATCH = 192 + 3 * 68 * 4;
template <bool JOIN>
__device__ static void start_or_given(const DevProof& P, uint32_t* S0, Fr* u, Fr* v, void* msg) {
  uint32_t* S2 = S0 + 16;
  const int tid = threadIdx.x;
  if (P.given) {
    for (int i = tid; i < P.d0 + P.d2; i += blockDim.x) {
      if (i < P.d0) u[i] = P.given->u[i];
      else v[i - P.d0] = P.given->v[i - P.d0];
    }
    if (tid < 32) P.scr->state[tid] = P.given->state[tid];
    __syncthreads();
    return;
  }
  const int warp = tid >> 5;
  uint32_t(*wk)[68] = reinterpret_cast<uint32_t(*)[68]>(static_cast<uint8_t*>(msg) + 192);
  if (warp == 0) {
    // the message of ts_start (a product of a batch: of ts_start_member)
    WarpMsg h(msg);
    if (P.member1 > 0) h.bytes("verilora-gb300/zkbatch/v1/member", 32);
    else h.bytes("verilora-gb300/zkmat/v1", 23);
    h.u64le(P.seed);
    if (P.member1 > 0) {
      h.u32le((uint32_t)P.nmembers);
      h.u32le((uint32_t)(P.member1 - 1));
    }
    h.u32le((uint32_t)P.m);
    h.u32le((uint32_t)P.k);
    h.u32le((uint32_t)P.n);
    h.byte((uint32_t)(P.tp & 1));
    h.byte((uint32_t)(P.tq & 1));
    h.bytes(P.binds, 96);
    if (JOIN) {
      h.pad();  // 141 or 158 bytes: three blocks
      named_sync(10, 128);
      ShaState st = sha_iv_state();
#pragma unroll 1
      for (int b = 0; b < 3; b++) st = sha_rounds_ni(st, h.block(b), wk[b], 1 + 3 * b);
      store_digest(S0, st.h);
    } else {
      uint32_t d[8];
      h.hash(d);
      store_digest(S0, d);
    }
  } else if (JOIN && warp < 4) {
    named_sync(10, 128);
    WarpMsg h(msg);
    sha_sched_ni(h.block(warp - 1), wk[warp - 1], 1 + 3 * (warp - 1));
  }
  __syncthreads();
  if (JOIN) {
    squeeze2_dev(S0, LBL_U, P.d0, u, LBL_V, P.d2, v, S2);
  } else {
    squeeze_dev(S0, LBL_U, P.d0, u, S0 + 8);
    squeeze_dev(S0 + 8, LBL_V, P.d2, v, S2);
  }
  if (tid < 32) P.scr->state[tid] = (uint8_t)(S2[tid >> 2] >> (24 - 8 * (tid & 3)));
}

// Shared memory the prologue needs (PRO_SMEM bytes), laid out below.
static_assert(PRO_SMEM == 128 + 2 * MAX_VARS * 32 + 2 * MAX_VARS * 32 + 2 * MAX_HALF * 32 + 8 * 32, "layout");

// Prologue of one proof by the whole block (any multiple of 32 threads, at
// least 128): transcript start, squeezes of u and v, eq tables, corrections.
static __device__ void prologue_block(const DevProof& P, uint8_t* smem) {
  uint32_t* S0 = reinterpret_cast<uint32_t*>(smem);
  Fr* u = reinterpret_cast<Fr*>(smem + 128 + 2 * MAX_VARS * 32);
  Fr* v = u + MAX_VARS;
  Fr* lo = v + MAX_VARS;
  Fr* hi = lo + MAX_HALF;
  Fr* red = hi + MAX_HALF;
  const int tid = threadIdx.x;

  start_or_given<true>(P, S0, u, v, v + MAX_VARS);

  Fr ca = build_eq(u, P.d0, P.m, P.tabA, P.eqA, P.eqA_soa, P.soa_pitchA, P.w8A, lo, hi, red);
  __syncthreads();
  Fr cb = build_eq(v, P.d2, P.n, P.tabB, P.eqB, P.eqB_soa, P.soa_pitchB, P.w8B, lo, hi, red);
  if (tid == 0) {
    P.scr->corrA = P.dtypeA == VL_I16 ? ca : fr_zero();
    P.scr->corrB = P.dtypeB == VL_I16 ? cb : fr_zero();
    P.scr->status = VL_OK;
  }
  __syncthreads();
}

// Factor tables of the eq tables of two sides x (dx variables) and y (dy),
// block-wide: side q's table is E[i] = hi[i >> s] . lo[i mod 2^s] with s =
// ceil(d / 2), lo over the last s variables (2^s entries), hi over the others
// (ceil(size / 2^s) entries); all in Montgomery form but lo of a side with
// `dbl` set, which is in double-Montgomery form.  Written to fac + 2 q EQ_FAC
// (lo) and EQ_FAC further (hi).  Each block of at most 8 variables is split
// once more into two of at most 4: 8 small tables of at most 16 entries, one
// entry per thread (four products on a thread's chain), then one product per
// factor entry, instead of one chain of up to eight products per entry.
// sub: 128 entries of shared memory.  By the block's first n threads (whole warps;
// barrier 11).
__device__ static void eq_factors(const Fr* x, int dx, int sizex, bool dblx, const Fr* y, int dy, int sizey, bool dbly,
                                  Fr* fac, Fr* sub, int n_threads) {
  const int tid = threadIdx.x;
  for (int e = tid; e < 128; e += n_threads) {
    const int q = e >> 4, j = e & 15;  // q: side, hi block, low half
    const bool second = q & 4;
    const int d = second ? dy : dx, s = (d + 1) >> 1;
    const int nv = (q & 2) ? d - s : s, base = (q & 2) ? 0 : d - s;
    const int nl = nv >> 1, n = (q & 1) ? nl : nv - nl, v0 = base + ((q & 1) ? nv - nl : 0);
    if (j < (1 << n)) {
      const Fr* z = second ? y : x;
      Fr acc = fr_r1();
      for (int t = 0; t < n; t++) {
        const Fr& xt = z[v0 + t];
        const Fr f = ((j >> (n - 1 - t)) & 1) ? xt : fr_sub(fr_r1(), xt);
        acc = t == 0 ? f : mont_mul_ni(acc, f);
      }
      // double-Montgomery: one factor of R more, on the low block's high half
      if ((q & 3) == 0 && (second ? dbly : dblx)) acc = to_mont_ni(acc);
      sub[e] = acc;
    }
  }
  named_sync(11, n_threads);
  const int sx = (dx + 1) >> 1, sy = (dy + 1) >> 1;
  const int lx = 1 << sx, hx = (sizex + lx - 1) >> sx, ly = 1 << sy, hy = (sizey + ly - 1) >> sy;
  for (int e = tid; e < lx + hx + ly + hy; e += n_threads) {
    const bool second = e >= lx + hx;
    const int e2 = second ? e - (lx + hx) : e, nlo = second ? ly : lx;
    const bool hi = e2 >= nlo;
    const int j = hi ? e2 - nlo : e2, d = second ? dy : dx, s = second ? sy : sx;
    const int nl = (hi ? d - s : s) >> 1;
    const Fr* tab = sub + 64 * second + 32 * hi;
    fac[(second ? 2 * EQ_FAC : 0) + (hi ? EQ_FAC : 0) + j] =
        nl ? mont_mul_ni(tab[j >> nl], tab[16 + (j & ((1 << nl) - 1))]) : tab[j];
  }
}

// sum_{i < size} eq(x, bits(i)) (Montgomery), in closed form: i < size
// exactly when, at the first bit (from the top) where i and size differ, i
// has 0 and size has 1; the bits below are free and their eq factors sum to
// 1.  So the sum runs over the 1-bits t of size: prod of the factors of size's
// bits above t, times (1 - x_t).  By one warp: lane t holds variable t, the
// products above it by a scan (five products deep instead of 2 d); every lane
// returns the sum.
__device__ static Fr eq_prefix_sum(const Fr* x, int d, int size) {
  if (size >= (1 << d)) return fr_r1();  // the whole cube: sum 1
  const int lane = threadIdx.x & 31;
  const bool in = lane < d, one = in && ((size >> (d - 1 - lane)) & 1);
  const Fr xt = in ? x[lane] : fr_zero(), om = fr_sub(fr_r1(), xt);
  Fr pre = in ? (one ? xt : om) : fr_r1();
  for (int off = 1; off < d; off <<= 1) {  // inclusive products
    Fr up;
#pragma unroll
    for (int l = 0; l < 8; l++) up.v[l] = __shfl_up_sync(0xffffffffu, pre.v[l], off);
    const Fr p = mont_mul_ni(pre, up);
    if (lane >= off) pre = p;
  }
  Fr above;
#pragma unroll
  for (int l = 0; l < 8; l++) above.v[l] = __shfl_up_sync(0xffffffffu, pre.v[l], 1);
  if (lane == 0) above = fr_r1();
  const Fr term = mont_mul_ni(above, om);
  return warp_sum_fr(one ? term : fr_zero());
}

// Offset correction 2^15 . sum_i E[i] (Montgomery) of one side, by one warp.
__device__ static void prologue_corr(const DevProof& P, const Fr* u, const Fr* v, bool a) {
  const Fr c = to_mont_ni(fr_small(1u << 15));
  // sum . R times 2^15 . R, reduced once: 2^15 . sum (Montgomery)
  const Fr corr = mont_mul_ni(a ? eq_prefix_sum(u, P.d0, P.m) : eq_prefix_sum(v, P.d2, P.n), c);
  if ((threadIdx.x & 31) == 0) {
    const bool i16 = (a ? P.dtypeA : P.dtypeB) == VL_I16;
    (a ? P.scr->corrA : P.scr->corrB) = i16 ? corr : fr_zero();
  }
}

// First launch of the prologue, one proof per block of THREADS (128 or 192):
// transcript start, squeezes of u and v, then the factor tables of both eq tables
// (to P.fac; four warps) and the offset corrections (one warp each; of 192
// threads beside the factors).  A chain: three and two compressions, the factors'
// five products or the corrections' seven.
template <int THREADS>
static __device__ void transcript_block(const DevProof& P, uint8_t* smem) {
  uint32_t* S0 = reinterpret_cast<uint32_t*>(smem);
  Fr* u = reinterpret_cast<Fr*>(smem + 128 + 2 * MAX_VARS * 32);
  Fr* v = u + MAX_VARS;
  const int warp = threadIdx.x >> 5;
  constexpr int CORR = THREADS >= 192 ? 4 : 0;  // first of the two warps of the corrections
  start_or_given<(THREADS >= 192)>(P, S0, u, v, v + MAX_VARS);
  if (warp < 4) {
    eq_factors(u, P.d0, P.m, true, v, P.d2, P.n, true, P.fac, v + MAX_VARS, 128);
    if (threadIdx.x == 0) P.scr->status = VL_OK;
  }
  if (warp == CORR || warp == CORR + 1) prologue_corr(P, u, v, warp == CORR);
}

// Second launch: entries [i0, i1) of one eq table, E[i] = hi[i >> s] . lo[i
// mod 2^s] (double-Montgomery), written in the formats the side's fold
// engines read; tensor-core tables are zero from the last entry to their
// padded end.
static __device__ void eq_chunk(const EqItem& it, const DevProof& P) {
  const bool b = it.side != 0;
  const int d = b ? P.d2 : P.d0, size = b ? P.n : P.m, tabs = b ? P.tabB : P.tabA;
  const int s = (d + 1) >> 1, mask = (1 << s) - 1;
  const Fr* lo = P.fac + (b ? 2 * EQ_FAC : 0);
  const Fr* hi = lo + EQ_FAC;
  Fr* out = b ? P.eqB : P.eqA;
  uint32_t* soa = b ? P.eqB_soa : P.eqA_soa;
  const int pitch = b ? P.soa_pitchB : P.soa_pitchA;
  uint32_t* w8 = b ? P.w8B : P.w8A;
  for (int i = it.i0 + threadIdx.x; i < it.i1; i += blockDim.x) {
    const Fr e = i < size ? mont_mul_ni(hi[i >> s], lo[i & mask]) : fr_zero();
    if ((tabs & TAB_LIMBS) && i < size) {
      out[i] = e;
#pragma unroll
      for (int l = 0; l < 8; l++) soa[l * pitch + i] = e.v[l];
    }
    if (tabs & TAB_BYTES) store_w8(w8, i, e);
  }
}

}  // namespace vl
