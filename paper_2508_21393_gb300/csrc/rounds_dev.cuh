// Claim and sumcheck rounds of each proof (Sec. II-B; Eq. eq:zk-mle-matmul).
//
// One CTA per proof, or a cluster of them.  The fold accumulators become the vectors
// f_A[w] = A~(u, w), f_B[w] = B~(w, v) over the padded cube w < 2^d1 (zeros
// for w >= k).  Round i (h = 2^(d1 - i)) has the degree-2 round polynomial
// g(X) = sum_j (a0 + X (a1 - a0)) (b0 + X (b1 - b0)) with a0 = f_A[j],
// a1 = f_A[j + h] (likewise b); its values at 0, 1, 2 are the message, g(0)
// and g(2) are absorbed, r_i squeezed and both vectors folded,
// f[j] <- f[j] + r_i (f[j + h] - f[j]) (variables bound most-significant
// first).  Finally a_r = f_A[0], b_r = f_B[0] are absorbed and the proof is
// written in canonical form.
//
// Work per pair: only g(0) = sum a0 b0 and the leading coefficient
// G = sum (a1 - a0)(b1 - b0) are summed; g(1) is the running claim minus g(0)
// (the claim of round 1 is formed from its g(1), summed too), g(2) =
// 2 g(1) - g(0) + 2 G, and the next claim is g(r) = g(0) + r (g(1) - g(0) - G
// + r G).  A thread sums its products unreduced (wide_mac) and reduces once.
// So a pair costs four fold products and two half products, against seven
// products for the three values evaluated one by one.
//
// Schedule (one proof's rounds are a serial chain of hashes):
//  * pass 0 reads (or reduces) f and evaluates round 1; each later pass folds
//    with r_i and evaluates round i + 1 in the same loop;
//  * short rounds spread a pair over four lanes of a warp: one fold each, then
//    one term on two of them (two products on the chain instead of six);
//    vectors of at most RND_VEC entries live in shared memory, and the last
//    rounds run on warp 0 alone, whose last lane forms the next claim;
//  * blocks with warps to spare have more to gain there: the next message is ready but for the challenge:
//    g(0) and G of round i + 1 are quadratics in r_i, as are the claim and g(2), and
//    other warps sum their coefficients from the unfolded vectors while warps 0
//    to 2 hash.  From the challenge to the next message are two products then,
//    and the fold with r_i runs beside the next hash (look_terms).  So r_i is read
//    while r_(i+1) is made, by warps that meet the hash's warps only at the block
//    barrier that ends each transcript step: odd and even rounds have a slot each,
//    and between a slot's last read and its next write lies the other slot's barrier;
//  * the transcript runs on warps 0 to 2: the rounds of each SHA-256
//    compression on warp 0, its message schedule on warp 1 (of an absorb's
//    second block: on warp 2); the two halves of the challenge and the
//    closing state update are three lanes of one compression.
#pragma once
#include "common.cuh"
#include "reduce.cuh"
#include "fr_dev.cuh"
#include "transcript_dev.cuh"

namespace vl {

static constexpr int RND_VEC = 256;      // vectors of at most this many entries are kept in shared memory
static constexpr int RND_MAX_WARPS = 16;
static constexpr int RND_MAX_CTAS = 8;   // CTAs of a cluster

// Shared memory of the rounds.
struct RndShared {
  alignas(16) uint32_t msg[32];    // an absorb's message: two blocks
  alignas(16) uint32_t wk[3][68];  // schedule words: of an absorb's two blocks, of a squeeze's three lanes
  alignas(16) uint32_t S[8];       // transcript state
  alignas(16) uint32_t sq[8];      // state before a squeeze
  Fr g[4];                         // g(0), g(1), g(2), G of the round (canonical)
  Fr claim;                        // the running claim (canonical)
  Fr r[2];                         // challenge r_i (Montgomery) of round i (1-based) at i mod 2
  alignas(16) unsigned long long red[3 * 8 * RND_MAX_WARPS];
  Fr fa[RND_VEC], fb[RND_VEC];
  // look-ahead and clusters only:
  Fr part[RND_MAX_CTAS][4];        // each CTA's g(0), G, g(1), in the first CTA
  Fr look[2][4][3];                // coefficients in r of the next g(0), G, claim, g(2) (canonical), two rounds
  Fr lsum[RND_MAX_WARPS][6];       // look_terms: the warps' sums
};
static_assert(offsetof(RndShared, part) <= RND_SMEM && sizeof(RndShared) <= RND_SMEM_LOOK, "shared memory of the rounds");

__device__ __forceinline__ Fr load_acc_fr(const unsigned long long* acc, int w, const Fr& corr) {
  U64x8 a;
#pragma unroll
  for (int l = 0; l < 8; l++) a.v[l] = acc[(size_t)w * 8 + l];
  return fr_sub(redc_columns_ni(a), corr);
}

__device__ __forceinline__ void store_fr(vl_fr* dst, const Fr& x) {
#pragma unroll
  for (int l = 0; l < 8; l++) dst->limb[l] = x.v[l];
}

__device__ __forceinline__ Fr fold1(const Fr& x0, const Fr& x1, const Fr& r) {
  return fr_add(x0, mont_mul_ni(r, fr_sub(x1, x0)));
}

__device__ __forceinline__ Fr shfl_fr(const Fr& x, int src) {
  Fr y;
#pragma unroll
  for (int l = 0; l < 8; l++) y.v[l] = __shfl_sync(0xffffffffu, x.v[l], src);
  return y;
}

// Fold the pair's four entries with r and add its terms to the wide sums
// w0 += a0 b0, wi += (a1 - a0)(b1 - b0).
__device__ __forceinline__ void fold_pair(const Fr* sA, const Fr* sB, Fr* dA, Fr* dB, int j, int h, const Fr& r,
                                          uint32_t (&w0)[17], uint32_t (&wi)[17]) {
  const int hh = h >> 1;
  const Fr a0 = fold1(sA[j], sA[j + h], r), a1 = fold1(sA[j + hh], sA[j + hh + h], r);
  const Fr b0 = fold1(sB[j], sB[j + h], r), b1 = fold1(sB[j + hh], sB[j + hh + h], r);
  dA[j] = a0;
  dA[j + hh] = a1;
  dB[j] = b0;
  dB[j + hh] = b1;
  wide_mac(w0, a0, b0);
  wide_mac(wi, fr_sub(a1, a0), fr_sub(b1, b0));
}

// Round 1's terms of one pair of unfolded entries: g(0), g(1), G.
__device__ __forceinline__ void first_pair(const Fr& a0, const Fr& a1, const Fr& b0, const Fr& b1, uint32_t (&w0)[17],
                                           uint32_t (&w1)[17], uint32_t (&wi)[17]) {
  wide_mac(w0, a0, b0);
  wide_mac(w1, a1, b1);
  wide_mac(wi, fr_sub(a1, a0), fr_sub(b1, b0));
}

// Four lanes of a pair: lane q (mod 4) folds x (+ d r: a0, a1, b0, b1); returned
// are the pair's terms, a0 b0 on lane 0 and (a1 - a0)(b1 - b0) on lane 1.  A
// lane with `clm` set forms (x + d r) r instead.
__device__ __forceinline__ Fr quad_terms(Fr& x, const Fr& d, const Fr& r, bool clm) {
  const int q = threadIdx.x & 3;
  x = fr_add(x, mont_mul_ni(d, r));
  const Fr y = shfl_xor_fr(x, 1);
  Fr z = (q & 1) ? fr_sub(x, y) : x;
  Fr w = shfl_xor_fr(z, 2);
  if (clm) z = x, w = r;
  return mont_mul_ni(z, w);
}

__device__ __forceinline__ void wide_zero(uint32_t (&w)[17]) {
#pragma unroll
  for (int i = 0; i < 17; i++) w[i] = 0;
}

// The message words of an absorb of N = 1 or 2 elements (33 + 32 N bytes: two
// blocks), one word per lane.
__device__ __forceinline__ void absorb_words(RndShared& sh, uint32_t label, const Fr& x, const Fr& y, int n) {
  const int lane = threadIdx.x & 31;
  const uint32_t* xs = x.v;
  const uint32_t* ys = y.v;
  auto limb = [&](int q) { return q < 8 ? xs[q & 7] : ys[q & 7]; };  // x, y are in memory
  uint32_t w = 0;
  const int q = lane - 8;
  if (q < 0) w = sh.S[lane];
  else if (q < 8 * n) w = __byte_perm(limb(q), q == 0 ? label << 24 : limb(q - 1), 0x7012);
  else if (q == 8 * n) w = (limb(q - 1) & 0xff000000u) | 0x00800000u;
  else if (lane == 31) w = (uint32_t)(33 + 32 * n) * 8u;
  sh.msg[lane] = w;
}

// SHA256 of the two blocks in sh.msg.  Warp 0 (returns the digest in every
// lane), with warps 1 and 2 in absorb_help.
__device__ __forceinline__ ShaState absorb_run(RndShared& sh) {
  named_sync(7, 96);
  ShaState st = sha_rounds_ni(sha_iv_state(), sha_load(sh.msg), sh.wk[0], 1);
  return sha_rounds_ni(st, sha_load(sh.msg + 16), sh.wk[1], 4);
}
__device__ __forceinline__ void absorb_help(RndShared& sh, int warp) {
  named_sync(7, 96);
  sha_sched_ni(sha_load(sh.msg + 16 * (warp - 1)), sh.wk[warp - 1], 1 + 3 * (warp - 1));
}

// The lane's block of the squeeze of one challenge from state S: lanes 0 and 1
// the challenge's halves, the others the closing update.
__device__ __forceinline__ ShaBlock squeeze_lane_block(const uint32_t (&S)[8]) {
  const int lane = threadIdx.x & 31, kind = lane < 2 ? lane : 2;
  ShaBlock b;
#pragma unroll
  for (int i = 0; i < 8; i++) b.w[i] = S[i];
  b.w[8] = ((uint32_t)LBL_R << 24) | (kind == 2 ? 1u << 16 : 0u);          // label, t = 0 or count = 1 (LE)
  b.w[9] = kind == 2 ? 0x00800000u : ((uint32_t)kind << 16) | 0x00008000u;  // (half,) padding
#pragma unroll
  for (int i = 10; i < 15; i++) b.w[i] = 0;
  b.w[15] = kind == 2 ? 37u * 8u : 38u * 8u;
  return b;
}

// The challenge from the two halves' digests (lanes 0 and 1), in Montgomery
// form: (lo + hi 2^256) mod r times R = REDC(lo R^2) + REDC(hi R^3), one
// product on the chain.  Valid in lane 0.
__device__ __forceinline__ Fr challenge_of(const uint32_t (&d)[8]) {
  const int lane = threadIdx.x & 31;
  Fr half = fr_zero();
  if (lane < 2) half = mont_mul_ni(digest_le(d), lane == 0 ? fr_r2() : fr_r3());
  const Fr other = shfl_fr(half, 1);
  return fr_add(half, other);
}

// The transcript step of round t (1-based): warps 0 to 2 of the block.  Warp 0
// has the message in sh.g; with_claim: the claim is absorbed before it.  At the
// end sh.r[t & 1], sh.S are set (visible after the block's next barrier).  msg: where
// the proof takes the message, written beside the hashes, g(1) being the claim
// less g(0) (null: round_message wrote it).
__device__ __forceinline__ void transcript_step(RndShared& sh, int warp, int t, bool with_claim, Fr* rch,
                                                vl_fr* msg = nullptr) {
  const int lane = threadIdx.x & 31;
  if (warp == 0) {
    if (with_claim) {
      absorb_words(sh, LBL_C, sh.claim, sh.claim, 1);
      const ShaState c = absorb_run(sh);
      if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 8; i++) sh.S[i] = c.h[i];
      }
      __syncwarp();
    }
    absorb_words(sh, LBL_G, sh.g[0], sh.g[2], 2);  // g(1) is fixed by the running claim
    ShaState st = absorb_run(sh);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < 8; i++) sh.sq[i] = st.h[i];
    }
    named_sync(8, 64);
    st = sha_rounds_ni(sha_iv_state(), squeeze_lane_block(st.h), sh.wk[lane < 2 ? lane : 2], 1);
    if (lane == 2) {
#pragma unroll
      for (int i = 0; i < 8; i++) sh.S[i] = st.h[i];
    }
    const Fr r = challenge_of(st.h);
    if (lane == 0) {
      sh.r[t & 1] = r;
      if (rch) *rch = r;  // chained proofs continue from this point
    }
  } else if (warp < 3) {
    if (with_claim) absorb_help(sh, warp);
    absorb_help(sh, warp);
    if (msg && warp == 2) {
      if (lane == 0) sh.g[1] = fr_sub(sh.claim, sh.g[0]);
      __syncwarp();
      if (lane < 24) msg[lane >> 3].limb[lane & 7] = sh.g[lane >> 3].v[lane & 7];
    }
    if (warp == 1) {
      named_sync(8, 64);
      uint32_t S[8];
#pragma unroll
      for (int i = 0; i < 8; i++) S[i] = sh.sq[i];
      sha_sched_ni(squeeze_lane_block(S), sh.wk[lane < 2 ? lane : 2], 1);
    }
  }
}

// Warp 0: the round's message from g(0) and G (canonical, in every lane; first:
// g(1) too, which makes the claim), into sh.g and the proof.
__device__ __forceinline__ void round_message(RndShared& sh, const Fr& g0, const Fr& G, const Fr* g1_first, vl_proof* pf,
                                              int i) {
  const int lane = threadIdx.x & 31;
  __syncwarp();  // the claim may come from another lane
  const Fr g1 = g1_first ? *g1_first : fr_sub(sh.claim, g0);
  const Fr s = fr_add(g1, G);
  const Fr g2 = fr_sub(fr_dbl(s), g0);
  __syncwarp();
  if (lane == 0) {
    sh.g[0] = g0;
    sh.g[1] = g1;
    sh.g[2] = g2;
    sh.g[3] = G;
    if (g1_first) {
      sh.claim = fr_add(g0, g1);
      store_fr(&pf->c, sh.claim);
    }
  }
  __syncwarp();
  if (lane < 24) pf->g[i][lane >> 3].limb[lane & 7] = sh.g[lane >> 3].v[lane & 7];
}

// One lane: the claim of the next round, g(r), from round t's message and challenge.
__device__ __forceinline__ void next_claim(RndShared& sh, int t) {
  const Fr r = sh.r[t & 1], b = fr_sub(fr_sub(sh.g[1], sh.g[0]), sh.g[3]);
  sh.claim = fr_add(sh.g[0], mont_mul_ni(r, fr_add(b, mont_mul_ni(r, sh.g[3]))));
}

__device__ __forceinline__ void store_state(uint8_t* dst, const ShaState& st) {
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int q = 0; q < 8; q++) reinterpret_cast<uint32_t*>(dst)[q] = bswap32(st.h[q]);
  }
}

// Entries j and j + h of f from the fold: reduced already (direct), or column
// sums to reduce here; j + h may be padding (!real).  They are written to dst
// where the vector does not hold them yet (write: always).
__device__ __forceinline__ void first_entries(const Fr* f, bool direct, const unsigned long long* acc, const Fr& corr,
                                              int j, int h, bool real, bool write, Fr* dst, Fr& x0, Fr& x1) {
  x0 = direct ? f[j] : load_acc_fr(acc, j, corr);
  x1 = fr_zero();
  if (real) x1 = direct ? f[j + h] : load_acc_fr(acc, j + h, corr);
  if (write || !direct) dst[j] = x0;
  if (write || !direct || !real) dst[j + h] = x1;
}

// One pass of a pair per four lanes over hh pairs (4 hh at most the threads of
// the calling warps): the vectors sA, sB (2h = 4 hh entries) folded with r into
// dA, dB, and the round's terms, summed over the warp: lane 0 g(0), lane 1 G
// (Montgomery form).  j: the thread's pair.  clm: this lane forms the next claim.
__device__ __forceinline__ Fr quad_pass(RndShared& sh, const Fr* sA, const Fr* sB, Fr* dA, Fr* dB, int j, bool act,
                                        int h, const Fr& r, bool clm) {
  const int hh = h >> 1, q = threadIdx.x & 3;
  Fr x = fr_zero(), d = fr_zero();
  if (act) {
    const Fr* f = (q < 2 ? sA : sB) + j + (q & 1) * hh;
    x = f[0];
    d = fr_sub(f[h], x);
  } else if (clm) {
    x = fr_sub(fr_sub(sh.g[1], sh.g[0]), sh.g[3]);
    d = sh.g[3];
  }
  __syncwarp();
  Fr p = quad_terms(x, d, r, clm);
  if (act) ((q < 2 ? dA : dB) + j + (q & 1) * hh)[0] = x;
  if (clm) sh.claim = fr_add(sh.g[0], p);
  if (!act) p = fr_zero();
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) p = fr_add(p, shfl_xor_fr(p, off));
  return p;
}

// The block's sums of quad_pass's terms, canonical, in lanes 0 and 1 of warp 0
// (one block barrier).
__device__ __forceinline__ Fr quad_block_sum(RndShared& sh, Fr p, int warp, int last) {
  const int lane = threadIdx.x & 31;
  Fr* red = reinterpret_cast<Fr*>(sh.red);
  if (lane < 2) red[2 * warp + lane] = p;
  __syncthreads();
  if (warp == 0) {
    p = lane < 2 * (last + 1) ? red[lane] : fr_zero();
#pragma unroll
    for (int off = 2; off < 32; off <<= 1) p = fr_add(p, shfl_xor_fr(p, off));
    p = from_mont_ni(p);
  }
  return p;
}

// ----------------------------------------------------------------- look-ahead
//
// With p = x[j], q = x[j + h] the vectors fold to p + r (q - p), so the next
// round's g(0) = sum_j a b and G = sum_j (a' - a)(b' - b) (a' hh = h / 2 entries
// on) are quadratics in r, fixed by their values at 0 and 1 and their leading
// coefficients: six products per pair of the next round instead of two, off
// the chain of hashes.  A short round of a lone proof: 8.5 -> 6.5 us (a 64 x 128 x
// 64 product 139 -> 122 us, one 7B projection 207 -> 190); with 128 threads, where
// many proofs share the GPU, slower (rounds of the 7B step 427 -> 437 us).
static constexpr int LOOK_THREADS = 256;  // blocks of at least this many threads have the warps to spare

// The warps that look ahead: of the schedulers 2 and 3 (warp mod 4), so that they
// take no issue slots from the hash's rounds (warp 0) and schedule (warp 1); warp
// 2's schedule of an absorb's second block has time.  (Warps 3 up: the first
// compression of a round 3400 cycles instead of 2700.)
__device__ __forceinline__ bool look_warp(int warp) { return (warp & 2) && warp != 2; }
__device__ __forceinline__ int look_rank(int warp) { return ((warp >> 2) << 1 | (warp & 1)) - 1; }
__device__ __forceinline__ int look_warps() { return (int)(blockDim.x >> 6) - 1; }

// The look-ahead warps: the coefficients of the message after round i's, whose vectors of
// N entries are in sh.fa, sh.fb, into sh.look[par].  Barrier 9: these warps; 10:
// warp 0 arrives once round i's message is in sh.g.
__device__ __forceinline__ void look_terms(RndShared& sh, int warp, int N, int par) {
  const int lane = threadIdx.x & 31, nwk = look_warps(), wk = look_rank(warp);
  const int h = N >> 1, hh = N >> 2, s = lane & 7, g = lane >> 3, v = s % 3;
  named_sync(9, 32 * nwk);  // the folded vectors
  Fr acc = fr_zero();
  for (int b = 4 * wk; b < hh; b += 4 * nwk) {
    const int j = b + g;
    const bool act = j < hh && s < 6;
    Fr z[2];
#pragma unroll
    for (int m = 0; m < 2; m++) {
      const Fr* f = (m ? sh.fb : sh.fa) + (act ? j : 0);
      Fr x = f[0], y = f[h];  // at r = 0, 1
      if (s >= 3) x = fr_sub(f[hh], x), y = fr_sub(f[h + hh], y);
      z[m] = v == 0 ? x : v == 1 ? y : fr_sub(y, x);
    }
    const Fr p = mont_mul_ni(z[0], z[1]);
    if (act) acc = fr_add(acc, p);
  }
  acc = fr_add(acc, shfl_xor_fr(acc, 8));
  acc = fr_add(acc, shfl_xor_fr(acc, 16));
  if (lane < 6) sh.lsum[wk][lane] = acc;
  named_sync(9, 32 * nwk);
  if (wk != 0) return;
  acc = fr_zero();
  if (s < 6)
    for (int w = g; w < nwk; w += 4) acc = fr_add(acc, sh.lsum[w][s]);
  acc = fr_add(acc, shfl_xor_fr(acc, 8));
  acc = fr_add(acc, shfl_xor_fr(acc, 16));
  acc = from_mont_ni(acc);
  // coefficient k on lane k (g(0)), 3 + k (G): 1 is the value at 1 less the others
  const Fr lead = shfl_fr(acc, (lane + 1) & 31), low = shfl_fr(acc, (lane + 31) & 31);
  const Fr c = v == 1 ? fr_sub(fr_sub(acc, low), lead) : acc;
  if (lane < 6) sh.look[par][lane / 3][v] = c;
  const Fr cg = shfl_fr(c, (lane + 3) & 31);
  named_sync(10, 64);  // round i's message
  if (lane < 3) {
    const Fr g0 = sh.g[0], G = sh.g[3];
    const Fr cl = lane == 0 ? g0 : lane == 1 ? fr_sub(fr_sub(sh.claim, fr_dbl(g0)), G) : G;
    sh.look[par][2][lane] = cl;
    // g(2) = 2 (claim - g(0) + G) - g(0)
    sh.look[par][3][lane] = fr_sub(fr_dbl(fr_add(fr_sub(cl, c), cg)), c);
  }
}

// Warp 0: round i + 1's message and claim at r_i, into sh.g and sh.claim.
__device__ __forceinline__ void look_message(RndShared& sh, const Fr& r, int par) {
  const int lane = threadIdx.x & 31, q = lane & 3;
  const Fr* c = sh.look[par][q];
  const Fr x = fr_add(c[0], mont_mul_ni(r, fr_add(c[1], mont_mul_ni(r, c[2]))));
  if (lane < 4) (lane == 0 ? sh.g[0] : lane == 1 ? sh.g[3] : lane == 2 ? sh.claim : sh.g[2]) = x;
  __syncwarp();
}

// The look-ahead warps: the vectors of N entries in shared memory folded with r.
__device__ __forceinline__ void look_fold(RndShared& sh, int warp, int N, const Fr& r) {
  const int h = N >> 1;
  for (int i = 32 * look_rank(warp) + (threadIdx.x & 31); i < N; i += 32 * look_warps()) {
    Fr* f = i < h ? sh.fa + i : sh.fb + (i - h);
    f[0] = fold1(f[0], f[h], r);
  }
}

// ------------------------------------------------------------------ clusters
//
// The first rounds of one proof by a cluster of up to RND_MAX_CTAS CTAs: CTA c
// owns the entries j with (j / 32) mod CTAs = c, so folding moves no entry
// between CTAs while a round has at least 32 pairs per CTA.  A round costs two
// cluster barriers: each CTA writes its sums of the round's terms into the first
// CTA's shared memory, and the first CTA, after the transcript step, the
// challenge into the others'.  The rounds below RND_CL_PAIRS pairs are the
// first CTA's alone.  What bounds a lone proof's first rounds is one SM's field
// products (4096-entry vectors: about 43 us of them, 5 on eight SMs).
static constexpr int RND_CL_PAIRS = 32 * RND_MAX_CTAS;
// Rounds of a proof with d1 variables that a cluster runs: those with at least
// RND_CL_PAIRS pairs (round t has 2^(d1 - t)).
__host__ __device__ __forceinline__ int cluster_rounds(int d1) { return d1 > 8 ? d1 - 8 : 0; }
static_assert(RND_CL_PAIRS == 1 << 8, "cluster_rounds");

// CTAs per cluster for n chains: while every CTA finds an SM of its own.
static inline int cluster_ctas(int n, int sms) { return 8 * n <= sms ? 8 : 4 * n <= sms ? 4 : 2 * n <= sms ? 2 : 1; }

// n clusters of `ctas` CTAs.
template <class... P, class... A>
cudaError_t launch_clusters(void (*kernel)(P...), int n, int ctas, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ctas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(n * ctas);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t x;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(x));
  return x;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t x;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(x));
  return x;
}
// Every thread of the cluster arrives; what was written before is visible after.
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Write `v` to `p` (shared memory of this CTA) in CTA `rank` of the cluster.
__device__ __forceinline__ void st_cluster(const void* p, uint32_t rank, uint32_t v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Rounds 1 to n = cluster_rounds(d1) >= 1 of the proof, the fold with r_n left
// out.  The first CTA returns with r_n in its slot and the vectors in memory as round
// n saw them (rounds_block goes on from there); the others may leave.
static __device__ void rounds_cluster(const DevProof& P, vl_proof* pf, RndShared& sh, int n) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x, last = (nthr >> 5) - 1;
  const int rank = (int)cluster_rank(), C = (int)cluster_size();
  const int K = 1 << P.d1;
  Fr* fA = P.fA;
  Fr* fB = P.fB;
  const bool da = P.fdirA, db = P.fdirB;
  cluster_sync();  // every CTA has started: its shared memory may be written
  for (int t = 1; t <= n; t++) {
    const int hh = K >> t, own = hh / C;  // the round's pairs, this CTA's
    auto pair = [&](int l) { return ((l >> 5) * C + rank) * 32 + (l & 31); };
    Fr s;
    if (t == 1) {
      uint32_t w0[17], w1[17], wi[17];
      wide_zero(w0), wide_zero(w1), wide_zero(wi);
      const Fr corrA = P.scr->corrA, corrB = P.scr->corrB;
      for (int l = tid; l < own; l += nthr) {
        const int j = pair(l);
        const bool real = j + hh < P.k;
        Fr a0, a1, b0, b1;
        first_entries(fA, da, P.accA, corrA, j, hh, real, false, fA, a0, a1);
        first_entries(fB, db, P.accB, corrB, j, hh, real, false, fB, b0, b1);
        first_pair(a0, a1, b0, b1, w0, w1, wi);
      }
      unsigned long long col[3][8];
      wide_redc(w0, col[0]);
      wide_redc(wi, col[1]);
      wide_redc(w1, col[2]);
      s = block_sum_columns<3>(col, sh.red);
    } else {
      const Fr r = sh.r[(t - 1) & 1];
      const int h = 2 * hh;
      if (rank == 0 && warp == last && lane == 0) next_claim(sh, t - 1);
      if (4 * own <= nthr) {
        const int l = tid >> 2;
        s = quad_pass(sh, fA, fB, fA, fB, pair(l), l < own, h, r, false);
        s = quad_block_sum(sh, s, warp, last);
      } else {
        uint32_t w0[17], wi[17];
        wide_zero(w0), wide_zero(wi);
        for (int l = tid; l < own; l += nthr) fold_pair(fA, fB, fA, fB, pair(l), h, r, w0, wi);
        unsigned long long col[2][8];
        wide_redc(w0, col[0]);
        wide_redc(wi, col[1]);
        s = block_sum_columns<2>(col, sh.red);
      }
    }
    if (warp == 0 && lane < 3) {
#pragma unroll
      for (int q = 0; q < 8; q++) st_cluster(&sh.part[rank][lane].v[q], 0, s.v[q]);
    }
    cluster_sync();
    if (rank == 0) {
      if (warp == 0) {
        // lane 4 c + q: value q of CTA c
        Fr v = (lane >> 2) < C && (lane & 3) < 3 ? sh.part[lane >> 2][lane & 3] : fr_zero();
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) v = fr_add(v, shfl_xor_fr(v, off));
        const Fr g1 = shfl_fr(v, 2);
        round_message(sh, shfl_fr(v, 0), shfl_fr(v, 1), t == 1 ? &g1 : nullptr, pf, t - 1);
      }
      transcript_step(sh, warp, t, t == 1, P.rch ? P.rch + (t - 1) : nullptr);
      if (warp == 0 && t < n) {
        __syncwarp();
        const Fr& r = sh.r[t & 1];
        for (int i = lane; i < 8 * (C - 1); i += 32) st_cluster(&r.v[i & 7], 1 + (i >> 3), r.v[i & 7]);
      }
    }
    if (t < n) cluster_sync();
  }
  __syncthreads();
}

// Claim, rounds and proof of one proof by the whole block (a multiple of 32
// threads, 128 to 512), from round t0 on.  t0 = 1: everything (clustered: the
// first cluster_rounds(d1) rounds by the cluster).  t0 > 1: the earlier rounds
// ran batched over many proofs (kernels_rounds.cu): their messages are in the
// proof already, the transcript state, the claim and r_(t0-1) are in the
// scratch, and the vectors hold the round-(t0-1) values, 2^(d1-t0+2) entries each.
// LOOK: blocks of LOOK_THREADS threads or more.
template <bool LOOK>
static __device__ void rounds_block(const DevProof& P, vl_proof* pf, uint8_t* smem, int t0 = 1,
                                    bool clustered = false) {
  RndShared& sh = *reinterpret_cast<RndShared*>(smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x, last = (nthr >> 5) - 1;
  const int d1 = P.d1, K = 1 << d1;
  const int ncl = clustered ? cluster_rounds(d1) : 0;
  const bool lead = !clustered || cluster_rank() == 0;
  if (!lead && ncl == 0) return;
  if (tid < 8) {
    sh.S[tid] = bswap32(reinterpret_cast<const uint32_t*>(P.scr->state)[tid]);
    if (t0 > 1) sh.claim.v[tid] = P.scr->claim.v[tid];
  }
  if (t0 == 1 && lead) {
    if (tid == 0) {
      pf->m = P.m; pf->k = P.k; pf->n = P.n;
      pf->d0 = P.d0; pf->d1 = P.d1; pf->d2 = P.d2;
      pf->reserved = 0;
    }
    for (int i = P.d1 * 24 + tid; i < VL_MAX_ROUNDS * 24; i += nthr) pf->g[i / 24][(i >> 3) % 3].limb[i & 7] = 0u;
  }
  Fr* fA = P.fA;
  Fr* fB = P.fB;
  __syncthreads();

  if (d1 == 0) {  // k = 1: no rounds, c = a_r . b_r
    if (tid == 0) {
      const Fr a = P.fdirA ? fA[0] : load_acc_fr(P.accA, 0, P.scr->corrA);
      const Fr b = P.fdirB ? fB[0] : load_acc_fr(P.accB, 0, P.scr->corrB);
      const Fr fin[2] = {from_mont_ni(a), from_mont_ni(b)};
      const Fr c[1] = {from_mont_ni(mont_mul_ni(a, b))};
      store_fr(&pf->c, c[0]);
      store_fr(&pf->a_r, fin[0]);
      store_fr(&pf->b_r, fin[1]);
      ShaState st;
#pragma unroll
      for (int i = 0; i < 8; i++) st.h[i] = sh.S[i];
      dev_absorb_fr<1>(st.h, LBL_C, c);
      dev_absorb_fr<2>(st.h, LBL_F, fin);
      store_state(pf->state, st);
      pf->status = P.scr->status;
    }
    __syncthreads();
    return;
  }

  if (ncl > 0) {
    rounds_cluster(P, pf, sh, ncl);
    if (!lead) return;
  } else {
    // The first evaluation: of round 1 on f from the fold (fdir: reduced; else
    // column sums to reduce here), or of round t0 after folding with r_(t0-1).
    uint32_t w0[17], w1[17], wi[17];
    wide_zero(w0), wide_zero(w1), wide_zero(wi);
    Fr v[3];  // g(0), G, g(1)
    if (t0 > 1) {
      const Fr r = P.scr->r;
      const int h = K >> (t0 - 1);
      Fr* dA = h <= RND_VEC ? sh.fa : fA;
      Fr* dB = h <= RND_VEC ? sh.fb : fB;
      for (int j = tid; j < (h >> 1); j += nthr) fold_pair(fA, fB, dA, dB, j, h, r, w0, wi);
    } else {
      const Fr corrA = P.scr->corrA, corrB = P.scr->corrB;
      const bool da = P.fdirA, db = P.fdirB, vec = K <= RND_VEC;
      Fr* dA = vec ? sh.fa : fA;
      Fr* dB = vec ? sh.fb : fB;
      const int h = K >> 1;
      for (int j = tid; j < h; j += nthr) {
        // K/2 < k <= K, so j < k always; j + h may be padding
        const bool real = j + h < P.k;
        Fr a0, a1, b0, b1;
        first_entries(fA, da, P.accA, corrA, j, h, real, vec, dA, a0, a1);
        first_entries(fB, db, P.accB, corrB, j, h, real, vec, dB, b0, b1);
        first_pair(a0, a1, b0, b1, w0, w1, wi);
      }
    }
    unsigned long long col[3][8];
    wide_redc(w0, col[0]);
    wide_redc(wi, col[1]);
    wide_redc(w1, col[2]);
    const Fr s = block_sum_columns<3>(col, sh.red);
    if (warp == 0) {
#pragma unroll
      for (int q = 0; q < 3; q++) v[q] = shfl_fr(s, q);
      round_message(sh, v[0], v[1], t0 == 1 ? &v[2] : nullptr, pf, t0 - 1);
    }
  }

  bool looked = false;  // the round's message is look_message's
  for (int i = ncl > 0 ? ncl - 1 : t0 - 1; i < d1; i++) {
    const int h = K >> (i + 1);  // the vectors hold 2h entries
    const bool look = LOOK && 2 * h <= RND_VEC && h > 1;  // prepare the next message
    if (i >= ncl) {
      if (look && warp == 0) {
        __syncwarp();
        named_arrive(10, 64);
      }
      if (look && look_warp(warp)) look_terms(sh, warp, 2 * h, i & 1);
      else transcript_step(sh, warp, i + 1, i == 0, P.rch ? P.rch + i : nullptr, looked ? pf->g[i] : nullptr);
      __syncthreads();
    }
    const Fr r = sh.r[(i + 1) & 1];
    const Fr* sA = 2 * h <= RND_VEC ? sh.fa : fA;
    const Fr* sB = 2 * h <= RND_VEC ? sh.fb : fB;
    if (i + 1 == d1) {
      // Last fold: a_r, b_r; absorb them and write the proof.
      if (warp == 0) {
        if (lane < 2) {
          const Fr* f = lane == 0 ? sA : sB;
          const Fr x = from_mont_ni(fold1(f[0], f[1], r));
          store_fr(lane == 0 ? &pf->a_r : &pf->b_r, x);
          sh.g[lane] = x;
        }
        __syncwarp();
        absorb_words(sh, LBL_F, sh.g[0], sh.g[1], 2);
        store_state(pf->state, absorb_run(sh));
        if (lane == 0) pf->status = P.scr->status;
      } else if (warp < 3) {
        absorb_help(sh, warp);
      }
      break;
    }
    looked = look;
    if (look) {
      if (warp == 0) look_message(sh, r, i & 1);
      else if (look_warp(warp)) look_fold(sh, warp, 2 * h, r);
      continue;
    }
    const int hh = h >> 1;
    Fr* dA = h <= RND_VEC ? sh.fa : fA;
    Fr* dB = h <= RND_VEC ? sh.fb : fB;
    if (4 * hh > nthr) {
      // Fold with r_i and evaluate round i + 2 (1-based; pairs j, j + hh) in one pass.
      if (warp == last && lane == 0) next_claim(sh, i + 1);
      uint32_t w0[17], wi[17];
      wide_zero(w0), wide_zero(wi);
      for (int j = tid; j < hh; j += nthr) fold_pair(sA, sB, dA, dB, j, h, r, w0, wi);
      unsigned long long col[2][8];
      wide_redc(w0, col[0]);
      wide_redc(wi, col[1]);
      const Fr s = block_sum_columns<2>(col, sh.red);
      if (warp == 0) round_message(sh, shfl_fr(s, 0), shfl_fr(s, 1), nullptr, pf, i + 1);
      continue;
    }
    // Four lanes per pair j: lane q folds a0, a1, b0, b1; lane 0 then forms a0
    // b0, lane 1 (a1 - a0)(b1 - b0).  With at most four pairs warp 0 does all,
    // its last lane the next claim in the same products.
    const bool alone = hh <= 4;
    if (alone && warp != 0) continue;
    const int j = tid >> 2;
    if (!alone && warp == last && lane == 0) next_claim(sh, i + 1);
    Fr p = quad_pass(sh, sA, sB, dA, dB, j, j < hh, h, r, alone && j >= hh && lane == 31);
    p = alone ? from_mont_ni(p) : quad_block_sum(sh, p, warp, last);
    if (warp == 0) round_message(sh, shfl_fr(p, 0), shfl_fr(p, 1), nullptr, pf, i + 1);
  }
  __syncthreads();
}

}  // namespace vl
