// Batched-claim matmul sumcheck (Sec. IV, composition of proving steps by
// random aggregation of claims under one Fiat-Shamir transcript).
//
// The products' prologues (member transcripts, eq tables) and folds are the
// single-proof kernels; then:
//   claims  (one CTA per product): c_i = sum_w f_A[w] f_B[w] and round 1's terms
//           of the product from the same loop, the Merkle leaf
//           SHA256(0x00 || S_i || c_i);
//   start   (one CTA): the Merkle root, the batch transcript start, rho, the
//           weights rho^i, the combined claim sum_i rho^i c_i, round 1's
//           transcript step;
//   rounds  t >= 2, one launch each: every product's pairs (fold with the
//           previous challenge, then rho^i-weighted sums of g(0) and the leading
//           coefficient, see rounds_dev.cuh); the CTA that finishes last runs
//           the transcript step (g(1) = claim - g(0));
//   tail    (one cluster) of up to BT_TAIL_PRODUCTS products the rounds of at most
//           BT_TAIL_PAIRS pairs, then a_i, b_i and their leaves (of more products:
//           one CTA per product);
//   close   (one CTA) the root, absorb 'f', the proof.
#include "prologue_dev.cuh"
#include "rounds_dev.cuh"

namespace vl {

namespace {

constexpr int BT_THREADS = 256;
constexpr int BT_TAIL_THREADS = 512;
constexpr uint8_t LBL_P = 'p';

// f_A[w] (side 0) or f_B[w] (side 1) of the unfolded vectors; 0 past k.
__device__ __forceinline__ Fr bt_level0(const DevProof& P, int side, int w) {
  if (w >= P.k) return fr_zero();
  if (side == 0) return P.fdirA ? P.fA[w] : load_acc_fr(P.accA, w, P.scr->corrA);
  return P.fdirB ? P.fB[w] : load_acc_fr(P.accB, w, P.scr->corrB);
}

// The 32 serialised bytes of a canonical element as big-endian words Y[at..at + 8).
template <int N>
__device__ __forceinline__ void bt_words(uint32_t (&Y)[N], int at, const Fr& canonical) {
#pragma unroll
  for (int l = 0; l < 8; l++) Y[at + l] = bswap32(canonical.v[l]);
}

// Tree node `i` (32 bytes, 16-byte aligned) as big-endian words, and back.
template <int N>
__device__ __forceinline__ void bt_load_node(const uint8_t* tree, int i, uint32_t (&Y)[N], int at) {
  const uint4* p = reinterpret_cast<const uint4*>(tree + (size_t)i * 32);
  const uint4 a = p[0], b = p[1];
  Y[at] = bswap32(a.x), Y[at + 1] = bswap32(a.y), Y[at + 2] = bswap32(a.z), Y[at + 3] = bswap32(a.w);
  Y[at + 4] = bswap32(b.x), Y[at + 5] = bswap32(b.y), Y[at + 6] = bswap32(b.z), Y[at + 7] = bswap32(b.w);
}

// One block per product: the claim, round 1's g(0) and leading coefficient;
// f_A, f_B left reduced in their vectors (zeros past k) for the later rounds.
__global__ void __launch_bounds__(BT_THREADS) bt_claims_kernel(const DevProof* dp, BtState* B) {
  __shared__ unsigned long long red[3 * 8 * (BT_THREADS / 32)];
  const DevProof& P = dp[blockIdx.x];
  const int i = P.member1 - 1, K = 1 << P.d1, h = K >> 1;
  uint32_t w0[17], w1[17], wi[17];
  wide_zero(w0), wide_zero(w1), wide_zero(wi);
  for (int j = threadIdx.x; j < max(h, 1); j += blockDim.x) {
    const Fr a0 = bt_level0(P, 0, j), b0 = bt_level0(P, 1, j);
    if (h == 0) {  // k = 1: no rounds
      P.fA[0] = a0, P.fB[0] = b0;
      wide_mac(w0, a0, b0);
      break;
    }
    const Fr a1 = bt_level0(P, 0, j + h), b1 = bt_level0(P, 1, j + h);
    P.fA[j] = a0, P.fA[j + h] = a1;
    P.fB[j] = b0, P.fB[j + h] = b1;
    first_pair(a0, a1, b0, b1, w0, w1, wi);
  }
  unsigned long long col[3][8];
  wide_redc(w0, col[0]);
  wide_redc(w1, col[1]);
  wide_redc(wi, col[2]);
  const Fr s = block_sum_columns<3>(col, red);
  if (threadIdx.x < 32) {
    const Fr g0 = shfl_fr(s, 0), g1 = shfl_fr(s, 1), G = shfl_fr(s, 2), c = fr_add(g0, g1);
    uint32_t Y[16], node[8];  // leaf: 0x00 || S_i || c_i
    const uint32_t* st = reinterpret_cast<const uint32_t*>(P.scr->state);
#pragma unroll
    for (int l = 0; l < 8; l++) Y[l] = bswap32(st[l]);
    bt_words(Y, 8, c);
    dev_hash_tagged<16>(0u, Y, node);
    if (threadIdx.x == 0) {
      B->c[3 * (size_t)i] = c;
      B->c[3 * (size_t)i + 1] = g0;
      B->c[3 * (size_t)i + 2] = G;
      store_fr(&B->c_out[i], c);
      store_digest_bytes(B->tree + (size_t)(B->P2 + i) * 32, node);
      if (P.scr->status != VL_OK) atomicExch(&B->status, P.scr->status);
    }
  }
}

// Root of the Merkle tree whose K leaves are in place (block-wide): zero
// padding leaves, then the levels bottom up.
__device__ void bt_tree(BtState* B) {
  uint8_t* t = B->tree;
  for (int i = B->K + threadIdx.x; i < B->P2; i += blockDim.x)
    for (int b = 0; b < 32; b++) t[(size_t)(B->P2 + i) * 32 + b] = 0;
  __syncthreads();
  for (int lvl = B->P2 >> 1; lvl >= 1; lvl >>= 1) {
    for (int j = lvl + threadIdx.x; j < 2 * lvl; j += blockDim.x) {
      uint32_t Y[16], node[8];  // 0x01 || left || right
      bt_load_node(t, 2 * j, Y, 0);
      bt_load_node(t, 2 * j + 1, Y, 8);
      dev_hash_tagged<16>(1u, Y, node);
      store_digest_bytes(t + (size_t)j * 32, node);
    }
    __syncthreads();
  }
}

// Warp 0: round t's message from g(0) and G, into sh.g and the proof.
__device__ __forceinline__ void bt_message(BtState* B, RndShared& sh, int t, const Fr& g0, const Fr& G) {
  const int lane = threadIdx.x & 31;
  const Fr g1 = fr_sub(sh.claim, g0), g2 = fr_sub(fr_dbl(fr_add(g1, G)), g0);
  if (lane == 0) {
    sh.g[0] = g0;
    sh.g[1] = g1;
    sh.g[2] = g2;
    sh.g[3] = G;
  }
  __syncwarp();
  if (lane < 24) B->out->g[t - 1][lane >> 3].limb[lane & 7] = sh.g[lane >> 3].v[lane & 7];
}

// Round t's transcript step by the whole block (at least 4 warps) from g(0)
// and the leading coefficient G (canonical, valid in warp 0): message, absorb,
// squeeze r_t, the next claim.
__device__ void bt_step(BtState* B, RndShared& sh, int t, const Fr& g0, const Fr& G) {
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid < 8) sh.S[tid] = B->St[tid];
  if (tid == 0) sh.claim = B->claim;
  __syncthreads();
  if (warp == 0) bt_message(B, sh, t, g0, G);
  transcript_step(sh, warp, t, false, &B->r[t - 1]);
  __syncthreads();
  if (tid < 8) B->St[tid] = sh.S[tid];
  if (tid == 0) {
    next_claim(sh, t);
    B->claim = sh.claim;
  }
}

// One block: batch start, rho, weights, combined claim, round 1.
__global__ void __launch_bounds__(BT_THREADS) bt_start_kernel(BtState* B) {
  __shared__ RndShared sh;
  __shared__ uint32_t S0[8], S1[8];
  __shared__ Fr ch[1];
  __shared__ Fr red[3 * (BT_THREADS / 32)];
  bt_tree(B);
  if (threadIdx.x < 32) {
    __shared__ __align__(16) uint8_t msg[128];
    WarpMsg h(msg);  // the message of ts_start_batch
    h.bytes("verilora-gb300/zkbatch/v1", 25);
    h.u64le(B->seed);
    h.u32le((uint32_t)B->K);
    h.bytes(B->tree + 32, 32);
    uint32_t d[8];
    h.hash(d);
    store_digest(S0, d);
  }
  __syncthreads();
  squeeze_dev(S0, LBL_P, 1, ch, S1);
  const Fr rho = ch[0];
  Fr acc[3] = {fr_zero(), fr_zero(), fr_zero()};  // claim, g(0), G
  for (int i = threadIdx.x; i < B->K; i += blockDim.x) {
    Fr w = fr_r1(), base = rho;  // rho^i by squaring
    for (int e = i; e; e >>= 1) {
      if (e & 1) w = mont_mul_ni(w, base);
      base = mont_mul_ni(base, base);
    }
    B->w[i] = w;
    for (int q = 0; q < 3; q++) acc[q] = fr_add(acc[q], mont_mul_ni(w, B->c[3 * (size_t)i + q]));
  }
  block_sum_fr<3>(acc, red);
  if (threadIdx.x == 0) B->claim = acc[0];
  if (threadIdx.x < 8) B->St[threadIdx.x] = S1[threadIdx.x];
  __syncthreads();
  if (B->d1 > 0) bt_step(B, sh, 1, acc[1], acc[2]);
}

// Round t >= 2 over pairs [k0, k1) of one product per CTA (item.proof = its
// DevProof index): fold with r_{t-1} in place, then the rho^i-weighted sums of
// a0 b0 and (a1 - a0)(b1 - b0).  Short rounds take four lanes per pair.  The CTA
// that finishes last adds the partial sums and runs the transcript step (a
// launch of its own per round cost 30 us, most of it launch and one thread's
// serial hashes and products).
__global__ void __launch_bounds__(BT_THREADS) bt_round_kernel(const DevProof* dp, BtState* B, int t,
                                                               const LkItem* items) {
  __shared__ RndShared sh;
  __shared__ bool last;
  const LkItem it = items[blockIdx.x];
  const DevProof& P = dp[it.proof];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, hh = 1 << (B->d1 - t), h = 2 * hh;
  const Fr r = B->r[t - 2];
  Fr s = fr_zero();
  if (4 * hh <= BT_THREADS) {
    const int j = tid >> 2, q = tid & 3;
    const bool act = j < hh;
    Fr* f = (q < 2 ? P.fA : P.fB) + j + (q & 1) * hh;
    Fr x = fr_zero(), d = fr_zero();
    if (act) {
      x = f[0];
      d = fr_sub(f[h], x);
    }
    __syncwarp();
    Fr p = quad_terms(x, d, r, false);
    if (act) f[0] = x;
    else p = fr_zero();
    Fr* red = reinterpret_cast<Fr*>(sh.red);
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) p = fr_add(p, shfl_xor_fr(p, off));
    if (lane < 2) red[2 * warp + lane] = p;
    __syncthreads();
    if (warp == 0) {
      p = lane < 2 * (BT_THREADS / 32) ? red[lane] : fr_zero();
#pragma unroll
      for (int off = 2; off < 32; off <<= 1) p = fr_add(p, shfl_xor_fr(p, off));
      s = from_mont_ni(p);
    }
  } else {
    uint32_t w0[17], wi[17];
    wide_zero(w0), wide_zero(wi);
    for (int j = it.k0 + tid; j < it.k1; j += BT_THREADS) fold_pair(P.fA, P.fB, P.fA, P.fB, j, h, r, w0, wi);
    unsigned long long col[2][8];
    wide_redc(w0, col[0]);
    wide_redc(wi, col[1]);
    s = block_sum_columns<2>(col, sh.red);
  }
  if (tid < 2) {
    B->part[(size_t)it.slot * 2 + tid] = mont_mul_ni(B->w[P.member1 - 1], s);
    __threadfence();  // the partial sums before the ticket
  }
  __syncthreads();
  if (tid == 0) last = atomicAdd(&B->ticket, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid == 0) B->ticket = 0;
  Fr acc[2] = {fr_zero(), fr_zero()};
  for (int i = B->pbeg[t] + tid; i < B->pend[t]; i += BT_THREADS) {
    const uint4* p = reinterpret_cast<const uint4*>(B->part + (size_t)i * 2);
    Fr v[2];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint4 a = __ldcg(p + q);  // other CTAs' writes: past the L1
      v[q >> 1].v[4 * (q & 1)] = a.x, v[q >> 1].v[4 * (q & 1) + 1] = a.y;
      v[q >> 1].v[4 * (q & 1) + 2] = a.z, v[q >> 1].v[4 * (q & 1) + 3] = a.w;
    }
    acc[0] = fr_add(acc[0], v[0]);
    acc[1] = fr_add(acc[1], v[1]);
  }
  __syncthreads();
  block_sum_fr<2>(acc, reinterpret_cast<Fr*>(sh.red));
  bt_step(B, sh, t, acc[0], acc[1]);
}

// One warp: a_i (lane 0) and b_i (lane 1) of a product, the last pair folded with
// r_d1, their canonical outputs and Merkle leaf.
__device__ __forceinline__ void bt_final(const DevProof& P, BtState* B, const Fr& r) {
  const int i = P.member1 - 1, d1 = B->d1, lane = threadIdx.x & 31;
  Fr x = fr_zero();
  if (lane < 2) {
    const Fr* f = lane == 0 ? P.fA : P.fB;
    x = d1 == 0 ? f[0] : fold1(f[0], f[1], r);
    x = from_mont_ni(x);
    store_fr(lane == 0 ? &B->a_out[i] : &B->b_out[i], x);
  }
  __syncwarp();
  const Fr ac = shfl_fr(x, 0), bc = shfl_fr(x, 1);
  uint32_t Y[17], node[8];  // leaf: 0x00 || i u32le || a_i || b_i
  Y[0] = bswap32((uint32_t)i);
  bt_words(Y, 1, ac);
  bt_words(Y, 9, bc);
  dev_hash_tagged<17>(0u, Y, node);
  if (lane == 0) store_digest_bytes(B->tree + (size_t)(B->P2 + i) * 32, node);
}

__global__ void __launch_bounds__(32) bt_final_kernel(const DevProof* dp, BtState* B) {
  bt_final(dp[blockIdx.x], B, B->d1 > 0 ? B->r[B->d1 - 1] : fr_zero());
}

// Rounds t0 .. d1 and the final values by one cluster: CTA c takes the products
// i = c (mod CTAs), four lanes per pair, so no vector entry changes hands; the
// sums go to the first CTA, which makes the transcript step, and the challenge
// comes back (as in rounds_cluster).  A round this short is latency, about 16 us as
// a launch of its own: 128 products of a 7B model 773 -> 762 us (from 8192 pairs
// on, with twice the products per pair of bt_round_kernel's loop, 794).
__global__ void __launch_bounds__(BT_TAIL_THREADS, 1) bt_tail_kernel(const DevProof* dp, BtState* B, int t0) {
  __shared__ RndShared sh;
  const int rank = (int)cluster_rank(), C = (int)cluster_size();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = tid & 3, last = BT_TAIL_THREADS / 32 - 1;
  const int d1 = B->d1, np = (B->K - rank + C - 1) / C;  // this CTA's products
  if (tid < 8) {
    sh.S[tid] = B->St[tid];
    sh.claim.v[tid] = B->claim.v[tid];
    sh.r[(t0 - 1) & 1].v[tid] = d1 > 0 ? B->r[t0 - 2].v[tid] : 0u;
  }
  cluster_sync();
  for (int t = t0; t <= d1; t++) {
    const int lg = d1 - t, hh = 1 << lg, h = 2 * hh;
    const Fr r = sh.r[(t - 1) & 1];
    if (rank == 0 && t > t0 && warp == last && lane == 0) next_claim(sh, t - 1);
    Fr acc = fr_zero();
    for (int b = 0; b < np << lg; b += BT_TAIL_THREADS / 4) {
      const int e = b + (tid >> 2);
      const bool act = e < np << lg;
      Fr x = fr_zero(), d = fr_zero(), w = fr_zero();
      Fr* f = nullptr;
      if (act) {
        const DevProof& P = dp[rank + C * (e >> lg)];
        f = (q < 2 ? P.fA : P.fB) + (e & (hh - 1)) + (q & 1) * hh;
        x = f[0];
        d = fr_sub(f[h], x);
        w = B->w[P.member1 - 1];
      }
      __syncwarp();
      const Fr p = mont_mul_ni(quad_terms(x, d, r, false), w);
      if (act) {
        f[0] = x;
        acc = fr_add(acc, p);
      }
    }
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) acc = fr_add(acc, shfl_xor_fr(acc, off));
    const Fr s = quad_block_sum(sh, acc, warp, last);
    if (warp == 0 && lane < 2) {
#pragma unroll
      for (int l = 0; l < 8; l++) st_cluster(&sh.part[rank][lane].v[l], 0, s.v[l]);
    }
    cluster_sync();
    if (rank == 0) {
      if (warp == 0) {
        Fr v = (lane >> 2) < C && q < 2 ? sh.part[lane >> 2][q] : fr_zero();
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) v = fr_add(v, shfl_xor_fr(v, off));
        bt_message(B, sh, t, shfl_fr(v, 0), shfl_fr(v, 1));
      }
      transcript_step(sh, warp, t, false, &B->r[t - 1]);
      if (warp == 0) {
        __syncwarp();
        const Fr& rt = sh.r[t & 1];
        for (int i = lane; i < 8 * (C - 1); i += 32) st_cluster(&rt.v[i & 7], 1 + (i >> 3), rt.v[i & 7]);
      }
    }
    cluster_sync();
  }
  for (int i = warp; i < np; i += BT_TAIL_THREADS / 32) bt_final(dp[rank + C * i], B, sh.r[d1 & 1]);
  if (rank == 0 && tid < 8) B->St[tid] = sh.S[tid];
}

// One block: the root of the final values, absorb 'f', the proof.
__global__ void __launch_bounds__(BT_THREADS) bt_close_kernel(BtState* B, int k) {
  bt_tree(B);
  vl_batch_proof* out = B->out;
  for (int i = threadIdx.x; i < (VL_MAX_ROUNDS - B->d1) * 24; i += blockDim.x)
    out->g[B->d1 + i / 24][(i / 8) % 3].limb[i & 7] = 0u;
  if (threadIdx.x != 0) return;
  uint32_t S[8], Y[8];
  for (int i = 0; i < 8; i++) S[i] = B->St[i];
  bt_load_node(B->tree, 1, Y, 0);
  dev_absorb_words<8>(S, LBL_F, Y);
  store_digest_bytes(out->state, S);
  out->K = B->K;
  out->k = k;
  out->d1 = B->d1;
  out->status = B->status;
}

}  // namespace

cudaError_t launch_batch_claims(const DevProof* dp, int np, BtState* B, cudaStream_t st) {
  bt_claims_kernel<<<np, BT_THREADS, 0, st>>>(dp, B);
  bt_start_kernel<<<1, BT_THREADS, 0, st>>>(B);
  return cudaGetLastError();
}

cudaError_t launch_batch_round(const DevProof* dp, BtState* B, int t, const LkItem* items, int nitems,
                               cudaStream_t st) {
  bt_round_kernel<<<nitems, BT_THREADS, 0, st>>>(dp, B, t, items);
  return cudaGetLastError();
}

// tail: the first round of the tail, 0 without one.
cudaError_t launch_batch_finish(const DevProof* dp, int np, BtState* B, int k, int tail, cudaStream_t st) {
  if (tail) {
    const cudaError_t e = launch_clusters(bt_tail_kernel, 1, RND_MAX_CTAS, BT_TAIL_THREADS, 0, st, dp, B, tail);
    if (e != cudaSuccess) return e;
  } else {
    bt_final_kernel<<<np, 32, 0, st>>>(dp, B);
  }
  bt_close_kernel<<<1, BT_THREADS, 0, st>>>(B, k);
  return cudaGetLastError();
}

}  // namespace vl
