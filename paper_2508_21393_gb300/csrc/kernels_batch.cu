// Batched-claim matmul sumcheck (Sec. IV, composition of proving steps by
// random aggregation of claims under one Fiat-Shamir transcript).
//
// The products' prologues (member transcripts, eq tables) and folds are the
// single-proof kernels; then:
//   claims  (one CTA per product): c_i = sum_w f_A[w] f_B[w], its Merkle leaf
//           SHA256(0x00 || S_i || c_i);
//   start   (one CTA): the Merkle root, the batch transcript start, rho, the
//           weights rho^i, the combined claim sum_i rho^i c_i;
//   rounds  per variable: a pass over every product's pairs (fold with the
//           previous challenge, then rho^i-weighted sums of g(0), g(2)) and
//           one CTA for the transcript step (g(1) = claim - g(0));
//   finish  (one CTA per product) a_i, b_i and their leaves; (one CTA) the
//           root, absorb 'f', the proof.
#include "prologue_dev.cuh"
#include "rounds_dev.cuh"

namespace vl {

namespace {

constexpr int BT_THREADS = 256;
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

// One block per product.
__global__ void __launch_bounds__(BT_THREADS) bt_claims_kernel(const DevProof* dp, BtState* B) {
  __shared__ Fr red[BT_THREADS / 32];
  const DevProof& P = dp[blockIdx.x];
  const int i = P.member1 - 1;
  Fr acc[1] = {fr_zero()};
  for (int w = threadIdx.x; w < P.k; w += blockDim.x)
    acc[0] = fr_add(acc[0], mont_mul_ni(bt_level0(P, 0, w), bt_level0(P, 1, w)));
  block_sum_fr<1>(acc, red);
  if (threadIdx.x == 0) {
    B->c[i] = acc[0];
    const Fr c = from_mont_ni(acc[0]);
    for (int l = 0; l < 8; l++) B->c_out[i].limb[l] = c.v[l];
    uint32_t Y[16], node[8];  // leaf: 0x00 || S_i || c_i
    const uint32_t* st = reinterpret_cast<const uint32_t*>(P.scr->state);
#pragma unroll
    for (int l = 0; l < 8; l++) Y[l] = bswap32(st[l]);
    bt_words(Y, 8, c);
    dev_hash_tagged<16>(0u, Y, node);
    store_digest_bytes(B->tree + (size_t)(B->P2 + i) * 32, node);
    if (P.scr->status != VL_OK) atomicExch(&B->status, P.scr->status);
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

// One block: batch start, rho, weights, combined claim.
__global__ void __launch_bounds__(BT_THREADS) bt_start_kernel(BtState* B) {
  __shared__ uint32_t S0[8], S1[8];
  __shared__ uint32_t dig[3][8];
  __shared__ Fr ch[1];
  __shared__ Fr red[BT_THREADS / 32];
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
  squeeze_dev(S0, LBL_P, 1, ch, S1, dig);
  const Fr rho = ch[0];
  Fr acc[1] = {fr_zero()};
  for (int i = threadIdx.x; i < B->K; i += blockDim.x) {
    Fr w = fr_r1(), base = rho;  // rho^i by squaring
    for (int e = i; e; e >>= 1) {
      if (e & 1) w = mont_mul_ni(w, base);
      base = mont_mul_ni(base, base);
    }
    B->w[i] = w;
    acc[0] = fr_add(acc[0], mont_mul_ni(w, B->c[i]));
  }
  block_sum_fr<1>(acc, red);
  if (threadIdx.x == 0) {
    B->rho = rho;
    B->claim = acc[0];
    for (int i = 0; i < 8; i++) B->St[i] = S1[i];
  }
}

// Round t over pairs [k0, k1) of one product (item.proof = its DevProof
// index): fold with r_{t-1} (the first round reads the unfolded vectors, the
// second folds them into fA/fB, later rounds fold in place), then the
// rho^i-weighted sums of a0 b0 and (2a1 - a0)(2b1 - b0).
__global__ void __launch_bounds__(BT_THREADS) bt_pass_kernel(const DevProof* dp, BtState* B, int t,
                                                              const LkItem* items) {
  __shared__ Fr red[2 * (BT_THREADS / 32)];
  const LkItem it = items[blockIdx.x];
  const DevProof& P = dp[it.proof];
  const int h = 1 << (B->d1 - t);
  Fr acc[2] = {fr_zero(), fr_zero()};
  for (int j = it.k0 + threadIdx.x; j < it.k1; j += blockDim.x) {
    Fr a0, a1, b0, b1;
    if (t == 1) {
      a0 = bt_level0(P, 0, j), a1 = bt_level0(P, 0, j + h);
      b0 = bt_level0(P, 1, j), b1 = bt_level0(P, 1, j + h);
    } else if (t == 2) {
      const Fr r = B->r[0];
      a0 = fold1(bt_level0(P, 0, j), bt_level0(P, 0, j + 2 * h), r);
      a1 = fold1(bt_level0(P, 0, j + h), bt_level0(P, 0, j + 3 * h), r);
      b0 = fold1(bt_level0(P, 1, j), bt_level0(P, 1, j + 2 * h), r);
      b1 = fold1(bt_level0(P, 1, j + h), bt_level0(P, 1, j + 3 * h), r);
      P.fA[j] = a0, P.fA[j + h] = a1, P.fB[j] = b0, P.fB[j + h] = b1;
    } else {
      const Fr r = B->r[t - 2];
      a0 = fold1(P.fA[j], P.fA[j + 2 * h], r);
      a1 = fold1(P.fA[j + h], P.fA[j + 3 * h], r);
      b0 = fold1(P.fB[j], P.fB[j + 2 * h], r);
      b1 = fold1(P.fB[j + h], P.fB[j + 3 * h], r);
      P.fA[j] = a0, P.fA[j + h] = a1, P.fB[j] = b0, P.fB[j + h] = b1;
    }
    acc[0] = fr_add(acc[0], mont_mul_ni(a0, b0));
    acc[1] = fr_add(acc[1], mont_mul_ni(fr_sub(fr_dbl(a1), a0), fr_sub(fr_dbl(b1), b0)));
  }
  block_sum_fr<2>(acc, red);
  if (threadIdx.x == 0) {
    const Fr w = B->w[P.member1 - 1];
    B->part[(size_t)it.slot * 2] = mont_mul_ni(w, acc[0]);
    B->part[(size_t)it.slot * 2 + 1] = mont_mul_ni(w, acc[1]);
  }
}

// One block: round t's polynomial from the partial sums, its values in the
// proof, absorb, squeeze r_t, new claim.
__global__ void __launch_bounds__(BT_THREADS) bt_round_kernel(BtState* B, int t) {
  __shared__ Fr red[2 * (BT_THREADS / 32)];
  __shared__ uint32_t Sw[8], Sn[8];
  __shared__ uint32_t dig[3][8];
  __shared__ Fr ch[1];
  __shared__ Fr gsh[3];
  Fr acc[2] = {fr_zero(), fr_zero()};
  for (int s = B->pbeg[t] + threadIdx.x; s < B->pend[t]; s += blockDim.x) {
    acc[0] = fr_add(acc[0], B->part[(size_t)s * 2]);
    acc[1] = fr_add(acc[1], B->part[(size_t)s * 2 + 1]);
  }
  block_sum_fr<2>(acc, red);
  if (threadIdx.x == 0) {
    const Fr g[3] = {acc[0], fr_sub(B->claim, acc[0]), acc[1]};
    Fr gc[3];
    for (int q = 0; q < 3; q++) {
      gsh[q] = g[q];
      gc[q] = from_mont_ni(g[q]);
      for (int l = 0; l < 8; l++) B->out->g[t - 1][q].limb[l] = gc[q].v[l];
    }
    uint32_t S[8];
    for (int i = 0; i < 8; i++) S[i] = B->St[i];
    const Fr m2[2] = {gc[0], gc[2]};
    dev_absorb_fr<2>(S, LBL_G, m2);
    for (int i = 0; i < 8; i++) Sw[i] = S[i];
  }
  __syncthreads();
  squeeze_dev(Sw, LBL_R, 1, ch, Sn, dig);
  if (threadIdx.x == 0) {
    const Fr r = ch[0];
    B->r[t - 1] = r;
    for (int i = 0; i < 8; i++) B->St[i] = Sn[i];
    // g(r) through (0, g0), (1, g1), (2, g2): g0 (r-1)(r-2)/2 - g1 r(r-2) + g2 r(r-1)/2
    const Fr one = fr_r1(), two = fr_add(one, one);
    const Fr r1 = fr_sub(r, one), r2 = fr_sub(r, two);
    const Fr l0 = mont_mul_ni(mont_mul_ni(r1, r2), B->inv2);
    const Fr l1 = fr_neg(mont_mul_ni(r, r2));
    const Fr l2 = mont_mul_ni(mont_mul_ni(r, r1), B->inv2);
    B->claim = fr_add(fr_add(mont_mul_ni(gsh[0], l0), mont_mul_ni(gsh[1], l1)), mont_mul_ni(gsh[2], l2));
  }
}

// One warp per product: a_i, b_i (the last pair folded with r_d1), their
// canonical outputs and Merkle leaf.
__global__ void __launch_bounds__(32) bt_final_kernel(const DevProof* dp, BtState* B) {
  if (threadIdx.x != 0) return;
  const DevProof& P = dp[blockIdx.x];
  const int i = P.member1 - 1, d1 = B->d1;
  Fr a, b;
  if (d1 == 0) {
    a = bt_level0(P, 0, 0);
    b = bt_level0(P, 1, 0);
  } else if (d1 == 1) {
    a = fold1(bt_level0(P, 0, 0), bt_level0(P, 0, 1), B->r[0]);
    b = fold1(bt_level0(P, 1, 0), bt_level0(P, 1, 1), B->r[0]);
  } else {
    a = fold1(P.fA[0], P.fA[1], B->r[d1 - 1]);
    b = fold1(P.fB[0], P.fB[1], B->r[d1 - 1]);
  }
  const Fr ac = from_mont_ni(a), bc = from_mont_ni(b);
  for (int l = 0; l < 8; l++) {
    B->a_out[i].limb[l] = ac.v[l];
    B->b_out[i].limb[l] = bc.v[l];
  }
  uint32_t Y[17], node[8];  // leaf: 0x00 || i u32le || a_i || b_i
  Y[0] = bswap32((uint32_t)i);
  bt_words(Y, 1, ac);
  bt_words(Y, 9, bc);
  dev_hash_tagged<17>(0u, Y, node);
  store_digest_bytes(B->tree + (size_t)(B->P2 + i) * 32, node);
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
  if (nitems) bt_pass_kernel<<<nitems, BT_THREADS, 0, st>>>(dp, B, t, items);
  bt_round_kernel<<<1, BT_THREADS, 0, st>>>(B, t);
  return cudaGetLastError();
}

cudaError_t launch_batch_finish(const DevProof* dp, int np, BtState* B, int k, cudaStream_t st) {
  bt_final_kernel<<<np, 32, 0, st>>>(dp, B);
  bt_close_kernel<<<1, BT_THREADS, 0, st>>>(B, k);
  return cudaGetLastError();
}

}  // namespace vl
