// Rounds kernels: one CTA or one cluster per proof (see rounds_dev.cuh).
#include <atomic>

#include "rounds_dev.cuh"

namespace vl {

template <int MINB, int THREADS>
__global__ void __launch_bounds__(THREADS, MINB) rounds_kernel(const DevProof* __restrict__ proofs,
                                                               vl_proof* __restrict__ out) {
  extern __shared__ __align__(128) uint8_t rnd_smem[];
  const DevProof& P = proofs[blockIdx.x];
  rounds_block<(THREADS >= LOOK_THREADS)>(P, out + P.job, rnd_smem);
}

// A cluster of CTAs per proof, its first rounds over the cluster.
__global__ void __launch_bounds__(512, 1) rounds_cluster_kernel(const DevProof* __restrict__ proofs,
                                                                vl_proof* __restrict__ out) {
  extern __shared__ __align__(128) uint8_t rnd_smem[];
  const DevProof& P = proofs[blockIdx.x / cluster_size()];
  rounds_block<true>(P, out + P.job, rnd_smem, 1, true);
}

// variant: CTAs per SM.  7, 6, 5 and 4 set the register allocation (7: one
// wave of 1064 proofs, tighter registers; 4: more registers per thread).  3 and 2
// use the variant-4 code and cap residency by reserving shared memory, for
// fewer co-resident proofs competing for issue slots.  threads: 128, 192,
// 256 or 512 per proof (more threads shorten the vector passes of large
// proofs; the register budget follows from variant x threads).
// Both 0: by the number of proofs.  A proof's rounds are a chain, so while
// there are SMs for all of them each proof gets a cluster of 8, 4 or 2 CTAs of
// 512 threads (max_d1: the largest of the batch; 0: no clusters), or as many
// threads as an SM holds at 128 registers (up to one proof per SM: 512, two:
// 256); beyond that 128 threads, four proofs per SM.  Measured, one CTA per
// proof: one 7B projection (8 proofs) 320 -> 232 us, one 13B projection from
// host memory 750 -> 578, the 7B step (1024 proofs) 2.60 -> 2.48 ms; with the
// clusters: the 7B projection 230 -> 207 us (rounds 154 -> 131), the 13B one 460 ->
// 411, a lone product of 2057 terms 294 -> 250.
// Batches of a server's four streams, one beside the other, gain too: 1,000 requests of 8
// proofs a second have a median latency of 0.40 ms, on one CTA of 512 threads per
// proof 0.45, of 128 threads 0.52; at 10,000 and 20,000 the throughput is the same.
cudaError_t launch_rounds(const DevProof* proofs, int nproofs, vl_proof* out, int variant, int threads, int max_d1,
                          cudaStream_t st) {
  if (nproofs <= 0) return cudaSuccess;
  if (variant == 0 && threads == 0) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int ctas = cluster_rounds(max_d1) > 0 ? cluster_ctas(nproofs, sms) : 1;
    if (ctas > 1) return launch_clusters(rounds_cluster_kernel, nproofs, ctas, 512, RND_SMEM_LOOK, st, proofs, out);
    if (nproofs <= sms) threads = 512;
    else if (nproofs <= 2 * sms) threads = 256;
    else variant = 4;
  }
  if (threads == 512) {
    rounds_kernel<1, 512><<<nproofs, 512, RND_SMEM_LOOK, st>>>(proofs, out);
  } else if (threads == 192) {
    rounds_kernel<4, 192><<<nproofs, 192, RND_SMEM, st>>>(proofs, out);
  } else if (threads == 256) {
    rounds_kernel<2, 256><<<nproofs, 256, RND_SMEM_LOOK, st>>>(proofs, out);
  } else if (variant == 2 || variant == 3) {
    static std::atomic<int> set{0};  // launches come from several host threads
    const int smem = variant == 2 ? 100 * 1024 : 70 * 1024;
    if (set.load(std::memory_order_acquire) < smem) {
      cudaError_t e =
          cudaFuncSetAttribute(rounds_kernel<4, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
      if (e != cudaSuccess) return e;
      set.store(100 * 1024, std::memory_order_release);
    }
    rounds_kernel<4, 128><<<nproofs, 128, smem, st>>>(proofs, out);
  } else if (variant == 4) {
    rounds_kernel<4, 128><<<nproofs, 128, RND_SMEM, st>>>(proofs, out);
  } else if (variant == 5) {
    rounds_kernel<5, 128><<<nproofs, 128, RND_SMEM, st>>>(proofs, out);
  } else if (variant == 6) {
    rounds_kernel<6, 128><<<nproofs, 128, RND_SMEM, st>>>(proofs, out);
  } else {
    rounds_kernel<7, 128><<<nproofs, 128, RND_SMEM, st>>>(proofs, out);
  }
  return cudaGetLastError();
}

}  // namespace vl

// ----------------------------------------------------------- batched rounds --
//
// The same claim and rounds as rounds_block, with the heavy first rounds
// organised by round instead of by proof: while a proof's round has more
// than 2^RB_TAIL_LOG pairs, the round's vector work (fold with the previous
// challenge, the sums of g(0) and the leading coefficient, in round 1 of g(1)
// too) for all such proofs is one launch of many CTAs, each on a range of one
// proof's pairs, and the round's transcript step is one launch with one warp
// per proof.  The first rounds'
// vector work (three quarters of a proof's) then spreads over the whole GPU
// instead of one CTA per proof; the rounds after that, short vector passes
// between serial hashes, run as before, one CTA per proof (rounds_block from
// the proof's first unbatched round), in one launch.

namespace vl {
namespace {

__global__ void __launch_bounds__(RB_THREADS, 4) rounds_pass_kernel(const DevProof* __restrict__ proofs,
                                                                    const RoundItem* __restrict__ items,
                                                                    Fr* __restrict__ partials, int t) {
  __shared__ unsigned long long red[3 * 8 * (RB_THREADS / 32)];
  const RoundItem it = items[blockIdx.x];
  const DevProof& P = proofs[it.proof];
  const int tid = threadIdx.x, K = 1 << P.d1;
  Fr* fA = P.fA;
  Fr* fB = P.fB;
  uint32_t w0[17], wi[17];
  wide_zero(w0), wide_zero(wi);
  Fr s;
  if (t == 1) {
    // f from the fold (reduced, or column sums to reduce here), round 1 on
    // pairs (j, j + K/2); j + K/2 may be padding (written as zeros)
    uint32_t w1[17];
    wide_zero(w1);
    const int h = K >> 1;
    const bool da = P.fdirA, db = P.fdirB;
    const Fr corrA = P.scr->corrA, corrB = P.scr->corrB;
    for (int j = it.j0 + tid; j < it.j1; j += RB_THREADS) {
      const Fr a0 = da ? fA[j] : load_acc_fr(P.accA, j, corrA);
      const Fr b0 = db ? fB[j] : load_acc_fr(P.accB, j, corrB);
      const bool real = j + h < P.k;
      Fr a1 = fr_zero(), b1 = fr_zero();
      if (real) {
        a1 = da ? fA[j + h] : load_acc_fr(P.accA, j + h, corrA);
        b1 = db ? fB[j + h] : load_acc_fr(P.accB, j + h, corrB);
      }
      if (!da) fA[j] = a0;
      if (!da || !real) fA[j + h] = a1;
      if (!db) fB[j] = b0;
      if (!db || !real) fB[j + h] = b1;
      first_pair(a0, a1, b0, b1, w0, w1, wi);
    }
    unsigned long long col[3][8];
    wide_redc(w0, col[0]);
    wide_redc(wi, col[1]);
    wide_redc(w1, col[2]);
    s = block_sum_columns<3>(col, red);
  } else {
    // fold with r_(t-1) (vectors of 2h entries) and evaluate round t on the
    // folded pairs (j, j + hh)
    const Fr r = P.scr->r;
    const int h = K >> (t - 1);
    for (int j = it.j0 + tid; j < it.j1; j += RB_THREADS) fold_pair(fA, fB, fA, fB, j, h, r, w0, wi);
    unsigned long long col[2][8];
    wide_redc(w0, col[0]);
    wide_redc(wi, col[1]);
    s = block_sum_columns<2>(col, red);
  }
  if (tid < (t == 1 ? 3 : 2)) partials[3 * (size_t)blockIdx.x + tid] = s;  // g(0), G, and round 1's g(1)
}

// Transcript step of round t for proofs [0, np) (each has more rounds after
// t: the last rounds are the tail's), one warp per proof.
__global__ void __launch_bounds__(32 * RB_WARPS) rounds_hash_kernel(const DevProof* __restrict__ proofs, int np,
                                                                    const int* __restrict__ ibase,
                                                                    const Fr* __restrict__ partials,
                                                                    vl_proof* __restrict__ out, int t) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p = blockIdx.x * RB_WARPS + warp;
  if (p >= np) return;  // whole warps leave together
  const DevProof& P = proofs[p];
  vl_proof* pf = out + P.job;
  if (t == 1) {
    if (lane == 0) {
      pf->m = P.m; pf->k = P.k; pf->n = P.n;
      pf->d0 = P.d0; pf->d1 = P.d1; pf->d2 = P.d2;
      pf->reserved = 0;
    }
    for (int i = P.d1 * 24 + lane; i < VL_MAX_ROUNDS * 24; i += 32) pf->g[i / 24][(i >> 3) % 3].limb[i & 7] = 0u;
  }
  // lane 4 e + q sums value q over every eighth item
  Fr v = fr_zero();
  if ((lane & 3) < (t == 1 ? 3 : 2))
    for (int i = ibase[p] + (lane >> 2); i < ibase[p + 1]; i += 8) v = fr_add(v, partials[3 * (size_t)i + (lane & 3)]);
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) v = fr_add(v, shfl_xor_fr(v, off));
  const Fr g0 = shfl_fr(v, 0), G = shfl_fr(v, 1);
  Fr g1 = shfl_fr(v, 2);
  uint32_t st[8];
#pragma unroll
  for (int i = 0; i < 8; i++) st[i] = bswap32(reinterpret_cast<const uint32_t*>(P.scr->state)[i]);
  if (t == 1) {
    const Fr c[1] = {fr_add(g0, g1)};
    if (lane == 0) store_fr(&pf->c, c[0]);
    dev_absorb_fr<1>(st, LBL_C, c);
  } else {
    g1 = fr_sub(P.scr->claim, g0);
  }
  const Fr g02[2] = {g0, fr_sub(fr_dbl(fr_add(g1, G)), g0)};  // g(2) = 2 g(1) - g(0) + 2 G
  if (lane == 0) {
    store_fr(&pf->g[t - 1][0], g0);
    store_fr(&pf->g[t - 1][1], g1);
    store_fr(&pf->g[t - 1][2], g02[1]);
  }
  dev_absorb_fr<2>(st, LBL_G, g02);
  uint32_t d[8];
  dev_squeeze_block(st, LBL_R, lane < 2 ? 0u : 1u, lane < 2 ? lane : 2, d);
  Fr r = challenge_of(d);
  if (lane == 0) {
    P.scr->r = r;
    if (P.rch) P.rch[t - 1] = r;  // chained proofs continue from this point
    const Fr b = fr_sub(fr_sub(g1, g0), G);
    P.scr->claim = fr_add(g0, mont_mul_ni(r, fr_add(b, mont_mul_ni(r, G))));
  }
  if (lane == 2) {
#pragma unroll
    for (int i = 0; i < 8; i++) reinterpret_cast<uint32_t*>(P.scr->state)[i] = bswap32(d[i]);
  }
}

// The rounds after the batched ones, one CTA per proof.
__global__ void __launch_bounds__(128, 4) rounds_tail_kernel(const DevProof* __restrict__ proofs,
                                                             vl_proof* __restrict__ out) {
  extern __shared__ __align__(128) uint8_t rnd_smem[];
  const DevProof& P = proofs[blockIdx.x];
  rounds_block<false>(P, out + P.job, rnd_smem, 1 + batched_rounds(P.d1));
}

}  // namespace

cudaError_t launch_rounds_pass(const DevProof* proofs, const RoundItem* items, int nitems, Fr* partials, int t,
                               cudaStream_t st) {
  if (nitems <= 0) return cudaSuccess;
  rounds_pass_kernel<<<nitems, RB_THREADS, 0, st>>>(proofs, items, partials, t);
  return cudaGetLastError();
}

cudaError_t launch_rounds_hash(const DevProof* proofs, int nproofs, const int* ibase, const Fr* partials,
                               vl_proof* out, int t, cudaStream_t st) {
  if (nproofs <= 0) return cudaSuccess;
  rounds_hash_kernel<<<(nproofs + RB_WARPS - 1) / RB_WARPS, 32 * RB_WARPS, 0, st>>>(proofs, nproofs, ibase,
                                                                                    partials, out, t);
  return cudaGetLastError();
}

cudaError_t launch_rounds_tail(const DevProof* proofs, int nproofs, vl_proof* out, cudaStream_t st) {
  if (nproofs <= 0) return cudaSuccess;
  rounds_tail_kernel<<<nproofs, 128, RND_SMEM, st>>>(proofs, out);
  return cudaGetLastError();
}

}  // namespace vl
