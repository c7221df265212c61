// Prologue kernels (see prologue_dev.cuh): the transcript part one CTA per
// proof, then the eq tables in chunks of EQ_CHUNK entries.
#include "prologue_dev.cuh"

namespace vl {

template <int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) transcript_kernel(const DevProof* __restrict__ proofs, int p0) {
  extern __shared__ __align__(128) uint8_t pro_smem[];
  transcript_block<THREADS>(proofs[p0 + blockIdx.x], pro_smem);
}

__global__ void __launch_bounds__(256) eq_kernel(const EqItem* __restrict__ items,
                                                  const DevProof* __restrict__ proofs) {
  const EqItem it = items[blockIdx.x];
  eq_chunk(it, proofs[it.proof]);
}

// While all proofs' blocks fit on the GPU at a time (four of 192 threads per SM) the
// corrections have warps of their own and both squeezes run at once: one proof 20.0
// -> 15.1 us; more proofs run in blocks of 128, eight per SM (1024 proofs in
// blocks of 192: 53 us against 39).
cudaError_t launch_prologue(const DevProof* proofs, int p0, int p1, const EqItem* items, int nitems,
                            cudaStream_t st) {
  if (p1 <= p0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (p1 - p0 <= 4 * sms) transcript_kernel<192, 4><<<p1 - p0, 192, PRO_SMEM, st>>>(proofs, p0);
  else transcript_kernel<128, 8><<<p1 - p0, 128, PRO_SMEM, st>>>(proofs, p0);
  if (nitems > 0) eq_kernel<<<nitems, 256, 0, st>>>(items, proofs);
  return cudaGetLastError();
}

}  // namespace vl
