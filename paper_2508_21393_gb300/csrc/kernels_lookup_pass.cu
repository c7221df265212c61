// Lookup-argument sumcheck: the batched round passes (the rounds of every
// proof before its tail).  Kept apart from kernels_lookup.cu so the two compile
// in parallel.
#include <type_traits>

#include "lookup_dev.cuh"

namespace vl {

namespace {

// Column sums over the warp's lanes of NV values, reduced: lane q < NV returns
// value q in Montgomery form, value q < nf multiplied by hf (Montgomery).
template <int NV>
__device__ __forceinline__ Fr lk_warp_sum(const unsigned long long (&c)[NV][8], int nf, const Fr* hf) {
  const int lane = threadIdx.x & 31;
  unsigned long long a[32];
#pragma unroll
  for (int i = 0; i < 32; i++) a[i] = i < NV * 8 ? c[i / 8 < NV ? i / 8 : 0][i % 8] : 0ull;
  const unsigned long long t = warp_transpose_sum<32>(a);
  U64x8 col;
#pragma unroll
  for (int l = 0; l < 8; l++) col.v[l] = __shfl_sync(0xffffffffu, t, (lane * 8 + l) & 31);
  Fr x = redc_columns_ni(col);  // canonical
  if (hf && lane < nf) x = mont_mul_ni(x, *hf);
  return to_mont_ni(x);
}

// Round t, one warp per item (pairs [k0, k1) of one proof, lanes strided by
// one: coalesced loads): the item's partial sums into its slot.  The item's
// pairs lie in one block of 2^sE pairs (LK_PAIRS, 2^sE), so a high round's hiP
// factor multiplies the item's sums once.
template <bool JR, int MODE>
__global__ void __launch_bounds__(LK_PASS_THREADS, JR ? 3 : 4) lk_pass_kernel(LkDev* Ls, int t, const LkItem* items, int n) {
  const int i = blockIdx.x * LK_PASS_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;  // whole warps leave together
  const LkItem it = items[i];
  LkDev* L = Ls + it.proof;
  const int h = 1 << (L->L - t);
  const LkEq q(L, t);
  const Fr r = t > 1 ? L->r[t - 2] : fr_zero();
  const Fr* hf = q.high ? q.hi_tab + (it.k0 >> L->sE) : nullptr;
  {
    LkSumA s;
    s.zero();
#pragma unroll 1
    for (int k = it.k0 + lane; k < it.k1; k += 32) lk_pair_a<MODE>(L, k, h, q.f_tab[k & q.f_mask], r, s);
    unsigned long long col[3][8];
    s.columns(col);
    const Fr x = lk_warp_sum<3>(col, 2, hf);
    if (lane < 3) L->part[(size_t)it.slot * LK_PART + lane] = x;
  }
  if constexpr (JR) {
    const int tj = t - (L->L - L->log2_n);  // table round number (1-based)
    const Fr toff = L->run.toff;
    LkSumB s;
    s.zero();
#pragma unroll 1
    for (int k = it.k0 + lane; k < it.k1; k += 32) lk_pair_b(L, tj, k, h, q.f_tab[k & q.f_mask], r, toff, s);
    unsigned long long col[4][8];
    s.columns(col);
    const Fr x = lk_warp_sum<4>(col, 2, hf);
    if (lane < 4) L->part[(size_t)it.slot * LK_PART + 3 + lane] = x;
  }
}

}  // namespace

// Round t's passes: nhi items of proofs in their high rounds, then nlo items
// of proofs in their table rounds.
cudaError_t launch_lookup_passes(LkDev* Ls, int t, const LkItem* items, int nhi, int nlo, cudaStream_t st) {
  const int ghi = (nhi + LK_PASS_WARPS - 1) / LK_PASS_WARPS, glo = (nlo + LK_PASS_WARPS - 1) / LK_PASS_WARPS;
  auto run = [&](auto jr, const LkItem* it, int n, int grid) {
    constexpr bool JR = decltype(jr)::value;
    if (t == 1) lk_pass_kernel<JR, 0><<<grid, LK_PASS_THREADS, 0, st>>>(Ls, t, it, n);
    else if (t == 2) lk_pass_kernel<JR, 1><<<grid, LK_PASS_THREADS, 0, st>>>(Ls, t, it, n);
    else if (t == 3) lk_pass_kernel<JR, 2><<<grid, LK_PASS_THREADS, 0, st>>>(Ls, t, it, n);
    else lk_pass_kernel<JR, 3><<<grid, LK_PASS_THREADS, 0, st>>>(Ls, t, it, n);
  };
  if (nhi) run(std::false_type{}, items, nhi, ghi);
  if (nlo) run(std::true_type{}, items + nhi, nlo, glo);
  return cudaGetLastError();
}

}  // namespace vl
