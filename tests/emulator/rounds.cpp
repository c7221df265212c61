// The rounds of one proof (rounds_dev.cuh, its barriers and cluster accesses
// replaced by the emulator's) on the CPU.
#include "cta.h"

#include <string.h>

#include "fr.cuh"

namespace vl {
// What fr.cuh has for the device only: 17-limb sums of products and their
// Montgomery reduction, here a reduced value in the low columns.
inline void wide_mac(uint32_t (&w)[17], const Fr& a, const Fr& b) {
  for (int i = 0; i < 8; i++) {
    uint64_t c = 0;
    for (int j = 0; j < 8; j++) {
      c += (uint64_t)a.v[i] * b.v[j] + w[i + j];
      w[i + j] = (uint32_t)c;
      c >>= 32;
    }
    for (int j = i + 8; c && j < 17; j++) {
      c += w[j];
      w[j] = (uint32_t)c;
      c >>= 32;
    }
  }
}
inline void wide_redc(const uint32_t (&w)[17], unsigned long long (&col)[8]) {
  Fr lo, hi;
  for (int i = 0; i < 8; i++) lo.v[i] = w[i], hi.v[i] = w[8 + i];
  // w / 2^256: the low half reduced by a product with 1, the others as they are (2^512 / 2^256 = R)
  Fr x = mont_mul(lo, fr_small(1));
  cond_sub_r(hi.v, 0), cond_sub_r(hi.v, 0);
  x = fr_add(x, hi);
  for (uint32_t t = 0; t < w[16]; t++) x = fr_add(x, fr_r1());
  for (int i = 0; i < 8; i++) col[i] = x.v[i];
}
}  // namespace vl

#include "rounds_dev.cuh"

using namespace vl;

namespace {
std::vector<std::vector<uint8_t>>* shared;
}
namespace emu {
void st_cluster(const void* p, uint32_t rank, uint32_t v) {
  const uint8_t* base = (*shared)[machine->now->cta].data();
  memcpy((*shared)[rank].data() + (static_cast<const uint8_t*>(p) - base), &v, 4);
}
}  // namespace emu

// f_A = a, f_B = b (k entries of int16), the transcript state before the claim;
// 1: the proof is in out, 0: every warp waits for another.
extern "C" int emu_rounds(int k, const int16_t* a, const int16_t* b, const uint8_t* state, int ctas, int threads,
                          int look, const int* order, vl_proof* out) {
  int d1 = 0;
  while ((1 << d1) < k) d1++;
  auto vec = [&](const int16_t* x) {
    std::vector<Fr> f((size_t)1 << d1);
    memset(f.data(), 0xa5, f.size() * sizeof(Fr));  // past k: whatever the fold left there
    for (int i = 0; i < k; i++) f[i] = to_mont(fr_from_i64(x[i]));
    return f;
  };
  std::vector<Fr> fa = vec(a), fb = vec(b);
  ProofScratch scr{};
  memcpy(scr.state, state, 32);
  DevProof P{};
  P.m = P.n = 1, P.k = k, P.d1 = d1;
  P.fA = fa.data(), P.fB = fb.data(), P.fdirA = P.fdirB = 1, P.scr = &scr;
  std::vector<std::vector<uint8_t>> sh(ctas, std::vector<uint8_t>(sizeof(RndShared) + 16, 0x5a));
  shared = &sh;
  memset(out, 0, sizeof(*out));
  emu::Machine m;
  return m.run(ctas, threads, order, [&] {
    uint8_t* mem = sh[emu::machine->now->cta].data();
    if (look) rounds_block<true>(P, out, mem, 1, ctas > 1);
    else rounds_block<false>(P, out, mem, 1, false);
  });
}
