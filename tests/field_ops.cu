// The device arithmetic of fr.cuh on single operands, for tests/test_gpu_field.py:
// row i of `in` (IN words) -> row i of `out` (OUT words).
#include <cuda_runtime.h>

#include "fr.cuh"

using namespace vl;

constexpr int IN = 40, OUT = 20;

template <int N>
__device__ void load(uint32_t (&x)[N], const uint32_t* p) {
  for (int i = 0; i < N; i++) x[i] = p[i];
}
__device__ Fr fr_at(const uint32_t* p) {
  Fr x;
  for (int i = 0; i < 8; i++) x.v[i] = p[i];
  return x;
}

__global__ void field_op(int op, const uint32_t* in, uint32_t* out, int n) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= n) return;
  const uint32_t* p = in + (size_t)row * IN;
  uint32_t* o = out + (size_t)row * OUT;
  auto put = [&](const Fr& x) { for (int i = 0; i < 8; i++) o[i] = x.v[i]; };
  uint32_t w[17], t9[9], z9[9];
  switch (op) {
    case 0: put(fr_add(fr_at(p), fr_at(p + 8))); break;
    case 1: put(fr_sub(fr_at(p), fr_at(p + 8))); break;
    case 2: put(mont_mul(fr_at(p), fr_at(p + 8))); break;
    case 3: put(from_mont(fr_at(p))); break;
    case 4: {
      uint64_t c[8];
      for (int i = 0; i < 8; i++) c[i] = p[2 * i] | ((uint64_t)p[2 * i + 1] << 32);
      put(redc_columns(c));
      break;
    }
    case 5:
      load(w, p);
      wide_mac(w, fr_at(p + 17), fr_at(p + 25));
      for (int i = 0; i < 17; i++) o[i] = w[i];
      break;
    case 6: {
      unsigned long long c[8];
      load(w, p);
      wide_redc(w, c);
      for (int i = 0; i < 8; i++) o[2 * i] = (uint32_t)c[i], o[2 * i + 1] = (uint32_t)(c[i] >> 32);
      break;
    }
    case 7: load(t9, p); put(small_reduce(t9)); break;
    case 8: put(small_mul_mod(fr_at(p), p[8])); break;
    case 9:
      load(w, p);
      load(z9, p + 25);
      wide_mac9(w, fr_at(p + 17), z9);
      for (int i = 0; i < 17; i++) o[i] = w[i];
      break;
    case 10:
      load(w, p);
      wide_mac_small(w, fr_at(p + 17), fr_at(p + 25), p[33]);
      for (int i = 0; i < 17; i++) o[i] = w[i];
      break;
    case 11: {
      uint64_t c[8];
      uint32_t t[10];
      for (int i = 0; i < 8; i++) c[i] = p[2 * i] | ((uint64_t)p[2 * i + 1] << 32);
      column_limbs(c, t);
      for (int i = 0; i < 10; i++) o[i] = t[i];
      break;
    }
    case 12:
      load(t9, p);
      sum9_add(t9, fr_at(p + 9));
      for (int i = 0; i < 9; i++) o[i] = t9[i];
      break;
    case 13:
      load(t9, p);
      load(z9, p + 9);
      add9(t9, z9);
      for (int i = 0; i < 9; i++) o[i] = t9[i];
      break;
    case 14: put(fr_inv_canonical(fr_at(p))); break;
  }
}

extern "C" int field_ops(int op, const uint32_t* in, uint32_t* out, int n) {
  uint32_t *di = nullptr, *dout = nullptr;
  cudaError_t e = cudaMalloc(&di, (size_t)n * IN * 4);
  if (e == cudaSuccess) e = cudaMalloc(&dout, (size_t)n * OUT * 4);
  if (e == cudaSuccess) e = cudaMemcpy(di, in, (size_t)n * IN * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(dout, 0, (size_t)n * OUT * 4);
  if (e == cudaSuccess) field_op<<<(n + 127) / 128, 128>>>(op, di, dout, n), e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(out, dout, (size_t)n * OUT * 4, cudaMemcpyDeviceToHost);
  cudaFree(di);
  cudaFree(dout);
  return (int)e;
}
