// Linear zkMat: sum_q c_q M_q = 0 by MLE linearity (Sec. IV; Eq. eq:MLE).
//
// M~(x, y) = sum_i sum_j eq(x, i) M[i, j] eq(y, j) is computed as a fold
// over one dimension (the shorter, "reduced") followed by a dot product over
// the other ("lines"):
//   start:  per proof, transcript start over the statement, squeezes of x
//           (d0) and y (d1), the eq factor tables of both sides, the offset
//           corrections (closed form); then, in chunks, the reduced side's eq
//           table in the form its fold reads;
//   reductions of more than LIN_SHORT_MAX entries: the tensor-core fold writes
//           f_q, the reduced vector of every matrix, and the lines side's eq
//           table is never formed: with E[w] = hi[w >> s] . lo[w mod 2^s],
//             e_q = sum_j hi[j] . (sum_l f_q[j 2^s + l] . lo[l]),
//           one warp per inner sum;
//   shorter ones: fold and dot product in one kernel (lin_short_kernel), with
//           the lines side's eq table;
//   finish: per proof the outer sums, the absorb of 'e' and the proof.
#include "fold_dev.cuh"
#include "prologue_dev.cuh"
#include "rounds_dev.cuh"

namespace vl {

namespace {

constexpr uint8_t LBL_X = 'x', LBL_Y = 'y', LBL_E = 'e';
constexpr int LIN_THREADS = 256;

// One block per proof.
__global__ void __launch_bounds__(LIN_THREADS) lin_start_kernel(LinDev* Ls) {
  LinDev* L = Ls + blockIdx.x;
  __shared__ uint32_t S0[8], S2[8];
  __shared__ Fr xs[MAX_VARS], ys[MAX_VARS];
  __shared__ __align__(16) Fr sub[128];  // factor tables; before them the statement's message (at most 17 blocks)
  static_assert(sizeof(sub) >= 64 * ((23 + 20 + 64 * VL_LIN_MAX + 9 + 63) / 64), "message buffer");
  const int tid = threadIdx.x;
  if (tid < 32) {
    WarpMsg h(sub);  // the message of ts_start_linear
    h.bytes("verilora-gb300/zklin/v1", 23);
    h.u64le(L->seed);
    h.u32le((uint32_t)L->rows);
    h.u32le((uint32_t)L->cols);
    h.u32le((uint32_t)L->nmats);
    h.bytes(L->coeffs, 32 * L->nmats);
    h.bytes(L->binds, 32 * L->nmats);
    uint32_t d[8];
    h.hash(d);
    store_digest(S0, d);
  }
  __syncthreads();
  squeeze2_dev(S0, LBL_X, L->d0, xs, LBL_Y, L->d1, ys, S2);
  if (tid < 8) L->S[tid] = S2[tid];
  const bool rr = L->red_rows != 0;
  eq_factors(xs, L->d0, L->rows, rr, ys, L->d1, L->cols, !rr, L->fac, sub, LIN_THREADS);
  if (tid < 32) {
    const Fr sx = eq_prefix_sum(xs, L->d0, L->rows), sy = eq_prefix_sum(ys, L->d1, L->cols);
    const Fr corr = mont_mul_ni(rr ? sx : sy, to_mont_ni(fr_small(1u << 15)));
    const Fr lcorr = mont_mul_ni(corr, rr ? sy : sx);
    if (tid == 0) {
      L->corr = corr;
      L->lcorr = lcorr;
      L->scr->status = VL_OK;
    }
  }
}

__device__ __forceinline__ uint32_t f16_of(uint32_t x) {
  uint16_t h;
  asm("cvt.rn.f16.u16 %0, %1;" : "=h"(h) : "h"((uint16_t)x));
  return h;
}

// Entries [i0, i1) of one side's eq table of one proof.  Reduced side (side 1):
// the tensor-core fold's fp16 byte table (zero up to a multiple of 128 entries),
// or of a short reduction (one item) the weight bytes as B fragments of
// mma.m16n8k16 -- word pair (16-entry step, 8-byte group, lane): entries 16 ks +
// 2 (lane % 4) + {0, 1} and + {8, 9} of byte 8 nt + lane / 4, zero past the last
// entry.  Lines side (side 0, short reductions): the table itself.
__global__ void __launch_bounds__(LIN_THREADS) lin_eq_kernel(const LinDev* Ls, const EqItem* items) {
  __shared__ __align__(16) uint8_t eb[LIN_SHORT_MAX][32];
  const EqItem it = items[blockIdx.x];
  const LinDev* L = Ls + it.proof;
  const bool xside = (L->red_rows != 0) == (it.side == 1);
  const int d = xside ? L->d0 : L->d1, size = xside ? L->rows : L->cols;
  const int s = (d + 1) >> 1, mask = (1 << s) - 1, tid = threadIdx.x;
  const Fr* lo = L->fac + (xside ? 0 : 2 * EQ_FAC);
  const Fr* hi = lo + EQ_FAC;
  if (it.side == 0) {
    for (int i = it.i0 + tid; i < it.i1; i += LIN_THREADS) L->el[i] = mont_mul_ni(hi[i >> s], lo[i & mask]);
    return;
  }
  if (!L->el) {
    for (int i = it.i0 + tid; i < it.i1; i += LIN_THREADS)
      store_w8(L->w8, i, i < size ? mont_mul_ni(hi[i >> s], lo[i & mask]) : fr_zero());  // eq . R^2
    return;
  }
  if (tid < LIN_SHORT_MAX)
    *reinterpret_cast<Fr*>(eb[tid]) = tid < size ? mont_mul_ni(hi[tid >> s], lo[tid & mask]) : fr_zero();
  __syncthreads();
  const int steps = (size + 15) >> 4;
  for (int w = tid; w < steps * 256; w += LIN_THREADS) {
    const int half = w & 1, ln = (w >> 1) & 31, nt = (w >> 6) & 3, ks = w >> 8;
    const int k = 16 * ks + 8 * half + 2 * (ln & 3), n = 8 * nt + (ln >> 2);
    L->bf[w] = f16_of(eb[k][n]) | (f16_of(eb[k + 1][n]) << 16);
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
template <bool TRANS>
__device__ __forceinline__ void lin_ldmatrix4(uint32_t addr, uint32_t (&r)[4]) {
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint2& b) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// Dynamic shared memory of lin_short_kernel: B fragments, then two tiles of 32
// lines per warp.
constexpr int LS_TILES = (LIN_SHORT_MAX / 16) * 1024;
__host__ __device__ constexpr int ls_tile_bytes(int red) { return ((red + 15) / 16) * 1024; }
constexpr int ls_smem(int red) { return LS_TILES + 2 * (LIN_SHORT_THREADS / 32) * ls_tile_bytes(red); }

// Short reductions (red <= LIN_SHORT_MAX): sum over the item's lines w of
// E[w] . V[w], V[w] = sum_j e_j p_j with the weights e = E R^2 (32 bytes) and p =
// x + 2^15 -- the same byte products as the tensor-core fold, on mma.sync, whose
// operands come straight from registers: a warp takes 32 lines at a time (16-byte
// asynchronous copies two tiles ahead of use, ldmatrix fragments), takes lo and hi
// bytes as fp16 subnormals (byte . 2^-24) and accumulates both planes against the 32
// weight bytes from 1/2 on: exact as there, 128 entries a period.  Two shuffle
// steps leave each lane the eight column sums of one line.  V stays unreduced
// (below 2^278): times E it is added to a 17-limb sum over the thread's lines
// (at most four: below 2^535), reduced once per thread; the offset correction is
// 2^15 (sum e)(sum E), taken off per matrix at the end.
// On the 768 update matrices of a 7B step (84.1 M entries, 3.15 M lines) 175 us,
// spent by instruction count on mma.sync (about 65 us), the column assembly (60)
// and 72 multiply-adds per line (25).  Eight 64-bit multiply-adds per entry and a
// reduction per line took 154 us, the inner sums over the folded lines in memory
// most of 94 more.
__global__ void __launch_bounds__(LIN_SHORT_THREADS, 2) lin_short_kernel(const LinDev* Ls, const LinShort* items) {
  extern __shared__ __align__(16) uint8_t ls[];
  __shared__ unsigned long long red_sh[8 * (LIN_SHORT_THREADS / 32)];
  const LinShort it = items[blockIdx.x];
  const LinDev* L = Ls + it.proof;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = lane & 3, g = lane >> 2;
  const int steps = (it.red + 15) >> 4, tile_bytes = ls_tile_bytes(it.red);
  for (int i = tid; i < steps * 64; i += LIN_SHORT_THREADS)
    reinterpret_cast<uint4*>(ls)[i] = reinterpret_cast<const uint4*>(L->bf)[i];
  const uint32_t buf = smem_addr(ls + LS_TILES) + (uint32_t)(2 * warp) * (uint32_t)tile_bytes;
  const bool rowdot = it.mode == MODE_ROWDOT;
  const int end = it.w0 + it.nw, ntile = (it.nw + 31) >> 5;
  const int nch = (it.red + 7) >> 3;                            // 16-byte chunks of a row (row dots)
  const uint32_t inv = (65536u + (uint32_t)nch - 1) / (uint32_t)nch;  // idx / nch for idx < 512
  // Tile of 32 lines from w.  Row dots: chunk c of line m at 16 (32 c + (m ^ c % 8));
  // column sums: chunk lc (8 lines) of entry k at 16 (16 steps lc + (k ^ 2 lc)).
  auto load_tile = [&](int tile, uint32_t dst) {
    const int w = it.w0 + 32 * tile;
    if (rowdot) {
      for (int i = lane; i < 32 * nch; i += 32) {
        const int m = (int)(((uint32_t)i * inv) >> 16), c = i - m * nch;
        const bool in = w + m < end;
        const int16_t* src = in ? it.base + (int64_t)(w + m) * it.ld + 8 * c : it.base;
        cp_async16(dst + 16u * (uint32_t)(32 * c + (m ^ (c & 7))), src, in ? min(16, 2 * (it.red - 8 * c)) : 0);
      }
    } else {
      for (int i = lane; i < 4 * it.red; i += 32) {
        const int k = i >> 2, lc = i & 3, left = end - (w + 8 * lc);
        const int16_t* src = left > 0 ? it.base + (int64_t)k * it.ld + w + 8 * lc : it.base;
        cp_async16(dst + 16u * (uint32_t)(16 * steps * lc + (k ^ (2 * lc))), src, left > 0 ? min(16, 2 * left) : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  __syncthreads();
  const uint2* bf = reinterpret_cast<const uint2*>(ls);
  uint32_t W[17];
  wide_zero(W);
  constexpr int NW = LIN_SHORT_THREADS / 32;
  if (warp < ntile) load_tile(warp, buf);
  int par = 0;
#pragma unroll 1
  for (int tile = warp; tile < ntile; tile += NW, par ^= 1) {
    if (tile + NW < ntile) {
      load_tile(tile + NW, buf + (uint32_t)((par ^ 1) * tile_bytes));
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    const uint32_t src = buf + (uint32_t)(par * tile_bytes);
    float acc[2][4][2][4];  // [16 lines][8 bytes][lo, hi]
#pragma unroll
    for (int i = 0; i < 64; i++) acc[i >> 5][(i >> 3) & 3][(i >> 2) & 1][i & 3] = 0.5f;
    const int l7 = lane & 7, lm = (lane >> 3) & 1, lk = lane >> 4;
#pragma unroll 1
    for (int ks = 0; ks < steps; ks++) {
      uint32_t lo[2][4], hi[2][4];
#pragma unroll
      for (int T = 0; T < 2; T++) {
        uint32_t r[4];
        if (rowdot) {
          const int m = 16 * T + 8 * lm + l7, c = 2 * ks + lk;
          lin_ldmatrix4<false>(src + 16u * (uint32_t)(32 * c + (m ^ (c & 7))), r);
        } else {
          const int k = 16 * ks + 8 * lk + l7, lc = 2 * T + lm;
          lin_ldmatrix4<true>(src + 16u * (uint32_t)(16 * steps * lc + (k ^ (2 * lc))), r);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
          lo[T][i] = r[i] & 0x00ff00ffu;
          hi[T][i] = __byte_perm(r[i], 0, 0x4341) ^ 0x00800080u;
        }
      }
#pragma unroll
      for (int nt = 0; nt < 4; nt++) {
        const uint2 b = bf[(ks * 4 + nt) * 32 + lane];
#pragma unroll
        for (int T = 0; T < 2; T++) {
          mma_f16(acc[T][nt][0], lo[T], b);
          mma_f16(acc[T][nt][1], hi[T], b);
        }
      }
    }
    __syncwarp();  // the tile's buffer is free for the copy after next
    // Column sums: this lane's digits 8 nt + 2 q + {0, 1} of lines g, g + 8 of
    // each 16 belong to column 2 nt + q / 2, at bit 16 (q % 2).
    auto digits = [&](const float (&clo)[4], const float (&chi)[4], int r) {
      const uint32_t l0 = __float_as_uint(clo[2 * r]) - 0x3F000000u, l1 = __float_as_uint(clo[2 * r + 1]) - 0x3F000000u;
      const uint32_t h0 = __float_as_uint(chi[2 * r]) - 0x3F000000u, h1 = __float_as_uint(chi[2 * r + 1]) - 0x3F000000u;
      unsigned long long v = l0 + (unsigned long long)(l1 + h0) * 256u;
      v += (unsigned long long)h1 * 65536u;
      return v << (16 * (q & 1));
    };
    uint64_t col[8];
#pragma unroll
    for (int nt = 0; nt < 4; nt++) {
      unsigned long long s[2];
#pragma unroll
      for (int T = 0; T < 2; T++) {
        const unsigned long long va = digits(acc[T][nt][0], acc[T][nt][1], 0), vb = digits(acc[T][nt][0], acc[T][nt][1], 1);
        const bool odd = q & 1;
        s[T] = (odd ? vb : va) + __shfl_xor_sync(0xffffffffu, odd ? va : vb, 1);
      }
      const bool up = q & 2;
      const unsigned long long keep = up ? s[1] : s[0], got = __shfl_xor_sync(0xffffffffu, up ? s[0] : s[1], 2);
      col[2 * nt] = up ? got : keep;
      col[2 * nt + 1] = up ? keep : got;
    }
    const int line = it.w0 + 32 * tile + 8 * (q & 1) + 8 * (q & 2) + g;
    if (line < end) {
      uint32_t t[10], z[9];
      column_limbs(col, t);
#pragma unroll
      for (int i = 0; i < 9; i++) z[i] = t[i];
      wide_mac9(W, L->el[line], z);
    }
  }
  unsigned long long c[8];
  wide_redc(W, c);
  const unsigned long long s = warp_transpose_sum<8>(c);
  if (lane < 8) red_sh[8 * warp + lane] = s;
  __syncthreads();
  if (warp == 0) {
    unsigned long long t = 0;
    if (lane < 8)
      for (int w = 0; w < NW; w++) t += red_sh[8 * w + lane];
    U64x8 cs;
#pragma unroll
    for (int l = 0; l < 8; l++) cs.v[l] = __shfl_sync(0xffffffffu, t, l);
    const Fr x = redc_columns_ni(cs);
    if (lane == 0) L->part[(size_t)it.q * L->nblk + it.part] = x;
  }
}

// Warp w of block (b, q, proof) sums inner block j = 8 b + w of matrix q:
// part[q][j] = sum_l f_q[j 2^s + l] . lo[l] (Montgomery; f from the
// accumulators when the fold ran in several segments).
__global__ void __launch_bounds__(LIN_THREADS) lin_dot_kernel(LinDev* Ls) {
  LinDev* L = Ls + blockIdx.z;
  const int q = blockIdx.y, lane = threadIdx.x & 31;
  const int j = blockIdx.x * (LIN_THREADS / 32) + (threadIdx.x >> 5);
  if (q >= L->nmats || j >= L->nblk || L->el) return;  // short reductions sum in their own kernel
  const bool xside = L->red_rows == 0;  // the lines side
  const int d = xside ? L->d0 : L->d1, lines = L->lines;
  const int s = (d + 1) >> 1, hb = 1 << s;
  const Fr* lo = L->fac + (xside ? 0 : 2 * EQ_FAC);
  const Fr corr = L->corr;
  // f_q[w] (Montgomery), from the accumulators when the fold ran in several segments
  auto load_f = [&](int w) {
    const size_t i = (size_t)q * lines + w;
    if (!L->acc) return L->f[i];
    U64x8 a;
#pragma unroll
    for (int l = 0; l < 8; l++) a.v[l] = L->acc[i * 8 + l];
    return fr_sub(redc_columns_ni(a), corr);
  };
  Fr acc = fr_zero();
  const int w1 = min(lines, (j + 1) * hb);
  int w = j * hb + lane;
  // Two independent inline products per step: the carry chains interleave.
  for (; w + 32 < w1; w += 64) {
    const Fr f0 = load_f(w), f1 = load_f(w + 32);
    const Fr p0 = mont_mul(f0, lo[w & (hb - 1)]), p1 = mont_mul(f1, lo[(w + 32) & (hb - 1)]);
    acc = fr_add(acc, fr_add(p0, p1));
  }
  if (w < w1) acc = fr_add(acc, mont_mul_ni(load_f(w), lo[w & (hb - 1)]));
  acc = warp_sum_fr(acc);
  if (lane == 0) L->part[(size_t)q * L->nblk + j] = acc;
}

// One block per proof: e_q = sum_j part[q][j] . hi[j] (short reductions: sum_j
// part[q][j] minus the offset correction), one warp per matrix; absorb, proof.
__global__ void __launch_bounds__(LIN_THREADS) lin_finish_kernel(const LinDev* Ls, vl_lin_proof* outs) {
  __shared__ Fr ev[VL_LIN_MAX];
  __shared__ __align__(16) uint8_t msg[64 * ((33 + 32 * VL_LIN_MAX + 9 + 63) / 64)];
  const LinDev* L = Ls + blockIdx.x;
  vl_lin_proof* out = outs + blockIdx.x;
  const int tid = threadIdx.x, nm = L->nmats, lane = tid & 31;
  const Fr* hi = L->fac + (L->red_rows ? 2 * EQ_FAC : 0) + EQ_FAC;  // the lines side's outer factors
  for (int q = tid >> 5; q < nm; q += LIN_THREADS / 32) {
    Fr acc = fr_zero();
    for (int j = lane; j < L->nblk; j += 32) {
      const Fr p = L->part[(size_t)q * L->nblk + j];
      acc = fr_add(acc, L->el ? p : mont_mul_ni(p, hi[j]));
    }
    acc = warp_sum_fr(acc);
    if (L->el) acc = fr_sub(acc, L->lcorr);
    acc = from_mont_ni(acc);
    if (lane == 0) ev[q] = acc;
  }
  __syncthreads();
  if (tid < 32) {
    WarpMsg h(msg);  // absorb 'e'
    h.state(L->S);
    h.byte(LBL_E);
    h.bytes(ev, 32 * nm);
    uint32_t S[8];
    h.hash(S);
    if (tid == 0) {
      out->rows = L->rows;
      out->cols = L->cols;
      out->d0 = L->d0;
      out->d1 = L->d1;
      out->nmats = nm;
      out->status = L->scr->status;
      store_digest_bytes(out->state, S);
    }
  }
  for (int i = tid; i < VL_LIN_MAX * 8; i += blockDim.x)
    out->evals[i >> 3].limb[i & 7] = (i >> 3) < nm ? ev[i >> 3].v[i & 7] : 0u;
}

}  // namespace

cudaError_t launch_linear_start(LinDev* Ls, int nproofs, const EqItem* items, int nitems, cudaStream_t st) {
  lin_start_kernel<<<nproofs, LIN_THREADS, 0, st>>>(Ls);
  if (nitems > 0) lin_eq_kernel<<<nitems, LIN_THREADS, 0, st>>>(Ls, items);
  return cudaGetLastError();
}

cudaError_t linear_short_prepare() {
  return cudaFuncSetAttribute(lin_short_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ls_smem(LIN_SHORT_MAX));
}

cudaError_t launch_linear_short(const LinDev* Ls, const LinShort* items, int nitems, int max_red, cudaStream_t st) {
  if (nitems > 0) lin_short_kernel<<<nitems, LIN_SHORT_THREADS, ls_smem(max_red), st>>>(Ls, items);
  return cudaGetLastError();
}

cudaError_t launch_linear_finish(LinDev* Ls, int nproofs, int max_nblk, int max_nmats, vl_lin_proof* out,
                                 cudaStream_t st) {
  const int bx = (max_nblk + LIN_THREADS / 32 - 1) / (LIN_THREADS / 32);
  if (bx > 0) lin_dot_kernel<<<dim3(bx, max_nmats, nproofs), LIN_THREADS, 0, st>>>(Ls);
  lin_finish_kernel<<<nproofs, LIN_THREADS, 0, st>>>(Ls, out);
  return cudaGetLastError();
}

}  // namespace vl
