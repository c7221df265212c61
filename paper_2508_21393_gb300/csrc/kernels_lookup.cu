// Lookup-argument sumcheck (Sec. II, lookup arguments; Protocol 1; Eq.
// eq:lookup-sumcheck) for range tables T_j = t0 + j, j < N, over a batch of
// proofs.
//
// The sumcheck runs over k = (i, j) in {0,1}^L, L = log2 D, binding the most
// significant variable first, on
//   P(k) = alpha A(k) E(k) S'(k) + A(k) + (N/D)(alpha^2 B(j) Ej(j) T'(j) - B(j) m(j))
// with A = 1/(beta + S), E = eq(u, .), S' = S + beta, B = 1/(beta + T),
// Ej = eq(u_low, .), T' = T + beta.  The table side depends on the low
// log2 N variables only, so in the first L - log2 N rounds its contribution
// to g_t(X) is the constant 2^-t . Cb, Cb = alpha^2 sum B Ej T' - sum B m;
// in the last log2 N rounds its four vectors are folded like the others.
//
// E = eq(u, .) is never formed: folded by r_1 .. r_{t-1} it is
//   E_t(X, k) = c_t . eqf(u_t, X) . eq(u_{t+1..L}, k),
//   c_t = prod_{v<t} eqf(u_v, r_v), eqf(u, x) = u x + (1 - u)(1 - x),
// so a pass sums eq(u_{t+1..L}, k) . (A S')(X, k) and the transcript step
// multiplies by the scalar c_t eqf(u_t, X).  eq(u_{t+1..L}, k) is read from
// suffix tables: while t binds one of the first L - sE variables it is
// hiP[k >> sE] . loP_sE[k mod 2^sE], later loP_(L-t)[k].
//
// Launches: start (per proof: transcript, beta, alpha, u, N/D, the suffix eq
// tables), histogram (multiplicities, range check), table (batch inversion of
// beta + T per 4096-entry block, B, T', m, partial sums of B m; the inverses
// of the u_t ride in the first block); per round a pass over all proofs' pairs
// (fold with the previous challenge, then the partial sums, lookup_dev.cuh) and
// a transcript step per proof; tail.
// A never exists as a vector: its entries are gathered from B by value
// (A_k = B_{S_k - t0}), and S' from T'.  The table side's cube sum is
// Cb = alpha^2 sum Ej B T' - sum B m = alpha^2 - sum B m (B T' = 1, sum Ej = 1).
#include "lookup_dev.cuh"

namespace vl {

namespace {

// One block per proof.
__global__ void __launch_bounds__(LK_THREADS) lk_start_kernel(LkDev* Ls) {
  LkDev* L = Ls + blockIdx.x;
  __shared__ uint32_t S0[8], S1[8], S2[8], S3[8];
  __shared__ __align__(16) uint8_t msg[128];
  __shared__ Fr ch[LK_MAX_L];
  __shared__ Fr beta_sh, alpha_sh;
  const int tid = threadIdx.x;
  if (tid < 32) {
    WarpMsg h(msg);  // the message of ts_start_lookup (86 bytes)
    h.bytes("verilora-gb300/zklookup/v1", 26);
    h.u64le(L->seed);
    h.u32le((uint32_t)L->n);
    h.u32le((uint32_t)L->L);
    h.u32le((uint32_t)L->log2_n);
    h.u64le((uint64_t)L->t0);
    h.bytes(L->bind, 32);
    uint32_t d[8];
    h.hash(d);
    store_digest(S0, d);
  }
  __syncthreads();
  squeeze_dev(S0, LBL_BETA, 1, ch, S1);
  if (tid == 0) beta_sh = ch[0];
  __syncthreads();
  squeeze_dev(S1, LBL_ALPHA, 1, ch, S2);
  if (tid == 0) alpha_sh = ch[0];
  __syncthreads();
  squeeze_dev(S2, LBL_U, L->L, ch, S3);
  if (tid < L->L) L->u[tid] = ch[tid];
  if (tid < 8) L->run.St[tid] = S3[tid];
  if (tid == 0) {
    const Fr alpha = alpha_sh, one = fr_small(1);
    Fr c = fr_r1();  // N / D = 2^-(L - log2 N)
    for (int i = 0; i < L->L - L->log2_n; i++) c = mont_mul_ni(c, L->inv2);
    const Fr a2 = mont_mul_ni(alpha, alpha);
    L->beta = beta_sh;
    L->c_nd = c;
    L->asq = from_mont_ni(a2);
    L->run.ac = alpha;
    L->run.fc = mont_mul_ni(c, a2);
    L->run.Tc = one;  // sum eq(u, .) A S' = sum eq(u, .) = 1
    L->run.Uc = one;
    L->run.toff = fr_zero();
    L->scr->status = VL_OK;
    const uint32_t pad = (uint32_t)((1 << L->L) - L->n);  // padding entries hold t0: table index 0
    if (pad) atomicAdd(&L->counts[0], pad);
  }
  // Suffix eq tables by doubling, loP on the first half of the block, hiP on
  // the second: level m (entries 2^m - 1 ..) is eq over the last m variables of
  // u (loP, m <= sE) or of its first L - sE (hiP, m < L - sE); entry i of it is
  // the factor of its highest variable's bit times entry i mod 2^(m-1) below.
  const bool lo = tid < LK_THREADS / 2;
  const int id = lo ? tid : tid - LK_THREADS / 2, top = lo ? L->L : L->L - L->sE;
  const int levels = lo ? L->sE : L->L - L->sE - 1;  // above level 0
  Fr* out = lo ? L->loP : L->hiP;
  if (id == 0 && levels >= 0) out[0] = fr_r1();
  const int most = L->sE > L->L - L->sE - 1 ? L->sE : L->L - L->sE - 1;
  for (int m = 1; m <= most; m++) {
    __syncthreads();
    if (m <= levels) {
      const Fr x = ch[top - m], y = fr_sub(fr_r1(), x);
      const int half = 1 << (m - 1);
      for (int i = id; i < 2 * half; i += LK_THREADS / 2)
        out[2 * half - 1 + i] = mont_mul_ni(i & half ? x : y, out[half - 1 + (i & (half - 1))]);
    }
  }
}

// Multiplicities and table indices of cube entries [k0, k1): S's entries, then the
// padding (index 0, counted by lk_start_kernel).  A value outside the table marks
// the proof VL_ELOOKUP (its index is clamped).  Tables up to 4096 entries count in
// shared memory.
__global__ void __launch_bounds__(LK_THREADS) lk_hist_kernel(LkDev* Ls, const LkItem* items) {
  __shared__ uint32_t h[4096];
  const LkItem it = items[blockIdx.x];
  LkDev* L = Ls + it.proof;
  const int N = 1 << L->log2_n, end = min(it.k1, L->n);
  const bool local = N <= 4096;
  uint16_t* idx = L->idx;
  if (local)
    for (int j = threadIdx.x; j < N; j += blockDim.x) h[j] = 0;
  __syncthreads();
  bool bad = false;
  auto count = [&](int k, int64_t v) {
    const int64_t j = v - L->t0;
    const bool in = j >= 0 && j < N;
    idx[k] = (uint16_t)(in ? j : j < 0 ? 0 : N - 1);
    if (!in) bad = true;
    else if (local) atomicAdd(&h[j], 1u);
    else atomicAdd(&L->counts[j], 1u);
  };
  int k = it.k0 + threadIdx.x;
  if (L->dense) {
    const int16_t* S = L->S;
    for (; k + 3 * (int)blockDim.x < end; k += 4 * blockDim.x) {  // four loads in flight
      int16_t v[4];
#pragma unroll
      for (int i = 0; i < 4; i++) v[i] = S[k + i * (int)blockDim.x];
#pragma unroll
      for (int i = 0; i < 4; i++) count(k + i * (int)blockDim.x, v[i]);
    }
    for (; k < end; k += blockDim.x) count(k, S[k]);
  } else {
    for (; k < end; k += blockDim.x) {
      const int row = k / (int)L->cols, col = k - row * (int)L->cols;
      count(k, L->S[(int64_t)row * L->ld + col]);
    }
  }
  for (; k < it.k1; k += blockDim.x) idx[k] = 0;
  if (bad) atomicExch(&L->scr->status, VL_ELOOKUP);
  __syncthreads();
  if (local)
    for (int j = threadIdx.x; j < N; j += blockDim.x)
      if (h[j]) atomicAdd(&L->counts[j], h[j]);
}

// Table entries [k0, k1) (at most 16 per thread, consecutive): x_j = beta + t0 +
// j, its inverse by one batch inversion per block (the products before each entry
// within its thread, left in Binv; scans over the threads; one field inversion;
// back substitution, two products per entry), the table-side vectors, and this
// block's share of sum B m (canonical, its slot's first entry).  The first
// block of a proof also inverts the u_t (one more element per thread).  Bound
// by products and the serial inversion: the tables of the 512 lookups of a 7B
// step take 258 us, with 1024-entry blocks (one inversion for 1024) 456.
__global__ void __launch_bounds__(LK_THREADS, 2) lk_table_kernel(LkDev* Ls, const LkItem* items) {
  __shared__ Fr pre[LK_THREADS], suf[LK_THREADS];
  __shared__ Fr inv_tot;
  __shared__ unsigned long long red[8 * (LK_THREADS / 32)];
  const LkItem it = items[blockIdx.x];
  LkDev* L = Ls + it.proof;
  const int tid = threadIdx.x, E = (it.k1 - it.k0 + LK_THREADS - 1) / LK_THREADS;
  const int j0 = it.k0 + E * tid, j1 = min(j0 + E, it.k1);
  const bool has_u = it.k0 == 0 && tid < L->L;
  const Fr ux = has_u ? L->u[tid] : fr_r1();
  Fr x = fr_add(L->beta, to_mont_ni(fr_from_i64(L->t0 + j0))), run = ux;
  for (int j = j0; j < j1; j++) {
    L->Binv[j] = run;
    run = mont_mul_ni(run, x);
    x = fr_add(x, fr_r1());
  }
  // inclusive prefix and suffix products of the thread totals (Hillis-Steele)
  pre[tid] = run;
  suf[tid] = run;
  __syncthreads();
  for (int off = 1; off < LK_THREADS; off <<= 1) {
    const Fr a = tid >= off ? mont_mul_ni(pre[tid - off], pre[tid]) : pre[tid];
    const Fr b = tid + off < LK_THREADS ? mont_mul_ni(suf[tid], suf[tid + off]) : suf[tid];
    __syncthreads();
    pre[tid] = a;
    suf[tid] = b;
    __syncthreads();
  }
  if (tid == 0) inv_tot = fr_inv_mont(pre[LK_THREADS - 1]);
  __syncthreads();
  if (fr_is_zero(inv_tot)) {  // beta + t0 + j = 0 for some j, or a u_t = 0 (probability ~2^-238)
    if (tid == 0) atomicExch(&L->scr->status, VL_ELOOKUP);
    return;
  }
  // 1 / (this thread's total) = inv_tot . (the totals of the threads before) . (of those after)
  Fr inv = inv_tot;
  if (tid > 0) inv = mont_mul_ni(inv, pre[tid - 1]);
  if (tid + 1 < LK_THREADS) inv = mont_mul_ni(inv, suf[tid + 1]);
  unsigned long long bm[1][8];
#pragma unroll
  for (int l = 0; l < 8; l++) bm[0][l] = 0;
  for (int j = j1 - 1; j >= j0; j--) {
    x = fr_sub(x, fr_r1());
    const Fr b = mont_mul_ni(inv, L->Binv[j]);
    inv = mont_mul_ni(inv, x);
    const uint32_t m = L->counts[j];
    L->Binv[j] = b;
    L->WB[j] = b;
    L->Tb[j] = x;
    L->WM[j] = to_mont_ni(fr_small(m));
#pragma unroll
    for (int l = 0; l < 8; l++) bm[0][l] += (unsigned long long)b.v[l] * m;  // sum m <= 2^24
  }
  if (has_u) L->uinv[tid] = inv;
  const Fr s = block_sum_columns<1>(bm, red);
  if (tid == 0) L->part[(size_t)it.slot * LK_PART] = s;
}

// The tables of round 2 (entries of a table item): UB = (1 - r_1) B, VB = r_1 B.
// One product per entry (51 us for the 512 lookups of a 7B step) against two per
// pair: with S' left to round 3, round 2's pass went from 1068 us to 892.
__global__ void __launch_bounds__(LK_THREADS) lk_tables2_kernel(LkDev* Ls, const LkItem* items) {
  const LkItem it = items[blockIdx.x];
  LkDev* L = Ls + it.proof;
  if (!L->round2) return;
  const Fr r = L->r[0];
  for (int j = it.k0 + threadIdx.x; j < it.k1; j += LK_THREADS) {
    const Fr b = L->Binv[j], v = mont_mul_ni(r, b);
    L->VB[j] = v;
    L->UB[j] = fr_sub(b, v);
  }
}

// Shared memory of a transcript step.
struct LkShared {
  alignas(16) uint32_t msg[48];     // an absorb's message: three blocks
  alignas(16) uint32_t wk[3][68];   // schedule words
  alignas(16) uint32_t sq[8];       // state before a squeeze
  LkRun run;
  Fr s[LK_PART];                    // the round's sums (canonical): T0, Tinf, A0 | U0, Uinf / h, V0, Vinf
  Fr quad[4][3];                    // T, A, U, V as (value at 0, value at 1, leading coefficient)
  Fr g[4];                          // g(0..3), or the final evaluations (canonical)
  Fr r;
  Fr kc[2];                         // R^2 2^(L-t), R^3 2^(L-t) mod r
  alignas(16) unsigned long long red[32 * LK_MAX_WARPS];
};

// SHA256 of the three blocks in sh.msg: warp 0 (digest in every lane), with
// warps 1 to 3 in lk_absorb_help.
__device__ __forceinline__ ShaState lk_absorb_run(LkShared& sh) {
  named_sync(10, 128);
  ShaState st = sha_rounds_ni(sha_iv_state(), sha_load(sh.msg), sh.wk[0], 1);
  st = sha_rounds_ni(st, sha_load(sh.msg + 16), sh.wk[1], 4);
  return sha_rounds_ni(st, sha_load(sh.msg + 32), sh.wk[2], 7);
}
__device__ __forceinline__ void lk_absorb_help(LkShared& sh, int warp) {
  named_sync(10, 128);
  sha_sched_ni(sha_load(sh.msg + 16 * (warp - 1)), sh.wk[warp - 1], 1 + 3 * (warp - 1));
}
// The message S || label || x_0 .. x_{n-1} (n = 3 or 4: three blocks), by warp 0;
// x(i): element i in shared memory.
template <class X>
__device__ __forceinline__ void lk_absorb_words(LkShared& sh, uint32_t label, int n, X x) {
  for (int i = threadIdx.x & 31; i < 48; i += 32) {
    const int q = i - 8;
    uint32_t w = 0;
    if (q < 0) w = sh.run.St[i];
    else if (q <= 8 * n) {
      const uint32_t prev = q == 0 ? label << 24 : x((q - 1) >> 3).v[(q - 1) & 7];
      w = q < 8 * n ? __byte_perm(x(q >> 3).v[q & 7], prev, 0x7012) : (prev & 0xff000000u) | 0x00800000u;
    } else if (i == 47) w = (uint32_t)(33 + 32 * n) * 8u;
    sh.msg[i] = w;
  }
}

// The round polynomial of round t from the sums in sh.s, by warp 0: g(X) =
// E_X T(X) + A(X) + table side for X = 0..3 (three products deep: T(1), U(1)
// from the claims, then all products of the four values at once), into sh.g and
// the proof.  tj: the table round's number, <= 0 in a high round; qform: the
// first sum is Q with T(0) = 1 - r_1 (1 - r_1) Q (round 2).
__device__ void lk_step_g(const LkDev* L, LkShared& sh, int t, int tj, bool qform, vl_lookup_proof* out) {
  const int lane = threadIdx.x & 31;
  const bool jr = tj > 0;
  const Fr ut = L->u[t - 1], ui = L->uinv[t - 1], one = fr_small(1);
  const LkRun& R = sh.run;
  Fr t0 = t == 1 ? one : sh.s[0];
  if (qform) {
    const Fr r1 = L->r[0];
    t0 = fr_sub(one, mont_mul_ni(mont_mul_ni(r1, fr_sub(fr_r1(), r1)), t0));
  }
  // lanes 0, 1: T(1), U(1) = (claim - (1 - u) value(0)) / u; lane 2: U's leading coefficient times h
  const Fr v0 = lane == 0 ? t0 : lane == 1 ? (tj == 1 ? one : sh.s[3]) : fr_small(1u << (L->L - t));
  const Fr x = mont_mul_ni(lane < 2 ? fr_sub(fr_r1(), ut) : fr_r2(), v0);
  const Fr y = mont_mul_ni(lane < 2 ? ui : sh.s[4], lane < 2 ? fr_sub(lane == 0 ? R.Tc : R.Uc, x) : x);
  if (lane == 0) {
    sh.quad[0][0] = v0;
    sh.quad[0][1] = y;
    sh.quad[0][2] = sh.s[1];
    sh.quad[1][0] = sh.s[2];
    sh.quad[1][1] = fr_sub(R.Ac, sh.s[2]);
    sh.quad[1][2] = fr_zero();
  } else if (lane == 1) {
    sh.quad[2][0] = v0;
    sh.quad[2][1] = y;
  } else if (lane == 2) {
    sh.quad[2][2] = y;
  } else if (lane == 3) {
    sh.quad[3][0] = sh.s[5];
    sh.quad[3][1] = fr_sub(R.Vc, sh.s[5]);
    sh.quad[3][2] = sh.s[6];
  }
  __syncwarp();
  // lane 4 i + X: part i = T, A, U, V at X, by differences (q(X + 1) - q(X) = q(1) - q(0) + 2 X lead)
  const int i = (lane >> 2) & 3, X = lane & 3;
  Fr v = sh.quad[i][0], d = fr_sub(sh.quad[i][1], v);
  const Fr dd = fr_dbl(sh.quad[i][2]);
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const Fr vn = fr_add(v, d);
    if (e < X) v = vn;
    d = fr_add(d, dd);
  }
  const Fr p = mont_mul_ni(i == 0 ? R.E[X] : i == 2 ? R.F[X] : L->c_nd, v);
  const Fr tx = shfl_fr(p, X), ax = shfl_fr(v, 4 + X), ux = shfl_fr(p, 8 + X), vx = shfl_fr(p, 12 + X);
  const Fr g = fr_add(fr_add(tx, ax), jr ? fr_sub(ux, vx) : R.tabc);
  if (lane < 4) {
    sh.g[lane] = g;
    for (int l = 0; l < 8; l++) out->g[t - 1][lane].limb[l] = g.v[l];
  }
  __syncwarp();
}

// After the squeeze of r_t, one warp: the running claims T(r), A(r), U(r), V(r),
// the scalars of the next round.  Three products deep.
__device__ void lk_step_r(LkDev* L, LkShared& sh, int t) {
  const int lane = threadIdx.x & 31, i = lane & 3;
  LkRun& R = sh.run;
  const Fr r = sh.r, ut = L->u[t - 1], one = fr_r1();
  const bool tabvar = t > L->L - L->log2_n;
  // lanes 0..3: claim i = q0 + r (q1 - q0 - lead + r lead); lanes 4, 5: eqf(u, r) = u r + (1 - u)(1 - r);
  // lane 7: the next tabc
  Fr a = r, b = sh.quad[i][2];
  if (lane == 4) b = ut;
  if (lane == 5) a = fr_sub(one, r), b = fr_sub(one, ut);
  if (lane == 7) a = L->inv2, b = R.tabc;
  const Fr p = mont_mul_ni(a, b);
  const Fr ef = fr_add(shfl_fr(p, 4), shfl_fr(p, 5));
  const Fr q0 = sh.quad[i][0];
  Fr c = r, e = fr_add(fr_sub(fr_sub(sh.quad[i][1], q0), sh.quad[i][2]), p);
  if (lane == 4) c = R.ac, e = ef;
  if (lane == 5) c = R.fc, e = ef;
  const Fr w = mont_mul_ni(c, e);
  const Fr ac = shfl_fr(w, 4), fc = tabvar ? shfl_fr(w, 5) : R.fc;
  __syncwarp();
  if (lane < 4) {
    const Fr cl = fr_add(q0, w);
    if (lane == 0) R.Tc = cl;
    else if (lane == 1) R.Ac = cl;
    else if (tabvar) (lane == 2 ? R.Uc : R.Vc) = cl;
  }
  if (lane == 4) R.ac = ac;
  if (lane == 5) R.fc = fc;
  if (lane == 7) R.tabc = p;
  if (t == 2) {  // the weights of round 3's S'
    const Fr r1 = L->r[0], p11 = mont_mul_ni(r1, r);
    if (lane == 0) {
      L->w4[3] = p11;
      L->w4[2] = fr_sub(r1, p11);
      L->w4[1] = fr_sub(r, p11);
      L->w4[0] = fr_sub(fr_sub(one, r1), fr_sub(r, p11));
    }
  }
  // E_X, F_X of round t + 1: eqf(u, X) = (1 - u) + X (2 u - 1)
  if (t < L->L) {
    const Fr un = L->u[t], e0 = fr_sub(one, un), d = fr_sub(un, e0);
    Fr v = e0;
#pragma unroll
    for (int q = 0; q < 3; q++)
      if (q < i) v = fr_add(v, d);
    const Fr z = mont_mul_ni(lane < 4 ? ac : fc, v);
    if (lane < 4) R.E[lane] = z;
    else if (lane < 8) R.F[lane - 4] = z;
  }
  __syncwarp();
}

// Round 1's scalars and the table side's claims and cube sum, from the table
// kernel's partials (block-wide).
__device__ void lk_first_step(const LkDev* L, LkShared& sh) {
  Fr x[1] = {fr_zero()};
  for (int s = L->xbeg + threadIdx.x; s < L->xend; s += blockDim.x) x[0] = fr_add(x[0], L->part[(size_t)s * LK_PART]);
  block_sum_fr<1>(x, reinterpret_cast<Fr*>(sh.red));
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x, i = lane & 3;
    const Fr bm = x[0], ac = sh.run.ac, fc = sh.run.fc, one = fr_r1();
    if (L->L > 0) {
      const Fr u = L->u[0], e0 = fr_sub(one, u), d = fr_sub(u, e0);
      Fr v = e0;
#pragma unroll
      for (int q = 0; q < 3; q++)
        if (q < i) v = fr_add(v, d);
      const Fr z = mont_mul_ni(lane < 4 ? ac : fc, v);
      if (lane < 4) sh.run.E[lane] = z;
      else if (lane < 8) sh.run.F[lane - 4] = z;
    }
    if (lane == 0) {
      sh.run.Ac = bm;  // sum A = sum B m
      sh.run.Vc = bm;
      sh.run.tabc = mont_mul_ni(L->inv2, fr_sub(L->asq, bm));
    }
  }
  __syncthreads();
}

// Absorb the round message and squeeze r_t: warps 0 to 3; sh.run.St and sh.r
// are set for the block after its next barrier.
__device__ __forceinline__ void lk_transcript(LkDev* L, LkShared& sh, int warp, int t) {
  const int lane = threadIdx.x & 31;
  const bool tabvar = t > L->L - L->log2_n;
  if (warp == 0) {
    lk_absorb_words(sh, LBL_G, 3, [&](int i) -> const Fr& { return sh.g[i == 0 ? 0 : i + 1]; });  // g(0), g(2), g(3)
    ShaState st = lk_absorb_run(sh);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < 8; i++) sh.sq[i] = st.h[i];
    }
    named_sync(11, 64);
    st = sha_rounds_ni(sha_iv_state(), squeeze_lane_block(st.h), sh.wk[lane < 2 ? lane : 2], 1);
    if (lane == 2) {
#pragma unroll
      for (int i = 0; i < 8; i++) sh.run.St[i] = st.h[i];
    }
    // challenge_of on lanes 0, 1; in a table round lanes 2, 3 form r 2^(L-t), the
    // variable's share of T' (Tb[k] + toff), from the same digests at once
    if (tabvar) named_sync(12, 64);
    uint32_t d[8];
#pragma unroll
    for (int i = 0; i < 8; i++) d[i] = __shfl_sync(0xffffffffu, st.h[i], lane & 1);
    Fr half = fr_zero();
    if (lane < 2 || (tabvar && lane < 4))
      half = mont_mul_ni(digest_le(d), lane == 0 ? fr_r2() : lane == 1 ? fr_r3() : sh.kc[lane - 2]);
    const Fr r = fr_add(half, shfl_xor_fr(half, 1));
    if (lane == 0) {
      sh.r = r;
      L->r[t - 1] = r;
    }
    if (tabvar && lane == 2) sh.run.toff = fr_add(sh.run.toff, r);
  } else if (warp < 4) {
    lk_absorb_help(sh, warp);
    if (tabvar && warp == 2) {
      Fr x = lane == 0 ? fr_r2() : fr_r3();
      for (int i = 0; i < L->L - t; i++) x = fr_dbl(x);
      if (lane < 2) sh.kc[lane] = x;
      __syncwarp();
      named_arrive(12, 64);
    }
    if (warp == 1) {
      named_sync(11, 64);
      uint32_t S[8];
#pragma unroll
      for (int i = 0; i < 8; i++) S[i] = sh.sq[i];
      sha_sched_ni(squeeze_lane_block(S), sh.wk[lane < 2 ? lane : 2], 1);
    }
  }
}

__device__ __forceinline__ void lk_copy_run(LkRun* dst, const LkRun* src) {
  const uint4* a = reinterpret_cast<const uint4*>(src);
  uint4* b = reinterpret_cast<uint4*>(dst);
  for (int i = threadIdx.x; i < (int)(sizeof(LkRun) / 16); i += blockDim.x) b[i] = a[i];
}
static_assert(sizeof(LkRun) % 16 == 0, "copied by 16 bytes");

// Round t of one proof before its tail (one block each): the round
// polynomial from the partial sums, absorb, squeeze r_t, new claims.
__global__ void __launch_bounds__(LK_STEP_THREADS) lk_round_kernel(LkDev* Ls, int t, vl_lookup_proof* outs) {
  __shared__ LkShared sh;
  LkDev* L = Ls + blockIdx.x;
  if (t >= L->tail) return;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int tj = t - (L->L - L->log2_n);
  lk_copy_run(&sh.run, &L->run);
  __syncthreads();
  if (t == 1) lk_first_step(L, sh);
  // the items' partial sums (Montgomery): threads stride over the slots
  Fr acc[3], accb[4];
  for (int i = 0; i < 3; i++) acc[i] = fr_zero();
  for (int i = 0; i < 4; i++) accb[i] = fr_zero();
  for (int s = L->pbeg[t] + tid; s < L->pend[t]; s += blockDim.x) {
    const Fr* p = L->part + (size_t)s * LK_PART;
    for (int i = 0; i < 3; i++) acc[i] = fr_add(acc[i], p[i]);
    if (tj > 0)
      for (int i = 0; i < 4; i++) accb[i] = fr_add(accb[i], p[3 + i]);
  }
  unsigned long long col[4][8];
  {
    unsigned long long c3[3][8];
    for (int i = 0; i < 3; i++)
      for (int l = 0; l < 8; l++) c3[i][l] = acc[i].v[l];
    const Fr x = block_sum_columns<3>(c3, sh.red);
    if (tid < 3) sh.s[tid] = x;
  }
  if (tj > 0) {
    for (int i = 0; i < 4; i++)
      for (int l = 0; l < 8; l++) col[i][l] = accb[i].v[l];
    const Fr x = block_sum_columns<4>(col, sh.red + 32 * (LK_STEP_THREADS / 32));
    if (tid < 4) sh.s[3 + tid] = x;
  }
  __syncwarp();
  if (warp == 0) lk_step_g(L, sh, t, tj, t == 2, outs + blockIdx.x);
  lk_transcript(L, sh, warp, t);
  __syncthreads();
  if (warp == 0) lk_step_r(L, sh, t);
  __syncthreads();
  lk_copy_run(&L->run, &sh.run);
}

// The final evaluations (the last pair folded with r_L), absorb 'f', the
// proof.  Warps 0 to 3.
__device__ void lk_finish(LkDev* L, LkShared& sh, vl_lookup_proof* out) {
  for (int i = threadIdx.x; i < (VL_LOOKUP_MAX_LOG_D - L->L) * 32; i += blockDim.x)  // unused rounds
    out->g[L->L + i / 32][(i / 8) & 3].limb[i & 7] = 0u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, Lp = L->L;
  if (warp > 0) {
    if (warp < 4) lk_absorb_help(sh, warp);
    return;
  }
  if (lane < 4) {  // a, s, b, m
    Fr x0, x1 = fr_zero();
    const bool fold = lane < 2 ? Lp > 0 : L->log2_n > 0;
    if (lane < 2) {
      if (Lp <= 1) {
        const Fr* tab = lane == 0 ? L->Binv : L->Tb;
        x0 = tab[lk_table_index(*L, 0)];
        if (fold) x1 = tab[lk_table_index(*L, 1)];
      } else if (Lp == 2 && lane == 1) {  // rounds 1 and 2 leave S' unfolded
        const Fr r1 = L->r[0];
        x0 = lk_fold(L->Tb[lk_table_index(*L, 0)], L->Tb[lk_table_index(*L, 2)], r1);
        x1 = lk_fold(L->Tb[lk_table_index(*L, 1)], L->Tb[lk_table_index(*L, 3)], r1);
      } else {
        const Fr* v = lane == 0 ? L->VA : L->VS;
        x0 = v[0], x1 = v[1];
      }
    } else {
      const Fr* v = lane == 2 ? L->WB : L->WM;
      x0 = v[0];
      if (fold) x1 = v[1];
    }
    if (fold) x0 = lk_fold(x0, x1, L->r[Lp - 1]);
    if (lane == 1) x0 = fr_sub(x0, L->beta);
    x0 = from_mont_ni(x0);
    sh.g[lane] = x0;
    vl_fr* dst = lane == 0 ? &out->a_r : lane == 1 ? &out->s_r : lane == 2 ? &out->b_r : &out->m_r;
    for (int l = 0; l < 8; l++) dst->limb[l] = x0.v[l];
  }
  __syncwarp();
  lk_absorb_words(sh, LBL_F, 4, [&](int i) -> const Fr& { return sh.g[i]; });
  const ShaState st = lk_absorb_run(sh);
  if (lane == 0) {
    store_state(out->state, st);
    out->n = L->n;
    out->log2_d = Lp;
    out->log2_n = L->log2_n;
    out->t0 = L->t0;
    out->status = L->scr->status;
  }
}

// One block or cluster per proof: its rounds from L->tail on, each a pass over the pairs, a block reduction and the
// transcript step in this block, then the final evaluations and the proof.
// In a table round the first half of the warps take the A side's pairs, the
// second half the table side's.  Short rounds spread a pair over four lanes
// (one fold each, then one product and one product by f).  The last warp forms
// the claims and scalars of the next round, of 512 threads beside the pass of the
// others, of 128 before its share.
// In a cluster (CL) the rounds of at least LK_CL_PAIRS pairs are spread over its
// CTAs as in rounds_cluster (CTA c owns the entries k with (k / 8) mod CTAs = c);
// the first CTA makes the transcript steps and, alone, the rounds after those.
template <int THREADS, int MINB, bool CL>
__global__ void __launch_bounds__(THREADS, MINB) lk_tail_kernel(LkDev* Ls, vl_lookup_proof* outs) {
  __shared__ LkShared sh;
  __shared__ Fr part[CL ? RND_MAX_CTAS : 1][8];  // each CTA's sums of a spread round, in the first CTA
  const int C = CL ? (int)cluster_size() : 1, rank = CL ? (int)cluster_rank() : 0;
  const int proof = CL ? (int)blockIdx.x / C : (int)blockIdx.x;
  LkDev* L = Ls + proof;
  vl_lookup_proof* out = outs + proof;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NW = THREADS / 32, NP = THREADS >= 512 ? NW - 1 : NW;  // warps, of them in the passes
  lk_copy_run(&sh.run, &L->run);
  if (tid < 8 && L->tail > 1) sh.r.v[tid] = L->r[L->tail - 2].v[tid];
  __syncthreads();
  if (L->tail == 1 && L->L >= 1) lk_first_step(L, sh);
  if (CL) cluster_sync();  // every CTA has started: its shared memory may be written
  for (int t = L->tail; t <= L->L; t++) {
    const int h = 1 << (L->L - t);
    const bool spread = CL && h >= LK_CL_PAIRS;
    if (CL && !spread && rank > 0) return;
    const int own = spread ? h / C : h;  // this CTA's pairs
    auto pair = [&](int l) { return spread ? ((l >> 3) * C + rank) * 8 + (l & 7) : l; };
    const int tj = t - (L->L - L->log2_n);
    const bool jr = tj > 0;
    if (t > L->tail) {
      if (t == 3) {  // round 3 needs the weights that the step leaves
        if (warp == NW - 1 && rank == 0) lk_step_r(L, sh, t - 1);
        __syncthreads();
        if (spread) cluster_sync();
      } else if (warp == NW - 1 && rank == 0) {
        lk_step_r(L, sh, t - 1);
      }
    }
    const LkEq q(L, t);
    const Fr r = sh.r;
    const int na = jr ? NW / 2 : NP;  // warps of the A side
    const bool sideb = warp >= na;
    const int id = sideb ? tid - 32 * na : tid, nid = 32 * (sideb ? NP - na : na);
    const bool loop = 4 * own > 32 * (jr ? NP - na : na), qform = t == 2 && loop;
    if (loop) {
      unsigned long long a[32];
#pragma unroll
      for (int i = 0; i < 32; i++) a[i] = 0;
      if (warp >= NP) {
      } else if (!sideb) {
        LkSumA s;
        s.zero();
#pragma unroll 1
        for (int l = id; l < own; l += nid) {
          const int k = pair(l);
          Fr f = q.f_tab[k & q.f_mask];
          if (q.high) f = mont_mul_ni(f, q.hi_tab[k >> L->sE]);
          if (t == 1) lk_pair_a<0>(L, k, h, f, r, s);
          else if (t == 2) lk_pair_a<1>(L, k, h, f, r, s);
          else if (t == 3) lk_pair_a<2>(L, k, h, f, r, s);
          else lk_pair_a<3>(L, k, h, f, r, s);
        }
        unsigned long long col[3][8];
        s.columns(col);
#pragma unroll
        for (int i = 0; i < 24; i++) a[i] = col[i / 8][i % 8];
      } else {
        const Fr toff = sh.run.toff;
        LkSumB s;
        s.zero();
#pragma unroll 1
        for (int l = id; l < own; l += nid) {
          const int k = pair(l);
          Fr f = q.f_tab[k & q.f_mask];
          if (q.high) f = mont_mul_ni(f, q.hi_tab[k >> L->sE]);
          lk_pair_b(L, tj, k, h, f, r, toff, s);
        }
        unsigned long long col[4][8];
        s.columns(col);
#pragma unroll
        for (int i = 0; i < 32; i++) a[i] = col[i / 8][i % 8];
      }
      if (warp < NP) sh.red[32 * warp + lane] = warp_transpose_sum<32>(a);
      __syncthreads();
      if (warp == 0) {
        unsigned long long ta = 0, tb = 0;
        for (int w = 0; w < na; w++) ta += sh.red[32 * w + lane];
        for (int w = na; w < NP; w++) tb += sh.red[32 * w + lane];
        U64x8 col;
#pragma unroll
        for (int l = 0; l < 8; l++) {
          const int src = 8 * (lane & 3) + l;
          const unsigned long long ca = __shfl_sync(0xffffffffu, ta, src), cb = __shfl_sync(0xffffffffu, tb, src);
          col.v[l] = lane < 4 ? ca : cb;
        }
        const Fr x = redc_columns_ni(col);
        if (lane < 3) sh.s[lane] = x;
        else if (lane >= 4 && lane < 8) sh.s[lane - 1] = x;
      }
    } else {
      const int j = pair(id >> 2), qd = id & 3, at = j + (qd & 1) * h;
      const bool act = warp < NP && (id >> 2) < own;
      Fr p = fr_zero();
      if (warp < NP && ((id & ~31) >> 2) < own) {  // warps without a pair leave their slots to zeros
      Fr x = fr_zero(), x1 = fr_zero(), f = fr_zero(), u0 = fr_zero();
      bool fold = false;
      Fr* dst = nullptr;
      if (act) {
        f = q.f_tab[j & q.f_mask];
        if (q.high) f = mont_mul_ni(f, q.hi_tab[j >> L->sE]);
        if (!sideb && t <= 2) {
          const Fr* tab = qd < 2 ? L->Binv : L->Tb;
          x = tab[lk_table_index(*L, at)];
          fold = t == 2;
          if (fold) x1 = tab[lk_table_index(*L, at + 2 * h)];
          if (fold && qd < 2) dst = L->VA;  // S' is formed in round 3
        } else if (!sideb && t == 3 && qd >= 2) {
          x = lk_s_round3(L, at, L->L - 2);
          dst = L->VS;
        } else {
          Fr* v = sideb ? (qd < 2 ? L->WB : L->WM) : (qd < 2 ? L->VA : L->VS);
          x = v[at];
          fold = !sideb || tj > 1;
          if (fold) x1 = v[at + 2 * h], dst = v;
        }
        if (sideb) u0 = fr_add(L->Tb[j], sh.run.toff);
      }
      __syncwarp();
      if (t > 1 && (!sideb || tj > 1)) {
        const Fr fx = fr_add(x, mont_mul_ni(r, fr_sub(x1, x)));
        if (fold) x = fx;
      }
      if (dst) dst[at] = x;
      const Fr y = shfl_xor_fr(x, 1);
      const Fr z = (qd & 1) ? fr_sub(x, y) : x;  // A: a0, da, s0, ds; table: b0, db, m0, dm
      Fr w = shfl_xor_fr(z, 2);
      const Fr a0 = w;
      if (sideb && qd == 0) w = u0;
      if (sideb && qd == 1) w = f;
      p = mont_mul_ni(z, w);
      const Fr pf = mont_mul_ni(p, f);
      if (sideb ? qd == 0 : qd < 2) p = pf;
      if (!sideb && qd == 2) p = a0;
      if (!act || (!sideb && qd == 3)) p = fr_zero();
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) p = fr_add(p, shfl_xor_fr(p, off));
      }
      Fr* red = reinterpret_cast<Fr*>(sh.red);
      if (lane < 4 && warp < NP) red[4 * warp + lane] = p;
      __syncthreads();
      if (warp == 0) {
        Fr va = fr_zero(), vb = fr_zero();
        for (int w2 = lane >> 2; w2 < NP; w2 += 8) {
          const Fr v = red[4 * w2 + qd];
          if (w2 < na) va = fr_add(va, v);
          else vb = fr_add(vb, v);
        }
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
          va = fr_add(va, shfl_xor_fr(va, off));
          if (jr) vb = fr_add(vb, shfl_xor_fr(vb, off));
        }
        const Fr v = from_mont_ni(lane < 4 ? va : vb);
        if (lane < 3) sh.s[lane] = v;
        else if (lane >= 4 && lane < 8) sh.s[lane - 1] = v;
      }
    }
    __syncwarp();
    if (spread) {
      if (warp == 0 && lane < 7) {
#pragma unroll
        for (int l = 0; l < 8; l++) st_cluster(&part[rank][lane].v[l], 0, sh.s[lane].v[l]);
      }
      cluster_sync();
      if (rank == 0 && warp == 0) {
        // lane 8 (c mod 4) + q: value q of CTAs c, c + 4
        const int c = lane >> 3;
        Fr v = c < C ? part[c][lane & 7] : fr_zero();
        if (c + 4 < C) v = fr_add(v, part[c + 4][lane & 7]);
#pragma unroll
        for (int off = 8; off < 32; off <<= 1) v = fr_add(v, shfl_xor_fr(v, off));
        if (lane < 7) sh.s[lane] = v;
        __syncwarp();
      }
    }
    if (rank == 0) {
      if (warp == 0) lk_step_g(L, sh, t, tj, qform, out);
      lk_transcript(L, sh, warp, t);
    }
    if (spread && (h >> 1) >= LK_CL_PAIRS) {
      // the other CTAs need r_t and T''s offset
      if (rank == 0 && warp == 0) {
        __syncwarp();
        for (int i = lane; i < 8 * (C - 1); i += 32) {
          st_cluster(&sh.r.v[i & 7], 1 + (i >> 3), sh.r.v[i & 7]);
          st_cluster(&sh.run.toff.v[i & 7], 1 + (i >> 3), sh.run.toff.v[i & 7]);
        }
      }
      cluster_sync();
    }
    __syncthreads();  // r_t and the folded vectors are visible to the next round
  }
  if (rank == 0) lk_finish(L, sh, out);
}

}  // namespace

cudaError_t launch_lookup_setup(LkDev* Ls, int np, const LkItem* hist_items, int nhist, const LkItem* tab_items,
                                int ntab, cudaStream_t st) {
  lk_start_kernel<<<np, LK_THREADS, 0, st>>>(Ls);
  if (nhist) lk_hist_kernel<<<nhist, LK_THREADS, 0, st>>>(Ls, hist_items);
  if (ntab) lk_table_kernel<<<ntab, LK_THREADS, 0, st>>>(Ls, tab_items);
  return cudaGetLastError();
}

cudaError_t launch_lookup_tables2(LkDev* Ls, const LkItem* tab_items, int ntab, cudaStream_t st) {
  lk_tables2_kernel<<<ntab, LK_THREADS, 0, st>>>(Ls, tab_items);
  return cudaGetLastError();
}

cudaError_t launch_lookup_round(LkDev* Ls, int np, int t, const LkItem* items, int nhi, int nlo,
                                vl_lookup_proof* out, cudaStream_t st) {
  const cudaError_t e = launch_lookup_passes(Ls, t, items, nhi, nlo, st);
  if (e != cudaSuccess) return e;
  lk_round_kernel<<<np, LK_STEP_THREADS, 0, st>>>(Ls, t, out);
  return cudaGetLastError();
}

// A proof's tail is a chain of rounds: with SMs to spare it runs on a cluster of 8,
// 4 or 2 CTAs (one lookup of 512 x 16 remainders 423 -> 355 us, its tail now from
// 2^LK_TAIL_LOG_FEW pairs), with an SM for every proof on 512 threads, else on 128, four proofs per SM (one lookup of 512 x 16 remainders
// 0.98 -> 0.42 ms, the 512 of a 7B step 8.86 -> 3.69 ms with the other changes
// described in lookup_dev.cuh).
cudaError_t launch_lookup_finish(LkDev* Ls, int np, vl_lookup_proof* out, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int ctas = cluster_ctas(np, sms);
  if (ctas > 1) return launch_clusters(lk_tail_kernel<512, 1, true>, np, ctas, 512, 0, st, Ls, out);
  if (np <= sms) lk_tail_kernel<512, 1, false><<<np, 512, 0, st>>>(Ls, out);
  else lk_tail_kernel<128, 4, false><<<np, 128, 0, st>>>(Ls, out);
  return cudaGetLastError();
}

}  // namespace vl
