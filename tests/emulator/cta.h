// Runs device code of a few thread blocks on the CPU, one fibre per CUDA thread,
// in an order that the caller chooses: a warp runs only while every warp ahead of
// it in the order waits at a barrier or has left.  What a kernel orders by time
// alone (a value read after a barrier and written again by a warp that no longer
// meets the reader) comes out wrong under the order that puts the reader last.
//
// Waiting is what the hardware's barriers make it: named barriers count threads
// (bar.sync arrives and waits, bar.arrive only arrives), a shuffle or __syncwarp
// is a meeting of the warp's 32 lanes, a cluster barrier one of all blocks.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <ucontext.h>

#include <functional>
#include <memory>
#include <vector>

namespace emu {

struct Barrier {
  int arrived = 0, phase = 0;
  void arrive(int n) {
    if (++arrived == n) arrived = 0, phase++;
  }
};
struct Warp {
  Barrier meet;
  uint32_t slot[2][32];
};
struct Fibre {
  ucontext_t ctx;
  std::unique_ptr<char[]> stack;
  const int* phase = nullptr;  // blocked while *phase == seen
  int seen = 0, cta = 0, tid = 0;
  bool done = false;
};

struct Machine {
  int ctas, threads;
  std::vector<Fibre> fibres;
  std::vector<Warp> warps;         // cta-major
  std::vector<Barrier> named;      // 16 per block
  Barrier cluster;
  ucontext_t scheduler;
  Fibre* now = nullptr;
  std::function<void()> body;

  void block(const int* phase, int seen) {
    if (*phase != seen) return;
    now->phase = phase, now->seen = seen;
    Fibre* self = now;
    swapcontext(&self->ctx, &scheduler);
  }
  void sync(Barrier& b, int n) {
    const int seen = b.phase;
    b.arrive(n);
    block(&b.phase, seen);
  }
  Warp& warp() { return warps[now->cta * (threads / 32) + now->tid / 32]; }
  uint32_t shuffle(uint32_t v, int src) {
    Warp& w = warp();
    const int par = w.meet.phase & 1;
    w.slot[par][now->tid & 31] = v;
    sync(w.meet, 32);
    return w.slot[par][src & 31];
  }
  // order: every warp (block-major index) once.  False: all warps that are left wait.
  bool run(int n_ctas, int n_threads, const int* order, std::function<void()> f);
};
inline Machine* machine = nullptr;

inline void entry() {
  machine->body();
  machine->now->done = true;
  swapcontext(&machine->now->ctx, &machine->scheduler);
}

inline bool Machine::run(int n_ctas, int n_threads, const int* order, std::function<void()> f) {
  machine = this;
  ctas = n_ctas, threads = n_threads, body = std::move(f);
  const int nw = ctas * threads / 32;
  constexpr size_t STACK = 48 << 10;
  fibres = std::vector<Fibre>(ctas * threads);
  warps = std::vector<Warp>(nw);
  named = std::vector<Barrier>(16 * ctas);
  cluster = Barrier();
  for (int i = 0; i < ctas * threads; i++) {
    Fibre& x = fibres[i];
    x.cta = i / threads, x.tid = i % threads;
    x.stack.reset(new char[STACK]);
    getcontext(&x.ctx);
    x.ctx.uc_stack.ss_sp = x.stack.get();
    x.ctx.uc_stack.ss_size = STACK;
    makecontext(&x.ctx, entry, 0);
  }
  for (size_t left = fibres.size(); left > 0;) {
    bool ran = false;
    for (int q = 0; q < nw && !ran; q++)
      for (int lane = 0; lane < 32; lane++) {
        Fibre& x = fibres[32 * order[q] + lane];
        if (x.done || (x.phase && *x.phase == x.seen)) continue;
        x.phase = nullptr;
        now = &x;
        swapcontext(&scheduler, &x.ctx);
        ran = true;
        if (x.done) left--;
      }
    if (!ran) return false;
  }
  return true;
}

struct Dim {
  struct X {
    int (*get)();
    operator int() const { return get(); }
  } x;
};

inline void bar_sync(int id, int n) { machine->sync(machine->named[16 * machine->now->cta + id], n); }
inline void bar_arrive(int id, int n) { machine->named[16 * machine->now->cta + id].arrive(n); }
inline void cluster_sync() { machine->sync(machine->cluster, machine->ctas * machine->threads); }
inline uint32_t cluster_rank() { return machine->now->cta; }
inline uint32_t cluster_size() { return machine->ctas; }

}  // namespace emu

#ifndef __noinline__
#define __noinline__ __attribute__((noinline))
#endif

namespace vl {
inline const emu::Dim threadIdx{{[] { return emu::machine->now->tid; }}};
inline const emu::Dim blockDim{{[] { return emu::machine->threads; }}};
}  // namespace vl

inline uint32_t __shfl_sync(uint32_t, uint32_t v, int src) { return emu::machine->shuffle(v, src); }
inline uint32_t __shfl_xor_sync(uint32_t, uint32_t v, int m) {
  return emu::machine->shuffle(v, (emu::machine->now->tid & 31) ^ m);
}
inline unsigned long long __shfl_sync(uint32_t m, unsigned long long v, int src) {
  const uint32_t lo = __shfl_sync(m, (uint32_t)v, src), hi = __shfl_sync(m, (uint32_t)(v >> 32), src);
  return lo | ((unsigned long long)hi << 32);
}
inline unsigned long long __shfl_xor_sync(uint32_t m, unsigned long long v, int x) {
  return __shfl_sync(m, v, (emu::machine->now->tid & 31) ^ x);
}
inline void __syncwarp() { emu::machine->sync(emu::machine->warp().meet, 32); }
inline void __syncthreads() { emu::bar_sync(0, emu::machine->threads); }
inline uint32_t __byte_perm(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t out = 0;
  for (int i = 0; i < 4; i++) {
    const int s = (sel >> (4 * i)) & 7;
    out |= ((s < 4 ? a >> (8 * s) : b >> (8 * (s - 4))) & 255u) << (8 * i);
  }
  return out;
}
inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t n) {
  return (uint32_t)((((unsigned long long)hi << 32) | lo) >> (n & 31));
}
