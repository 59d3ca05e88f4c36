// common.cuh -- shared definitions of the CUDA path (device helpers, status
// bits, workspace layout structs). Nothing here is shared with the CPU oracle.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#define MOND_HD __host__ __device__ __forceinline__

// Device status bits, OR-ed into a word in the workspace and read at
// synchronising calls.
enum : uint32_t {
  ST_DOMAIN = 1u,    // particle cell/offset outside the domain (skipped)
  ST_NAN = 2u,       // non-finite value in a field or particle
  ST_TIMEOUT = 4u,   // a bounded device wait gave up
  ST_OVERFLOW = 8u,  // fixed-point bound violated
};

// ---------------------------------------------------------------------------
// Early launches. A kernel launched by launch_early is started, where it
// follows another kernel in its stream, as that one's last CTAs leave, ahead of
// the write-back and the bookkeeping between two kernels (about 2 us of a
// stream launch); its tables are read meanwhile. Before kernel_wait, which
// returns when the kernel before has completed with its writes visible,
// nothing that an earlier kernel writes is read and nothing is written. What
// others write is read after the wait by plain loads, or through a pointer from
// after_wait: the compiler may move read-only loads and __ldcs, whose assembly
// it does not take for a memory access, past the wait. Every thread waits, so a
// completed kernel implies that all before it have completed. After a copy, a
// memset or an event a launch waits as any other.
// Solve at 96^3: 290 -> 222 us; force step at 64^3, 1e4 particles: 284 -> 181
// us, at 192^3, 4e5 particles: 1.91 -> 1.80 ms; surrogate: inference 64^3 ->
// 256^3 (34 launches) 581 -> 501 us, training step at 32^3 1.66 -> 1.49 ms. A
// graph's kernels follow each other as closely without it (no change). Letting
// the next kernel in when the first has started (launch_dependents) was slower:
// 250 us, 260 us, 1.86 ms, and 7% with eight systems side by side.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void kernel_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename T>
__device__ __forceinline__ T* after_wait(T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
template <typename... P, typename... A>
cudaError_t launch_early(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... a) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(a)...);
}

// ---------------------------------------------------------------------------
// Complex arithmetic on float2 (x = real, y = imaginary).
// ---------------------------------------------------------------------------
// The sums are one packed instruction on both parts (each rounded as the
// scalar ones): a fifth fewer instructions in a transform. 256^3: x-passes 2%,
// potential's inverse x-pass 5%, staged final z-pass 1%; 512^3 z-passes 5%.
__device__ __forceinline__ uint64_t pack2(float2 a) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// a * (DIR * i): DIR = -1 gives a * (-i), DIR = +1 gives a * i
template <int DIR>
__device__ __forceinline__ float2 cmul_i(float2 a) {
  return DIR < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
}
// e^{DIR * i * theta} from the table entry (cos theta, sin theta)
template <int DIR>
__device__ __forceinline__ float2 twid(float2 t) {
  return DIR < 0 ? make_float2(t.x, -t.y) : t;
}

// signed frequency of index i on an axis of length n (Nyquist n/2 -> -n/2)
MOND_HD int freq_of(int i, int n) { return i < (n + 1) / 2 ? i : i - n; }

__device__ __forceinline__ int wrapi(int i, int n) {
  int r = i % n;
  return r < 0 ? r + n : r;
}

__device__ __forceinline__ void set_status(uint32_t* st, uint32_t bit) { atomicOr(st, bit); }
