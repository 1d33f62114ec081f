// Shared definitions of the GB300 LOBPCG library (device and host side).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include <cstdio>
#include <string>

#include "../../include/lobpcg.h"

#define LOBPCG_EXPORT extern "C" __attribute__((visibility("default")))

namespace lob {

constexpr int kMaxSeg = 4;

__host__ __device__ inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
inline int64_t round_up(int64_t a, int64_t b) { return ceil_div(a, b) * b; }

// A row-major block presented as up to kMaxSeg column segments, each with its
// own base pointer and leading dimension: S = [X, P, W] without copies.
struct SegList {
  const double* ptr[kMaxSeg];
  int64_t ld[kMaxSeg];
  int off[kMaxSeg + 1];  // prefix sums of segment widths; off[nseg] = total columns
  int nseg;
};

inline SegList seg1(const double* p, int64_t ld, int cols) {
  SegList s{};
  s.ptr[0] = p; s.ld[0] = ld; s.off[0] = 0; s.off[1] = cols; s.nseg = 1;
  for (int i = 2; i <= kMaxSeg; ++i) s.off[i] = cols;
  return s;
}

inline void seg_push(SegList& s, const double* p, int64_t ld, int cols) {
  if (cols <= 0) return;
  s.ptr[s.nseg] = p; s.ld[s.nseg] = ld;
  s.off[s.nseg + 1] = s.off[s.nseg] + cols;
  s.nseg++;
  for (int i = s.nseg + 1; i <= kMaxSeg; ++i) s.off[i] = s.off[s.nseg];
}

inline SegList seg_empty() {
  SegList s{};
  s.nseg = 0;
  return s;
}

__device__ __forceinline__ double seg_load(const SegList& s, int c, int64_t row) {
  int i = 0;
#pragma unroll
  for (int t = 1; t < kMaxSeg; ++t) i += (t < s.nseg && c >= s.off[t]) ? 1 : 0;
  return s.ptr[i][row * s.ld[i] + (c - s.off[i])];
}

// Output block split into up to two destinations by column (e.g. [X_new, P_new]).
struct OutList {
  double* ptr[2];
  int64_t ld[2];
  int split;  // columns < split go to ptr[0], the rest to ptr[1]
};

__device__ __forceinline__ double* out_addr(const OutList& o, int c, int64_t row) {
  return c < o.split ? o.ptr[0] + row * o.ld[0] + c : o.ptr[1] + row * o.ld[1] + (c - o.split);
}

// Device scratch in stream order from this library's pool (scratch.cu).
int scratch_alloc(void** p, size_t bytes, cudaStream_t st);
void scratch_free(void* p, cudaStream_t st);
void scratch_trim(int device);  // the memory kept on a device goes back

// Launches that follow one another on a stream without the gap of a full
// completion (programmatic dependent launch): the next kernel's CTAs take their
// places while this one runs and wait in chain_wait(), which every thread of a
// chained kernel calls before its first access to memory (and before any
// return, so that a kernel's end implies the end of all before it).  Such
// kernels take their inputs by plain pointers, without __restrict__ or __ldg:
// loads of data declared constant need not stay behind the wait.  A solver
// iteration has about 80 small kernels, each of which otherwise pays a launch
// gap of its own length: 32 x 32 solve 60.4 -> 55.0 ms, 48 x 40 x 36 solve 150 ->
// 120 ms, syev of order 213 1.13 -> 1.07 ms.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t shared,
                           cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = shared;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Kernel launch counter (host side, per process) used for the stats.
extern int64_t g_launches;

}  // namespace lob

#define LOB_CUDA_OK(expr)                                  \
  do {                                                     \
    cudaError_t _e = (expr);                               \
    if (_e != cudaSuccess) return LOBPCG_ERR_CUDA;         \
  } while (0)

#define LOB_LAUNCHED()                                     \
  do {                                                     \
    ++lob::g_launches;                                     \
    if (cudaPeekAtLastError() != cudaSuccess) return LOBPCG_ERR_CUDA; \
  } while (0)
