// Per-kernel launch statistics of a context: a launch counter that is always on, and, while
// profiling is enabled, CUDA events around every launch on the launching stream together
// with the launch's algorithmic bytes (operands read once, results written once) and flops.
#ifndef PV_PROF_CUH
#define PV_PROF_CUH
#include <cuda_runtime.h>
#include <utility>
#include <cstring>
#include <string>
#include <vector>

namespace pv {

struct KProf {
  struct Rec {
    const char* name;
    double bytes, flops;
  };
  struct Acc {
    std::string name;
    long long launches = 0;
    double ms = 0, bytes = 0, flops = 0;
  };
  bool on = false;
  bool gemm_only = false;   // time only the batched GEMM kernels (names kb_gemm*)
  long long launches = 0;
  std::vector<cudaEvent_t> pool;
  size_t used = 0;
  std::vector<Rec> recs;
  std::vector<Acc> acc;

  ~KProf() {
    for (cudaEvent_t e : pool) cudaEventDestroy(e);
  }
  bool wanted(const char* name) const {
    return on && (!gemm_only || strncmp(name, "kb_gemm", 7) == 0);
  }
  void begin(cudaStream_t st, const char* name) {
    ++launches;
    if (!wanted(name)) return;
    if (used + 2 > pool.size()) {
      for (int i = 0; i < 4096; ++i) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) {
          cudaGetLastError();
          on = false;
          return;
        }
        pool.push_back(e);
      }
    }
    cudaEventRecord(pool[used], st);
  }
  void end(cudaStream_t st, const char* name, double bytes, double flops) {
    if (!wanted(name) || used + 2 > pool.size()) return;
    cudaEventRecord(pool[used + 1], st);
    used += 2;
    recs.push_back(Rec{name, bytes, flops});
  }
  // Folds the recorded launches into the per-kernel sums; the caller has synchronised.
  void fold() {
    for (size_t i = 0; i < recs.size(); ++i) {
      float ms = 0;
      cudaEventElapsedTime(&ms, pool[2 * i], pool[2 * i + 1]);
      Acc* a = nullptr;
      for (Acc& x : acc)
        if (x.name == recs[i].name) a = &x;
      if (!a) {
        acc.push_back(Acc());
        a = &acc.back();
        a->name = recs[i].name;
      }
      a->launches += 1;
      a->ms += ms;
      a->bytes += recs[i].bytes;
      a->flops += recs[i].flops;
    }
    recs.clear();
    used = 0;
  }
  void reset() {
    recs.clear();
    used = 0;
    acc.clear();
  }
};

// Programmatic dependent launch: the batched engine is thousands of short kernels in a row, and a
// kernel's launch, its index tables and its tensor-memory allocation need nothing of the one before.
// A kernel launched with pdl() may start while its predecessor in the stream ends, and calls pdl_wait()
// before its first access to device memory (the wait covers the predecessor's completion and its writes,
// and, as the predecessor waited itself, everything before).  pdl_go() lets the successor start;
// a kernel that allocates tensor memory calls it only when it holds its columns (a successor's
// block that took them first would wait for this kernel's end).  Launched without pdl() both do
// nothing.
#if defined(__CUDACC__)
// Lets a kernel that is about to be launched with `bytes` of dynamic shared memory have more than the
// default 48 KB (its static arrays, a few hundred bytes, included): up to `cap`, the same for every
// caller, so that no context lowers it under another.  Set where the kernel is launched, since the
// attribute loads the kernel's code: forty of them set by the first context took it 17 of 49 ms.
template <typename K>
inline void smem_cap(K kern, size_t bytes, int cap) {
  if (bytes > 44 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline void pdl_if(bool early, void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A&&... a) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = at;
  c.numAttrs = early ? 1 : 0;
  cudaLaunchKernelEx(&c, kern, P(a)...);
}
template <typename... P, typename... A>
inline void pdl(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A&&... a) {
  pdl_if(true, kern, grid, threads, smem, st, std::forward<A>(a)...);
}
#endif

// Brackets one launch statement: counts it and, when profiling, times it.
#define PV_KLAUNCH(prof, st, name, bytes, flops, ...) \
  do {                                                \
    if (prof) (prof)->begin(st, name);                \
    __VA_ARGS__;                                      \
    if (prof) (prof)->end(st, name, bytes, flops);    \
  } while (0)

}  // namespace pv
#endif
