// Kernel launches that the runtime refuses, on call: loaded with its symbols global ahead of a library, this takes
// the place of the runtime's two launch entries and passes every launch on, the chosen one with more shared memory
// than any GPU has, so that the runtime turns it down (nothing reaches the GPU) and leaves its error as ever.  It
// also counts the shared-memory limits that were set to another value than before, and the graphs made.
#include <cuda_runtime_api.h>
#include <dlfcn.h>

#include <map>

static int countdown = -1, seen = 0, changed = 0, graphs = 0;
static std::map<const void *, int> limits;

static size_t smem_of(size_t asked) {
  ++seen;
  return countdown >= 0 && countdown-- == 0 ? (size_t)1 << 30 : asked;
}
static void *real(const char *name) {
  static void *rt = dlopen("libcudart.so.13", RTLD_LAZY);
  return dlsym(rt, name);
}

extern "C" {

// Refuse launch n (from 0) of those that follow; n < 0: none.
void refuse_launch(int n) {
  countdown = n;
  seen = 0;
}
int launches_seen() { return seen; }
int limits_changed() { return changed; }
int graphs_made() { return graphs; }

cudaError_t cudaGraphInstantiate(cudaGraphExec_t *ex, cudaGraph_t g, unsigned long long flags) {
  static auto f = (cudaError_t(*)(cudaGraphExec_t *, cudaGraph_t, unsigned long long))real("cudaGraphInstantiate");
  ++graphs;
  return f(ex, g, flags);
}

cudaError_t cudaFuncSetAttribute(const void *k, cudaFuncAttribute what, int value) {
  static auto f = (cudaError_t(*)(const void *, cudaFuncAttribute, int))real("cudaFuncSetAttribute");
  if (what == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    const auto it = limits.emplace(k, value).first;
    changed += it->second != value;
    it->second = value;
  }
  return f(k, what, value);
}

cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t st) {
  static auto f = (cudaError_t(*)(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t))real("__cudaLaunchKernel");
  return f(k, grid, block, args, smem_of(smem), st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *k, void **args) {
  static auto f = (cudaError_t(*)(const cudaLaunchConfig_t *, const void *, void **))real("cudaLaunchKernelExC");
  cudaLaunchConfig_t c = *cfg;
  c.dynamicSmemBytes = smem_of(c.dynamicSmemBytes);
  return f(&c, k, args);
}

}  // extern "C"
