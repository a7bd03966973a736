// Launches of the library's objects on two devices of one process, linked against a model of the CUDA runtime that keeps
// the shared-memory opt-in of a kernel per device, as the runtime does: a launch beyond 48 KB fails where the
// device has not been told. exit status 0 and "ok" if every launch is allowed
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

#include "fs_engine.h"

#ifndef __CUDA_ARCH__  // (host code only)
namespace {
int device = 0, launches = 0, refused = 0, big = 0;
std::map<std::pair<int, const void*>, size_t> allowed;
struct Config { dim3 grid, block; size_t smem; cudaStream_t stream; };
std::vector<Config> config;
cudaError_t launch(const void* f, size_t smem) {
  launches++;
  if (smem > 48 * 1024) {
    big++;
    auto it = allowed.find({device, f});
    if (it == allowed.end() || it->second < smem) {
      refused++;
      printf("device %d: a launch with %zu bytes of shared memory, not opted in\n", device, smem);
      return cudaErrorInvalidValue;
    }
  }
  return cudaSuccess;
}
}  // namespace

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
char __cudaInitModule(void**) { return 1; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  config.push_back({g, b, smem, s});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  const Config c = config.back();
  config.pop_back();
  *g = c.grid; *b = c.block; *smem = c.smem; *(cudaStream_t*)s = c.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  allowed[{device, f}] = (size_t)v;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaMalloc(void** p, size_t) { *p = malloc(16); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t, cudaStream_t) { *p = malloc(16); return cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}

int main() {
  using namespace fs;
  int failed = 0;
  for (device = 0; device < 2; device++)
    for (int lt : {4, 64, 256}) {  // the cluster kernel's lattices, the tile kernels'
      Ctx c;
      c.device = device;
      c.nsm = 152;
      c.g.L[0] = c.g.L[1] = c.g.L[2] = 4;
      c.g.L[3] = lt;
      c.g.Lh0 = 2;
      c.g.Vh = 32 * lt;
      c.g.V = 64 * lt;
      c.stream = (cudaStream_t)16;
      if (lt == 256) {  // 16384 sites
        c.g.L[0] = 8;
        c.g.Lh0 = 4;
        c.g.Vh *= 2;
        c.g.V *= 2;
      }
      for (int prec : {PREC_F64, PREC_F32, PREC_F16, PREC_BF16})
        for (int N : {2, 8, 16, 32}) {
          TileBase* T = c.tile(prec, N, 18);
          if (!T || T->enqueue_init() || T->enqueue_iters(1) || T->enqueue_recon()) failed++;
        }
      std::vector<ContractPair> pairs;
      for (int k = 0; k < 4; k++) pairs.push_back(ContractPair{0, k, 0, k});
      std::vector<double> gamma(32, 0.0), result;
      gamma[0] = 1.0;
      if (contract_tile(&c, c.tile(PREC_F64, 8, 18), pairs, gamma.data(), {0}, result, 4)) failed++;
    }
  printf("%d launches, %d beyond 48 KB, %d refused\n", launches, big, refused);
  const bool ok = failed == 0 && refused == 0 && big > 0;
  printf("%s\n", ok ? "ok" : "failed");
  return ok ? 0 : 1;
}
#endif
