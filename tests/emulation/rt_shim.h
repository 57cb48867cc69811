// Host stand-ins for the CUDA runtime calls the library's host code makes, and the launch of
// a kernel as blocks of host threads (one cluster after another).
#pragma once
#include "shim.h"
typedef int cudaError_t;
enum : int { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2 };
typedef void* cudaStream_t;
typedef void* cudaEvent_t;
enum cudaDeviceAttr { cudaDevAttrMultiProcessorCount = 16, cudaDevAttrMaxSharedMemoryPerBlockOptin = 97 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
#define cudaStreamNonBlocking 1u
#define cudaEventDisableTiming 2u
inline cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
inline cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  const char* sms = getenv("EMU_SMS");   // another number of SMs than GB300's, for clusters of few blocks
  *v = a == cudaDevAttrMultiProcessorCount ? (sms ? atoi(sms) : 152) : 232448;
  return cudaSuccess;
}
inline cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t = nullptr) {
  std::memset(p, v, n);
  return cudaSuccess;
}
inline cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t = nullptr) { return cudaSuccess; }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned = 0) { return cudaSuccess; }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (void*)1; return cudaSuccess; }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (void*)1; return cudaSuccess; }

// Shared memory is filled with 0xff bytes (NaN in either float type), so a read before the
// kernel writes shows up in the results.
template <class P>
void emu_launch_clusters(void (*kernel)(const P), int count, int blocks, size_t smem, const P& params) {
  constexpr int kThreads = 512;
  for (int c = 0; c < count; ++c) {
    std::barrier<> cluster(kThreads * blocks);
    std::vector<EmuBlock> blk(blocks);
    std::vector<void*> dyn(blocks);
    for (int r = 0; r < blocks; ++r) {
      blk[r].cluster = &cluster;
      blk[r].block = std::make_unique<std::barrier<>>(kThreads);
      for (int w = 0; w < 32; ++w) blk[r].warp[w] = std::make_unique<std::barrier<>>(32);
      if (posix_memalign(&dyn[r], 128, smem ? smem : 16) != 0) abort();
      std::memset(dyn[r], 0xff, smem ? smem : 16);
    }
    std::vector<std::thread> th;
    for (int r = 0; r < blocks; ++r)
      for (int t = 0; t < kThreads; ++t)
        th.emplace_back([&, r, t, c] {
          emu_blk = &blk[r];
          emu_dyn_smem = (unsigned char*)dyn[r];
          threadIdx.x = t;
          blockIdx.x = c * blocks + r;
          kernel(params);
          emu_blk->warp[t >> 5]->arrive_and_drop();
          emu_blk->block->arrive_and_drop();
          cluster.arrive_and_drop();
        });
    for (auto& x : th) x.join();
    for (void* p : dyn) free(p);
  }
}
template <class P>
void emu_launch(void (*kernel)(const P), int grid, size_t smem, const P& params) {
  emu_launch_clusters(kernel, grid, 1, smem, params);
}
