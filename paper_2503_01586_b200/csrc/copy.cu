// Copy between device memory and pinned host memory by a kernel.
//
// A decode step that starts and ends in host memory is a copy in, three kernels and a copy out.  As
// copy-engine operations the two copies cost about 6 us of hand-over each way beside their 1.5 and
// 3.5 us; as kernels they are links of the chain of programmatic dependent launches.
// A 7B step from host arrays to a host result, with copy-engine copies and with these: B1
// 45.6 -> 39.3 us, B16 82.7 -> 72.7, B64 (0.8 MB in, 0.5 MB out) 205 -> 186.
#include "common.cuh"
#include "copy.cuh"

namespace {

constexpr int kCopyThreads = 256;
constexpr int kCopyBatch = 4;        // 16-byte requests of a thread in flight

__global__ void __launch_bounds__(kCopyThreads)
copy_kernel(unsigned char* dst, const unsigned char* src, long long bytes) {
  ekv_pdl_trigger();
  ekv_pdl_wait();       // src may be an earlier kernel's output, dst its input
  const long long n = bytes >> 4, step = (long long)gridDim.x * kCopyThreads;
  const long long t = (long long)blockIdx.x * kCopyThreads + threadIdx.x;
  for (long long i = t; i < n; i += kCopyBatch * step) {
    uint4 v[kCopyBatch];
#pragma unroll
    for (int k = 0; k < kCopyBatch; ++k)
      if (i + k * step < n) v[k] = __ldcv((const uint4*)src + i + k * step);
#pragma unroll
    for (int k = 0; k < kCopyBatch; ++k)
      if (i + k * step < n) ((uint4*)dst)[i + k * step] = v[k];
  }
  if (t < (bytes & 15)) dst[(n << 4) + t] = __ldcv(src + (n << 4) + t);
}

bool device_reads(const void* p, int device) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return ekv_addressable(at, p, device);
}

}  // namespace

extern "C" int elitekv_copy(void* dst, const void* src, int64_t bytes, elitekv_stream_t stream) {
  if (!dst || !src || bytes < 0 || (((uintptr_t)dst | (uintptr_t)src) & 15)) return ELITEKV_ERR_INVALID_ARG;
  int device = 0;
  EKV_CUDA_OK(cudaGetDevice(&device));
  if (!device_reads(dst, device) || !device_reads(src, device)) return ELITEKV_ERR_INVALID_ARG;
  if (bytes == 0) return ELITEKV_OK;
  const long long per_block = 16ll * kCopyThreads;
  long long blocks = (bytes + per_block - 1) / per_block;
  if (blocks > 512) blocks = 512;
  EKV_CUDA_OK(ekv_launch_pdl(copy_kernel, dim3((unsigned)blocks), dim3(kCopyThreads), 0, (cudaStream_t)stream,
                             (unsigned char*)dst, (const unsigned char*)src, (long long)bytes));
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}
