// Host arrays of the C ABI: what kind of memory one is, and the page writes
// ahead of a copy from the device.  Host code only.
#pragma once
#include <cuda_runtime.h>
#include <unistd.h>

// mapped: device address of an array in page-locked memory that the GPU can
// address (cudaHostAlloc / cudaHostRegister), or null; kernels then read or write
// it in place over the CPU-GPU link instead of going through a staging copy.
// plain: ordinary pageable memory, which the host may write to.  Neither: device
// or managed memory, an array that only part of is page-locked; the CUDA copy
// takes such a pointer or refuses it.
struct WbHostArray {
  void* mapped;
  bool plain;
};

// From the attributes of the first and the last element, span bytes apart.
inline WbHostArray wb_host_array_of(const cudaPointerAttributes& first, const cudaPointerAttributes& last, size_t span) {
  WbHostArray a = {nullptr, false};
  a.plain = first.type == cudaMemoryTypeUnregistered && last.type == cudaMemoryTypeUnregistered;
  if (first.type == cudaMemoryTypeHost && last.type == cudaMemoryTypeHost && first.devicePointer && last.devicePointer &&
      (size_t)(static_cast<char*>(last.devicePointer) - static_cast<char*>(first.devicePointer)) == span)
    a.mapped = first.devicePointer;
  return a;
}

// The array of n doubles at p (nothing of it is read or written).
inline WbHostArray wb_host_array(const void* p, long long n) {
  if (!p || n <= 0) return {nullptr, false};
  const size_t span = sizeof(double) * (size_t)(n - 1);
  cudaPointerAttributes first, last;
  if (cudaPointerGetAttributes(&first, p) != cudaSuccess ||
      cudaPointerGetAttributes(&last, static_cast<const char*>(p) + span) != cudaSuccess) {
    cudaGetLastError();
    return {nullptr, false};
  }
  return wb_host_array_of(first, last, span);
}

// Brings in the pages of a host buffer that a copy from the device is about to
// fill.  The copy writes pageable memory in place over the CPU-GPU link, and a
// page nobody has written yet then costs a fault taken from the GPU: 129 MB into
// fresh arrays took 37 to 49 ms (64 KB pages), into written ones 3.1; writing
// to each page here costs 3.9.  (Reading a page first maps the zero page, and the
// write after it is as slow as the GPU's fault.)
inline void wb_touch_pages(void* p, size_t bytes) {
  const long page = sysconf(_SC_PAGESIZE);
  if (page <= 0 || !bytes) return;
  volatile char* c = static_cast<volatile char*>(p);
  for (size_t at = 0; at < bytes; at += (size_t)page) c[at] = 0;
  c[bytes - 1] = 0;
}

// Whether everything enqueued on s so far is done (false: unknown).
inline bool wb_stream_idle(cudaStream_t s) {
  if (cudaPeekAtLastError() != cudaSuccess) return false;  // an earlier error is the caller's to see
  const cudaError_t e = cudaStreamQuery(s);
  if (e == cudaErrorNotReady) cudaGetLastError();
  return e == cudaSuccess;
}

// The same ahead of a copy on stream s, in the stream's order: work enqueued
// earlier may still read the buffer (a copy out of it, a host function), so unless
// the stream was idle before this call enqueued anything (*idle; what the call
// enqueues uses no other of the caller's arrays) it is waited for first.
inline cudaError_t wb_touch_in_order(void* p, size_t bytes, cudaStream_t s, bool* idle) {
  if (!*idle) {
    const cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    *idle = true;
  }
  wb_touch_pages(p, bytes);
  return cudaSuccess;
}
