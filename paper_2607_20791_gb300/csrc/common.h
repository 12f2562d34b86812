// Host-side helpers shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstdarg>
#include <cstdint>
#include <cstdio>

#include "rgd.h"

namespace rgd {

// Sets the calling thread's error string and returns `code`.
int set_error(int code, const char* fmt, ...);
void clear_error();

inline int cuda_error(cudaError_t e, const char* what) {
  return set_error(RGD_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Launches a kernel as a programmatic dependent of the previous kernel on the
// stream: it is scheduled while that kernel finishes, and waits for it
// (griddepcontrol.wait) before it reads or writes memory.
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), int grid, int block, int smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

constexpr int kMaxDevices = 64;  // devices whose state is kept (others are asked on every call)

// Opts a kernel into `bytes` of dynamic shared memory on the current device (the
// attribute is a device's own), once for each: `done`, one flag a device, is the
// kernel's.
template <typename Kernel>
int ensure_smem(Kernel k, int bytes, std::atomic<bool> (&done)[kMaxDevices]) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  std::atomic<bool>* d = dev < kMaxDevices ? &done[dev] : nullptr;
  if (d && d->load(std::memory_order_acquire)) return RGD_OK;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute");
  if (d) d->store(true, std::memory_order_release);
  return RGD_OK;
}

// Argument checks of rgd_sample_head_gated (shared with rgd_decode_step, which
// checks them before launching its first kernel).
int check_gated_head(const char* fn, int32_t rows, int32_t vocab, int32_t dtype, const void* logits,
                     const float* temperature, const float* min_p, const uint64_t* seed, const int32_t* token_out,
                     const rgd_trie* trie, int32_t rows_per_group, int32_t max_len, const rgd_gate_state* state);

// rgd_sample_head_gated with its arguments checked under the name `fn`.  early:
// the previous kernel on the stream writes no input of the head and lets it
// start only once every input was complete, so the head may read them before
// that kernel ends (it still waits for it before it writes anything).
int launch_gated_head(const char* fn, int32_t rows, int32_t vocab, int32_t dtype, const void* logits,
                      const uint8_t* is_probe, const float* temperature, const float* min_p, const uint64_t* seed,
                      uint64_t step, uint8_t* row_active, int32_t* token_out, int32_t* kept_count,
                      const rgd_trie* trie, int32_t rows_per_group, int32_t eos_token, int32_t max_len,
                      rgd_gate_state* state, int32_t* dev_status, rgd_stream_t stream, bool early);

}  // namespace rgd

#define RGD_CHECK_ARG(cond, ...)                                        \
  do {                                                                  \
    if (!(cond)) return ::rgd::set_error(RGD_ERR_INVALID_ARG, __VA_ARGS__); \
  } while (0)
