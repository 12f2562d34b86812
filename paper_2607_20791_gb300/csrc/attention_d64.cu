// The attention kernel for head dimension 64 (one translation unit per head
// dimension, compiled in parallel).
#include "attention_kernel.cuh"

namespace rgd {

int launch_attn_d64(const CUtensorMap& tmK, const CUtensorMap& tmV, const AttnParams& p, int smem_bytes,
                    cudaStream_t st) {
  return launch_attn<64>(tmK, tmV, p, smem_bytes, st);
}

}  // namespace rgd
