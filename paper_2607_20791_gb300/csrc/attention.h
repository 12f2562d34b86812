// Shared by the attention's translation units: the kernel's parameters, the
// query configurations and the shared-memory plan of a call.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "common.h"

namespace rgd {

constexpr int kPage = 16;                      // tokens per KV page
constexpr int kGroupPages = 8;                 // pages per group: 128 tokens, the MMA's M
constexpr int kMaxQueries = 128;               // rows_per_group * Hq / Hkv
// A split job of at most this many other pieces is folded in the merging block's K
// ring.  With ten (a page each) the fold's loops took 17 us where the merge from
// global memory by every thread takes 12; with one or two the fold saves 1.7 us of
// 33 (16 groups x 5 rows) and 6 of 40 (200 x 16 rows, D 64).
constexpr int kMaxFold = 4;
constexpr int kRingMax = 4;                    // K or V areas at most
constexpr int kSmemLimit = 226 * 1024;         // dynamic part; static shared memory needs the rest

// Partial (m, l) pairs are stored nq rounded up to even per piece.
__host__ __device__ constexpr int ml_stride(int nq) { return (nq + 1) & ~1; }
inline int align_up(int x, int a) { return (x + a - 1) / a * a; }

// Softmax sets (four warps each) and queries per set for a job of nq queries.
// Every thread of a set keeps its token's scores and sums of all the set's
// queries in registers, so a set takes as few queries as threads allow: 8 up to
// 32 queries; then three or four sets of 16, 24 or 32, the smallest that holds
// the count, since the MMAs' columns and the P^T writes go with sets x per_set.
// Per query count (us; 64 or 32 query heads, 8 kv heads), against a kernel that
// held 128 rows of query copies whatever the count: 12 in (2, 8): 54 (73 with
// copies), 16: 62 (82), 32 in (4, 8): 57 (75), 36 in (3, 16): 47 (70), 56 in
// (4, 16): 71 (100), 72 in (3, 24): 115 (202), 96 in (4, 24): 92 (138), 128 in
// (4, 32): 121 (150).
struct QueryConfig {
  int sets, per_set;
};
constexpr QueryConfig query_config(int nq) {
  return nq <= 8    ? QueryConfig{1, 8}
         : nq <= 16 ? QueryConfig{2, 8}
         : nq <= 24 ? QueryConfig{3, 8}
         : nq <= 32 ? QueryConfig{4, 8}
         : nq <= 48 ? QueryConfig{3, 16}
         : nq <= 64 ? QueryConfig{4, 16}
         : nq <= 72 ? QueryConfig{3, 24}
         : nq <= 96 ? QueryConfig{4, 24}
                    : QueryConfig{4, 32};
}
// Query columns of the MMAs (their N is a multiple of 16).
__host__ __device__ constexpr int query_cols(int sets, int per_set) { return (sets * per_set + 15) / 16 * 16; }

// Shared-memory carve-up, laid out by the host.  Rings, P^T and Q are
// 1024-byte aligned (swizzle atoms).
struct AttnLayout {
  int kring, vring, p, q, wmax, lw, mfin, mref, einv, erow, desc, gpre, plen, rowbits, slen, total;
};
inline AttnLayout attn_layout(int D, int sets, int per_set, int hk, int hv, int np, int nqb, int G, int R,
                              bool slen_in_smem) {
  const int area = kGroupPages * kPage * D * 2, N = query_cols(sets, per_set), nq = sets * per_set;
  AttnLayout L;
  L.kring = 0;                                // [hk][8 pages][2 row groups][D/64 halves][8 rows][128 B]
  L.vring = L.kring + hk * area;              // [hv][8 pages][D/64 halves][16 rows][128 B]
  L.p = L.vring + hv * area;                  // [np] P^T: 128 tokens x (N high parts, N residuals) bf16
  L.q = L.p + np * 512 * N;                   // [nqb][D/64 halves][N rows][128 B]
  L.wmax = L.q + nqb * N * D * 2;             // [4][nq] per-quarter query maxima of a group
  L.lw = L.wmax + 4 * nq * 4;                 // [2 pieces][4][nq] per-warp query sums
  L.mfin = L.lw + 8 * nq * 4;                 // [2 pieces][nq] reference maxima at the piece end
  L.mref = L.mfin + 2 * nq * 4;               // [2 versions][nq] current reference maxima
  L.einv = L.mref + 2 * nq * 4;               // piece end, per query: 1 / sum, output row (-1: none)
  L.erow = L.einv + kMaxQueries * 4;
  L.desc = L.erow + kMaxQueries * 4;          // [8 groups][8 pages] tokens and row of a page
  L.gpre = L.desc + 8 * kGroupPages * 4;      // [G + 1] pages of the groups before
  L.plen = align_up(L.gpre + (G + 1) * 4, 16);
  L.rowbits = align_up(L.plen + G * 4, 16);   // one bit per row: active
  L.slen = align_up(L.rowbits + (R + 31) / 32 * 4, 16);
  L.total = align_up(L.slen + (slen_in_smem ? R * 4 : 0), 16) + 1024;  // + slack for the 1024-byte aligned base
  return L;
}

struct AttnParams {
  const __nv_bfloat16* q;
  const int32_t* prompt_bt;
  const int32_t* prompt_len;
  const int32_t* suffix_bt;
  const int32_t* suffix_len;
  const uint8_t* row_active;
  __nv_bfloat16* out;
  float* lse;
  float* slot_o;    // [(C + J - 1) * nq, D]
  float2* slot_ml;  // [(C + J - 1) * ml_stride(nq)]
  int32_t* ticket;  // [J] pieces of a split job that have finished (zero between calls)
  int32_t* dev_status;
  int32_t G, rpg, Hq, Hkv, gq, num_pages, max_pp, max_sp;
  int32_t nq, C;
  int32_t end_pages;     // pages that a job's end counts for when the pages are dealt to the blocks
  int32_t hk, hv;        // K and V areas of the ring
  uint64_t rpg_mul, hk_mul, hv_mul;  // ceil(2^32 / rpg), / hk, / hv: x / n = x n_mul >> 32 while x n < 2^32
  int32_t np, nqb;       // P^T and Q buffers (1 or 2)
  int32_t fold;          // a split job of at most this many other pieces is folded in the K ring
  int32_t slen_in_smem;  // the rows' suffix lengths are kept in shared memory
  float scale_log2;
  AttnLayout L;      // the shared-memory carve-up
  uint64_t wait_ns;  // limit of every wait on another role or block (rgd_set_wait_limit_ns)
};

// The kernel for one head dimension (attention_d64.cu, attention_d128.cu).
int launch_attn_d64(const CUtensorMap& tmK, const CUtensorMap& tmV, const AttnParams& p, int smem_bytes,
                    cudaStream_t st);
int launch_attn_d128(const CUtensorMap& tmK, const CUtensorMap& tmV, const AttnParams& p, int smem_bytes,
                     cudaStream_t st);

}  // namespace rgd
