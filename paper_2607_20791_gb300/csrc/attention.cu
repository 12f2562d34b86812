// Shared-prefix decode attention: the entry points, the plan of a call and its
// tensor maps.  The kernel is in attention_kernel.cuh.
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>

#include "attention.h"
#include "ptx.cuh"

namespace rgd {
namespace {

constexpr int kTicketSlots = 8192;  // job counters at the start of every workspace (at least)
constexpr float kLog2e = 1.4426950408889634f;

PFN_cuTensorMapEncodeTiled_v12000 get_encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  });
  return fn;
}

// The K or V pool ([rows][D] bf16) for copies of whole 16-token page-head tiles, one
// box each, with the 128-byte swizzle (16-byte chunk index XOR row index mod 8).
// V: 64 columns x 16 rows x D/64 halves, so a tile lands half-major.  K: 64 columns x
// 8 rows x D/64 halves x 2 row groups, so that consecutive 8-row groups of a half
// are D/64 KB apart within a tile and across tiles: a group's K is one 128-row
// operand per half although each page is one box (with a box per half the K
// producer's issue, ~75 cycles a box, was twice the V producer's).
int make_kv_map(CUtensorMap* map, const void* base, int64_t rows, int D, bool is_k) {
  auto fn = get_encode_fn();
  if (!fn) return set_error(RGD_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
  const cuuint32_t halves = (cuuint32_t)(D / 64);
  const cuuint64_t row = (cuuint64_t)D * 2;
  const cuuint64_t dims_k[4] = {64, 8, halves, (cuuint64_t)rows / 8}, strides_k[3] = {row, 128, 8 * row};
  const cuuint64_t dims_v[3] = {64, (cuuint64_t)rows, halves}, strides_v[2] = {row, 128};
  const cuuint32_t box_k[4] = {64, 8, halves, kPage / 8}, box_v[3] = {64, (cuuint32_t)kPage, halves};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, is_k ? 4 : 3, const_cast<void*>(base), is_k ? dims_k : dims_v,
                  is_k ? strides_k : strides_v, is_k ? box_k : box_v, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(RGD_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return RGD_OK;
}

// Limit of the kernel's waits on other roles and blocks, for the calls that
// follow (rgd_set_wait_limit_ns).
std::atomic<uint64_t> g_wait_ns{kWaitLimitNs};

int device_sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return n;
}

struct Plan {
  int nq, C, J;
  int hk, hv, np, nqb;  // K and V areas of the ring, P^T and Q buffers
  bool slen_in_smem;
  AttnLayout layout;
  size_t ticket_off, ml_off, o_off, total;
};

int check_shape(const rgd_attn_shape* s) {
  RGD_CHECK_ARG(s != nullptr, "attention shape is NULL");
  RGD_CHECK_ARG(s->num_groups >= 1 && s->rows_per_group >= 1, "num_groups and rows_per_group must be >= 1");
  RGD_CHECK_ARG(s->num_kv_heads >= 1 && s->num_q_heads >= s->num_kv_heads &&
                    s->num_q_heads % s->num_kv_heads == 0,
                "num_q_heads must be a positive multiple of num_kv_heads");
  if (s->head_dim != 64 && s->head_dim != 128)
    return set_error(RGD_ERR_UNSUPPORTED, "head_dim %d unsupported (64 or 128)", s->head_dim);
  if (s->page_size != kPage) return set_error(RGD_ERR_UNSUPPORTED, "page_size %d unsupported (16)", s->page_size);
  RGD_CHECK_ARG(s->num_pages >= 1, "num_pages must be >= 1");
  RGD_CHECK_ARG((int64_t)s->num_pages * s->num_kv_heads * kPage < (int64_t)1 << 31,
                "num_pages * num_kv_heads * page_size must be < 2^31");
  RGD_CHECK_ARG(s->max_prompt_pages >= 1 && s->max_suffix_pages >= 1, "block tables need >= 1 column");
  RGD_CHECK_ARG(s->num_ctas >= 0 && s->num_ctas <= 65535 && s->reserved == 0,
                "num_ctas must be in [0, 65535] and reserved 0");
  RGD_CHECK_ARG((int64_t)s->num_groups * (s->max_prompt_pages + (int64_t)s->rows_per_group * s->max_suffix_pages) *
                        s->num_kv_heads <
                    ((int64_t)1 << 31),
                "too many KV pages in one call (must be < 2^31)");
  const int nq = s->rows_per_group * (s->num_q_heads / s->num_kv_heads);
  if (nq > kMaxQueries)
    return set_error(RGD_ERR_UNSUPPORTED, "rows_per_group * Hq/Hkv = %d exceeds %d", nq, kMaxQueries);
  return RGD_OK;
}

int make_plan(const rgd_attn_shape* s, Plan* pl) {
  if (int rc = check_shape(s)) return rc;
  pl->nq = s->rows_per_group * (s->num_q_heads / s->num_kv_heads);
  pl->C = s->num_ctas > 0 ? s->num_ctas : device_sm_count();
  if (pl->C <= 0) return set_error(RGD_ERR_CUDA, "could not query the device's SM count");
  pl->J = s->num_groups * s->num_kv_heads;
  // Shared memory: a block needs a K and a V area, a P^T and a Q buffer.  Second
  // P^T and Q buffers let a group's softmax run ahead of the PV before it and a
  // short job's QK ahead of the piece end before it; they are taken while five
  // areas are left (one more than a group in flight and a group in use), then
  // the rest goes to more areas: 5 at the Llama-3-8B shape and for 72 queries, up
  // to 8 at head dim 64.  The rows' suffix lengths leave shared memory only when
  // a call has so many rows that not even two areas fit beside them.
  const int D = s->head_dim, rows = s->num_groups * s->rows_per_group;
  const QueryConfig qc = query_config(pl->nq);
  const int area = kGroupPages * kPage * D * 2;
  pl->hk = pl->hv = 0;
  if (s->num_groups > kSmemLimit / 8)  // two words a group: refused before a sum of sizes can overflow
    return set_error(RGD_ERR_UNSUPPORTED, "shape needs more shared memory than an SM has (too many groups?)");
  const struct {
    int np, nqb, areas;
    bool slen_in_smem;
  } tries[] = {{2, 2, 5, true}, {1, 2, 5, true}, {1, 1, 2, true}, {1, 1, 2, false}};
  for (const auto& t : tries) {
    pl->slen_in_smem = t.slen_in_smem;
    pl->np = t.np;
    pl->nqb = t.nqb;
    const int fixed = attn_layout(D, qc.sets, qc.per_set, 0, 0, t.np, t.nqb, s->num_groups, rows, t.slen_in_smem).total;
    const int n = std::min((kSmemLimit - fixed) / area, 2 * kRingMax);
    if (fixed > kSmemLimit || n < t.areas) continue;
    pl->hk = n / 2;  // (K areas come back sooner than V areas)
    pl->hv = n - n / 2;
    break;
  }
  if (pl->hk == 0)
    return set_error(RGD_ERR_UNSUPPORTED, "shape needs more shared memory than an SM has (too many groups?)");
  pl->layout = attn_layout(D, qc.sets, qc.per_set, pl->hk, pl->hv, pl->np, pl->nqb, s->num_groups, rows,
                           pl->slen_in_smem);
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  const size_t n_part = (size_t)pl->C + pl->J - 1;  // partial-result slots
  // The job counters come first, in an area of at least kTicketSlots counters
  // whatever the shape, so that a workspace reused for another shape with up to
  // kTicketSlots jobs finds its counters where earlier calls left zeros, not
  // where they wrote partials.
  pl->ticket_off = 0;
  pl->ml_off = up((size_t)std::max(pl->J, kTicketSlots) * sizeof(int32_t));
  pl->o_off = pl->ml_off + up(n_part * ml_stride(pl->nq) * sizeof(float2));
  pl->total = pl->o_off + up(n_part * pl->nq * s->head_dim * sizeof(float));
  return RGD_OK;
}

// Workspace fields used by the allocation-free entry point below.
size_t ws_total(const rgd_attn_shape* s) {
  Plan pl;
  return make_plan(s, &pl) == RGD_OK ? pl.total : 0;
}

}  // namespace
}  // namespace rgd

using namespace rgd;

extern "C" int rgd_set_wait_limit_ns(uint64_t limit_ns) {
  clear_error();
  g_wait_ns.store(limit_ns == 0 ? kWaitLimitNs : limit_ns, std::memory_order_relaxed);
  return RGD_OK;
}

extern "C" size_t rgd_prefix_decode_attn_workspace_size(const rgd_attn_shape* shape) {
  clear_error();
  Plan pl;
  if (make_plan(shape, &pl) != RGD_OK) return 0;
  return pl.total;
}

extern "C" int rgd_prefix_decode_attn(const rgd_attn_shape* shape, const rgd_bf16* q, const rgd_bf16* k_pages,
                                      const rgd_bf16* v_pages, const int32_t* prompt_block_table,
                                      const int32_t* prompt_len, const int32_t* suffix_block_table,
                                      const int32_t* suffix_len, const uint8_t* row_active, float softmax_scale,
                                      rgd_bf16* out, float* lse, void* workspace, size_t workspace_bytes,
                                      int32_t* dev_status, rgd_stream_t stream) {
  clear_error();
  Plan pl;
  if (int rc = make_plan(shape, &pl)) return rc;
  const rgd_attn_shape& s = *shape;
  RGD_CHECK_ARG(q && k_pages && v_pages && prompt_block_table && prompt_len && suffix_block_table && suffix_len &&
                    out && workspace,
                "rgd_prefix_decode_attn: a required pointer is NULL");
  RGD_CHECK_ARG(aligned16(q) && aligned16(k_pages) && aligned16(v_pages) && aligned16(out),
                "rgd_prefix_decode_attn: q, k_pages, v_pages and out must be 16-byte aligned");
  RGD_CHECK_ARG((reinterpret_cast<uintptr_t>(workspace) & 255) == 0, "workspace must be 256-byte aligned");
  RGD_CHECK_ARG(std::isfinite(softmax_scale) && softmax_scale > 0.f, "softmax_scale must be > 0");
  RGD_CHECK_ARG(workspace_bytes >= pl.total, "workspace too small: %zu < %zu", workspace_bytes, pl.total);

  CUtensorMap tmK, tmV;
  const int64_t kv_rows = (int64_t)s.num_pages * s.num_kv_heads * kPage;
  if (int rc = make_kv_map(&tmK, k_pages, kv_rows, s.head_dim, true)) return rc;
  if (int rc = make_kv_map(&tmV, v_pages, kv_rows, s.head_dim, false)) return rc;

  AttnParams p;
  p.q = reinterpret_cast<const __nv_bfloat16*>(q);
  p.prompt_bt = prompt_block_table;
  p.prompt_len = prompt_len;
  p.suffix_bt = suffix_block_table;
  p.suffix_len = suffix_len;
  p.row_active = row_active;
  p.out = reinterpret_cast<__nv_bfloat16*>(out);
  p.lse = lse;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  p.ticket = reinterpret_cast<int32_t*>(ws + pl.ticket_off);
  p.slot_ml = reinterpret_cast<float2*>(ws + pl.ml_off);
  p.slot_o = reinterpret_cast<float*>(ws + pl.o_off);
  p.dev_status = dev_status;
  p.G = s.num_groups;
  p.rpg = s.rows_per_group;
  p.Hq = s.num_q_heads;
  p.Hkv = s.num_kv_heads;
  p.gq = s.num_q_heads / s.num_kv_heads;
  p.num_pages = s.num_pages;
  p.max_pp = s.max_prompt_pages;
  p.max_sp = s.max_suffix_pages;
  p.nq = pl.nq;
  p.C = pl.C;
  // A job's end takes its block's warps about 2300 cycles and more with many
  // queries, a page 340 cycles at head dim 128 and the copy rate.  In pages, 0 / 6 /
  // 16: 16 groups x 5 rows 30.4 / 29.7 / 30.2 us; 32 x 16 rows of 128 queries a job
  // 87.6 / 83.9 / 82.8; 32 x 4 rows at head dim 64 37.3 / 36.5 / 35.4.
  p.end_pages = (6 + pl.nq / 16) * 128 / s.head_dim;
  if (((int64_t)s.num_groups * (s.max_prompt_pages + (int64_t)s.rows_per_group * s.max_suffix_pages + p.end_pages)) *
          s.num_kv_heads >=
      (int64_t)1 << 31)
    p.end_pages = 0;  // (the positions must fit 31 bits)
  p.hk = pl.hk;
  auto mul_of = [](int n) { return ((1ull << 32) + n - 1) / n; };
  p.rpg_mul = mul_of(s.rows_per_group);  // (at most kSmemLimit / 8 groups of 128 rows: x n < 2^32)
  p.hk_mul = mul_of(pl.hk);
  p.hv_mul = mul_of(pl.hv);
  p.hv = pl.hv;
  p.np = pl.np;
  p.nqb = pl.nqb;
  p.fold = std::min(kMaxFold, pl.hk * kGroupPages * kPage * s.head_dim * 2 /
                                  (pl.nq * s.head_dim * 4 + ml_stride(pl.nq) * 8));
  p.slen_in_smem = pl.slen_in_smem ? 1 : 0;
  p.L = pl.layout;
  p.scale_log2 = softmax_scale * kLog2e;
  p.wait_ns = g_wait_ns.load(std::memory_order_relaxed);

  cudaStream_t st = (cudaStream_t)stream;
  return s.head_dim == 128 ? launch_attn_d128(tmK, tmV, p, pl.layout.total, st)
                           : launch_attn_d64(tmK, tmV, p, pl.layout.total, st);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of rgd_prefix_decode_attn
// ---------------------------------------------------------------------------
// The split partials live in a fixed file-scope device array
// instead of a caller-provided workspace.  The array exists once per device in
// every process that loads the library, for the life of the process.
namespace rgd {
namespace {

constexpr size_t kStaticScratchBytes = size_t(8) << 20;  // 8 MiB
__device__ __align__(256) uint8_t g_attn_scratch[kStaticScratchBytes];

std::mutex g_scratch_mu;
void* g_scratch_ptr[kMaxDevices] = {};

}  // namespace
}  // namespace rgd

extern "C" int rgd_prefix_decode_attn_noalloc(const rgd_attn_shape* shape, const rgd_bf16* q,
                                              const rgd_bf16* k_pages, const rgd_bf16* v_pages,
                                              const int32_t* prompt_block_table, const int32_t* prompt_len,
                                              const int32_t* suffix_block_table, const int32_t* suffix_len,
                                              const uint8_t* row_active, float softmax_scale, rgd_bf16* out,
                                              float* lse, int32_t* dev_status, rgd_stream_t stream) {
  clear_error();
  if (int rc = check_shape(shape)) return rc;
  // The counters must sit in the fixed area at the start of the array for every
  // shape (a larger job count would move the partials over them).
  if ((int64_t)shape->num_groups * shape->num_kv_heads > kTicketSlots)
    return set_error(RGD_ERR_UNSUPPORTED,
                     "rgd_prefix_decode_attn_noalloc: num_groups * num_kv_heads = %lld exceeds %d",
                     (long long)shape->num_groups * shape->num_kv_heads, kTicketSlots);
  const size_t need = ws_total(shape);
  if (need > kStaticScratchBytes)
    return set_error(RGD_ERR_UNSUPPORTED,
                     "rgd_prefix_decode_attn_noalloc: this shape needs %zu bytes of scratch; the static "
                     "scratch holds %zu (use rgd_prefix_decode_attn with a workspace)",
                     need, kStaticScratchBytes);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return set_error(RGD_ERR_UNSUPPORTED, "device ordinal %d >= %d", dev, kMaxDevices);
  void* scratch = nullptr;
  {
    // once per device, with that device current: the host-side symbol is only a
    // stand-in, so the kernel gets the device address of the array
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (g_scratch_ptr[dev] == nullptr) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_attn_scratch);
      if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(g_attn_scratch)");
      g_scratch_ptr[dev] = p;
    }
    scratch = g_scratch_ptr[dev];
  }
  // the array is zero when the module is loaded (device variables without an
  // initializer are zero-filled); every call leaves the counters of its jobs at
  // zero, and no call writes anything else into the fixed counter area
  return rgd_prefix_decode_attn(shape, q, k_pages, v_pages, prompt_block_table, prompt_len, suffix_block_table,
                                suffix_len, row_active, softmax_scale, out, lse, scratch, kStaticScratchBytes,
                                dev_status, stream);
}
