// Refusal-prefix gate: host-built token trie + per-token hard-gate kernel.
//
// The compatibility predicate C(q, P) of Sec. 3 holds when q is a prefix of some
// refusal prefix pi, or some pi (with |pi| >= min_confirm, the two-token minimum
// of App. D) is a prefix of q.  On a trie of P this becomes a walk: while q is a
// trie path it is a prefix of some pi; once q reaches a node that ends a pi of
// length >= min_confirm ("confirmed") every extension stays compatible; leaving
// the trie before that is incompatible.  The hard gate of Alg. 1 applies the
// predicate after every greedy probe token (the cap c does not change the
// outcome of the hard gate).
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <map>
#include <vector>

#include "common.h"
#include "ptx.cuh"
#include "trie.cuh"

namespace rgd {
namespace cg = cooperative_groups;
namespace {

__global__ void gate_state_init_kernel(rgd_gate_state* st, int32_t groups) {
  const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (a dependent waits for this kernel's end)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (g >= groups) return;
  rgd_gate_state s;
  s.node = 0;
  s.length = 0;
  s.steps = 0;
  s.decisive_step = -1;
  s.decision = RGD_PENDING;
  s.confirmed = 0;
  s.done = 0;
  s.reserved = 0;
  st[g] = s;
}

// A trie node during a warp's walk: its first edge and their number.
struct WalkNode {
  int32_t begin, count;
};

// The edge labelled `tok` out of node n, by a warp: 32 edges a step, so a node of
// up to 32 children takes one load, the root of a thousand two.  {node it leads
// to, whether that node confirms}, or {-1, 0}; n becomes that node.
__device__ __forceinline__ int2 warp_child(const TrieView& t, WalkNode& n, int32_t tok, int lane) {
  int32_t lo = n.begin, cnt = n.count;
#pragma unroll 1
  while (cnt > 32) {  // the last of 32 evenly spaced edges that is not above tok
    const int32_t step = (cnt + 31) >> 5, i = lane * step;
    const bool le = i < cnt && __ldg(&t.edges[lo + i].x) <= tok;
    const int32_t k = __popc(__ballot_sync(0xffffffffu, le));
    if (k == 0) return make_int2(-1, 0);
    lo += (k - 1) * step;
    cnt = min(step, cnt - (k - 1) * step);
  }
  int4 e = make_int4(-1, -1, 0, 0);
  if (lane < cnt) e = __ldg(t.edges + lo + lane);
  const uint32_t hit = __ballot_sync(0xffffffffu, lane < cnt && e.x == tok);
  if (hit == 0) return make_int2(-1, 0);
  const int src = __ffs(hit) - 1;
  n.begin = __shfl_sync(0xffffffffu, e.z, src);
  const int32_t w = __shfl_sync(0xffffffffu, e.w, src);
  n.count = w & 0x7fffffff;
  return make_int2(__shfl_sync(0xffffffffu, e.y, src), w < 0 ? 1 : 0);
}

// One warp per group.  The walk is a chain of dependent loads, an L2 round trip
// each, and nothing else: so the tokens come 32 at a time, a token takes one
// round trip (two or three out of a large node), and the state and the rows' mask
// are the lanes' together.  Every lane holds the same gate state.  Inside a graph:
// 1024 probes of 32 tokens against 1000 prefixes 14.5 us with a thread a group and
// a binary search over separate arrays, 6.4 so; 4096 of 64 tokens against 2000:
// 20 us, 7.7; one probe of 32 tokens: 7.5 us, 2.6.
constexpr int kGateThreads = 128;
__global__ void __launch_bounds__(kGateThreads)
    probe_gate_kernel(TrieView t, int32_t groups, int32_t rows_per_group, const int32_t* __restrict__ tokens,
                      int32_t n_tokens, int64_t stride, int32_t eos, int32_t max_len,
                      rgd_gate_state* __restrict__ state, uint8_t* __restrict__ row_active, int32_t* dev_status) {
  const int lane = threadIdx.x & 31;
  const int32_t g = blockIdx.x * (kGateThreads / 32) + (int)(threadIdx.x >> 5);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (a dependent waits for this kernel's end)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (g >= groups) return;
  const bool root_has_children = __ldg(t.child_begin + 1) > 0;
  const int32_t* toks = tokens + (int64_t)g * stride;
  int32_t mine = lane < n_tokens ? __ldg(toks + lane) : 0;
  rgd_gate_state s = state[g];
  WalkNode n{0, 0};
  if (!s.done && !s.confirmed) {
    n.begin = __ldg(t.child_begin + s.node);
    n.count = __ldg(t.child_begin + s.node + 1) - n.begin;
  }
  bool bad_token = false;
#pragma unroll 1
  for (int32_t k = 0; k < n_tokens && !s.done; ++k) {
    const int32_t at = k & 31;
    if (k > 0 && at == 0) mine = k + lane < n_tokens ? __ldg(toks + k + lane) : 0;
    if (s.confirmed) {
      // every further token only counts, up to the stop token or the one that
      // reaches max_len: all of the chunk's before that at once
      const bool in = lane >= at && k - at + lane < n_tokens;
      const bool stop = eos >= 0 && mine == eos;
      const uint32_t good = __ballot_sync(0xffffffffu, in && !stop && mine >= 0);
      const bool last = ((good >> lane) & 1u) != 0 &&
                        __popc(good & (0xffffffffu >> (31 - lane))) == max(1, max_len - s.length);
      const uint32_t end = __ballot_sync(0xffffffffu, in && (stop || last));
      const uint32_t bad = __ballot_sync(0xffffffffu, in && !stop && mine < 0);
      const int n_chunk = end ? __ffs(end) - 1 : 32;  // (chunk position of the token that ends the probe)
      const uint32_t before = n_chunk == 32 ? 0xffffffffu : (1u << n_chunk) - 1u;
      const int counted = __popc(good & before);
      s.steps += counted;
      s.length += counted;
      bad_token = bad_token || (bad & before) != 0;
      k += n_chunk - at;
      if (n_chunk == 32) {
        --k;  // (the next chunk's first token)
        continue;
      }
    }
    const int32_t y = __shfl_sync(0xffffffffu, mine, k & 31);
    if (y < 0 && !(eos >= 0 && y == eos)) {
      bad_token = true;
      continue;
    }
    consume_token_with(s, y, eos, max_len, root_has_children,
                       [&](int32_t tok) { return warp_child(t, n, tok, lane); });
  }
  if (lane == 0) {
    state[g] = s;
    if (bad_token && dev_status) atomicOr(dev_status, RGD_DEV_BAD_TOKEN);
  }
  if (!row_active) return;
  uint8_t* ra = row_active + (int64_t)g * rows_per_group;
  if (s.done && lane == 0) ra[0] = 0;
  if (s.decision == RGD_REFUSAL)
    for (int32_t i = 1 + lane; i < rows_per_group; i += 32) ra[i] = 0;
}

// ---------------------------------------------------------------------------
// Soft compatibility gate (the appendix ablation's Alg. 2), one probe step.
// In the first c steps, a greedy token y that would leave the refusal-prefix
// set does not end the probe at once: among the top-K tokens of the probe's
// next-token distribution (softmax of its logits; ties to the lower index),
// the refusal-compatible ones -- the children of the probe's trie node, and
// the stop token, which d(q) drops -- are found, and if their probability
// mass m reaches rho the most probable of them is appended instead.
//
// One thread-block cluster of K CTAs per group (K by the number of groups, see
// rgd_soft_gate), each CTA taking an equal contiguous share of the probe's logits,
// copied into shared memory in chunks by bulk copies issued before anything else.
// While they are in flight, the children of the probe's trie node (token, node,
// confirm flag) are read into shared memory -- every trie lookup of the step is then a
// shared-memory scan -- and, when the soft branch can be taken at this step,
// the candidates' keys (logit, token) and the kProbe best of them.  A
// candidate's rank -- the number of logits above it -- grows along the
// candidates' order, so the candidates in the top K are a prefix of that
// order.  The pass finds the maximum, its lowest index (y) and the softmax
// normaliser Z and counts the logits above each of the kProbe best
// candidates, which settles the prefix unless all of them are in the top K;
// then the candidates are sorted (bitonic, in shared memory) and a search over
// the rest finishes it, one candidate a pass: the next, then ever wider steps
// until one is out (few are in the top K where most of a node's children are
// improbable: one pass then, a binary search takes six for 36), then halving.  A
// pass reads the share in shared memory if its chunks still hold all of it, else
// from L2.  After each pass every CTA pushes its partial
// results into every CTA's shared memory and all of them combine the same
// values in the same order, so every CTA takes the same decisions; CTA 0
// writes the step's outcome.  The kernel runs once per decode step behind
// kernels that sweep L2, so its own instructions are fetched cold: its loops
// stay rolled, which keeps the code it runs short.
constexpr int kSoftThreads = 512;
constexpr int kSoftCluster = 6;  // CTAs per group at most (6, 4 or 2)
constexpr int kMaxCand = 2048;  // a node's children + the stop token (a power of two: the sort's padding)
constexpr int kProbe = 4;       // candidates whose ranks the first pass counts
constexpr int kSoftChunk = 32768;  // bytes of logits per bulk copy
constexpr int kSoftStages = 3;     // chunk buffers

struct SoftPart {  // one CTA's share of the first pass
  float m, z;
  int32_t mi;
  int32_t c[kProbe];
};

struct SoftShared {
  uint64_t key[kMaxCand];       // slot k < nc: child k; slot nc: the stop token (no candidate: ~0)
  int32_t slot_tok[kMaxCand];   // child k: its token, the node it leads to, that node's confirm flag
  int32_t slot_node[kMaxCand];
  uint8_t slot_conf[kMaxCand];
  SoftPart part[kSoftCluster * kSoftThreads / 32];  // first pass, slot = CTA rank x warps + warp
  int32_t cnt[2][kSoftCluster];  // search passes, slot = CTA rank, by pass parity
  int32_t cnt_cta;
  uint64_t full[kSoftStages];    // chunk buffer s holds its chunk
  int32_t ncand;
};

template <typename LT>
__device__ __forceinline__ float logit_at(const LT* row, int64_t i);
template <>
__device__ __forceinline__ float logit_at<float>(const float* row, int64_t i) {
  return __ldg(row + i);
}
template <>
__device__ __forceinline__ float logit_at<uint16_t>(const uint16_t* row, int64_t i) {
  return __uint_as_float((uint32_t)__ldg(row + i) << 16);
}

// Element e of a 16-byte vector of logits.
template <typename LT>
__device__ __forceinline__ float vec_elem(const uint4& w, int e);
template <>
__device__ __forceinline__ float vec_elem<float>(const uint4& w, int e) {
  return __uint_as_float(e == 0 ? w.x : e == 1 ? w.y : e == 2 ? w.z : w.w);
}
template <>
__device__ __forceinline__ float vec_elem<uint16_t>(const uint4& w, int e) {
  const uint32_t u = (e >> 1) == 0 ? w.x : (e >> 1) == 1 ? w.y : (e >> 1) == 2 ? w.z : w.w;
  return __uint_as_float((e & 1) ? (u & 0xffff0000u) : (u << 16));
}

// Calls f(logit, index) for this thread's share of part `part` (of nparts
// equal contiguous parts) of a row, in increasing index order: 16-byte
// vectors when the row is 16-byte aligned (the few elements past the last
// whole vector, one per thread, go to the last part and come last), else
// single elements.  batch_end() follows every batch of loads.
template <int kThreads, int kBatchLoads, typename LT, typename F, typename B>
__device__ __forceinline__ void scan_row(const LT* row, int32_t vocab, bool vec, int part, int nparts, F&& f,
                                         B&& batch_end) {
  constexpr int E = 16 / (int)sizeof(LT);
  const int tid = threadIdx.x;
  if (vec) {
    const int32_t nvec = vocab / E;
    const int32_t lo = (int32_t)((int64_t)nvec * part / nparts), hi = (int32_t)((int64_t)nvec * (part + 1) / nparts);
    const uint4* rv = reinterpret_cast<const uint4*>(row);
    uint4 w[kBatchLoads];
    int32_t v0 = lo + tid;
#pragma unroll
    for (int b = 0; b < kBatchLoads; ++b)
      if (v0 + b * kThreads < hi) w[b] = __ldg(rv + v0 + b * kThreads);
    for (;;) {
#pragma unroll
      for (int b = 0; b < kBatchLoads; ++b) {
        const int32_t vi = v0 + b * kThreads;
        if (vi >= hi) break;
#pragma unroll
        for (int e = 0; e < E; ++e) f(vec_elem<LT>(w[b], e), vi * E + e);
      }
      batch_end();
      v0 += kBatchLoads * kThreads;
      if (v0 >= hi) break;
#pragma unroll
      for (int b = 0; b < kBatchLoads; ++b)
        if (v0 + b * kThreads < hi) w[b] = __ldg(rv + v0 + b * kThreads);
    }
    const int32_t i = nvec * E + tid;
    if (part == nparts - 1 && i < vocab) f(logit_at<LT>(row, i), i);
  } else {
    const int32_t lo = (int32_t)((int64_t)vocab * part / nparts), hi = (int32_t)((int64_t)vocab * (part + 1) / nparts);
    float v[kBatchLoads];
    int32_t i0 = lo + tid;
#pragma unroll
    for (int b = 0; b < kBatchLoads; ++b)
      if (i0 + b * kThreads < hi) v[b] = logit_at<LT>(row, i0 + b * kThreads);
    for (;;) {
#pragma unroll
      for (int b = 0; b < kBatchLoads; ++b) {
        if (i0 + b * kThreads >= hi) break;
        f(v[b], i0 + b * kThreads);
      }
      batch_end();
      i0 += kBatchLoads * kThreads;
      if (i0 >= hi) break;
#pragma unroll
      for (int b = 0; b < kBatchLoads; ++b)
        if (i0 + b * kThreads < hi) v[b] = logit_at<LT>(row, i0 + b * kThreads);
    }
  }
}

// Order-preserving key: ascending keys = logits descending, then tokens ascending.
__device__ __forceinline__ uint64_t rank_key(float v, int32_t tok) {
  uint32_t u = __float_as_uint(v);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);  // ascending with v
  return ((uint64_t)(~u) << 32) | (uint32_t)tok;
}
__device__ __forceinline__ float key_logit(uint64_t k) {
  uint32_t u = ~(uint32_t)(k >> 32);
  u = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
  return __uint_as_float(u);
}

// (v, i) ranks above (w, j): a larger logit, or the same logit and a lower index.
__device__ __forceinline__ bool above(float v, int32_t i, float w, int32_t j) { return v > w || (v == w && i < j); }

constexpr float kLog2e = 1.4426950408889634f;

// Online softmax state (m, z, mi): the maximum logit seen, z = sum e^(l - m)
// over the logits seen (e^x = 2^(x log2 e), by the SFU), and the lowest index
// of the maximum.  Merges (om, oz, oi).
__device__ __forceinline__ void merge_mz(float& m, float& z, int32_t& mi, float om, float oz, int32_t oi) {
  const float nm = fmaxf(m, om);
  if (nm != -INFINITY) z = z * ex2_approx((m - nm) * kLog2e) + oz * ex2_approx((om - nm) * kLog2e);
  if (om > m || (om == m && oi < mi)) mi = oi;
  m = nm;
}

// The SoftParts of a warp's lanes, and n more from shared memory (n a multiple
// of 32: lane l folds parts[l], parts[l + 32], ...), merged in a fixed order;
// every lane returns lane 0's result.  One rolled loop, not inlined: every
// merge of the step runs the same few lines of code.
__device__ __noinline__ SoftPart merge_lanes(SoftPart p, const SoftPart* parts, int n) {
  const int lane = threadIdx.x & 31;
  int i = lane, o = 16;
#pragma unroll 1
  for (;;) {
    SoftPart q;
    if (i < n) {  // (uniform: n is a multiple of 32)
      q = parts[i];
      i += 32;
    } else if (o > 0) {
      q.m = __shfl_xor_sync(0xffffffffu, p.m, o);
      q.z = __shfl_xor_sync(0xffffffffu, p.z, o);
      q.mi = __shfl_xor_sync(0xffffffffu, p.mi, o);
#pragma unroll
      for (int k = 0; k < kProbe; ++k) q.c[k] = __shfl_xor_sync(0xffffffffu, p.c[k], o);
      o >>= 1;
    } else {
      break;
    }
    merge_mz(p.m, p.z, p.mi, q.m, q.z, q.mi);
#pragma unroll
    for (int k = 0; k < kProbe; ++k) p.c[k] += q.c[k];
  }
  p.m = __shfl_sync(0xffffffffu, p.m, 0);  // (the lanes may differ in z's rounding)
  p.z = __shfl_sync(0xffffffffu, p.z, 0);
  p.mi = __shfl_sync(0xffffffffu, p.mi, 0);
  return p;
}

template <typename LT>
__global__ void __launch_bounds__(kSoftThreads, 1)
    soft_gate_kernel(TrieView t, int32_t rows_per_group, int32_t vocab, const LT* __restrict__ logits,
                     int64_t row_stride, bool vec, int32_t top_k, float rho, int32_t c, int32_t eos, int32_t max_len,
                     rgd_gate_state* __restrict__ state, uint8_t* __restrict__ row_active, int32_t* token_out,
                     float* mass_out, int32_t* dev_status) {
  constexpr int E = 16 / (int)sizeof(LT);   // logits per 16-byte vector
  constexpr int kVpc = kSoftChunk / 16;      // vectors per chunk
  constexpr int kWarps = kSoftThreads / 32;
  __shared__ SoftShared sh;
  extern __shared__ uint4 soft_buf[];  // kSoftStages chunks
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), K = (int)cluster.num_blocks();
  const int g = blockIdx.x / K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const LT* row = logits + (int64_t)g * row_stride;
  // this CTA's share of the row: vectors [lo, lo + nv) when the row is
  // 16-byte aligned (staged through shared memory), else elements [lo, hi_u)
  const int32_t nvec = vocab / E;
  const int32_t n_units = vec ? nvec : vocab;
  const int32_t lo = (int32_t)((int64_t)n_units * rank / K);
  const int32_t hi_u = (int32_t)((int64_t)n_units * (rank + 1) / K);
  const int32_t nv = vec ? hi_u - lo : 0;
  const int32_t nchunks = (nv + kVpc - 1) / kVpc;
  const uint4* rv = reinterpret_cast<const uint4*>(row);
  auto issue = [&](int32_t ck) {  // (thread 0) chunk ck into buffer ck % kSoftStages
    const uint32_t bytes = (uint32_t)min(kVpc, nv - ck * kVpc) * 16u;
    uint64_t* bar = &sh.full[ck % kSoftStages];
    mbar_arrive_expect_tx(bar, bytes);
    bulk_load(soft_buf + (ck % kSoftStages) * kVpc, rv + lo + ck * kVpc, bytes, bar);
  };
  bool timed_out = false;
  auto wait_chunk = [&](int32_t ck) {  // bounded; a second bounded wait after a timeout
    uint64_t* bar = &sh.full[ck % kSoftStages];
    const uint32_t par = (uint32_t)(ck / kSoftStages) & 1u;
    if (!mbar_wait(bar, par)) {
      timed_out = true;
      mbar_wait(bar, par);
    }
  };
  if (tid == 0) {
    for (int b = 0; b < kSoftStages; ++b) mbar_init(&sh.full[b], 1);
    fence_mbar_init();
    sh.ncand = 0;
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (a dependent waits for this kernel's end)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid == 0)
    for (int32_t ck = 0; ck < min(kSoftStages, nchunks); ++ck) issue(ck);
  // Every thread reads the state and takes the same decisions from it: the
  // kernel has no section where one warp works while the others wait.
  const rgd_gate_state s0 = state[g];
  __syncthreads();
  if (s0.done) {  // (uniform over the cluster) nothing to consume
    if (tid == 0) {
      for (int32_t ck = 0; ck < min(kSoftStages, nchunks); ++ck) wait_chunk(ck);  // (no copy outlives the CTA)
      if (timed_out && dev_status) atomicOr(dev_status, RGD_DEV_WAIT_TIMEOUT);
      if (rank == 0) {
        token_out[g] = -1;
        if (mass_out) mass_out[g] = -1.f;
      }
    }
    return;
  }
  cluster_arrive_relaxed();  // (waited for before the first push into another CTA)

  // ---- while the first chunks are in flight: the node's children (needed
  // unless the probe is confirmed) and, when the soft branch can be taken at
  // this step (the first c steps), the candidates' keys and the kProbe best ----
  const bool gather = !s0.confirmed;
  const bool maybe_soft = gather && s0.steps < c;
  int32_t cb = 0, nc = 0;
  if (gather) {
    cb = __ldg(t.child_begin + s0.node);
    nc = __ldg(t.child_begin + s0.node + 1) - cb;
  }
  const int32_t nslot = maybe_soft ? nc + 1 : nc;
  {
    int32_t mine = 0;
    for (int32_t k = tid; k < nslot; k += kSoftThreads) {
      int32_t a = eos;
      if (k < nc) {
        const int4 e = __ldg(t.edges + cb + k);
        a = e.x;
        sh.slot_tok[k] = a;
        sh.slot_node[k] = e.y;
        sh.slot_conf[k] = e.w < 0 ? 1 : 0;
      }
      if (maybe_soft) {
        const bool ok = a >= 0 && a < vocab && (k == nc || a != eos);
        sh.key[k] = ok ? rank_key(logit_at<LT>(row, a), a) : ~0ull;
        mine += ok ? 1 : 0;
      }
    }
    if (mine) atomicAdd(&sh.ncand, mine);
  }
  __syncthreads();
  const int32_t n = sh.ncand;        // candidates
  const int32_t hi = min(n, top_k);  // only the first hi of them can be in the top K
  const int32_t np_ = min(hi, kProbe);
  // the np_ smallest keys (every warp finds them: one warp-wide minimum each;
  // keys are distinct); their logits and tokens probe the pass
  float pv[kProbe];
  int32_t pi[kProbe], pc[kProbe];
  {
    uint64_t prev = 0;
#pragma unroll
    for (int q = 0; q < kProbe; ++q) {
      uint64_t best = ~0ull;
      if (q < np_) {
#pragma unroll 1
        for (int32_t k = lane; k < nslot; k += 32) {
          const uint64_t key = sh.key[k];
          if ((q == 0 || key > prev) && key < best) best = key;
        }
        const uint32_t bh = __reduce_min_sync(0xffffffffu, (uint32_t)(best >> 32));
        const uint32_t bl = __reduce_min_sync(0xffffffffu, (uint32_t)(best >> 32) == bh ? (uint32_t)best : ~0u);
        best = ((uint64_t)bh << 32) | bl;
      }
      prev = best;
      pv[q] = q < np_ ? key_logit(best) : INFINITY;  // (nothing ranks above +inf at index 0)
      pi[q] = q < np_ ? (int32_t)(uint32_t)best : 0;
      pc[q] = 0;
    }
  }
  const float p_min = np_ > 0 ? pv[np_ - 1] : INFINITY;  // only a logit >= this can rank above a probe

  // ---- the pass: maximum, its lowest index, z = sum e^(l - m), probe ranks ----
  float m = -INFINITY, z = 0.f, z_lo = 0.f;  // (z_lo: what z's sums round off)
  int32_t mi = 0x7fffffff;
  auto probe_counts = [&](float v, int32_t i) {
#pragma unroll
    for (int q = 0; q < kProbe; ++q) pc[q] += above(v, i, pv[q], pi[q]) ? 1 : 0;
  };
  auto add_z = [&](float x) {  // z += x, what the sum rounds off to z_lo
    const float sum = z + x, up = sum - z;
    z_lo += (z - (sum - up)) + (x - up);
    z = sum;
  };
  // a single logit (indices grow along a thread), summed in zs, which goes to z every
  // eight.  A thread's chain is as long as its CTA's share: added to z one by one,
  // without the rest that z_lo keeps, 262143 Zipf-ranked fp32 logits gave the mass an
  // rms error of 4.9e-7 with 6 CTAs a group and 1.2e-6 with 2; 1.7e-7 with either so
  float zs = 0.f;
  auto one = [&](float v, int32_t i) {
    if (v > m) {
      const float f = m == -INFINITY ? 0.f : ex2_approx((m - v) * kLog2e);
      z *= f;
      z_lo *= f;
      zs *= f;
      m = v;
      mi = i;
    }
    if (m != -INFINITY) zs += ex2_approx(fmaf(v, kLog2e, -m * kLog2e));
    if (v >= p_min) probe_counts(v, i);
  };
  if (vec) {
    for (int32_t ck = 0; ck < nchunks; ++ck) {
      wait_chunk(ck);
      const uint4* buf = soft_buf + (ck % kSoftStages) * kVpc;
      const int32_t cnt = min(kVpc, nv - ck * kVpc), base = lo + ck * kVpc;
      // this thread's vectors of the chunk: their maximum first, so that the
      // running maximum moves at most once per chunk
      float bm = -INFINITY;
#pragma unroll 1
      for (int32_t k = tid; k < cnt; k += kSoftThreads) {
        const uint4 x = buf[k];
#pragma unroll
        for (int e = 0; e < E; ++e) bm = fmaxf(bm, vec_elem<LT>(x, e));
      }
      if (bm > m) {  // the lowest index of bm here (indices grow along k, then e)
        int32_t bi = 0x7fffffff;
#pragma unroll 1
        for (int32_t k = tid; k < cnt && bi == 0x7fffffff; k += kSoftThreads) {
          const uint4 x = buf[k];
#pragma unroll
          for (int e = E - 1; e >= 0; --e)
            if (vec_elem<LT>(x, e) == bm) bi = (base + k) * E + e;
        }
        const float f = m == -INFINITY ? 0.f : ex2_approx((m - bm) * kLog2e);
        z *= f;
        z_lo *= f;
        m = bm;
        mi = bi;
      }
      // z, and the probes for the few logits at or above the weakest one
      if (m != -INFINITY) {
        const float ml = m * kLog2e;
        float zc = 0.f;  // (a chunk's share: short sums round less)
#pragma unroll 1
        for (int32_t k = tid; k < cnt; k += kSoftThreads) {
          const uint4 x = buf[k];
          float z0 = 0.f, z1 = 0.f;
#pragma unroll
          for (int e = 0; e < E; e += 2) {
            const float v0 = vec_elem<LT>(x, e), v1 = vec_elem<LT>(x, e + 1);
            z0 += ex2_approx(fmaf(v0, kLog2e, -ml));
            z1 += ex2_approx(fmaf(v1, kLog2e, -ml));
            if (v0 >= p_min) probe_counts(v0, (base + k) * E + e);
            if (v1 >= p_min) probe_counts(v1, (base + k) * E + e + 1);
          }
          zc += z0 + z1;
        }
        add_z(zc);
      } else if (bm >= p_min) {  // (every logit so far is -inf, and so is a probed candidate)
#pragma unroll 1
        for (int32_t k = tid; k < cnt; k += kSoftThreads) {
          const uint4 x = buf[k];
#pragma unroll
          for (int e = 0; e < E; ++e) probe_counts(vec_elem<LT>(x, e), (base + k) * E + e);
        }
      }
      if (ck + kSoftStages < nchunks) {
        __syncthreads();  // the buffer is free
        if (tid == 0) issue(ck + kSoftStages);
      }
    }
    // the few logits past the last whole vector
    const int32_t i = nvec * E + tid;
    if (rank == K - 1 && i < vocab) one(logit_at<LT>(row, i), i);
  } else {
    scan_row<kSoftThreads, 8, LT>(row, vocab, false, rank, K, one, [&] {
      add_z(zs);
      zs = 0.f;
    });
  }
  z += z_lo + zs;
  if (timed_out && dev_status) atomicOr(dev_status, RGD_DEV_WAIT_TIMEOUT);  // (the outputs are then not valid)

  // ---- every warp's share -> every CTA of the cluster ----
  {
    SoftPart p;
    p.m = m;
    p.z = z;
    p.mi = mi;
#pragma unroll
    for (int q = 0; q < kProbe; ++q) p.c[q] = pc[q];
    p = merge_lanes(p, nullptr, 0);
    cluster_wait();  // every CTA of the cluster has started
    if (lane < K) cluster.map_shared_rank(&sh, lane)->part[rank * kWarps + warp] = p;
  }
  cluster.sync();  // every warp's share is in every CTA's shared memory
  // ---- the same combination, in the same order, in every warp of the cluster ----
  SoftPart all;
  all.m = -INFINITY;
  all.z = 0.f;
  all.mi = 0x7fffffff;
#pragma unroll
  for (int q = 0; q < kProbe; ++q) all.c[q] = 0;
  all = merge_lanes(all, sh.part, K * kWarps);  // (K is even: a multiple of 32)
  const int32_t y = all.mi;
  // the children labelled y and a* (the best candidate), if any
  const int32_t a_star = np_ > 0 ? pi[0] : -1;
  int32_t sy = -1, sa = -1;
#pragma unroll 1
  for (int32_t k = lane; k < nc; k += 32) {
    const int32_t tk = sh.slot_tok[k];
    if (tk == y) sy = k;  // (a node's children have distinct tokens)
    if (tk == a_star) sa = k;
  }
  sy = __reduce_max_sync(0xffffffffu, sy);
  sa = __reduce_max_sync(0xffffffffu, sa);
  const bool stop = eos >= 0 && y == eos;
  const bool compatible = s0.confirmed || sy >= 0;
  const bool soft = !(s0.steps >= c || stop || compatible);  // else the hard step with y
  // the probed candidates in the top K (a prefix: ranks grow along the order)
  int32_t n_in = 0;
  if (soft)
    while (n_in < np_ && all.c[n_in] < top_k) ++n_in;
  if (soft && n_in == np_ && np_ < hi) {
    // ---- the rest: sort the candidates (bitonic, padded to a power of two;
    // the first np_ are the probed ones), then a search over
    // candidates np_ .. hi - 1 (every thread of the cluster takes the same steps) ----
    int32_t np2 = 1;
    while (np2 < nslot) np2 <<= 1;
    for (int32_t i = nslot + tid; i < np2; i += kSoftThreads) sh.key[i] = ~0ull;
    __syncthreads();
    for (int32_t k = 2; k <= np2; k <<= 1) {
      for (int32_t j = k >> 1; j > 0; j >>= 1) {
        for (int32_t i = tid; i < np2; i += kSoftThreads) {
          const int32_t ij = i ^ j;
          if (ij > i) {
            const uint64_t a = sh.key[i], b2 = sh.key[ij];
            if ((a > b2) == ((i & k) == 0)) {
              sh.key[i] = b2;
              sh.key[ij] = a;
            }
          }
        }
        __syncthreads();
      }
    }
    int32_t lo_c = np_, hi_c = hi, step = 1;
    bool out = false;  // a candidate outside the top K has been found
    const bool staged = vec && nchunks <= kSoftStages;  // (the share's chunks are contiguous and still there)
#pragma unroll 1
    for (int pass = 0; lo_c < hi_c; ++pass) {
      const int32_t mid = out ? (lo_c + hi_c) >> 1 : min(lo_c + step - 1, hi_c - 1);
      const uint64_t key = sh.key[mid];
      const float cv = key_logit(key);
      const int32_t ci = (int32_t)(uint32_t)key;
      if (tid == 0) sh.cnt_cta = 0;
      __syncthreads();
      int32_t cnt = 0;
      auto count = [&](float v, int32_t i) { cnt += above(v, i, cv, ci) ? 1 : 0; };
      if (staged) {
#pragma unroll 2
        for (int32_t k = tid; k < nv; k += kSoftThreads) {
          const uint4 x = soft_buf[k];
#pragma unroll
          for (int e = 0; e < E; ++e) count(vec_elem<LT>(x, e), (lo + k) * E + e);
        }
        const int32_t i = nvec * E + tid;
        if (rank == K - 1 && i < vocab) count(logit_at<LT>(row, i), i);
      } else {
        scan_row<kSoftThreads, 8, LT>(row, vocab, vec, rank, K, count, [] {});
      }
      cnt = __reduce_add_sync(0xffffffffu, cnt);
      if (lane == 0 && cnt) atomicAdd(&sh.cnt_cta, cnt);
      __syncthreads();
      // CTA r's slot of this pass's parity is next written two passes on,
      // after every CTA has passed the next cluster barrier (and read this one)
      if (warp == 0 && lane < K) cluster.map_shared_rank(&sh, lane)->cnt[pass & 1][rank] = sh.cnt_cta;
      cluster.sync();
      int32_t total = 0;
      for (int r = 0; r < K; ++r) total += sh.cnt[pass & 1][r];
      if (total < top_k) {
        lo_c = mid + 1;
        step *= 2;
      } else {
        hi_c = mid;
        out = true;
      }
    }
    n_in = lo_c;
  }
  // (no CTA touches another's shared memory after the last cluster barrier)
  if (warp != 0 || rank != 0) return;
  // ---- the step's outcome (warp 0 of CTA 0) ----
  float mass = -1.f;
  if (soft) {
    // m = the probability mass of the candidates in the top K
    const float ml = all.m * kLog2e;
    float part = 0.f;
    for (int32_t k = lane; k < n_in; k += 32) {
      float l = 0.f;
#pragma unroll
      for (int q = 0; q < kProbe; ++q)
        if (k == q) l = pv[q];
      if (k >= kProbe) l = key_logit(sh.key[k]);
      part += ex2_approx(fmaf(l, kLog2e, -ml));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    mass = part / all.z;
  }
  if (lane != 0) return;
  rgd_gate_state s = s0;
  auto child = [&](int32_t tok) {  // the gathered children: tok is y or a*
    const int32_t k = tok == y ? sy : sa;
    return k < 0 ? make_int2(-1, 0) : make_int2(sh.slot_node[k], (int)sh.slot_conf[k]);
  };
  const bool root_has_children = __ldg(t.child_begin + 1) > __ldg(t.child_begin);
  int32_t tok = -1;
  if (!soft) {
    tok = y;
    consume_token_with(s, tok, eos, max_len, root_has_children, child);
  } else if (n_in > 0 && mass >= rho) {
    tok = a_star;  // the most probable compatible token
    consume_token_with(s, tok, eos, max_len, root_has_children, child);
  } else {  // no refusal-like alternative with enough mass: discard the probe
    s.decision = RGD_NON_REFUSAL;
    s.decisive_step = s.steps;
    s.steps++;
    s.done = 1;
  }
  state[g] = s;
  token_out[g] = tok;
  if (mass_out) mass_out[g] = soft ? mass : -1.f;
  mask_rows(s, row_active, g, rows_per_group);
}

// Clusters of K CTAs of the soft gate that the current device holds at once, asked
// of the runtime once per device, logit type and K.
cudaError_t soft_clusters(cudaLaunchConfig_t cfg, int32_t dtype, int K, int* out) {
  constexpr int kMaxDev = 16;
  static std::atomic<int> cache[kMaxDev][2][kSoftCluster + 1] = {};  // clusters + 1; 0: not asked yet
  int dev = 0;
  if (cudaError_t e = cudaGetDevice(&dev); e != cudaSuccess) return e;
  std::atomic<int>* c = dev < kMaxDev ? &cache[dev][dtype == RGD_F32 ? 0 : 1][K] : nullptr;
  if (const int n = c ? c->load(std::memory_order_relaxed) : 0; n > 0) {
    *out = n - 1;
    return cudaSuccess;
  }
  cfg.gridDim = dim3((unsigned)K);
  cfg.numAttrs = 1;
  const cudaError_t e = dtype == RGD_F32 ? cudaOccupancyMaxActiveClusters(out, soft_gate_kernel<float>, &cfg)
                                         : cudaOccupancyMaxActiveClusters(out, soft_gate_kernel<uint16_t>, &cfg);
  if (e == cudaSuccess && c) c->store(*out + 1, std::memory_order_relaxed);
  return e;
}

}  // namespace
}  // namespace rgd

using namespace rgd;

extern "C" int rgd_trie_create(const int32_t* tokens, const int64_t* offsets, int32_t n_seq,
                               int32_t min_confirm, rgd_trie** out) {
  clear_error();
  RGD_CHECK_ARG(out != nullptr, "rgd_trie_create: out is NULL");
  *out = nullptr;
  RGD_CHECK_ARG(n_seq >= 0, "rgd_trie_create: n_seq < 0");
  RGD_CHECK_ARG(min_confirm >= 1, "rgd_trie_create: min_confirm must be >= 1");
  RGD_CHECK_ARG(n_seq == 0 || (tokens != nullptr && offsets != nullptr),
                "rgd_trie_create: tokens/offsets are NULL");
  if (n_seq > 0) RGD_CHECK_ARG(offsets[0] == 0, "rgd_trie_create: offsets[0] != 0");
  // host build: nodes with ordered children (std::map keeps tokens sorted)
  std::vector<std::map<int32_t, int32_t>> kids(1);
  std::vector<int32_t> depth(1, 0);
  std::vector<uint8_t> terminal(1, 0);
  for (int32_t s = 0; s < n_seq; ++s) {
    const int64_t b = offsets[s], e = offsets[s + 1];
    RGD_CHECK_ARG(e > b, "rgd_trie_create: sequence %d is empty or offsets decrease", s);
    int32_t node = 0;
    for (int64_t i = b; i < e; ++i) {
      const int32_t tok = tokens[i];
      RGD_CHECK_ARG(tok >= 0, "rgd_trie_create: negative token in sequence %d", s);
      auto it = kids[node].find(tok);
      if (it == kids[node].end()) {
        const int32_t nn = (int32_t)kids.size();
        kids[node][tok] = nn;
        kids.emplace_back();
        depth.push_back(depth[node] + 1);
        terminal.push_back(0);
        node = nn;
      } else {
        node = it->second;
      }
    }
    terminal[node] = 1;
  }
  const int32_t nn = (int32_t)kids.size();
  std::vector<int32_t> begin(nn + 1, 0);
  int32_t max_children = 0;
  for (int32_t n = 0; n < nn; ++n) {
    max_children = std::max(max_children, (int32_t)kids[n].size());
    begin[n + 1] = begin[n] + (int32_t)kids[n].size();
  }
  std::vector<int4> edges;
  for (int32_t n = 0; n < nn; ++n) {
    for (const auto& [tok, node] : kids[n]) {
      const uint32_t confirm = terminal[node] && depth[node] >= min_confirm ? 1u << 31 : 0u;
      edges.push_back(make_int4(tok, node, begin[node], (int32_t)((uint32_t)kids[node].size() | confirm)));
    }
  }
  if (edges.empty()) edges.push_back(make_int4(-1, 0, 0, 0));  // keep the device array non-empty
  rgd_trie* t = new rgd_trie();
  t->num_nodes = nn;
  t->num_edges = begin[nn];
  t->max_children = max_children;
  cudaGetDevice(&t->device);
  cudaError_t err = cudaSuccess;
  auto upload = [&](void** dst, const void* src, size_t bytes) {
    if (err != cudaSuccess) return;
    err = cudaMalloc(dst, bytes);
    if (err == cudaSuccess) err = cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice);
  };
  upload((void**)&t->child_begin, begin.data(), begin.size() * sizeof(int32_t));
  upload((void**)&t->edges, edges.data(), edges.size() * sizeof(int4));
  if (err != cudaSuccess) {
    rgd_trie_destroy(t);
    return cuda_error(err, "rgd_trie_create upload");
  }
  *out = t;
  return RGD_OK;
}

extern "C" int rgd_trie_destroy(rgd_trie* t) {
  if (!t) return RGD_OK;
  cudaFree(t->child_begin);
  cudaFree(t->edges);
  delete t;
  return RGD_OK;
}

extern "C" int rgd_trie_info(const rgd_trie* t, int32_t* num_nodes, int32_t* num_edges) {
  clear_error();
  RGD_CHECK_ARG(t != nullptr, "rgd_trie_info: trie is NULL");
  if (num_nodes) *num_nodes = t->num_nodes;
  if (num_edges) *num_edges = t->num_edges;
  return RGD_OK;
}

extern "C" int rgd_gate_state_init(rgd_gate_state* state, int32_t groups, rgd_stream_t stream) {
  clear_error();
  RGD_CHECK_ARG(groups >= 0, "rgd_gate_state_init: groups < 0");
  if (groups == 0) return RGD_OK;
  RGD_CHECK_ARG(state != nullptr, "rgd_gate_state_init: state is NULL");
  const int threads = 128;
  const cudaError_t e = launch_dependent(gate_state_init_kernel, (groups + threads - 1) / threads, threads, 0,
                                         (cudaStream_t)stream, state, groups);
  return e == cudaSuccess ? RGD_OK : cuda_error(e, "gate_state_init launch");
}

extern "C" int rgd_probe_gate(const rgd_trie* trie, int32_t groups, int32_t rows_per_group,
                              const int32_t* probe_tokens, int32_t n_tokens, int64_t token_stride,
                              int32_t eos_token, int32_t max_len, rgd_gate_state* state,
                              uint8_t* row_active, int32_t* dev_status, rgd_stream_t stream) {
  clear_error();
  RGD_CHECK_ARG(trie != nullptr, "rgd_probe_gate: trie is NULL");
  RGD_CHECK_ARG(groups >= 0 && rows_per_group >= 1, "rgd_probe_gate: bad groups/rows_per_group");
  RGD_CHECK_ARG(n_tokens >= 0 && token_stride >= n_tokens, "rgd_probe_gate: bad n_tokens/token_stride");
  RGD_CHECK_ARG(max_len >= 1, "rgd_probe_gate: max_len must be >= 1");
  if (groups == 0 || n_tokens == 0) return RGD_OK;
  RGD_CHECK_ARG(probe_tokens != nullptr && state != nullptr, "rgd_probe_gate: tokens/state NULL");
  TrieView v{trie->child_begin, trie->edges};
  constexpr int kPer = kGateThreads / 32;  // groups per block
  const cudaError_t e = launch_dependent(probe_gate_kernel, groups / kPer + (groups % kPer != 0), kGateThreads, 0,
                                         (cudaStream_t)stream, v, groups, rows_per_group, probe_tokens, n_tokens,
                                         token_stride, eos_token, max_len, state, row_active, dev_status);
  return e == cudaSuccess ? RGD_OK : cuda_error(e, "probe_gate launch");
}

extern "C" int rgd_soft_gate(const rgd_trie* trie, int32_t groups, int32_t rows_per_group, int32_t vocab,
                             int32_t dtype, const void* probe_logits, int64_t row_stride, int32_t top_k, float rho,
                             int32_t c, int32_t eos_token, int32_t max_len, rgd_gate_state* state,
                             uint8_t* row_active, int32_t* token_out, float* mass_out, int32_t* dev_status,
                             rgd_stream_t stream) {
  clear_error();
  RGD_CHECK_ARG(trie != nullptr, "rgd_soft_gate: trie is NULL");
  RGD_CHECK_ARG(groups >= 0 && groups <= INT32_MAX / 6 && rows_per_group >= 1 && vocab >= 1,
                "rgd_soft_gate: bad groups/rows/vocab");
  RGD_CHECK_ARG(dtype == RGD_F32 || dtype == RGD_BF16, "rgd_soft_gate: dtype must be RGD_F32 or RGD_BF16");
  RGD_CHECK_ARG(row_stride >= vocab, "rgd_soft_gate: row_stride < vocab");
  RGD_CHECK_ARG(top_k >= 1 && c >= 0 && max_len >= 1, "rgd_soft_gate: need top_k >= 1, c >= 0, max_len >= 1");
  RGD_CHECK_ARG(std::isfinite(rho), "rgd_soft_gate: rho must be finite");
  if (trie->max_children + 1 > kMaxCand)
    return set_error(RGD_ERR_UNSUPPORTED, "rgd_soft_gate: a trie node has %d children (max %d)",
                     trie->max_children, kMaxCand - 1);
  if (groups == 0) return RGD_OK;
  RGD_CHECK_ARG(probe_logits != nullptr && state != nullptr && token_out != nullptr,
                "rgd_soft_gate: logits/state/token_out NULL");
  TrieView tv{trie->child_begin, trie->edges};
  cudaStream_t st = (cudaStream_t)stream;
  const int es = dtype == RGD_F32 ? 4 : 2;
  const bool vec = aligned16(probe_logits) && (row_stride * es) % 16 == 0;  // 16-byte vector loads
  constexpr int kDyn = kSoftStages * kSoftChunk;  // chunk buffers (dynamic shared memory)
  static std::atomic<bool> done[2][kMaxDevices] = {};
  if (int rc = dtype == RGD_F32 ? ensure_smem(soft_gate_kernel<float>, kDyn, done[0])
                                : ensure_smem(soft_gate_kernel<uint16_t>, kDyn, done[1]))
    return rc;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kSoftThreads);
  cfg.dynamicSmemBytes = kDyn;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  // CTAs per group: as many as let every group's cluster run at once (one CTA on an
  // SM; clusters of 6 and 4 leave some of a processing cluster's SMs out): a second
  // wave costs more than a longer share.  6 / 4 / 2 CTAs inside a graph, K = 40, 128256
  // fp32 logits: 16 groups 13.7 / 16.1 / 23.7 us; 24 groups 19.7 / 16.3 / 23.7; 64
  // groups 33.8 / 29.6 / 25.2; 200 groups of 32000 64 / 46 / 31 (1 CTA: 29).
  int K = kSoftCluster;
  cudaError_t e = cudaSuccess;
  for (;; K -= 2) {
    attr[0].val.clusterDim = {(unsigned)K, 1, 1};
    if (K == 2) break;
    int n = 0;
    if ((e = soft_clusters(cfg, dtype, K, &n)) != cudaSuccess) return cuda_error(e, "soft_gate occupancy");
    if (groups <= n) break;
  }
  cfg.gridDim = dim3((unsigned)(groups * K));
  cfg.numAttrs = 2;
  if (dtype == RGD_F32)
    e = cudaLaunchKernelEx(&cfg, soft_gate_kernel<float>, tv, rows_per_group, vocab,
                           static_cast<const float*>(probe_logits), row_stride, vec, top_k, rho, c, eos_token, max_len,
                           state, row_active, token_out, mass_out, dev_status);
  else
    e = cudaLaunchKernelEx(&cfg, soft_gate_kernel<uint16_t>, tv, rows_per_group, vocab,
                           static_cast<const uint16_t*>(probe_logits), row_stride, vec, top_k, rho, c, eos_token,
                           max_len, state, row_active, token_out, mass_out, dev_status);
  if (e == cudaSuccess) e = cudaGetLastError();
  return e == cudaSuccess ? RGD_OK : cuda_error(e, "soft_gate launch");
}
