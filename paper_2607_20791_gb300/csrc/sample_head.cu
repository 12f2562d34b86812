// Sample head: the greedy step G_M and the truncated high-temperature sampler
// S_{T,theta} of Alg. 1, with min-p truncation and a Philox4x32-10 inverse-CDF
// draw.
//
// One thread-block cluster of K CTAs (K chosen per call) handles one row at a
// time and walks the rows cluster by cluster.  A row is read from HBM once: its
// 16-byte vectors are cut into K equal contiguous shares, and each CTA's copy warp
// brings its share into a ring of shared-memory slots of 1024 vectors, one bulk copy
// each.  A slot is eight stream warps' work, four stripes (32 vectors, one a lane)
// each, and holds the row until its second pass is over.  Pass 1 finds the row's max
// and lowest-index argmax (each warp sends its own to every CTA of the cluster);
// probe rows need no more.  Sample rows form the min-p cutoff from the max and, in
// pass 2, sum the kept weights of every stripe from shared memory; every slot that
// pass 2 has finished takes a slot of the cluster's next row at once, so the
// copies of the next row run behind this row's exchange and second pass.  The
// draw belongs to a ninth warp per CTA, which works on row i while the stream
// warps go on with row i + 1: the Philox target u * Z picks CTA, lane segment and
// stripe by prefix sums in index order, and that one stripe is read again to find
// the lane and the element.
//
// A stripe's weights (128 or 256) are summed in fp32 by a tree: 7 or 9 roundings one
// above the other, 8 or 12 in a slot that is not all the row's.  So a stripe's sum is
// at most 12 x 2^-24 = 7e-7 of itself off, and the cumulative sums no more of Z:
// inside the 1e-6 of Z within which a draw counts as a boundary case.  From there on
// sums are 64-bit fixed point, exact in any order; FP64 is slow on this part, and the
// only fp64 step is the cutoff's logarithm, off the stream warps' path.
//
// What bounds it: see launch_head (the split per size) for the measured figures.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.h"
#include "ptx.cuh"
#include "trie.cuh"

namespace rgd {
namespace {

constexpr int kMaxCluster = 16;  // CTAs per row at most (8 unless the row needs more)
constexpr int kHeadWarps = 8;    // stream warps per CTA; then the draw warp and the copy warp
constexpr int kHeadThreads = (kHeadWarps + 2) * 32;
constexpr int kSlotStripes = 4;  // stripes (32 vectors of 16 bytes) per stream warp and ring slot
constexpr int kSlotVecs = kHeadWarps * kSlotStripes * 32;
constexpr int kSlotBytes = kSlotVecs * 16;  // one bulk copy
constexpr int kMaxSlots = 13;    // ring slots

struct HeadParams {
  const uint8_t* logits;
  int32_t rows;
  int32_t vocab;
  int32_t cvec;    // vectors of a row per CTA (a multiple of 32)
  int32_t nslots;  // ring slots (at least a row's)
  int32_t early;   // the inputs are complete before the previous kernel on the stream (see rgd_decode_step)
  int64_t total_bytes;  // of logits
  const uint8_t* is_probe;
  const float* temperature;
  const float* min_p;
  const uint64_t* seed;
  uint64_t step;
  const uint8_t* row_active;
  int32_t* token_out;
  int32_t* kept_count;
  uint8_t* kept_mask;
  int32_t* dev_status;
  // the fused gate (gstate == nullptr: none): rows g * rpg .. g * rpg + rpg - 1
  // form group g, whose probe token (row g * rpg) goes through the hard gate
  TrieView trie;
  rgd_gate_state* gstate;
  uint8_t* gate_row_active;  // row_active, written by the gate
  int32_t rpg, eos, max_len;
};

// The fused gate.  The thread that writes a row's token then counts the row as
// finished in the top byte of its group's gate-state word {decision, confirmed,
// done, reserved}.  The probe row's thread first feeds its token to the hard
// gate (exactly rgd_probe_gate's step): it writes the state's integer fields
// directly and the decision, confirmed and done bytes by atomics, which leave
// the count in the top byte alone.  The group's last row to finish -- by then
// every row of the group has drawn its token and read its activity flag, and
// the probe's outcome is in the word its count returns -- masks the group's rows
// and sets the count back to zero.  Nothing waits, and the trie walk runs on
// the probe row, whose greedy path ends long before the sampled rows'.
__device__ __noinline__ void finish_row(const HeadParams& p, int row, int32_t tok) {
  const int g = row / p.rpg;
  rgd_gate_state* st = p.gstate + g;
  uint32_t* word = reinterpret_cast<uint32_t*>(&st->decision);
  if (row == g * p.rpg) {
    const uint32_t w0 = *reinterpret_cast<volatile uint32_t*>(word);  // (only this thread changes the low bytes)
    rgd_gate_state s;
    s.done = (uint8_t)((w0 >> 16) & 0xffu);
    if (!s.done) {
      if (tok < 0 && !(p.eos >= 0 && tok == p.eos)) {
        if (p.dev_status) atomicOr(p.dev_status, RGD_DEV_BAD_TOKEN);  // (an inactive or rejected probe row)
      } else {
        s.node = st->node;
        s.length = st->length;
        s.steps = st->steps;
        s.decisive_step = st->decisive_step;
        s.decision = (uint8_t)(w0 & 0xffu);
        s.confirmed = (uint8_t)((w0 >> 8) & 0xffu);
        const bool root_has_children = __ldg(p.trie.child_begin + 1) > __ldg(p.trie.child_begin);
        consume_token(p.trie, s, tok, p.eos, p.max_len, root_has_children);
        st->node = s.node;
        st->length = s.length;
        st->steps = s.steps;
        st->decisive_step = s.decisive_step;
        atomicAnd(word, 0xff000000u);
        atomicOr(word, (uint32_t)s.decision | ((uint32_t)s.confirmed << 8) | ((uint32_t)s.done << 16));
      }
    }
  }
  const uint32_t old = atomicAdd(word, 1u << 24);
  if ((int)(old >> 24) != p.rpg - 1) return;
  *word = old & 0x00ffffffu;  // the count back to 0 (every row of the group has counted itself)
  rgd_gate_state s;
  s.decision = (uint8_t)(old & 0xffu);
  s.done = (uint8_t)((old >> 16) & 0xffu);
  mask_rows(s, p.gate_row_active, g, p.rpg);
}

// Two fp32 values in one 64-bit register, and arithmetic on both at once.
__device__ __forceinline__ uint64_t pair(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float pair_sum(uint64_t a) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
  return x + y;
}
// 2^((l - M) kexp) of two logits, the same steps as kept_weight's.
__device__ __forceinline__ uint64_t weights2(uint64_t l, uint64_t neg_max, uint64_t kexp) {
  uint64_t t = add2(l, neg_max);
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(t), "l"(kexp));
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(t));
  return pair(ex2_approx(x), ex2_approx(y));
}
__device__ __forceinline__ uint4 lds128(uint32_t at) {
  uint4 w;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "r"(at));
  return w;
}

// 16 bytes of logits: 4 fp32 or 8 bf16 elements.
template <typename T>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int kN = 4, kSize = 4;
  static constexpr uint32_t kNegInf = 0xff800000u, kNegInfWord = 0xff800000u;
  __device__ static float get(const uint4& w, int k) {
    const uint32_t u = k == 0 ? w.x : k == 1 ? w.y : k == 2 ? w.z : w.w;
    return __uint_as_float(u);
  }
  __device__ static uint32_t scalar(const uint8_t* p) { return *reinterpret_cast<const uint32_t*>(p); }
  // The maximum of four vectors.
  __device__ static float max4(const uint4 (&w)[4]) {
    auto f = [](uint32_t u) { return __uint_as_float(u); };
    float m = f(w[0].x);
#pragma unroll
    for (int s = 0; s < 4; ++s) m = fmaxf(fmaxf(fmaxf(fmaxf(m, f(w[s].x)), f(w[s].y)), f(w[s].z)), f(w[s].w));
    return m;
  }
  // A row's cutoff, and what its weights need.
  struct Cut {
    float cut;
    uint64_t neg_max, kexp;
    __device__ Cut(float c, float M, float k) : cut(c), neg_max(pair(-M, -M)), kexp(pair(k, k)) {}
  };
  // The sum of a vector's kept weights; their number is added to cnt.
  __device__ static float kept(const uint4& w, const Cut& c, int32_t& cnt) {
    float l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool keep = get(w, k) >= c.cut;
      l[k] = keep ? get(w, k) : -INFINITY;
      cnt += keep ? 1 : 0;
    }
    return pair_sum(add2(weights2(pair(l[0], l[1]), c.neg_max, c.kexp), weights2(pair(l[2], l[3]), c.neg_max, c.kexp)));
  }
};
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int kN = 8, kSize = 2;
  static constexpr uint32_t kNegInf = 0xff80u, kNegInfWord = 0xff80ff80u;
  __device__ static float get(const uint4& w, int k) {
    const uint32_t u = (k >> 1) == 0 ? w.x : (k >> 1) == 1 ? w.y : (k >> 1) == 2 ? w.z : w.w;
    return __uint_as_float((k & 1) ? (u & 0xffff0000u) : (u << 16));
  }
  __device__ static uint32_t scalar(const uint8_t* p) { return *reinterpret_cast<const uint16_t*>(p); }
  __device__ static __nv_bfloat162 b2(uint32_t u) { return *reinterpret_cast<const __nv_bfloat162*>(&u); }
  __device__ static float max4(const uint4 (&w)[4]) {  // two elements at a time (NaN never wins, as with fmaxf)
    __nv_bfloat162 m = b2(w[0].x);
#pragma unroll
    for (int s = 0; s < 4; ++s) m = __hmax2(__hmax2(__hmax2(__hmax2(m, b2(w[s].x)), b2(w[s].y)), b2(w[s].z)), b2(w[s].w));
    const uint32_t u = *reinterpret_cast<const uint32_t*>(&m);
    return fmaxf(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
  }
  // A bf16 is >= the fp32 cutoff exactly if it is >= the cutoff rounded up to bf16.
  struct Cut {
    __nv_bfloat162 cut;
    uint64_t neg_max, kexp;
    __device__ Cut(float c, float M, float k)
        : cut(__bfloat162bfloat162(__float2bfloat16_ru(c))), neg_max(pair(-M, -M)), kexp(pair(k, k)) {}
  };
  __device__ static float kept(const uint4& w, const Cut& c, int32_t& cnt) {
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
    uint64_t s = 0;
    uint32_t bits = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t m = __hge2_mask(b2(u[i]), c.cut);
      bits |= m & (0x00010001u << i);
      const uint32_t l = (u[i] & m) | (kNegInfWord & ~m);
      const uint64_t x = weights2(pair(__uint_as_float(l << 16), __uint_as_float(l & 0xffff0000u)), c.neg_max, c.kexp);
      s = i ? add2(s, x) : x;
    }
    cnt += __popc(bits);
    return pair_sum(s);
  }
};

// A row as 16-byte vectors of memory: vector v of the row holds elements
// v * kN - shift + k.  Aligned rows start on a vector (shift 0) and hold a whole
// number of them; else the first and last vectors also hold other rows' elements
// (masked to -inf), and the last vector of the buffer may reach past its end.
struct RowView {
  const uint8_t* base;  // 16-byte aligned address of vector 0
  int32_t shift;
  int32_t nvec;
  int32_t nfull;  // vectors that lie within the buffer (nvec, or nvec - 1)
};

template <typename T, bool kAligned>
__device__ __forceinline__ RowView row_view(const HeadParams& p, int row) {
  constexpr int kSize = Vec<T>::kSize;
  const int64_t b0 = (int64_t)row * p.vocab * kSize, b1 = b0 + (int64_t)p.vocab * kSize;
  RowView r;
  if (kAligned) {
    r.base = p.logits + b0;
    r.shift = 0;
    r.nvec = r.nfull = (int32_t)((b1 - b0) >> 4);
  } else {
    const int64_t a0 = b0 & ~int64_t(15);
    r.base = p.logits + a0;
    r.shift = (int32_t)(b0 - a0) / kSize;
    r.nvec = (int32_t)((b1 - a0 + 15) >> 4);
    r.nfull = (int32_t)(min(b1 - a0 + 15, p.total_bytes - a0) >> 4);
  }
  return r;
}

// The elements of vector v that belong to the row; the others read as -inf.
template <typename T>
__device__ __forceinline__ void mask_vec(uint4& w, int64_t e0, int32_t vocab) {
  using V = Vec<T>;
  if (e0 >= 0 && e0 + V::kN <= vocab) return;
  uint32_t* u = reinterpret_cast<uint32_t*>(&w);
#pragma unroll
  for (int k = 0; k < V::kN; ++k) {
    if (e0 + k >= 0 && e0 + k < vocab) continue;
    if (V::kSize == 4) u[k] = 0xff800000u;
    else u[k >> 1] = (k & 1) ? ((u[k >> 1] & 0xffffu) | 0xff800000u) : ((u[k >> 1] & 0xffff0000u) | 0xff80u);
  }
}

// Vector v of a row read element by element from global memory (the last
// vector of a buffer that ends within it).
template <typename T>
__device__ __noinline__ uint4 load_vec_scalar(const RowView rv, int32_t v, int32_t vocab) {
  using V = Vec<T>;
  const int64_t e0 = (int64_t)v * V::kN - rv.shift;
  uint32_t u[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint8_t* q = rv.base + (int64_t)v * 16 + 4 * k;
    if (V::kSize == 4) {
      u[k] = (e0 + k >= 0 && e0 + k < vocab) ? V::scalar(q) : V::kNegInf;
    } else {
      const uint32_t lo = (e0 + 2 * k >= 0 && e0 + 2 * k < vocab) ? V::scalar(q) : V::kNegInf;
      const uint32_t hi = (e0 + 2 * k + 1 >= 0 && e0 + 2 * k + 1 < vocab) ? V::scalar(q + 2) : V::kNegInf;
      u[k] = lo | (hi << 16);
    }
  }
  return make_uint4(u[0], u[1], u[2], u[3]);
}

// Philox4x32-10 (Salmon et al., SC'11): word 0 of the block for (counter, key).
__device__ __forceinline__ uint32_t philox_word0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                 uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  return c0;
}

// What a row's passes need besides its logits.
struct RowParams {
  float theta;  // T ln p_min
  float kexp;   // log2(e) / T
  uint32_t u24;  // the draw's uniform, u = u24 2^-24
  uint8_t greedy, valid;
};

// Row buffers are doubled (row i of a cluster uses buffer i & 1).
struct Shared {
  // pushed by every stream warp of the cluster into every CTA (slot = 8 rank + warp): its max and argmax
  uint64_t wmax[2][kMaxCluster * kHeadWarps];
  // pushed by every CTA's draw warp into every CTA (slot = rank): its weight sum, its count
  uint64_t csum[2][kMaxCluster], ccnt[2][kMaxCluster];
  // this CTA's stream warps -> its draw warp
  uint64_t stripe_sum[2][kMaxSlots * 32];  // in index order
  uint64_t wsum[2][kHeadWarps];
  int32_t wcnt[2][kHeadWarps];
  float row_max[2];
  int32_t row_arg[2];
  RowParams prm[2][32];  // a block of the cluster's rows with an active one: the draw warp -> the stream warps
  uint64_t full_bar[kMaxSlots];   // a ring slot's copy has landed
  uint64_t empty_bar[kMaxSlots];  // every stream warp is done with the slot
  uint64_t max_bar[2];   // every warp's max is in wmax
  uint64_t sum_bar[2];   // this CTA's stream warps are done with the row
  uint64_t csum_bar[2];  // every CTA's sum is in csum
  uint64_t prm_bar[2];   // the block's parameters are in place (blocks without an active row have no phase)
  uint64_t free_bar[2];  // the draw warp is done with the row
  int32_t abort;         // a wait gave up: every later wait returns at once
};

// The address of a shared-memory object of this CTA in CTA `rank` of its cluster.
__device__ __forceinline__ uint32_t map_to(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// 8 bytes into a CTA of the cluster, counted on that CTA's barrier when they have arrived.
__device__ __forceinline__ void push8(uint32_t addr, uint64_t v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
               ::"r"(addr), "l"(v), "r"(bar) : "memory");
}
// As mbar_try_wait, ordering other CTAs' pushes before what follows.
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  return mbar_try_wait_cluster(smem_u32(bar), parity);
}
// Warp-wide maximum of a float that is no NaN.
__device__ __forceinline__ float warp_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// Weight sums as 64-bit fixed point with kFixBits binary places: a weight is at
// most 1 and a row has at most 2^20 of them, so sums fit, prefix sums are exact
// and in any order, and a stripe's fp32 sum loses less than 2^-44 (Z >= 1).
// (FP64 is slow on this part: a scan of doubles took the draw three times as long.)
constexpr int kFixBits = 43;
__device__ __forceinline__ uint64_t to_fix(float x) { return __float2ull_rn(x * (float)(1ull << kFixBits)); }

// The kept weight exp((l - M) / T) = 2^((l - M) log2(e) / T) of logit l, 0 below
// the cutoff; kexp = log2(e) / T per row.  The same fp32 steps everywhere, so
// pass 2 and the draw agree bit for bit.  Against exact weights the relative
// error is the factor's rounding times the exponent plus the 2^x unit's 2 ulp:
// a few 1e-7 for the weights that carry the mass (exponents near 0), inside the
// 1e-6 of Z within which a draw counts as a boundary case; weights below 2^-126
// flush to 0.
__device__ __forceinline__ float kept_weight(float l, float cut, float M, float kexp) {
  return l >= cut ? ex2_approx(__fsub_rn(l, M) * kexp) : 0.f;
}

// The loop of a bounded wait (for data of any CTA of the cluster).  After one
// wait has given up every other returns at once, and the block's remaining
// output is not valid.
__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, volatile int32_t* abort_flag, int32_t* status) {
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t i = 1; !*abort_flag; ++i) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((i & 63u) == 0 && globaltimer_ns() - t0 > kWaitLimitNs) {
      *abort_flag = 1;
      if (status) atomicOr(status, RGD_DEV_WAIT_TIMEOUT);
    }
  }
  return false;
}

// The draw of one sampled row, by the draw warp of every CTA of its cluster:
// the CTAs exchange their weight sums (exchange xc of the cluster), and the one
// whose range holds the target u * Z finds the slot and the stripe by prefix
// sums in index order, then reads that stripe again for the lane and the element.
template <typename T, bool kAligned>
__device__ __forceinline__ void draw_row(const HeadParams& p, Shared& sh, const RowParams rp, int row, int rank, int K,
                                         int buf, int xc, float M) {
  using V = Vec<T>;
  constexpr int kN = V::kN;
  const int lane = threadIdx.x & 31;
  const int xb = xc & 1;
  const float cut = __fadd_rn(M, rp.theta), kexp = rp.kexp;
  {
    uint64_t t = lane < kHeadWarps ? sh.wsum[buf][lane] : 0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    t = __shfl_sync(0xffffffffu, t, 0);
    const int32_t ct = __reduce_add_sync(0xffffffffu, lane < kHeadWarps ? sh.wcnt[buf][lane] : 0);
    if (lane == 0) mbar_arrive_expect_tx(&sh.csum_bar[xb], (uint32_t)K * 16u);
    __syncwarp();
    if (lane < K) {
      const uint32_t bar = map_to(smem_u32(&sh.csum_bar[xb]), lane);
      push8(map_to(smem_u32(&sh.csum[xb][rank]), lane), t, bar);
      push8(map_to(smem_u32(&sh.ccnt[xb][rank]), lane), (uint64_t)(uint32_t)ct, bar);
    }
  }
  const uint32_t par = (uint32_t)(xc >> 1) & 1u;
  const bool ok = mbar_try_wait_cluster(&sh.csum_bar[xb], par) ||
                  wait_slow(smem_u32(&sh.csum_bar[xb]), par, &sh.abort, p.dev_status);
  if (!__all_sync(0xffffffffu, ok)) return;
  const uint64_t cs = lane < K ? *reinterpret_cast<volatile uint64_t*>(&sh.csum[xb][lane]) : 0;
  int32_t cc = lane < K ? (int32_t)*reinterpret_cast<volatile uint64_t*>(&sh.ccnt[xb][lane]) : 0;
  cc = __reduce_add_sync(0xffffffffu, cc);
  // inclusive prefix sums over the first n lanes (the others hold 0)
  auto scan = [&](uint64_t v, int n) {
#pragma unroll 1
    for (int o = 1; o < n; o <<= 1) {
      const uint64_t t = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += t;
    }
    return v;
  };
  // the lane whose range [incl - v, incl) holds x; base is the range's start
  auto pick = [&](uint64_t v, uint64_t incl, uint64_t x, uint64_t& base) {
    const uint32_t hit = __ballot_sync(0xffffffffu, v != 0 && x < incl);
    const int L = hit ? __ffs(hit) - 1 : 0;  // (the ranges tile the whole: there is one)
    base = __shfl_sync(0xffffffffu, incl - v, L);
    return L;
  };
  const uint64_t ci = scan(cs, K);
  const uint64_t Z = __shfl_sync(0xffffffffu, ci, K - 1);
  // cumulative weight > u Z exactly if it is > floor(u Z), being whole
  const uint64_t target = __umul64hi(Z, (uint64_t)rp.u24 << 40);
  if (lane == 0 && rank == 0 && p.kept_count) p.kept_count[row] = cc;
  // a sampled row other than its group's probe is counted by the last CTA
  // (every warp of the cluster read its activity flag long ago)
  if (p.gstate && rank == K - 1 && lane == 0 && row % p.rpg != 0) finish_row(p, row, -1);
  __syncwarp();
  uint64_t base;
  if (pick(cs, ci, target, base) != rank) return;
  // this CTA's stripes, n to a lane in index order; then the lane's stripes
  const int n = (p.cvec / 32 + 31) / 32;
  uint64_t seg = 0;
  for (int i = 0; i < n; ++i) seg += sh.stripe_sum[buf][lane * n + i];
  const int sl = pick(seg, base + scan(seg, 32), target, base);
  const uint64_t sv = lane < n ? sh.stripe_sum[buf][sl * n + lane] : 0;
  uint64_t sbase;
  const int st = sl * n + pick(sv, base + scan(sv, 16), target, sbase);
  // the stripe's lanes: the same weights as pass 2, an inclusive scan in index order
  const RowView rv = row_view<T, kAligned>(p, row);
  const int v = rank * p.cvec + st * 32 + lane;
  uint4 w = make_uint4(V::kNegInfWord, V::kNegInfWord, V::kNegInfWord, V::kNegInfWord);
  if (v < rv.nvec) {
    if (kAligned || v < rv.nfull) w = __ldg(reinterpret_cast<const uint4*>(rv.base) + v);
    else w = load_vec_scalar<T>(rv, v, p.vocab);
    if (!kAligned) mask_vec<T>(w, (int64_t)v * kN - rv.shift, p.vocab);
  }
  uint64_t ls = 0;
#pragma unroll
  for (int k = 0; k < kN; ++k) ls += to_fix(kept_weight(V::get(w, k), cut, M, kexp));
  const uint64_t incl = sbase + scan(ls, 32);
  // (the stripe's fp32 sum and its elements differ by rounding: past every lane
  // means the last one with any weight)
  const uint32_t over = __ballot_sync(0xffffffffu, ls != 0 && target < incl);
  const uint32_t kept_lanes = __ballot_sync(0xffffffffu, ls != 0);
  const int L = over ? __ffs(over) - 1 : (kept_lanes ? 31 - __clz(kept_lanes) : 0);
  if (lane == L) {
    uint64_t r2 = incl - ls;
    int32_t tok = -1, lk = 0;
#pragma unroll
    for (int k = 0; k < kN; ++k) {
      const uint64_t wk = to_fix(kept_weight(V::get(w, k), cut, M, kexp));
      if (wk != 0) {
        lk = v * kN - rv.shift + k;
        r2 += wk;
        if (r2 > target && tok < 0) tok = lk;
      }
    }
    if (tok < 0) tok = lk;  // the lane's last kept token
    p.token_out[row] = tok;
    // (one lane of one CTA of the cluster writes the token; a sampled probe
    // row's token goes through the gate here)
    if (p.gstate && row % p.rpg == 0) finish_row(p, row, tok);
  }
}

// Sums one value per stripe of a slot (four per lane) over the lanes: every
// lane returns the sum of stripe 2 (lane / 16 & 1) + (lane / 8 & 1), formed by
// the pairwise tree of a butterfly (6 shuffles instead of 20).
__device__ __forceinline__ float slot_sums(const float (&v)[kSlotStripes], int lane) {
  static_assert(kSlotStripes == 4, "");
  const bool u16 = (lane & 16) != 0, u8 = (lane & 8) != 0;
  const float a0 = (u16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, u16 ? v[0] : v[2], 16);
  const float a1 = (u16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, u16 ? v[1] : v[3], 16);
  float b = (u8 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, u8 ? a0 : a1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
  return b;
}

template <typename T, bool kAligned>
__global__ void __launch_bounds__(kHeadThreads, 3) sample_head_kernel(const HeadParams p) {
  using V = Vec<T>;
  constexpr int kN = V::kN;
  __shared__ Shared sh;
  extern __shared__ __align__(128) uint8_t ring_mem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t rank_u, k_u, cid_u, ncl_u;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(k_u));
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(cid_u));
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(ncl_u));
  const int rank = (int)rank_u, K = (int)k_u, cid = (int)cid_u, stride = (int)ncl_u;
  volatile int32_t* abort_flag = &sh.abort;

  if (tid < p.nslots) {
    mbar_init(&sh.full_bar[tid], 1);
    mbar_init(&sh.empty_bar[tid], kHeadWarps);
  }
  if (tid == 32) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sh.max_bar[b], 1);
      mbar_init(&sh.sum_bar[b], kHeadWarps);
      mbar_init(&sh.csum_bar[b], 1);
      mbar_init(&sh.prm_bar[b], 1);
      mbar_init(&sh.free_bar[b], 1);
    }
    sh.abort = 0;
  }
  fence_mbar_init();
  __syncthreads();
  // arrived here, waited for before the first push into another CTA: by then
  // every CTA of the cluster has started and set its barriers up
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  // launched as a programmatic dependent of the previous kernel on the stream:
  // what follows may read what that kernel wrote, unless the caller knows that
  // the inputs were complete before it began
  if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");

  auto wait = [&](uint64_t* bar, uint32_t parity, bool cluster) {
    if (cluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity)) return true;
    return wait_slow(smem_u32(bar), parity, &sh.abort, p.dev_status);
  };
  auto wwait = [&](uint64_t* bar, uint32_t parity, bool cluster) {  // of a whole warp, one answer
    return __all_sync(0xffffffffu, wait(bar, parity, cluster));
  };
  // Round k gives the cluster row k * stride + (cid + k) % stride: shifted by
  // one each round, so that no cluster is left with one kind of row only where
  // the kinds repeat (probes and samples, temperatures).  Every warp takes the
  // rounds in blocks of 32, lane k % 32 reading round k's activity.  The gate may
  // clear the flag of an active row once the row is finished, by CTA 0's draw warp
  // alone if it is greedy, so every warp of the cluster must have read the block's
  // flags by then.  It has: a row is finished behind the exchange of its maxima, to
  // which every stream warp of the cluster contributes only after its own copy warp's
  // copies and its own draw warp's parameters of the block, and both of these read
  // the flags first.
  const int nblk = ((p.rows + stride - 1) / stride + 31) / 32;
  auto row_of = [&](int k) { return k * stride + (cid + k) % stride; };
  auto block_rows = [&](int blk) {
    const int r = row_of(blk * 32 + lane);
    return __ballot_sync(0xffffffffu, r < p.rows && (p.row_active == nullptr || p.row_active[r] != 0));
  };
  // CTA r holds vectors [r cvec, (r + 1) cvec) of a row, 1024 to a ring slot,
  // of which stream warp w takes 128 w .. 128 w + 127 (its four stripes)
  const int c0 = rank * p.cvec;
  const int nsl = p.nslots, spr = (p.cvec + kSlotVecs - 1) / kSlotVecs;  // ring slots; a row's slots

  if (warp == kHeadWarps + 1) {
    // ============================== copy warp ==============================
    // Slot after slot of the cluster's active rows, as far ahead as the ring goes.
    const uint64_t pol = policy_evict_first();
    int pos = 0, round = 0;  // ring position, and how often the ring has been filled
    bool ok = true;
    for (int blk = 0; blk < nblk && ok; ++blk) {
      for (uint32_t m = block_rows(blk); m && ok; m &= m - 1) {
        const RowView rv = row_view<T, kAligned>(p, row_of(blk * 32 + __ffs(m) - 1));
        const int c1 = min(rv.nfull, c0 + p.cvec);
        for (int a = c0; a < c0 + p.cvec; a += kSlotVecs) {
          if (round > 0 && !wwait(&sh.empty_bar[pos], (uint32_t)(round - 1) & 1u, false)) {
            ok = false;
            break;
          }
          if (lane == 0) {
            const int n = min(kSlotVecs, c1 - a);
            if (n > 0) {
              mbar_arrive_expect_tx(&sh.full_bar[pos], (uint32_t)n * 16u);
              bulk_load_hint(ring_mem + pos * kSlotBytes, rv.base + (int64_t)a * 16, (uint32_t)n * 16u,
                             &sh.full_bar[pos], pol);
            } else {
              mbar_arrive(&sh.full_bar[pos]);  // (nothing of the row here)
            }
          }
          if (++pos == nsl) {
            pos = 0;
            ++round;
          }
        }
      }
    }
    // every copy is issued: a programmatic dependent of this kernel may be
    // scheduled once every block has come this far
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*abort_flag && lane == 0) {  // the copies still in flight: each slot's last phase, bounded
      for (int i = 0; i < nsl; ++i) {
        if (--pos < 0) {
          pos = nsl - 1;
          --round;
        }
        if (round < 0) break;
        mbar_wait(&sh.full_bar[pos], (uint32_t)round & 1u);
      }
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else if (warp < kHeadWarps) {
    // ============================ stream warps ============================
    const uint32_t ring_s = smem_u32(ring_mem) + warp * (kSlotStripes * 512) + lane * 16;
    const int v0 = c0 + warp * (kSlotStripes * 32);
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    // the CTA's vectors of a row end at vend; [safe_lo, safe_hi) of them hold
    // elements of the row only
    int vend = kAligned ? min(p.vocab / kN, c0 + p.cvec) : 0, safe_lo = 0, safe_hi = vend;
    int pos = 0;
    uint32_t phase = 0;  // ring position of the next slot, and its phase
    int it = 0, nb = -1;  // rows so far, and the block's number among those with an active row
    for (int blk = 0; blk < nblk; ++blk) {
      uint32_t mask_rows32 = block_rows(blk);
      nb += mask_rows32 != 0 ? 1 : 0;
      bool have_prm = false;
      auto block_params = [&]() {  // (by the block's first row)
        if (!have_prm) wait(&sh.prm_bar[nb & 1], (uint32_t)(nb >> 1) & 1u, false);
        have_prm = true;
      };
      for (; mask_rows32; mask_rows32 &= mask_rows32 - 1, ++it) {
        const int kk = __ffs(mask_rows32) - 1;
        const int row = row_of(blk * 32 + kk);
        const RowParams& rp = sh.prm[nb & 1][kk];
        const int buf = it & 1;
        const uint32_t par = (uint32_t)(it >> 1) & 1u;
        RowView rv;
        if (!kAligned) {
          rv = row_view<T, kAligned>(p, row);
          vend = min(rv.nvec, c0 + p.cvec);
          safe_lo = rv.shift == 0 ? 0 : 1;
          safe_hi = min(vend, rv.nvec - 1);
        }
        const int shift = kAligned ? 0 : rv.shift;
        auto is_whole = [&](int j) {  // all of the warp's vectors in slot j (uniform)
          const int a = v0 + j * kSlotVecs;
          return a >= safe_lo && a + kSlotStripes * 32 <= safe_hi;
        };
        // stripe s of the slot at `at`, whose vectors start at v: any vector of
        // the range, elements of other rows and vectors past the end as -inf
        auto fetch_any = [&](uint32_t at, int v) {
          uint4 w = make_uint4(V::kNegInfWord, V::kNegInfWord, V::kNegInfWord, V::kNegInfWord);
          if (v < vend) {
            if (kAligned || v < rv.nfull) w = lds128(at);
            else w = load_vec_scalar<T>(rv, v, p.vocab);
            if (!kAligned) mask_vec<T>(w, (int64_t)v * kN - rv.shift, p.vocab);
          }
          return w;
        };
        auto fetch_slot = [&](uint32_t at, int vb, bool whole, uint4 (&w)[kSlotStripes]) {
          if (whole) {
#pragma unroll
            for (int s = 0; s < kSlotStripes; ++s) w[s] = lds128(at + s * 512);
          } else {
#pragma unroll
            for (int s = 0; s < kSlotStripes; ++s) w[s] = fetch_any(at + s * 512, vb + s * 32);
          }
        };
        // ---- pass 1: the lane's maximum and the first slot that holds it; lane j
        // also keeps slot j's maximum, which pass 2 looks at ----
        float lm = -INFINITY, slot_max = -INFINITY;
        int lj = -1;
        uint32_t lat = 0;
        {
          int ps = pos;
          uint32_t ph = phase;
          uint4 w[kSlotStripes];
          auto take = [&](int j) {  // slot j of the row into registers
            wait(&sh.full_bar[ps], ph, false);
            const uint32_t at = ring_s + ps * kSlotBytes;
            fetch_slot(at, v0 + j * kSlotVecs + lane, is_whole(j), w);
            if (++ps == nsl) {
              ps = 0;
              ph ^= 1u;
            }
            return at;
          };
#pragma unroll 1
          for (int j = 0; j < spr; ++j) {
            const uint32_t at = take(j);
            const float m = V::max4(w);
            if (m > lm) {  // slots only grow: strict > keeps the lowest
              lm = m;
              lj = j;
              lat = at;
            }
            const float sm = warp_max(m);
            if (lane == j) slot_max = sm;
          }
        }
        const float wm = warp_max(lm);
        block_params();
        const bool greedy = rp.greedy != 0;
        uint32_t idx = 0x7fffffffu;
        if (greedy) {  // the argmax is the answer: its lowest index
          if (lj >= 0 && lm == wm) {
            const int vb = v0 + lj * kSlotVecs + lane;
#pragma unroll 1
            for (int s = kSlotStripes - 1; s >= 0; --s) {
              const uint4 w = fetch_any(lat + s * 512, vb + s * 32);
#pragma unroll
              for (int k = kN - 1; k >= 0; --k)
                if (V::get(w, k) == wm) idx = (uint32_t)((vb + s * 32) * kN - shift + k);
            }
          }
          idx = __reduce_min_sync(0xffffffffu, idx);
        }
        // the warp's maximum to every CTA
        if (warp == 0 && lane == 0) mbar_arrive_expect_tx(&sh.max_bar[buf], (uint32_t)(K * kHeadWarps) * 8u);
        __syncwarp();
        if (lane < K) {
          const uint64_t v = ((uint64_t)idx << 32) | __float_as_uint(wm);
          push8(map_to(smem_u32(&sh.wmax[buf][rank * kHeadWarps + warp]), lane), v,
                map_to(smem_u32(&sh.max_bar[buf]), lane));
        }
        if (greedy) {  // no second pass: the slots take later rows at once
#pragma unroll 1
          for (int j = 0; j < spr; ++j) {
            if (lane == 0) mbar_arrive(&sh.empty_bar[pos]);
            if (++pos == nsl) {
              pos = 0;
              phase ^= 1u;
            }
          }
        }
        // the draw warp is done with the row before last (its sums and maxima may be overwritten)
        if (it >= 2) wait(&sh.free_bar[buf], par ^ 1u, false);
        wait(&sh.max_bar[buf], par, true);
        __syncwarp();
        float M = -INFINITY;
        for (int i = lane; i < K * kHeadWarps; i += 32)
          M = fmaxf(M, __uint_as_float(*reinterpret_cast<volatile uint32_t*>(&sh.wmax[buf][i])));
        M = warp_max(M);
        if (warp == 0) {
          uint32_t A = 0x7fffffffu;
          if (greedy) {
            for (int i = lane; i < K * kHeadWarps; i += 32) {
              const uint64_t v = *reinterpret_cast<volatile uint64_t*>(&sh.wmax[buf][i]);
              if (__uint_as_float((uint32_t)v) == M) A = min(A, (uint32_t)(v >> 32));
            }
            A = __reduce_min_sync(0xffffffffu, A);
          }
          if (lane == 0) {
            sh.row_max[buf] = M;
            sh.row_arg[buf] = (int32_t)A;
          }
        }
        if (!greedy) {
          // ---- pass 2: kept weights; the sum of every stripe and of the warp ----
          const float cut = __fadd_rn(M, rp.theta);  // the min-p cutoff fl32(M + fl32(T ln p_min))
          const float kexp = rp.kexp;
          // (a rejected row has no kept set: its mask is not written)
          uint8_t* mask =
              p.kept_mask && rp.valid && isfinite(M) ? p.kept_mask + (int64_t)row * p.vocab : nullptr;
          const uint32_t hits = mask ? ~0u : __ballot_sync(0xffffffffu, slot_max >= cut);
          const typename V::Cut vc(cut, M, kexp);
          int32_t cnt = 0;
          uint64_t fsum = 0;  // lanes 0, 8, 16, 24
#pragma unroll 1
          for (int j = 0; j < spr; ++j) {
            const uint32_t at = ring_s + pos * kSlotBytes;
            const int vb = v0 + j * kSlotVecs + lane;
            const bool hit = (hits >> j) & 1u, whole = is_whole(j);
            uint4 w[kSlotStripes];
            if (hit) fetch_slot(at, vb, whole, w);
            __syncwarp();  // every lane has read its part of the slot
            if (lane == 0) mbar_arrive(&sh.empty_bar[pos]);
            if (++pos == nsl) {
              pos = 0;
              phase ^= 1u;
            }
            float sum = 0.f;
            if (hit) {
              float ls[kSlotStripes];  // the lane's kept weights of each stripe
              if (whole) {
#pragma unroll
                for (int s = 0; s < kSlotStripes; ++s) ls[s] = V::kept(w[s], vc, cnt);
              } else {
#pragma unroll
                for (int s = 0; s < kSlotStripes; ++s) {
                  ls[s] = 0.f;
#pragma unroll
                  for (int k = 0; k < kN; ++k) {
                    const int e = (vb + s * 32) * kN - shift + k;
                    const float l = V::get(w[s], k);
                    const bool keep = l >= cut && vb + s * 32 < vend && e >= 0 && e < p.vocab;
                    ls[s] += keep ? kept_weight(l, cut, M, kexp) : 0.f;
                    cnt += keep ? 1 : 0;
                  }
                }
              }
              sum = slot_sums(ls, lane);
            }
            if ((lane & 7) == 0) {
              const uint64_t f = to_fix(sum);
              fsum += f;
              sh.stripe_sum[buf][(j * kHeadWarps + warp) * kSlotStripes + ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1)] = f;
            }
            if (mask) {
#pragma unroll
              for (int s = 0; s < kSlotStripes; ++s) {
                const int v = vb + s * 32;
#pragma unroll
                for (int k = 0; k < kN; ++k) {
                  const int e = v * kN - shift + k;
                  if (v < vend && e >= 0 && e < p.vocab) mask[e] = V::get(w[s], k) >= cut ? 1 : 0;
                }
              }
            }
          }
          cnt = __reduce_add_sync(0xffffffffu, cnt);
          fsum += __shfl_xor_sync(0xffffffffu, fsum, 16);
          fsum += __shfl_xor_sync(0xffffffffu, fsum, 8);
          if (lane == 0) {
            sh.wcnt[buf][warp] = cnt;
            sh.wsum[buf][warp] = fsum;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.sum_bar[buf]);
      }
    }
  } else {
    // ============================== draw warp ==============================
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    // The active rows of a block, and the parameters of its 32 rows, one lane each:
    // the min-p offset T ln p_min (fp64 logarithm) and the draw's uniform.  The
    // arrival that publishes the parameters comes after the flags have been read
    // (see above; read behind it, a flag could already be this launch's gate's).
    // Only blocks with an active row take a parameter buffer and a phase of prm_bar:
    // every stream warp waits for the phase before the block's first row counts as
    // summed, and this warp is through with a block's rows before it fills the
    // second block after it, so no phase is passed and no buffer overwritten early.
    // (In a block without an active row this warp waits for nothing; were it to
    // publish there, it could run ahead of a stream warp by two phases of one
    // barrier, which that warp could not tell from none.)
    int filled = 0;
    auto fill = [&](int blk) {
      if (blk >= nblk) return 0u;
      const int row = row_of(blk * 32 + lane);
      bool active = row < p.rows;
      if (active && p.row_active) active = p.row_active[row] != 0;
      RowParams rp{};
      if (row < p.rows) {
        const float temp = p.temperature[row], mp = p.min_p[row];
        const bool greedy = (p.is_probe && p.is_probe[row]) || temp == 0.0f;
        const uint64_t sd = p.seed[row];
        rp.theta = -INFINITY;
        if (mp > 0.0f && !greedy) rp.theta = (float)((double)temp * log((double)mp));
        rp.kexp = 1.4426950408889634f / temp;
        const uint32_t x0 = philox_word0((uint32_t)p.step, (uint32_t)(p.step >> 32), 0u, 0u, (uint32_t)sd,
                                         (uint32_t)(sd >> 32));
        rp.u24 = x0 >> 8;
        rp.greedy = greedy;
        rp.valid = temp >= 0.0f && isfinite(temp) && mp >= 0.0f && mp <= 1.0f;
      }
      const uint32_t rows = __ballot_sync(0xffffffffu, active);
      if (rows == 0) return 0u;
      sh.prm[filled & 1][lane] = rp;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.prm_bar[filled & 1]);
      ++filled;
      return rows;
    };
    uint32_t next_rows = fill(0);
    if (p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    int it = 0, xc = 0, nb = -1;  // rows and exchanges of weight sums so far; the block's number, as above
    for (int blk = 0; blk < nblk; ++blk) {
      uint32_t mask_rows32 = next_rows;
      nb += mask_rows32 != 0 ? 1 : 0;
      next_rows = fill(blk + 1);  // (over the parameters of an earlier block, which every warp is done with)
      if (rank == 0) {  // the block's inactive rows
        const int r = row_of(blk * 32 + lane);
        if (r < p.rows && !((mask_rows32 >> lane) & 1u)) {
          p.token_out[r] = -1;
          if (p.kept_count) p.kept_count[r] = 0;
          if (p.gstate) finish_row(p, r, -1);
        }
        __syncwarp();
      }
      for (; mask_rows32; mask_rows32 &= mask_rows32 - 1, ++it) {
        const int kk = __ffs(mask_rows32) - 1;
        const int row = row_of(blk * 32 + kk);
        const RowParams rp = sh.prm[nb & 1][kk];
        const int buf = it & 1;
        const bool fine = wwait(&sh.sum_bar[buf], (uint32_t)(it >> 1) & 1u, false);
        const float M = sh.row_max[buf];
        const int32_t A = sh.row_arg[buf];
        const bool bad = !rp.valid || !isfinite(M);
        if (rp.greedy || bad) {
          if (rank == 0 && lane == 0 && fine) {
            int32_t tok = -1;
            if (bad && !rp.greedy) {
              if (p.dev_status) atomicOr(p.dev_status, RGD_DEV_BAD_PARAM);
              if (p.kept_count) p.kept_count[row] = 0;
            } else {
              tok = A < p.vocab ? A : -1;
              if (p.kept_count) p.kept_count[row] = 1;
            }
            p.token_out[row] = tok;
            if (p.gstate) finish_row(p, row, tok);
          }
        } else {
          draw_row<T, kAligned>(p, sh, rp, row, rank, K, buf, xc++, M);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.free_bar[buf]);
      }
    }
  }
  // no CTA leaves while another may still push into it
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace
}  // namespace rgd

using namespace rgd;

namespace rgd {
namespace {

// How a call is cut: CTAs per row, and each CTA's share and ring.
struct HeadPlan {
  int K, cvec, nslots;
};

// Clusters of a plan that the current device holds at once (0: none), asked of
// the runtime once per device, kernel, cluster size and ring.
template <typename Kernel>
int max_clusters(Kernel k, int kernel_id, const cudaLaunchConfig_t& cfg, const HeadPlan& pl, int* out) {
  constexpr int kMaxDev = 16;
  static std::mutex mu;
  static int16_t cache[kMaxDev][4][5][kMaxSlots + 1] = {};  // clusters + 1; 0: not asked yet
  int dev = 0;
  if (cudaError_t e = cudaGetDevice(&dev); e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  const int kl = pl.K == 1 ? 0 : pl.K == 2 ? 1 : pl.K == 4 ? 2 : pl.K == 8 ? 3 : 4;
  std::lock_guard<std::mutex> lock(mu);
  int16_t* c = dev < kMaxDev ? &cache[dev][kernel_id][kl][pl.nslots] : nullptr;
  if (c && *c) {
    *out = *c - 1;
    return RGD_OK;
  }
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSlots * kSlotBytes);
  if (e == cudaSuccess && pl.K > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return cuda_error(e, "sample_head attributes");
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
  if (e != cudaSuccess) return cuda_error(e, "sample_head occupancy");
  n = std::min(std::max(n, 0), 32766);
  if (c) *c = (int16_t)(n + 1);
  *out = n;
  return RGD_OK;
}

// Launches the head by the first plan of `plans` that the device can hold, as a
// programmatic dependent of the previous kernel on the stream, so that its
// blocks are scheduled while that kernel finishes.
template <typename T, bool kAligned>
int launch_head_t(int kernel_id, const HeadPlan* plans, int n_plans, HeadParams& hp, cudaStream_t st) {
  auto k = sample_head_kernel<T, kAligned>;
  for (int i = 0; i < n_plans; ++i) {
    const HeadPlan& pl = plans[i];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.K);
    cfg.blockDim = dim3(kHeadThreads);
    cfg.dynamicSmemBytes = (size_t)pl.nslots * kSlotBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {(unsigned)pl.K, 1, 1};
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (int rc = max_clusters(k, kernel_id, cfg, pl, &n)) return rc;
    if (n < 1) continue;
    hp.cvec = pl.cvec;
    hp.nslots = pl.nslots;
    cfg.gridDim = dim3((unsigned)std::min(n, hp.rows) * pl.K);
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k, hp);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? RGD_OK : cuda_error(e, "sample_head launch");
  }
  return set_error(RGD_ERR_UNSUPPORTED, "sample_head: the device has no room for a row of %d logits", hp.vocab);
}

// The split.  A row must fit the shared memory of its cluster, and a cluster has
// one row's latency (loads, the exchange of maxima, pass 2, the draw) per row,
// so a CTA's share should be as large as still lets two or three CTAs share an
// SM and cover one another: at most 6 ring slots (96 KB) each.  Measured at
// 435 active rows x 152064 bf16: 42.5 us with 5 slots (4 CTAs per row, 2 on an
// SM) against 52 us with 3 (8 CTAs per row); 1024 x 262144 fp32: 205 us with 4
// slots (16 CTAs per row) against 300-375 us with 8 (8 CTAs per row, 1 on an
// SM).  With few rows more CTAs per row shorten the row itself (8 rows x 128256
// fp32: 12.1 us at 8 CTAs per row, 12.3 at 4, 22.5 with the share of 2), until
// the SMs have two CTAs each.  Rows above 1.7 MB need 16 CTAs; where a cluster
// of 16 cannot be placed the others fall back to 8.
//
// What bounds it: issue slots (about 2.4 of 4 a cycle; the two passes take ~50
// instructions per 512 bytes) with many rows, latency with few.  Against the
// two-pass kernel that read a row's kept stripes again from L2: 1024 x 262144
// fp32 205 us (0.78 of the measured copy bandwidth) from 380, bf16 112 from
// 307; 256 x 128256 bf16 24.8 from 59.9; 80 x 128256 fp32 18.6 from 22.6; one
// row of 32000 8.3 from 10.4.
int launch_head(int32_t rows, int32_t vocab, int32_t dtype, const HeadParams& hp0, cudaStream_t st) {
  const int es = dtype == RGD_F32 ? 4 : 2;
  HeadParams hp = hp0;
  hp.total_bytes = (int64_t)rows * vocab * es;
  const bool aligned = ((int64_t)vocab * es) % 16 == 0;
  const int64_t nvec = ((int64_t)vocab * es + 15) / 16 + (aligned ? 0 : 1);
  const int64_t stripes = (nvec + 31) / 32;
  auto cvec_of = [&](int K) { return (int)((stripes + K - 1) / K) * 32; };
  auto slots_of = [&](int K) { return (cvec_of(K) + kSlotVecs - 1) / kSlotVecs; };
  int K = 1;
  while (K < 8 && (slots_of(K) > 6 || ((int64_t)rows * K < 304 && slots_of(K) > 1))) K *= 2;
  while (K < 16 && slots_of(K) > 6) K *= 2;
  HeadPlan plans[2];
  int n_plans = 0;
  for (; K >= 8 || n_plans == 0; K /= 2) {
    if (slots_of(K) > kMaxSlots || n_plans == 2) break;
    // the largest ring that lets 3, 2 or 1 CTAs share an SM's 228 KB and holds a row's share
    int nslots = 0;
    for (int cps = 3; cps >= 1 && nslots < slots_of(K); --cps)
      nslots = std::min<int>(kMaxSlots, (233472 / cps - 1024 - (int)sizeof(Shared)) / kSlotBytes);
    plans[n_plans++] = HeadPlan{K, cvec_of(K), nslots};
  }
  if (dtype == RGD_F32)
    return aligned ? launch_head_t<float, true>(0, plans, n_plans, hp, st)
                   : launch_head_t<float, false>(1, plans, n_plans, hp, st);
  return aligned ? launch_head_t<__nv_bfloat16, true>(2, plans, n_plans, hp, st)
                 : launch_head_t<__nv_bfloat16, false>(3, plans, n_plans, hp, st);
}

// Argument checks shared by both entry points.
int check_head_args(const char* fn, int32_t rows, int32_t vocab, int32_t dtype, const void* logits,
                    const float* temperature, const float* min_p, const uint64_t* seed, const int32_t* token_out) {
  RGD_CHECK_ARG(rows >= 0, "%s: rows < 0", fn);
  RGD_CHECK_ARG(vocab >= 1, "%s: vocab < 1", fn);
  RGD_CHECK_ARG(dtype == RGD_F32 || dtype == RGD_BF16, "%s: dtype must be RGD_F32 or RGD_BF16", fn);
  if (rows == 0) return RGD_OK;
  RGD_CHECK_ARG(logits && temperature && min_p && seed && token_out,
                "%s: logits/temperature/min_p/seed/token_out must be non-NULL", fn);
  RGD_CHECK_ARG(aligned16(logits), "%s: logits must be 16-byte aligned", fn);
  RGD_CHECK_ARG(rows <= 0x7fffffff / 8, "%s: too many rows", fn);
  // a row is cut into at most 4096 stripes of 512 bytes
  const int64_t per_stripe = 512 / (dtype == RGD_F32 ? 4 : 2);
  if (vocab > 4096 * per_stripe)
    return set_error(RGD_ERR_UNSUPPORTED, "%s: vocab %d too large (max %lld)", fn, vocab, (long long)(4096 * per_stripe));
  return RGD_OK;
}

}  // namespace
}  // namespace rgd

extern "C" int rgd_sample_head(int32_t rows, int32_t vocab, int32_t dtype, const void* logits,
                               const uint8_t* is_probe, const float* temperature, const float* min_p,
                               const uint64_t* seed, uint64_t step, const uint8_t* row_active,
                               int32_t* token_out, int32_t* kept_count, uint8_t* kept_mask,
                               int32_t* dev_status, rgd_stream_t stream) {
  clear_error();
  if (int rc = check_head_args("rgd_sample_head", rows, vocab, dtype, logits, temperature, min_p, seed, token_out))
    return rc;
  if (rows == 0) return RGD_OK;
  HeadParams hp{};
  hp.logits = static_cast<const uint8_t*>(logits);
  hp.rows = rows;
  hp.vocab = vocab;
  hp.is_probe = is_probe;
  hp.temperature = temperature;
  hp.min_p = min_p;
  hp.seed = seed;
  hp.step = step;
  hp.row_active = row_active;
  hp.token_out = token_out;
  hp.kept_count = kept_count;
  hp.kept_mask = kept_mask;
  hp.dev_status = dev_status;
  return launch_head(rows, vocab, dtype, hp, (cudaStream_t)stream);
}

namespace rgd {

int check_gated_head(const char* fn, int32_t rows, int32_t vocab, int32_t dtype, const void* logits,
                     const float* temperature, const float* min_p, const uint64_t* seed, const int32_t* token_out,
                     const rgd_trie* trie, int32_t rows_per_group, int32_t max_len, const rgd_gate_state* state) {
  if (int rc = check_head_args(fn, rows, vocab, dtype, logits, temperature, min_p, seed, token_out)) return rc;
  RGD_CHECK_ARG(trie != nullptr, "%s: trie is NULL", fn);
  RGD_CHECK_ARG(rows_per_group >= 1 && rows_per_group <= 255, "%s: rows_per_group must be in [1, 255]", fn);
  RGD_CHECK_ARG(rows % rows_per_group == 0, "%s: rows must be a multiple of rows_per_group", fn);
  RGD_CHECK_ARG(max_len >= 1, "%s: max_len must be >= 1", fn);
  if (rows == 0) return RGD_OK;
  RGD_CHECK_ARG(state != nullptr, "%s: state is NULL", fn);
  RGD_CHECK_ARG((reinterpret_cast<uintptr_t>(state) & 3u) == 0, "%s: state must be 4-byte aligned", fn);
  return RGD_OK;
}

}  // namespace rgd

namespace rgd {

int launch_gated_head(const char* fn, int32_t rows, int32_t vocab, int32_t dtype, const void* logits,
                      const uint8_t* is_probe, const float* temperature, const float* min_p, const uint64_t* seed,
                      uint64_t step, uint8_t* row_active, int32_t* token_out, int32_t* kept_count,
                      const rgd_trie* trie, int32_t rows_per_group, int32_t eos_token, int32_t max_len,
                      rgd_gate_state* state, int32_t* dev_status, rgd_stream_t stream, bool early) {
  if (int rc = check_gated_head(fn, rows, vocab, dtype, logits, temperature, min_p, seed, token_out, trie,
                                rows_per_group, max_len, state))
    return rc;
  if (rows == 0) return RGD_OK;
  HeadParams hp{};
  hp.logits = static_cast<const uint8_t*>(logits);
  hp.rows = rows;
  hp.vocab = vocab;
  hp.early = early ? 1 : 0;
  hp.is_probe = is_probe;
  hp.temperature = temperature;
  hp.min_p = min_p;
  hp.seed = seed;
  hp.step = step;
  hp.row_active = row_active;
  hp.token_out = token_out;
  hp.kept_count = kept_count;
  hp.dev_status = dev_status;
  hp.trie = TrieView{trie->child_begin, trie->edges};
  hp.gstate = state;
  hp.gate_row_active = row_active;
  hp.rpg = rows_per_group;
  hp.eos = eos_token;
  hp.max_len = max_len;
  return launch_head(rows, vocab, dtype, hp, (cudaStream_t)stream);
}

}  // namespace rgd

extern "C" int rgd_sample_head_gated(int32_t rows, int32_t vocab, int32_t dtype, const void* logits,
                                     const uint8_t* is_probe, const float* temperature, const float* min_p,
                                     const uint64_t* seed, uint64_t step, uint8_t* row_active,
                                     int32_t* token_out, int32_t* kept_count, const rgd_trie* trie,
                                     int32_t rows_per_group, int32_t eos_token, int32_t max_len,
                                     rgd_gate_state* state, int32_t* dev_status, rgd_stream_t stream) {
  clear_error();
  return launch_gated_head("rgd_sample_head_gated", rows, vocab, dtype, logits, is_probe, temperature, min_p, seed,
                           step, row_active, token_out, kept_count, trie, rows_per_group, eos_token, max_len, state,
                           dev_status, stream, false);
}
