// Shared-prefix decode attention on the 5th-generation tensor cores.
//
// Sec. 3 reuses the prompt KV cache across the greedy probe and the high-
// temperature sampling stage.  Here that reuse is explicit: for every prompt
// group g and kv head h one "job" attends all rows_per_group * (Hq/Hkv) queries
// of the group that map to h.  A job's page list is the group's prompt pages
// (visible to every row) followed by the suffix pages of each active row
// (visible to that row's queries only, by a per-page row mask), so a row's
// suffix simply continues the online softmax of its prompt: the result is
// attention over [prompt KV | own suffix KV], and every KV page is read from
// HBM exactly once.
//
// Work distribution.  The jobs' page lists are laid end to end (job-major) and
// the grid's persistent blocks (one per SM) each take an equal contiguous range
// of pages and works through it in order.  Only the two jobs at the ends of a
// block's range can be split with a neighbour.  A split job is merged by
// log-sum-exp (Sec. 3's shared-prefix split is the same identity) in the block
// holding its first page, whose last piece it is: the job's other pieces -- each
// the first piece of its own block, behind no wait on another block -- write a
// partial (o, m, l) to workspace slot (block + job) and count themselves in the
// job's ticket.  The merging block fetches them into its idle K ring while its
// last group is in flight and folds them into its own piece on the way out; if
// the ring has no room for all, it writes its own piece to the workspace too and
// folds all of them from there.
//
// Inside a block the tokens are the MMA's M and the queries its N:
//   S^T = K Q^T      A = a group's K (128 tokens = 8 pages, K-major), B = Q,
//                    accumulator S^T: token t in lane t, a query per column;
//   O^T += V^T P^T   A = V^T of a page straight from its V tile (token rows, so
//                    MN-major), B = P^T of that page's 16 tokens (MN-major): a
//                    bf16 high part and a bf16 residual side by side, so one
//                    MMA a page; accumulator O^T: head dimension d in lane d.
// A softmax thread owns one token and its set's queries: it reads their scores
// from its lane, and the query maxima are shared through shared memory only
// when one of them has to move (the reference maximum of a query moves lazily,
// when a score exceeds it by more than 2^8; a piece's first group sets it).
//
// Warps: 4 per softmax set (token quarter = warp % 4), 4 for the piece ends
// (head-dimension quarter; they also write Q), then the K producer, the V
// producer, the QK issuer (which allocates the tensor memory) and the PV issuer.
// K areas go back to their producer when the group's QK is done, V areas when
// its PV is, so K runs ahead of V.
//
// What bounds it: HBM on large batches (2900-3300 cycles per 64 KB group and SM
// is the measured copy rate); with little KV per block the set-up chain (lengths
// -> block table -> data) and the merge at the end.  Measured inside a CUDA
// graph, against a kernel with the queries as the MMA's M (128 rows of query
// copies), P in tensor memory and one ring for K and V together (us):
//   256 groups x 2 rows, 32/8 heads, D 128, prompts of 128-8192    440 -> 353 (0.98 of the copy rate)
//   16 x 5, 32/8, 128, 512-2048                                     36 -> 29
//   1 x 5, 32/8, 128, 3000                                          25 -> 15.0
//   12 x 9, 32/8, 128, 500-6000                                     70 -> 46
//   4 x 9, 64/8, 128, 32768                                        202 -> 114
//   32 x 16, 64/8, 128, 200-800                                    107 -> 81
//   200 x 16, 4/1, 64, 50-100                                       35 -> 32
// Every wait on an mbarrier is bounded; a timeout is reported in the status
// word and every role stops.
#pragma once

#include <type_traits>

#include "attention.h"
#include "ptx.cuh"

namespace rgd {
namespace {

constexpr float kRescaleLog2 = 8.f;  // lazy rescale threshold (factor 256)
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kNoRef = 3.0e38f;    // the negated reference of a query that has seen no token yet

template <int D, int NS, int QS>
struct AttnCfg {
  static constexpr int kNq = NS * QS;                     // query columns with a softmax thread
  static constexpr int kN = query_cols(NS, QS);           // the MMAs' query columns
  static constexpr int kArea = kGroupPages * kPage * D * 2;  // a group's K or V
  static constexpr int kPBytes = 512 * kN;                // P^T of a group, both parts
  static constexpr int kQBytes = kN * D * 2;
  // P^T rows (tokens) are cut into swizzle atoms of kSw bytes of columns x 8 tokens
  static constexpr int kSw = kN % 64 == 0 ? 128 : kN % 32 == 0 ? 64 : 32;
  static constexpr int kSwLayout = kSw == 128 ? 2 : kSw == 64 ? 4 : 6;
  static constexpr int kOBufs = 6 * kN <= 512 ? 2 : 1;    // O^T buffers (by piece), 2 kN columns each
  static constexpr int kSCol = 0, kOCol = 2 * kN;         // S^T: two buffers of kN columns
  static constexpr int kCols = 2 * kN + kOBufs * 2 * kN;
  static constexpr int kTmemCols = kCols <= 128 ? 128 : kCols <= 256 ? 256 : 512;
  static constexpr int kThreads = (4 * NS + 8) * 32;
  static constexpr int kEpi = 4 * NS, kProdK = kEpi + 4, kProdV = kProdK + 1, kQk = kProdV + 1, kPv = kQk + 1;
  static_assert(kCols <= 512, "TMEM columns");
};

struct Job {
  int g, h, n;  // group, kv head, pages
  int start;    // first page in the global page order (fewer than 2^31 pages)
};


// What every role of a block looks up, in shared memory: the functions that
// take it are out of line and shared by the roles, which keeps the kernel's code
// (fetched cold by every launch) small.
struct BlockCtx {
  int b, e;        // this block's pages
  int T, Ceff;     // the dealt pages (see the set-up), which Ceff blocks share
  int jl_end;      // dealt position of the last job's last page
  int G, Hkv, rpg, max_pp, max_sp;
  const int32_t *prompt_bt, *suffix_bt, *suffix_len;
  const int32_t *gpre, *plen, *slen;  // slen: NULL when it is read from global memory
  const uint32_t* rowbits;
  Job j0, jl;  // first and last job of the range (the block's pieces are the jobs' parts in it, in order)
  int n0;      // the first job's pages in the range
};

__device__ __forceinline__ void flag(int32_t* status, int32_t bit) {
  if (status) atomicOr(status, bit);
}
__device__ __forceinline__ int clamp_len(int n, int max_pages) { return n < 0 ? 0 : min(n, max_pages * kPage); }
__device__ __forceinline__ int pages_of(int tokens) { return (tokens + kPage - 1) / kPage; }
__device__ __forceinline__ bool row_bit(const uint32_t* bits, int r) { return (bits[r >> 5] >> (r & 31)) & 1u; }

// a / b for a >= 0, b > 0: 32-bit division when both fit (the usual case;
// 64-bit division is a long instruction sequence on the GPU).
__device__ __noinline__ int64_t div_wide(int64_t a, int64_t b) { return a / b; }
__device__ __forceinline__ int div_nn(int64_t a, int b) {
  if ((uint64_t)a >> 32 == 0) return (int)((uint32_t)a / (uint32_t)b);
  return (int)div_wide(a, b);
}

// The job containing global page x (x < total pages).
__device__ __noinline__ Job job_at(const BlockCtx& c, int x) {
  int lo = 0, hi = c.G - 1;  // largest g with Hkv * gpre[g] <= x
#pragma unroll 1
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (c.Hkv * c.gpre[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  Job j;
  j.g = lo;
  j.n = c.gpre[lo + 1] - c.gpre[lo];
  const int base = c.Hkv * c.gpre[lo];
  j.h = (int)((uint32_t)(x - base) / (uint32_t)j.n);
  j.start = base + j.h * j.n;
  return j;
}

// The piece after (cur, n pages): its job and pages; false when there is none.
__device__ __noinline__ bool next_piece(const BlockCtx& c, Job& cur, int& n) {
  const int x = cur.start + cur.n;
  if (x >= c.e) return false;
  cur = x >= c.jl.start ? c.jl : job_at(c, x);
  n = min(c.e, cur.start + cur.n) - x;
  return true;
}

// Suffix tokens of a row (0 when it is inactive).
__device__ __forceinline__ int slen_of(const BlockCtx& c, int r) {
  if (c.slen) return c.slen[r];
  return row_bit(c.rowbits, r) ? clamp_len(__ldg(c.suffix_len + r), c.max_sp) : 0;
}

// An active row's suffix pages into its group's count (word g + 1 of gpre, whose top
// bit says that a row of the group is active).
constexpr uint32_t kAnyActive = 0x80000000u;
__device__ __forceinline__ void count_row(const AttnParams& p, int32_t* gpre, int r, int slen) {
  const int g = (int)(((uint64_t)(uint32_t)r * p.rpg_mul) >> 32);
  uint32_t* w = reinterpret_cast<uint32_t*>(gpre + g + 1);
  atomicAdd(w, (uint32_t)pages_of(slen));
  atomicOr(w, kAnyActive);
}
// A group's pages: its prompt pages if any row of it is active, plus its active
// rows' suffix pages.
__device__ __forceinline__ int pages_of_group(int word, int plen) {
  return word < 0 ? (int)((uint32_t)word & ~kAnyActive) + pages_of(plen) : 0;
}

// The lengths and activity of the rows past the first one per thread (G <= rows),
// four of a thread's rows in flight.  Out of line: a call with few rows does not
// fetch this code.
__device__ __noinline__ void more_rows(const AttnParams& p, int32_t* slen_s, int32_t* plen_s, uint32_t* rowbits,
                                       int32_t* gpre, int c, int tid, int nthreads) {
  constexpr int kU = 4;
  const int lane = tid & 31, nrows = p.G * p.rpg;
#pragma unroll 1
  for (int r0 = tid + nthreads; r0 - lane < nrows; r0 += kU * nthreads) {  // (whole warps: the ballots below)
    int act[kU], sl[kU], pl[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = r0 + u * nthreads;
      act[u] = sl[u] = pl[u] = 0;
      if (r < nrows) {
        act[u] = p.row_active == nullptr ? 1 : p.row_active[r];
        sl[u] = p.suffix_len[r];
        if (r < p.G) pl[u] = p.prompt_len[r];
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = r0 + u * nthreads;
      if (r < nrows) {
        if (c == 0 && (sl[u] < 0 || sl[u] > p.max_sp * kPage)) flag(p.dev_status, RGD_DEV_BAD_PAGE);
        sl[u] = act[u] ? clamp_len(sl[u], p.max_sp) : 0;
        if (p.slen_in_smem) slen_s[r] = sl[u];
        if (act[u]) count_row(p, gpre, r, sl[u]);
        if (r < p.G) {
          if (c == 0 && (pl[u] < 0 || pl[u] > p.max_pp * kPage)) flag(p.dev_status, RGD_DEV_BAD_PAGE);
          plen_s[r] = clamp_len(pl[u], p.max_pp);
        }
      }
      const uint32_t bits = __ballot_sync(0xffffffffu, r < nrows && act[u] != 0);
      if (lane == 0 && r - lane < nrows) rowbits[r >> 5] = bits;
    }
  }
}

// Page i of the block's range.
struct PageRef {
  int page, desc, h;   // pool page (-1: none); tokens | row << 16 (-1: every row); kv head
  int pos, ng;         // position in its group of 8, and the pages of that group
};
__device__ __noinline__ PageRef resolve_page(const BlockCtx& c, int i) {
  PageRef r{-1, 0, 0, 0, 0};
  const int x = c.b + i;
  if (x >= c.e) return r;
  const Job jb = i < c.n0 ? c.j0 : x >= c.jl.start ? c.jl : job_at(c, x);
  // this block's piece of the job starts at max(b, job start); groups restart there
  const int pstart = max(c.b, jb.start);
  const int kin = x - pstart;
  const int npiece = min(c.e, jb.start + jb.n) - pstart;
  r.pos = kin % kGroupPages;
  r.ng = min(kGroupPages, npiece - (kin - r.pos));
  r.h = jb.h;
  const int k = x - jb.start;
  const int plen = c.plen[jb.g];
  const int ppg = pages_of(plen);
  int row = -1, tok = 0;
  if (k < ppg) {
    r.page = __ldg(c.prompt_bt + (int64_t)jb.g * c.max_pp + k);
    tok = min(kPage, plen - k * kPage);
  } else {
    int ks = k - ppg;
#pragma unroll 1
    for (int rr = 0; rr < c.rpg; ++rr) {  // the active row holding suffix page ks
      const int slen = slen_of(c, jb.g * c.rpg + rr);
      const int np = pages_of(slen);
      if (ks < np) {
        r.page = __ldg(c.suffix_bt + (int64_t)(jb.g * c.rpg + rr) * c.max_sp + ks);
        tok = min(kPage, slen - ks * kPage);
        row = rr;
        break;
      }
      ks -= np;
    }
  }
  r.desc = tok | ((row & 0xffff) << 16);
  return r;
}

// Bounded wait that also gives up as soon as another role has given up.
// A waiting thread sleeps inside try_wait (woken when the phase completes), so
// warps parked on a barrier take no issue slots from the working ones.
__device__ __noinline__ bool wait_or_abort_slow(uint64_t* bar, uint32_t parity, volatile int32_t* abort_flag,
                                                uint64_t limit_ns) {
  if (*abort_flag) return false;
  const uint64_t t0 = globaltimer_ns();
#pragma unroll 1
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait_sleep(bar, parity, 20000u)) return true;
    if ((i & 63u) == 0) {
      if (*abort_flag) return false;
      if (globaltimer_ns() - t0 > limit_ns) {
        *abort_flag = 1;
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int32_t* abort_flag,
                                              uint64_t limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  return wait_or_abort_slow(bar, parity, abort_flag, limit_ns);
}

// Bounded wait (one thread) until a job's other pieces have counted themselves;
// the ticket, or -1.
__device__ __noinline__ int wait_ticket(const int32_t* ticket, int nparts, volatile int32_t* abort_flag,
                                        uint64_t limit_ns) {
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    const int tk = ld_acquire_gpu(ticket);
    if ((tk & 0xffff) == nparts) return tk;
    if (*abort_flag || globaltimer_ns() - t0 > limit_ns) {
      *abort_flag = 1;
      return -1;
    }
    __nanosleep(64);
  }
}

// 128-byte swizzle of a [rows][128 B] tile (16-byte chunk index XOR the row mod 8).
__device__ __forceinline__ uint32_t sw128_off(int row, int chunk) {
  return (uint32_t)(row * 128 + (((chunk ^ row) & 7) << 4));
}

// Byte of P^T's 16-byte chunk c8 (8 query columns of part 0, the high parts, or
// 1, the residuals) of token t.
template <typename C>
__device__ __forceinline__ uint32_t p_off(int t, int c8, int part) {
  const int byte = part * C::kN * 2 + c8 * 16, atom = byte / C::kSw, row = t & 7;
  const int chunk = ((byte % C::kSw) >> 4) ^ (C::kSw == 128 ? row : C::kSw == 64 ? (row >> 1) : (row >> 2));
  return (uint32_t)(atom * 128 * C::kSw + (t >> 3) * 8 * C::kSw + row * C::kSw + ((chunk & (C::kSw / 16 - 1)) << 4));
}

// Warp reduction of 8 values per lane over the lanes, ending with lane L
// holding the result for index L & 7: two butterfly steps over the lane
// quarters, then halving over 8 lanes.
template <typename Op>
__device__ __forceinline__ float transpose_reduce8(float (&v)[8], int lane, Op op) {
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = op(v[i], __shfl_xor_sync(0xffffffffu, v[i], 16));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = op(v[i], __shfl_xor_sync(0xffffffffu, v[i], 8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float send = up ? v[i] : v[i + o];
      const float keep = up ? v[i + o] : v[i];
      v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, o));
    }
  }
  return v[0];
}

// Two fp32 values in one 64-bit register, and a fused multiply-add or a sum of both
// at once (a softmax thread's arithmetic is all in pairs: half the issue slots).
__device__ __forceinline__ uint64_t pair(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpair(uint64_t a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// P = hi + lo with hi = p rounded to bf16 and lo = p - hi rounded to bf16
// (|p - hi - lo| <= 2^-17 |p| without a bias; truncating both gave 2^-15 and made
// every weight 7e-6 too small on average), two values per 32-bit word, the first in
// the low half.
__device__ __forceinline__ void split_bf16x2(float p0, float p1, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16x2(p0, p1);
  const uint64_t h = pair(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
  const float2 l = unpair(fma2(h, pair(-1.f, -1.f), pair(p0, p1)));  // (exact)
  lo = pack_bf16x2(l.x, l.y);
}

// The merge of a split job by every warp of the block that holds its first page,
// once all pieces are done: a warp takes a query, a lane D / 32 of its columns.
// The block's own piece (0) has its O in shared memory, the others in consecutive
// workspace slots (ml, which starts at the own piece: stride mls; o: stride nq * D).
// It sits at the end of the block and an L2 round trip takes 1-2 us while other
// blocks stream, so round trips are what counts: a lane brings a piece's (m, l),
// the weights go round by shuffles, and the first eight pieces' columns are in
// flight meanwhile.  (One prompt over 19 blocks, 20 queries: 4.6 us from the last
// partial with a table of weights in shared memory and a barrier on both sides of it,
// 2.4 so.)  A job of more than 32 pieces goes on in the same way, 32 at a time.
template <int D>
__device__ __noinline__ void merge_job(const float* own, const int32_t* erow, const float2* ml, const float* o,
                                       __nv_bfloat16* out, float* lse, int nq, int pieces, int warp, int nwarps) {
  constexpr int kV = D / 32;
  using Cols = typename std::conditional<D == 128, float4, float2>::type;
  const int lane = threadIdx.x & 31, mls = ml_stride(nq);
#pragma unroll 1
  for (int q = warp; q < nq; q += nwarps) {
    const Cols* src = reinterpret_cast<const Cols*>(o + (int64_t)q * D) + lane;
    const int64_t step = (int64_t)nq * 32;
    float M = -INFINITY, l = 0.f, acc[kV];
    {
      const Cols x = reinterpret_cast<const Cols*>(own + q * D)[lane];
#pragma unroll
      for (int i = 0; i < kV; ++i) acc[i] = reinterpret_cast<const float*>(&x)[i];
    }
#pragma unroll 1
    for (int k0 = 0; k0 < pieces; k0 += 32) {
      const int n = min(32, pieces - k0);
      Cols v[8];
      auto load = [&](int b) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (k0 + b + u > 0 && b + u < n) v[u] = __ldcg(src + (k0 + b + u) * step);
      };
      float2 x = make_float2(0.f, 0.f);
      if (lane < n) x = __ldcg(ml + (int64_t)(k0 + lane) * mls + q);
      load(0);
      float m = x.y > 0.f ? x.x : -INFINITY;
#pragma unroll 1
      for (int i = 16; i > 0; i >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, i));
      m = fmaxf(m, M);
      const float w = x.y > 0.f ? exp2f(x.x - m) : 0.f;
      float ls = w * x.y;
#pragma unroll 1
      for (int i = 16; i > 0; i >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, i);
      // what has been summed so far (the own piece at first) comes under the new maximum
      const float f = k0 == 0 ? __shfl_sync(0xffffffffu, w, 0) : M == -INFINITY ? 0.f : exp2f(M - m);
      l = (k0 == 0 ? 0.f : l * f) + ls;
      M = m;
#pragma unroll
      for (int i = 0; i < kV; ++i) acc[i] *= f;
#pragma unroll 1
      for (int b = 0; b < n; b += 8) {
        if (b > 0) load(b);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float wk = __shfl_sync(0xffffffffu, w, b + u);
          if (k0 + b + u > 0 && b + u < n) {
#pragma unroll
            for (int i = 0; i < kV; ++i) acc[i] += wk * reinterpret_cast<const float*>(&v[u])[i];
          }
        }
      }
    }
    const int row = erow[q];
    if (row < 0) continue;
    const float inv = l > 0.f ? 1.f / l : 0.f;
    uint32_t pk[kV / 2];
#pragma unroll
    for (int i = 0; i < kV / 2; ++i) pk[i] = pack_bf16x2(acc[2 * i] * inv, acc[2 * i + 1] * inv);
    uint32_t* dst = reinterpret_cast<uint32_t*>(out + (int64_t)row * D) + lane * (kV / 2);
    if constexpr (kV == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(pk[0], pk[1]);
    else *dst = pk[0];
    if (lse && lane == 0) lse[row] = l > 0.f ? (M + log2f(l)) * kLn2 : -INFINITY;
  }
}

// The weights of a split job's other partials for one query (in place of their
// maxima, over the whole job's sum) and of this block's own piece (m, l; returned
// unnormalised); m and l become the whole job's.
__device__ __noinline__ float fold_weights(float2* pml, int stride, int nparts, float& m, float& l) {
  float2 x[kMaxFold];
#pragma unroll
  for (int k = 0; k < kMaxFold; ++k) x[k] = k < nparts ? pml[k * stride] : make_float2(0.f, 0.f);
  float M = l > 0.f ? m : -INFINITY;
#pragma unroll
  for (int k = 0; k < kMaxFold; ++k) M = x[k].y > 0.f ? fmaxf(M, x[k].x) : M;
  const float own = l > 0.f ? exp2f(m - M) : 0.f;
  float L = own * l;
#pragma unroll
  for (int k = 0; k < kMaxFold; ++k) {
    x[k].x = x[k].y > 0.f ? exp2f(x[k].x - M) : 0.f;
    L += x[k].x * x[k].y;
  }
  const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
  for (int k = 0; k < kMaxFold; ++k)
    if (k < nparts) pml[k * stride].x = x[k].x * inv;
  m = M;
  l = L;
  return own;
}

// Q of job jb into a Q buffer by the 128 piece-end threads (this one: et):
// [D/64 halves][kN rows][128 B], 128-byte swizzle; rows >= nq are zero.
template <int D, int kN>
__device__ __noinline__ void write_q(const __nv_bfloat16* q, const Job& jb, uint32_t qbase, int et, int nq, int gq,
                                     int rpg, int Hq) {
  constexpr int kCc = D / 8;  // 16-byte chunks per query row
  constexpr int kPer = kN * kCc / 128, kB = kPer % 4 == 0 ? 4 : kPer % 2 == 0 ? 2 : 1;
#pragma unroll 1
  for (int i0 = 0; i0 < kPer; i0 += kB) {
    uint4 v[kB];
#pragma unroll
    for (int i = 0; i < kB; ++i) {
      const int idx = (i0 + i) * 128 + et, r = idx / kCc, cc = idx % kCc;
      v[i] = make_uint4(0u, 0u, 0u, 0u);
      if (r < nq) {
        const int rr = r / gq;
        v[i] = __ldg(reinterpret_cast<const uint4*>(
                         q + ((int64_t)(jb.g * rpg + rr) * Hq + jb.h * gq + (r - rr * gq)) * D) + cc);
      }
    }
#pragma unroll
    for (int i = 0; i < kB; ++i) {
      const int idx = (i0 + i) * 128 + et, r = idx / kCc, cc = idx % kCc;
      st_shared_v4(qbase + (cc >> 3) * (kN * 128) + sw128_off(r, cc & 7), v[i].x, v[i].y, v[i].z, v[i].w);
    }
  }
  fence_proxy_async_smem();
}

// The jobs with no pages at all (empty prompt and suffixes, some row active):
// out = 0, lse = -inf.
__device__ __noinline__ void write_empty_jobs(const BlockCtx& c, int block, int blocks, int et, int nq, int gq, int Hq,
                                              int D, __nv_bfloat16* out, float* lse) {
#pragma unroll 1
  for (int j = block; j < c.G * c.Hkv; j += blocks) {
    const int g = j / c.Hkv, h = j - g * c.Hkv;
    if (c.gpre[g + 1] != c.gpre[g]) continue;
#pragma unroll 1
    for (int i = 0; i < nq; ++i) {
      const int rr = g * c.rpg + i / gq;
      if (!row_bit(c.rowbits, rr)) continue;
      const int64_t row = (int64_t)rr * Hq + h * gq + i % gq;
      if (et < D) out[row * D + et] = __float2bfloat16(0.f);
      if (et == 0 && lse) lse[row] = -INFINITY;
    }
  }
}

// O^T columns c0, c0 + step, ... (eight a time) of a finished piece, by a warp of
// TMEM lane quarter d / 32: to the partial `part` of a split job, or, normalised,
// to the output rows, with the `nparts` other partials of a split job added by
// their weights (pml's x).  (part, out and po point at head dimension d; erow and
// einv have 128 entries, erow -1 past nq.)  A block's time after its last MMA is
// this function's, so the eight columns' loads go together and stores are
// predicated: with a branch or a dependent load per column it took 120 cycles a
// column (360 with a partial to add).
template <int D>
__device__ __noinline__ void write_columns(uint32_t col, int lo_off, int c0, int step, int nq, float* part,
                                           __nv_bfloat16* out, const int32_t* erow, const float* einv, int nparts,
                                           const float* po, const float2* pml) {
#pragma unroll 1
  for (; c0 < nq; c0 += step) {
    uint32_t hi[8], lo[8];
    tmem_ld8(col + c0, hi);
    tmem_ld8(col + lo_off + c0, lo);
    tmem_ld_wait8(hi);
    tmem_ld_wait8(lo);
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
    if (part) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (c0 + i < nq) part[(c0 + i) * D] = v[i];
      continue;
    }
    const int4 r0 = *reinterpret_cast<const int4*>(erow + c0), r1 = *reinterpret_cast<const int4*>(erow + c0 + 4);
    const float4 e0 = *reinterpret_cast<const float4*>(einv + c0), e1 = *reinterpret_cast<const float4*>(einv + c0 + 4);
    const int row[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
    const float ev[8] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] *= ev[i];
    const float* o = po + c0 * D;  // (past nq: other shared memory, for columns that are not stored)
    const float2* m = pml + c0;
#pragma unroll 1
    for (int k = 0; k < nparts; ++k, o += nq * D, m += ml_stride(nq)) {
      float x[8], y[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        x[i] = m[i].x;
        y[i] = o[i * D];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] += x[i] * y[i];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (row[i] >= 0) out[(int64_t)row[i] * D] = __float2bfloat16(v[i]);
  }
}

template <int D, int NS, int QS>
__global__ void __launch_bounds__(AttnCfg<D, NS, QS>::kThreads, 1)
    attn_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                const __grid_constant__ AttnParams p) {
  using C = AttnCfg<D, NS, QS>;
  constexpr int kTile = kPage * D * 2;  // one K or V page-head tile
  constexpr int kHalves = D / 64;
  constexpr int kThr = C::kThreads;
  constexpr uint32_t kIdQK = idesc_bf16_f32(128, C::kN, 0, 0);      // A = K, B = Q: both K-major
  constexpr uint32_t kIdPV = idesc_bf16_f32(128, 2 * C::kN, 1, 1);  // A = V^T, B = P^T (both parts): both MN-major
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int nrows = p.G * p.rpg;
  const AttnLayout& L = p.L;
  uint32_t* rowbits = reinterpret_cast<uint32_t*>(smem + L.rowbits);
  int32_t* gpre = reinterpret_cast<int32_t*>(smem + L.gpre);
  int32_t* plen_s = reinterpret_cast<int32_t*>(smem + L.plen);
  int32_t* slen_s = reinterpret_cast<int32_t*>(smem + L.slen);
  int32_t* descs = reinterpret_cast<int32_t*>(smem + L.desc);
  float* einv = reinterpret_cast<float*>(smem + L.einv);
  int32_t* erow = reinterpret_cast<int32_t*>(smem + L.erow);
  // (m, l) of a folded job's partials, behind their O in the K ring; l becomes the weights
  auto pml_of = [&](int parts) { return reinterpret_cast<float2*>(smem + L.kring + parts * p.nq * D * 4); };
  __shared__ uint64_t k_full[kRingMax], k_empty[kRingMax], v_full[kRingMax], v_empty[kRingMax];
  __shared__ uint64_t s_full[2], s_empty[2], p_full[2], p_empty[2], q_full[2], q_empty[2];
  __shared__ uint64_t o_full[2], o_free[2], ml_full[2], ml_empty[2], mma_done[2];
  // the split job that starts in this block: its pieces (0: none), its index, its
  // ticket, and whether its partials' copies (completing on m_full) were issued
  __shared__ uint64_t m_full;
  __shared__ int32_t s_abort, s_issued[2], s_mpieces, s_mjob, s_tick, s_mcopy;
  // the block's last piece: 0 none or given up, 2 to be written; its job + 1 if split; its O^T buffer
  __shared__ int32_t s_last_ok, s_last_split, s_last_ob;
  __shared__ uint32_t s_tmem;
  __shared__ BlockCtx ctx;
  volatile int32_t* abort_flag = &s_abort;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = blockIdx.x;
  const uint32_t sbase = smem_u32(smem);

  if (tid == 0) {
#pragma unroll 1
    for (int i = 0; i < kRingMax; ++i) {
      mbar_init(&k_full[i], kGroupPages);  // one arrival per page position (absent pages of a short group too)
      mbar_init(&k_empty[i], 1);           // the group's QK commit
      mbar_init(&v_full[i], kGroupPages);
      mbar_init(&v_empty[i], 1);           // the group's PV commit
    }
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_full[i], 2);  // the QK commit, and its thread (which orders the page descriptors)
      mbar_init(&s_empty[i], 4 * NS);
      mbar_init(&p_full[i], 4 * NS);
      mbar_init(&p_empty[i], 1);
      mbar_init(&q_full[i], 4);
      mbar_init(&q_empty[i], 1);
      mbar_init(&o_full[i], 1);
      mbar_init(&o_free[i], 4);
      mbar_init(&ml_full[i], 4 * NS);
      mbar_init(&ml_empty[i], 4);
      mbar_init(&mma_done[i], 1);
    }
    s_abort = 0;
    s_issued[0] = s_issued[1] = 0;
    mbar_init(&m_full, 1);
    s_mpieces = s_mcopy = 0;
    s_last_ok = s_last_split = 0;
    fence_mbar_init();
  }
  if (warp == C::kQk) {
    tmem_alloc(&s_tmem, C::kTmemCols);
    tmem_relinquish();
  }
  if (warp == C::kProdK && lane == 0) {  // the copies' descriptors, fetched while the set-up runs
    prefetch_tensormap(&tmK);
    prefetch_tensormap(&tmV);
  }
#pragma unroll 1
  for (int g = tid; g <= p.G; g += kThr) gpre[g] = 0;
  __syncthreads();
  // launched as a programmatic dependent of the previous kernel on the stream:
  // everything below may read what that kernel wrote
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // ---- lengths and activity flags, all loads issued together, kept in shared memory ----
  {
    int act = 0, sl = 0, pl = 0;
    auto load = [&](int r) {
      act = sl = pl = 0;
      if (r < nrows) {
        act = p.row_active == nullptr ? 1 : p.row_active[r];
        sl = p.suffix_len[r];
      }
      if (r < p.G) pl = p.prompt_len[r];
    };
    load(tid);
    // This block's share of the block tables and queries is asked of L2 while the
    // lengths load (each line once over the grid), so that the first block-table
    // and query loads of every block find them there.
    const int64_t nb_p = (int64_t)p.G * p.max_pp * 4, nb_s = (int64_t)nrows * p.max_sp * 4;
    const int64_t nb_q = (int64_t)nrows * p.Hq * D * 2;
    const int64_t lp = (nb_p + 127) / 128, ls = (nb_s + 127) / 128, lq = (nb_q + 127) / 128;
    const int64_t step = (int64_t)p.C * kThr;
#pragma unroll 1
    for (int64_t l = (int64_t)tid * p.C + c; l < lp + ls + lq; l += step) {
      if (l < lp) prefetch_l2(reinterpret_cast<const uint8_t*>(p.prompt_bt) + l * 128);
      else if (l < lp + ls) prefetch_l2(reinterpret_cast<const uint8_t*>(p.suffix_bt) + (l - lp) * 128);
      else prefetch_l2(reinterpret_cast<const uint8_t*>(p.q) + (l - lp - ls) * 128);
    }
    auto store = [&](int r) {
      if (r < nrows) {
        if (c == 0 && (sl < 0 || sl > p.max_sp * kPage)) flag(p.dev_status, RGD_DEV_BAD_PAGE);
        sl = act ? clamp_len(sl, p.max_sp) : 0;
        if (p.slen_in_smem) slen_s[r] = sl;
        if (act) count_row(p, gpre, r, sl);
      }
      if (r < p.G) {
        if (c == 0 && (pl < 0 || pl > p.max_pp * kPage)) flag(p.dev_status, RGD_DEV_BAD_PAGE);
        plen_s[r] = clamp_len(pl, p.max_pp);
      }
      const uint32_t bits = __ballot_sync(0xffffffffu, r < nrows && act != 0);
      if (lane == 0 && r - lane < nrows) rowbits[r >> 5] = bits;
    };
    store(tid);
    if (nrows > kThr) more_rows(p, slen_s, plen_s, rowbits, gpre, c, tid, kThr);
  }
  if (tid == 0) {
    ctx.G = p.G;
    ctx.Hkv = p.Hkv;
    ctx.rpg = p.rpg;
    ctx.max_pp = p.max_pp;
    ctx.max_sp = p.max_sp;
    ctx.prompt_bt = p.prompt_bt;
    ctx.suffix_bt = p.suffix_bt;
    ctx.suffix_len = p.suffix_len;
    ctx.gpre = gpre;
    ctx.plen = plen_s;
    ctx.slen = p.slen_in_smem ? slen_s : nullptr;
    ctx.rowbits = rowbits;
  }
  __syncthreads();
  if (warp == 0) {  // inclusive prefix sum of the groups' pages, then this block's range
    // (up to 32 groups, one per lane, stay in registers; every function called or
    // division made here is on the path to the first copy, and cold)
    const bool few = p.G <= 32;
    const int E = (p.G + 31) / 32;
    const int lo = 1 + lane * E, hi = min(p.G + 1, lo + E);
    int sum = 0;
    if (few) {
      if (lane < p.G) sum = pages_of_group(gpre[lane + 1], plen_s[lane]);
    } else {
#pragma unroll 1
      for (int i = lo; i < hi; ++i) {
        const int n = pages_of_group(gpre[i], plen_s[i - 1]);
        gpre[i] = n;
        sum += n;
      }
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (few) {
      if (lane < p.G) gpre[lane + 1] = incl;
    } else {
      int run = incl - sum;
#pragma unroll 1
      for (int i = lo; i < hi; ++i) {
        run += gpre[i];
        gpre[i] = run;
      }
    }
    __syncwarp();
    // The pages are dealt over Ceff = min(C, T) blocks, block c taking the positions
    // [floor(c T / Ceff), floor((c + 1) T / Ceff)) of T.  With up to 32 groups (more
    // give every block about as many job ends) and more pages than blocks, every job
    // counts p.end_pages more than it has, for the time of its end, so that a block
    // with more ends gets fewer pages; positions past a job's pages map to its end.
    // Every position is some block's, so a job's pieces are exactly the blocks from
    // that of its first page to that of its last.
    const int pages = p.Hkv * __shfl_sync(0xffffffffu, incl, 31);
    const int extra = few && pages > p.C ? p.end_pages : 0;
    const uint32_t some = __ballot_sync(0xffffffffu, few && sum > 0);
    const int ends = __popc(some & (0xffffffffu >> (31 - lane)));  // groups with pages, up to the lane's
    const int vincl = p.Hkv * (incl + extra * ends);
    const int T = __shfl_sync(0xffffffffu, vincl, 31), Ceff = min(p.C, T);
    int x = pages;  // lane 0: b; lane 1: e
    auto group_of = [&](int v, int at0, int at1) {  // the group in which lane 0's (1's) position lies, by prefix sums v
      const int g0 = __popc(__ballot_sync(0xffffffffu, lane < p.G && v <= at0));
      const int g1 = __popc(__ballot_sync(0xffffffffu, lane < p.G && v <= at1));
      return lane == 1 ? g1 : g0;
    };
    if (c < Ceff) {
      const int y = div_nn((int64_t)(c + (lane & 1)) * T, Ceff);
      if (extra == 0) {
        x = y;
      } else {
        const int g = group_of(vincl, __shfl_sync(0xffffffffu, y, 0), __shfl_sync(0xffffffffu, y, 1));
        const int n = __shfl_sync(0xffffffffu, sum, g), excl = __shfl_sync(0xffffffffu, incl, g) - n;
        const int off = y - (__shfl_sync(0xffffffffu, vincl, g) - p.Hkv * (n + extra));
        const int h = (int)((uint32_t)off / (uint32_t)max(1, n + extra));
        if (g < p.G) x = p.Hkv * excl + h * n + min(off - h * (n + extra), n);
      }
    }
    const int b = __shfl_sync(0xffffffffu, x, 0), e = __shfl_sync(0xffffffffu, x, 1);
    if (lane == 0) {
      ctx.b = b;
      ctx.e = e;
      ctx.T = T;
      ctx.Ceff = Ceff;
    }
    __syncwarp();
    if (b < e) {  // the jobs at the range's ends (lanes 0 and 1)
      const int at = lane == 1 ? e - 1 : b;
      Job j;
      int end;
      if (few) {  // (lane g holds the prefix sums up to group g)
        j.g = group_of(p.Hkv * incl, b, e - 1);
        j.n = __shfl_sync(0xffffffffu, sum, j.g);
        const int base = p.Hkv * (__shfl_sync(0xffffffffu, incl, j.g) - j.n);
        j.h = (int)((uint32_t)(at - base) / (uint32_t)j.n);
        j.start = base + j.h * j.n;
        end = __shfl_sync(0xffffffffu, vincl, j.g) - (p.Hkv - 1 - j.h) * (j.n + extra) - extra - 1;
      } else {
        j = job_at(ctx, at);
        end = j.start + j.n - 1;
      }
      if (lane == 0) {
        ctx.j0 = j;
        ctx.n0 = min(e, j.start + j.n) - b;
      }
      if (lane == 1) {
        ctx.jl = j;
        ctx.jl_end = end;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int b = ctx.b, e = ctx.e;
  const int hk = p.hk, hv = p.hv, np = p.np, nqb = p.nqb;

  if (warp == C::kProdK || warp == C::kProdV) {
    // ============================ producers ===========================
    // One warp for K and one for V, 32 pages (one per lane, one copy each) a round,
    // groups of 8 pages; a copy takes its issuer ~75 cycles, hence two warps.  A K
    // tile lands as [2 row groups][D/64][8 rows][128 B], so that a group is one
    // 128-row A operand per half, a V tile as [D/64][16 rows][128 B].  The next round's pages
    // are resolved (job by binary search, then the block-table entry) before the
    // first wait of a round, so the block-table loads are in flight meanwhile.
    const bool is_v = warp == C::kProdV;
    const int nr = is_v ? hv : hk;
    const uint64_t nr_mul = is_v ? p.hv_mul : p.hk_mul;
    uint64_t* full = is_v ? v_full : k_full;
    uint64_t* empty = is_v ? v_empty : k_empty;
    uint8_t* ring = smem + (is_v ? L.vring : L.kring);
    const uint64_t pol = policy_evict_first();
    const int n_pages = e - b;
    int gbase = 0;  // groups started before sequence position ib
    PageRef nxt = resolve_page(ctx, lane);
#pragma unroll 1
    for (int ib = 0; ib < n_pages; ib += 32) {
      const PageRef cur = nxt;
      bool have_next = false;
      const bool valid = ib + lane < n_pages;
      const bool start = valid && cur.pos == 0;
      const uint32_t starts = __ballot_sync(0xffffffffu, start);
      const uint32_t le = 0xffffffffu >> (31 - lane);
      const int gidx = gbase + __popc(starts & le) - 1;  // lane 0 may continue the last round's group
      const int g0 = __shfl_sync(0xffffffffu, gidx, 0);
      const int g1 = __shfl_sync(0xffffffffu, gidx, 31 - __clz(__ballot_sync(0xffffffffu, valid)));
      gbase += __popc(starts);
      const int gs = gidx - (int)(((uint64_t)(uint32_t)gidx * nr_mul) >> 32) * nr;  // gidx % nr
      bool aborted = false;
#pragma unroll 1
      for (int gq = g0; gq <= g1; ++gq) {
        if (gq >= nr) {
          if (!have_next && ib + 32 < n_pages) {
            nxt = resolve_page(ctx, ib + 32 + lane);
            have_next = true;
          }
          const int use = (int)(((uint64_t)(uint32_t)gq * nr_mul) >> 32);  // gq / nr
          const bool ok = wait_or_abort(&empty[gq - use * nr], (uint32_t)(use - 1) & 1u, abort_flag, p.wait_ns);
          if (!__all_sync(0xffffffffu, ok)) {
            aborted = true;
            break;
          }
        }
        if (valid && gidx == gq) {
          int32_t y = -2 * kPage;  // fully out of bounds: the TMA fills zeros
          if (cur.page >= 0 && cur.page < p.num_pages) y = (cur.page * p.Hkv + cur.h) * kPage;
          else flag(p.dev_status, RGD_DEV_BAD_PAGE);
          uint8_t* sl = ring + gs * C::kArea;
          // (the descriptor before the arrival, which releases it to the QK thread and so to the softmax)
          if (!is_v) descs[(gq & 7) * kGroupPages + cur.pos] = cur.desc;
          mbar_arrive_expect_tx(&full[gs], kTile);
          if (is_v) tma_load_3d_hint(sl + cur.pos * kTile, &tmV, &full[gs], 0, y, 0, pol);
          else tma_load_4d_hint(sl + cur.pos * kTile, &tmK, &full[gs], 0, 0, 0, y / 8, pol);
          if (cur.pos == cur.ng - 1 && cur.ng < kGroupPages) mbar_arrive_cnt(&full[gs], kGroupPages - cur.ng);
          if (start) atomicMax(&s_issued[is_v], gq + 1);
        }
      }
      if (aborted) break;
      if (!have_next && ib + 32 < n_pages) nxt = resolve_page(ctx, ib + 32 + lane);
      __syncwarp();
    }
    // Every copy of this warp is issued: a programmatic dependent of this kernel
    // (the sample head) may be scheduled once every block has got here or
    // exited.  It still waits for this kernel to complete before it writes.
    if (is_v) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // The split job that starts in this block is merged here, with the block's
    // last piece: its other pieces are the first ones of later blocks, behind no
    // wait on another block, so waiting for them ends (bounded anyway).  Their
    // partials, if few, are copied to the K ring, which nothing uses after the last QK.
    if (!is_v && lane == 0 && b < e) {
      const Job jb = ctx.jl;
      const int nparts = div_nn((int64_t)(ctx.jl_end + 1) * ctx.Ceff - 1, ctx.T) - c;
      if (jb.start >= b && nparts > 0) {
        const int j = jb.g * p.Hkv + jb.h;
        s_mpieces = nparts + 1;
        s_mjob = j;
        if (nparts > p.fold) {
          mbar_arrive(&m_full);  // (nothing to wait for here: the merge comes after the own partial)
        } else {
          int tick = wait_ticket(p.ticket + j, nparts, abort_flag, p.wait_ns);
#pragma unroll 1
          for (int g = max(0, gbase - hk); g < gbase; ++g)
            if (!wait_or_abort(&k_empty[g % hk], (uint32_t)(g / hk) & 1u, abort_flag, p.wait_ns)) tick = -1;
          s_tick = tick;
          if (tick > 0 && (tick >> 16) == 0) {
            const int64_t slot = (int64_t)c + j + 1;
            const uint32_t ob = nparts * p.nq * D * 4, mb = nparts * ml_stride(p.nq) * 8;
            fence_proxy_async_global();  // (the partials are other blocks' ordinary writes)
            s_mcopy = 1;
            mbar_arrive_expect_tx(&m_full, ob + mb);
            bulk_load(smem + L.kring, p.slot_o + slot * p.nq * D, ob, &m_full);
            bulk_load(smem + L.kring + ob, p.slot_ml + slot * ml_stride(p.nq), mb, &m_full);
          } else {
            mbar_arrive(&m_full);
          }
        }
      }
    }
  } else if (warp == C::kQk) {
    // ============================ QK issue ============================
    if (lane == 0 && b < e) {
      const uint64_t kdesc = smem_desc(sbase + L.kring, 16, kHalves * 1024, 2);
      const uint64_t qdesc = smem_desc(sbase + L.q, 16, 1024, 2);
      int gi = 0, pc = 0, gs = 0;
      uint32_t ph = 0;
      bool ok = true;
      Job cur = ctx.j0;
      int n_in = ctx.n0;
#pragma unroll 1
      for (bool more = true; ok && more; more = next_piece(ctx, cur, n_in)) {
        const int qb = nqb == 2 ? pc & 1 : 0;
        if (!wait_or_abort(&q_full[qb], (uint32_t)(nqb == 2 ? pc >> 1 : pc) & 1u, abort_flag, p.wait_ns)) break;
#pragma unroll 1
        for (int k0 = 0; k0 < n_in; k0 += kGroupPages) {
          const int sb = gi & 1;
          if (!wait_or_abort(&k_full[gs], ph, abort_flag, p.wait_ns) ||
              (gi >= 2 && !wait_or_abort(&s_empty[sb], (uint32_t)((gi >> 1) - 1) & 1u, abort_flag, p.wait_ns))) {
            ok = false;
            break;
          }
          tc_fence_after();
          uint64_t a = kdesc + (uint64_t)((gs * C::kArea) >> 4), bq = qdesc + (uint64_t)((qb * C::kQBytes) >> 4);
#pragma unroll 1
          for (int hf = 0; hf < kHalves; ++hf, a += 1024 >> 4, bq += C::kN * 128 >> 4) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)  // 16 of the half's 64 columns
              umma_bf16(tmem + C::kSCol + sb * C::kN, a + kk * 2, bq + kk * 2, kIdQK, (hf | kk) != 0 ? 1u : 0u);
          }
          umma_commit(&s_full[sb]);
          mbar_arrive(&s_full[sb]);
          umma_commit(&k_empty[gs]);  // the group's K is no longer read
          if (k0 + kGroupPages >= n_in) umma_commit(&q_empty[qb]);  // Q's buffer may take a later piece
          ++gi;
          if (++gs == hk) {
            gs = 0;
            ph ^= 1u;
          }
        }
        ++pc;
      }
    }
  } else if (warp == C::kPv) {
    // ============================ PV issue ============================
    // V: 64-column halves 2 KB apart (head dim 64 has one, read twice: lanes
    // 64..127 of O^T are not used), 8-token groups 1 KB apart
    if (lane == 0 && b < e) {
      const uint64_t vdesc = smem_desc(sbase + L.vring, D == 128 ? 2048 : 0, 1024, 2);
      const uint64_t pdesc = smem_desc(sbase + L.p, 128 * C::kSw, 8 * C::kSw, C::kSwLayout);
      int gi = 0, pc = 0, gs = 0;
      uint32_t ph = 0;
      bool ok = true;
      Job cur = ctx.j0;
      int n_in = ctx.n0;
#pragma unroll 1
      for (bool more = true; ok && more; more = next_piece(ctx, cur, n_in)) {
        const int ob = C::kOBufs == 2 ? pc & 1 : 0;
        const uint32_t od = tmem + C::kOCol + ob * 2 * C::kN;
        if (pc >= C::kOBufs &&
            !wait_or_abort(&o_free[ob], (uint32_t)((C::kOBufs == 2 ? pc >> 1 : pc) - 1) & 1u, abort_flag, p.wait_ns))
          break;
#pragma unroll 1
        for (int k0 = 0; k0 < n_in; k0 += kGroupPages) {
          const int ng = min(kGroupPages, n_in - k0);
          const int pb = np == 2 ? gi & 1 : 0;
          if (!wait_or_abort(&v_full[gs], ph, abort_flag, p.wait_ns) ||
              !wait_or_abort(&p_full[pb], (uint32_t)(np == 2 ? gi >> 1 : gi) & 1u, abort_flag, p.wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          uint64_t vd = vdesc + (uint64_t)((gs * C::kArea) >> 4), pd = pdesc + (uint64_t)((pb * C::kPBytes) >> 4);
#pragma unroll 1
          for (int j = 0; j < ng; ++j, vd += kTile >> 4, pd += C::kSw)  // (16 tokens of P^T are 16 kSw bytes)
            umma_bf16(od, vd, pd, kIdPV, (k0 | j) != 0 ? 1u : 0u);
          umma_commit(&p_empty[pb]);
          umma_commit(&v_empty[gs]);
          if (k0 + kGroupPages >= n_in) umma_commit(&o_full[ob]);
          ++gi;
          if (++gs == hv) {
            gs = 0;
            ph ^= 1u;
          }
        }
        ++pc;
      }
    }
  } else if (warp < C::kEpi) {
    // ============================ softmax ============================
    // Thread = token t of the group (lane quarter qd); set hs takes queries
    // QS hs .. + QS - 1.  The reference maxima of the queries (log2 units,
    // negated) live in shared memory, two versions: a group that moves a set's
    // maxima writes the other version and the set's threads switch after a
    // barrier, so all use the same reference for a group.  lacc[i] is this thread's running sum of
    // query QS hs + i.
    constexpr int kCh = QS / 8;  // 8-query chunks of a set
    const int qd = warp & 3, hs = warp >> 2;
    const int t = qd * 32 + lane, jp = t >> 4, tip = t & 15;
    const int q0 = hs * QS;
    const uint32_t tl = tmem + ((uint32_t)(qd * 32) << 16);
    float* wmax = reinterpret_cast<float*>(smem + L.wmax) + q0;
    float* lw = reinterpret_cast<float*>(smem + L.lw) + q0;
    float* mfin = reinterpret_cast<float*>(smem + L.mfin) + q0;
    float* nref = reinterpret_cast<float*>(smem + L.mref) + q0;  // [2 versions][kNq], negated
    constexpr uint32_t kAllQ = QS == 32 ? 0xffffffffu : (1u << QS) - 1u;
    // named barrier of the set's 128 threads (0 is __syncthreads, 1 the piece ends')
    auto set_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(hs + 2) : "memory"); };
    auto set_any = [&](bool x) {  // whether x holds in any of them
      int r;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\t"
          "bar.red.or.pred q, %2, 128, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
          : "=r"(r) : "r"((int)x), "r"(hs + 2) : "memory");
      return r != 0;
    };
    auto wwait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, wait_or_abort(bar, parity, abort_flag, p.wait_ns));
    };
    // the set's queries of row sel: a suffix page is visible to them only, a prompt page
    // to all (also to the columns past the job's nq: their Q is 0 and nothing reads them)
    auto row_mask = [&](int sel) {  // queries sel * gq .. + gq - 1
      const int lo = max(0, sel * p.gq - q0), hi = min(QS, (sel + 1) * p.gq - q0);
      if (hi <= lo) return 0u;
      return (hi - lo >= 32 ? 0xffffffffu : ((1u << (hi - lo)) - 1u)) << lo;
    };
    uint64_t lacc[QS / 2];  // (pairs)
#pragma unroll
    for (int i = 0; i < QS / 2; ++i) lacc[i] = 0;
    const uint64_t scale2 = pair(p.scale_log2, p.scale_log2);
    int mv = 0;         // current version of the reference maxima
    bool fresh = true;  // piece start: every reference is -inf (not read from shared memory)
    int gi = 0;
    bool ok = true;
    if (b < e) {
      Job cur = ctx.j0;
      int n_in = ctx.n0;
      int pc = 0;
#pragma unroll 1
      for (bool more = true; more; more = next_piece(ctx, cur, n_in)) {
        const int ob = C::kOBufs == 2 ? pc & 1 : 0;
#pragma unroll 1
        for (int k0 = 0; k0 < n_in; k0 += kGroupPages) {
          const int ng = min(kGroupPages, n_in - k0);
          const int sb = gi & 1;
          const bool has = jp < ng;
          if (ok && !wwait(&s_full[sb], (uint32_t)(gi >> 1) & 1u)) ok = false;
          tc_fence_after();
          uint32_t vis = 0;  // the visible queries of this token
          if (ok && has) {
            const int dsc = descs[(gi & 7) * kGroupPages + jp];
            const int sel = (int)(int16_t)(dsc >> 16);
            if (tip < (dsc & 0xffff)) vis = sel < 0 ? kAllQ : row_mask(sel);
          }
          const bool whole = __all_sync(0xffffffffu, vis == kAllQ);
          // queries that any of the warp's tokens is visible to: on suffix pages few
          // are, and the others' scores need not be looked at
          const uint32_t seen = whole ? kAllQ : __reduce_or_sync(0xffffffffu, vis);
          const uint32_t sa = tl + C::kSCol + sb * C::kN + q0;
          uint32_t sc[QS > 16 ? 2 : kCh][8];  // scores by chunks of 8 queries
          auto chunk_seen = [&](int ch) { return ((seen >> (8 * ch)) & 0xffu) != 0; };
          auto mask_chunk = [&](uint32_t (&x)[8], int ch) {  // -inf where the query does not see this token
            if (whole) return;
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = ((vis >> (ch * 8 + q)) & 1u) ? x[q] : 0xff800000u;
          };
          // does a score exceed its query's reference by 2^8?  (the set's four warps agree)
          float mx = -INFINITY;
          auto look = [&](const uint32_t (&x)[8], int ch) {
            const float* nr = nref + mv * C::kNq + ch * 8;
#pragma unroll
            for (int q = 0; q < 8; q += 4) {
              const float4 n4 = fresh ? make_float4(kNoRef, kNoRef, kNoRef, kNoRef) : *reinterpret_cast<const float4*>(nr + q);
              const float2 a = unpair(fma2(pair(__uint_as_float(x[q]), __uint_as_float(x[q + 1])), scale2, pair(n4.x, n4.y)));
              const float2 c2 = unpair(fma2(pair(__uint_as_float(x[q + 2]), __uint_as_float(x[q + 3])), scale2, pair(n4.z, n4.w)));
              mx = fmaxf(fmaxf(mx, a.x), a.y);
              mx = fmaxf(fmaxf(mx, c2.x), c2.y);
            }
          };
          if (QS <= 16) {  // the scores stay in registers
#pragma unroll
            for (int ch = 0; ch < kCh; ++ch) tmem_ld8(sa + ch * 8, sc[ch]);
#pragma unroll
            for (int ch = 0; ch < kCh; ++ch) {
              tmem_ld_wait8(sc[ch]);
              mask_chunk(sc[ch], ch);
              if (chunk_seen(ch)) look(sc[ch], ch);
            }
          } else {  // (too many: they are read twice, a chunk ahead of its use)
            tmem_ld8(sa, sc[0]);
#pragma unroll
            for (int ch = 0; ch < kCh; ++ch) {
              uint32_t(&x)[8] = sc[ch & 1];
              tmem_ld_wait8(x);
              if (ch + 1 < kCh) tmem_ld8(sa + (ch + 1) * 8, sc[(ch + 1) & 1]);
              if (chunk_seen(ch)) {
                mask_chunk(x, ch);
                look(x, ch);
              }
            }
          }
          if (set_any(mx > kRescaleLog2)) {
            // this warp's query maxima, then the new reference of each query
            // from the four warps and its factor
#pragma unroll 1
            for (int ch = 0; ch < kCh; ++ch) {  // (read again: rare, and it keeps the registers few)
              uint32_t x[8];
              float v[8];
              tmem_ld8(sa + ch * 8, x);
              tmem_ld_wait8(x);
#pragma unroll
              for (int q = 0; q < 8; ++q)
                v[q] = ((vis >> (ch * 8 + q)) & 1u) ? __uint_as_float(x[q]) * p.scale_log2 : -INFINITY;
              const float wm = transpose_reduce8(v, lane, [](float x, float y) { return fmaxf(x, y); });
              if (lane < 8) wmax[qd * C::kNq + ch * 8 + lane] = wm;
            }
            set_sync();
            const int qi = lane < QS ? lane : 0;
            const float no = fresh ? kNoRef : nref[mv * C::kNq + qi];
            const float mo = no == kNoRef ? -INFINITY : -no;
            const float mn = fmaxf(fmaxf(mo, wmax[qi]), fmaxf(fmaxf(wmax[C::kNq + qi], wmax[2 * C::kNq + qi]),
                                                             wmax[3 * C::kNq + qi]));
            const float fq = mo == -INFINITY ? 0.f : exp2f(mo - mn);
            if (qd == 0 && lane < QS) nref[(mv ^ 1) * C::kNq + qi] = mn == -INFINITY ? kNoRef : -mn;
#pragma unroll
            for (int q = 0; q < QS; q += 2) {
              const float2 l = unpair(lacc[q / 2]);
              lacc[q / 2] = pair(l.x * __shfl_sync(0xffffffffu, fq, q), l.y * __shfl_sync(0xffffffffu, fq, q + 1));
            }
            // O^T already holds this piece's earlier groups: once their PV is
            // done, the set's query columns (this warp's 32 head dimensions) are scaled
            if (k0 > 0) {
              const int pg = gi - 1;
              if (ok && !wwait(&p_empty[np == 2 ? pg & 1 : 0], (uint32_t)(np == 2 ? pg >> 1 : pg) & 1u)) ok = false;
              if (ok) {
                tc_fence_after();
#pragma unroll 1
                for (int part = 0; part < 2; ++part) {
#pragma unroll 1
                  for (int ch = 0; ch < kCh; ++ch) {
                    const uint32_t oc = tl + C::kOCol + (2 * ob + part) * C::kN + q0 + ch * 8;
                    uint32_t o8[8];
                    tmem_ld8(oc, o8);
                    tmem_ld_wait();
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                      o8[u] = __float_as_uint(__uint_as_float(o8[u]) * __shfl_sync(0xffffffffu, fq, ch * 8 + u));
                    tmem_st8(oc, o8);
                  }
                }
                tmem_st_wait();
              }
            }
            set_sync();  // the new version is written, wmax and the old version are read
            mv ^= 1;
            fresh = false;
          }
          // P = 2^(s - m) in bf16 high part + residual (ex2 of -inf is +0), 8 queries at a time
          const int pb = np == 2 ? gi & 1 : 0;
          const uint32_t pbase = sbase + L.p + pb * C::kPBytes;
          if (QS > 16) tmem_ld8(sa, sc[0]);
#pragma unroll
          for (int ch = 0; ch < kCh; ++ch) {
            uint32_t(&x)[8] = sc[QS > 16 ? ch & 1 : ch];
            if (QS > 16) {
              tmem_ld_wait8(x);
              if (ch + 1 < kCh) tmem_ld8(sa + (ch + 1) * 8, sc[(ch + 1) & 1]);  // (behind this chunk's exponentials)
              mask_chunk(x, ch);
            }
            if (ch == kCh - 1) {  // S^T is in registers
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&s_empty[sb]);
            }
            uint32_t hi[4] = {0u, 0u, 0u, 0u}, lo[4] = {0u, 0u, 0u, 0u};
            if (chunk_seen(ch)) {
              const float* nr = nref + mv * C::kNq + ch * 8;
#pragma unroll
              for (int q = 0; q < 8; q += 4) {
                const float4 n4 = fresh ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4*>(nr + q);
                const uint64_t nn[2] = {pair(n4.x, n4.y), pair(n4.z, n4.w)};
#pragma unroll
                for (int u = 0; u < 4; u += 2) {
                  const int i = q + u;
                  const float2 t2 = unpair(fma2(pair(__uint_as_float(x[i]), __uint_as_float(x[i + 1])), scale2, nn[u / 2]));
                  const float p0 = ex2_approx(t2.x), p1 = ex2_approx(t2.y);
                  lacc[(ch * 8 + i) / 2] = add2(lacc[(ch * 8 + i) / 2], pair(p0, p1));
                  split_bf16x2(p0, p1, hi[i / 2], lo[i / 2]);
                }
              }
            }
            // the P^T buffer is free once the PV that read it last is done
            if (ch == 0 && gi >= np && ok &&
                !wwait(&p_empty[pb], (uint32_t)((np == 2 ? gi >> 1 : gi) - 1) & 1u))
              ok = false;
            if (ok) {
              st_shared_v4(pbase + p_off<C>(t, hs * kCh + ch, 0), hi[0], hi[1], hi[2], hi[3]);
              st_shared_v4(pbase + p_off<C>(t, hs * kCh + ch, 1), lo[0], lo[1], lo[2], lo[3]);
            }
          }
          fence_proxy_async_smem();  // the MMAs read P^T through the async proxy
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&p_full[pb]);
          ++gi;
        }
        // piece end: per-warp query sums and the reference maxima to the piece-end warps
        const int mb = pc & 1;
        if (pc >= 2 && ok && !wwait(&ml_empty[mb], (uint32_t)((pc >> 1) - 1) & 1u)) ok = false;
#pragma unroll
        for (int ch = 0; ch < kCh; ++ch) {
          float v[8];
#pragma unroll
          for (int q = 0; q < 8; q += 2) {
            const float2 l = unpair(lacc[(ch * 8 + q) / 2]);
            v[q] = l.x;
            v[q + 1] = l.y;
            lacc[(ch * 8 + q) / 2] = 0;
          }
          const float ls = transpose_reduce8(v, lane, [](float x, float y) { return x + y; });
          if (lane < 8) {
            lw[(mb * 4 + qd) * C::kNq + ch * 8 + lane] = ls;
            if (qd == 0) {
              const float no = fresh ? kNoRef : nref[mv * C::kNq + ch * 8 + lane];
              mfin[mb * C::kNq + ch * 8 + lane] = no == kNoRef ? -INFINITY : -no;
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&ml_full[mb]);
        fresh = true;
        ++pc;
      }
    }
  } else {
    // ============================ piece ends ==========================
    // Thread = head dimension d of O^T (lane quarter w), and query et of the
    // job.  Writes Q of the next pieces, reads a finished piece's O^T, and writes
    // the output or the partial of a split job.
    const int w = warp - C::kEpi;
    const int d = w * 32 + lane, et = d;
    const uint32_t tl = tmem + ((uint32_t)(w * 32) << 16);
    const float* lw = reinterpret_cast<const float*>(smem + L.lw);
    const float* mfin = reinterpret_cast<const float*>(smem + L.mfin);
    auto epi_sync = [&]() { asm volatile("bar.sync 1, 128;" ::: "memory"); };
    auto wwait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, wait_or_abort(bar, parity, abort_flag, p.wait_ns));
    };
    const int nq = p.nq, gq = p.gq;
    const int mls = ml_stride(nq);
    bool ok = true;
    auto put_q = [&](const Job& jb, int qb) {
      write_q<D, C::kN>(p.q, jb, sbase + L.q + qb * C::kQBytes, et, nq, gq, p.rpg, p.Hq);
      __syncwarp();
      if (lane == 0) mbar_arrive(&q_full[qb]);
    };
    if (b < e) {
      Job cur = ctx.j0, nx1 = cur, nxq = cur;  // this piece, the next, the next whose Q is to be written
      int n_in = ctx.n0, n1 = n_in, nq_in = n_in;
      put_q(cur, 0);
      bool hasq = next_piece(ctx, nxq, nq_in);
      if (hasq && nqb == 2) {
        put_q(nxq, 1);
        hasq = next_piece(ctx, nxq, nq_in);
      }
      write_empty_jobs(ctx, c, p.C, et, nq, gq, p.Hq, D, p.out, p.lse);  // (while the first group's copies are in flight)
#pragma unroll 1
      for (int pc = 0;; ++pc) {
        const int ob = C::kOBufs == 2 ? pc & 1 : 0, mb = pc & 1;
        const int j = cur.g * p.Hkv + cur.h;
        const bool merger = cur.start >= b && cur.start + cur.n > e;  // the job goes on in later blocks
        const bool split = merger || cur.start < b;
        nx1 = cur;
        n1 = n_in;
        const bool more = next_piece(ctx, nx1, n1);
        // ---- Q of the piece nqb ahead, into this piece's Q buffer ----
        if (hasq) {
          const int qb = nqb == 2 ? pc & 1 : 0;
          if (ok && !wwait(&q_empty[qb], (uint32_t)(nqb == 2 ? pc >> 1 : pc) & 1u)) ok = false;
          if (ok) put_q(nxq, qb);
          else if (lane == 0) mbar_arrive(&q_full[qb]);  // (keeps the QK warp's waits bounded by the abort)
          hasq = next_piece(ctx, nxq, nq_in);
        }
        // ---- this piece's maxima, sums and output rows, one query per thread ----
        if (ok && !wwait(&ml_full[mb], (uint32_t)(pc >> 1) & 1u)) ok = false;
        if (merger && ok && !wwait(&m_full, 0u)) ok = false;
        const int nparts = merger && ok ? s_mpieces - 1 : 0;  // its other pieces
        const bool fold = nparts > 0 && nparts <= p.fold;
        float2* pml = pml_of(nparts);
        bool good = ok && !(fold && (s_tick <= 0 || (s_tick >> 16) != 0));
        const int64_t slot = (int64_t)c + j;  // of a split job's partial
        erow[et] = -1;
        if (et < nq) {
          float M = mfin[mb * C::kNq + et];
          float Ls = (lw[(mb * 4) * C::kNq + et] + lw[(mb * 4 + 1) * C::kNq + et]) +
                     (lw[(mb * 4 + 2) * C::kNq + et] + lw[(mb * 4 + 3) * C::kNq + et]);
          const int r = et / gq, rr = cur.g * p.rpg + r;
          const int row = row_bit(rowbits, rr) ? rr * p.Hq + cur.h * gq + (et - r * gq) : -1;
          erow[et] = row;
          float own = 1.f;
          if (fold && good) own = fold_weights(pml + et, mls, nparts, M, Ls);
          einv[et] = Ls > 0.f ? own / Ls : 0.f;
          if (good && split && !fold) p.slot_ml[slot * mls + et] = make_float2(M, Ls);
          if (good && (!split || fold) && p.lse && row >= 0) p.lse[row] = Ls > 0.f ? (M + log2f(Ls)) * kLn2 : -INFINITY;
        }
        if (ok && !wwait(&o_full[ob], (uint32_t)(C::kOBufs == 2 ? pc >> 1 : pc) & 1u)) ok = false;
        tc_fence_after();
        good = __all_sync(0xffffffffu, good && ok && !*abort_flag);
        epi_sync();
        if (!more) {  // the block's last piece: all softmax and piece-end warps share its columns
          if (et == 0) {
            s_last_ok = ok ? (good ? 2 : 1) : 0;
            s_last_split = split ? j + 1 : 0;
            s_last_ob = ob;
          }
          break;
        }
        if (good && d < D)
          write_columns<D>(tl + C::kOCol + 2 * ob * C::kN, C::kN, 0, 8, nq,
                           split ? p.slot_o + slot * nq * D + d : nullptr, p.out + d, erow, einv, 0, nullptr, nullptr);
        tc_fence_before();
        epi_sync();
        if (lane == 0) {
          mbar_arrive(&o_free[ob]);
          mbar_arrive(&ml_empty[mb]);
        }
        if (et == 96 && split) {  // (a later piece follows, so this job ends here; the last warp has least to do)
          // the partial was written by every piece-end warp before the barrier
          red_release_gpu_add(p.ticket + j, good && !*abort_flag ? 1 : 0x10001);
        }
        cur = nx1;
        n_in = n1;
      }
    }
    if (b >= e) write_empty_jobs(ctx, c, p.C, et, nq, gq, p.Hq, D, p.out, p.lse);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const int parts = s_mpieces - 1;  // of the split job merged here, without the block's own
  const bool fold = parts > 0 && parts <= p.fold;
  if (s_last_ok > 0) {  // (uniform) the last piece's O^T: set s and the piece-end warps take every (NS + 1)-th chunk
    const int split = s_last_split, j = split - 1;
    const int d = (warp & 3) * 32 + lane;
    if (warp < C::kEpi + 4 && s_last_ok == 2 && d < D)
      write_columns<D>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + C::kOCol + 2 * s_last_ob * C::kN, C::kN,
                       (warp >> 2) * 8, (NS + 1) * 8, p.nq,
                       parts > 0 ? (fold ? nullptr : reinterpret_cast<float*>(smem) + d)
                       : split   ? p.slot_o + ((int64_t)c + j) * p.nq * D + d
                                 : nullptr,
                       p.out + d, erow, einv,
                       fold ? parts : 0, reinterpret_cast<const float*>(smem + L.kring) + d, pml_of(parts));
    tc_fence_before();
    __syncthreads();
  }
  // (a split job's last piece counts itself also when this block has given up)
  if (tid == 0 && s_last_split > 0 && parts < 0)  // the partial was written by every warp before the barrier
    red_release_gpu_add(p.ticket + (s_last_split - 1), s_last_ok == 2 && !*abort_flag ? 1 : 0x10001);
  if (parts > 0) {  // (uniform) the merge of the split job that starts in this block
    const int j = s_mjob;
    if (!fold) {
      int tick = 0;
      if (lane == 0) tick = wait_ticket(p.ticket + j, parts, abort_flag, p.wait_ns);
      tick = __shfl_sync(0xffffffffu, tick, 0);
      __syncwarp();
      const int64_t slot = (int64_t)c + j;
      if (tick > 0 && (tick >> 16) == 0 && s_last_ok == 2)  // (the own O is in the rings, idle by now)
        merge_job<D>(reinterpret_cast<const float*>(smem), erow, p.slot_ml + slot * ml_stride(p.nq),
                     p.slot_o + slot * p.nq * D, p.out, p.lse, p.nq, parts + 1, warp, kThr / 32);
      __syncthreads();  // (every warp has seen the ticket)
    }
    if (tid == 0) p.ticket[j] = 0;  // every other piece has counted itself
  }
  if (*abort_flag) {
    // a wait gave up: report, and let copies and MMAs still in flight drain (bounded)
    if (tid == 0) {
      flag(p.dev_status, RGD_DEV_WAIT_TIMEOUT);
      if (s_mcopy) mbar_wait(&m_full, 0);
#pragma unroll 1
      for (int g = max(0, s_issued[0] - hk); g < s_issued[0]; ++g) mbar_wait(&k_full[g % hk], (g / hk) & 1);
#pragma unroll 1
      for (int g = max(0, s_issued[1] - hv); g < s_issued[1]; ++g) mbar_wait(&v_full[g % hv], (g / hv) & 1);
    }
    if ((warp == C::kQk || warp == C::kPv) && lane == 0) {
      uint64_t* md = &mma_done[warp == C::kQk ? 0 : 1];
      umma_commit(md);  // arrives once every MMA this thread issued has completed
      mbar_wait(md, 0);
    }
    __syncthreads();
  }
  tc_fence_after();
  if (warp == C::kQk) tmem_dealloc(tmem, C::kTmemCols);
}

template <int D, int NS, int QS>
int launch_attn_cfg(const CUtensorMap& tmK, const CUtensorMap& tmV, const AttnParams& p, int smem_bytes,
                    cudaStream_t st) {
  static std::atomic<bool> done[kMaxDevices] = {};
  if (int rc = ensure_smem(attn_kernel<D, NS, QS>, kSmemLimit, done)) return rc;
  // (its blocks are placed, and set up what needs no input, while the previous kernel finishes)
  const cudaError_t e = launch_dependent(attn_kernel<D, NS, QS>, p.C, AttnCfg<D, NS, QS>::kThreads, smem_bytes, st,
                                         tmK, tmV, p);
  return e == cudaSuccess ? RGD_OK : cuda_error(e, "attention launch");
}

// The kernel of the job size's configuration (query_config).
template <int D>
int launch_attn(const CUtensorMap& tmK, const CUtensorMap& tmV, const AttnParams& p, int smem_bytes, cudaStream_t st) {
  const QueryConfig qc = query_config(p.nq);
  switch (qc.sets * 100 + qc.per_set) {
    case 108: return launch_attn_cfg<D, 1, 8>(tmK, tmV, p, smem_bytes, st);
    case 208: return launch_attn_cfg<D, 2, 8>(tmK, tmV, p, smem_bytes, st);
    case 308: return launch_attn_cfg<D, 3, 8>(tmK, tmV, p, smem_bytes, st);
    case 408: return launch_attn_cfg<D, 4, 8>(tmK, tmV, p, smem_bytes, st);
    case 316: return launch_attn_cfg<D, 3, 16>(tmK, tmV, p, smem_bytes, st);
    case 416: return launch_attn_cfg<D, 4, 16>(tmK, tmV, p, smem_bytes, st);
    case 324: return launch_attn_cfg<D, 3, 24>(tmK, tmV, p, smem_bytes, st);
    case 424: return launch_attn_cfg<D, 4, 24>(tmK, tmV, p, smem_bytes, st);
    default: return launch_attn_cfg<D, 4, 32>(tmK, tmV, p, smem_bytes, st);
  }
}

}  // namespace
}  // namespace rgd
