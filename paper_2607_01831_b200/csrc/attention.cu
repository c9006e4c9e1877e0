// lynx_anchor_attention and lynx_merge_verify_attention: split-K decode attention over the
// packed nibble planes, dequantised on chip (sm_100a).  This file holds what the kernels share
// (parameters, PTX helpers, the joining of partial results and the accept / reject decision) and the host
// side; the kernels are in attention_pipe.cuh, attention_i8.cuh and attention_f16.cuh.
//
// What is computed (Section 2 attention equation on the states of Section 4.2; accept/reject
// of Section 4.3): for every (sequence, KV head) the G = Hq/Hkv query heads of each of the n_q
// query positions ("columns", n_q*G of them) share one pass over that head's K and V planes.
//
// Per-token groups make dequantisation almost free: with x^ = zero_t + scale_t * level,
//     q . K^_t        = scale_t * (q . level_t) + zero_t * sum_d q_d
//     sum_t p_t V^_t  = sum_t (p_t scale_t) level_t + (sum_t p_t zero_t) * 1
// so the two contractions run on the integer levels and the scalars are applied per token
// outside.  Anchor attention (any column count) and verification with up to 16 columns per launch run both contractions as exact integer products on
// tcgen05.mma kind::i8 (attention_pipe.cuh up to 16 columns, attention_i8.cuh above); verification with 17..64 columns per launch
// runs its scores on tcgen05.mma kind::f16, its values likewise with two-term FP16 weights or as integers (attention_f16.cuh).
//
// Common shape.  Persistent grid, one CTA per SM, flash-decoding split-K in stream-K form: the
// (sequence, KV head, stage-unit) list is cut into equal contiguous ranges, one per CTA.
// Producer warps stream 16-token sub-blocks of the planes (1 KiB each, contiguous in the paged
// layout) into a shared-memory ring with bulk copies (TMA) completing on mbarriers, and
// the queries of each piece into one of two slots.
// A range that covers a whole (sequence, KV head) writes the output directly (the FP16 kernel: its slot like the others),
// otherwise the partial (m, l, O) goes to the workspace, and a small dependent kernel joins them, row by row, and takes the
// accept/reject decision of a verification; anchor calls with many heads have the last contributor of a head join them
// (atomic ticket, no waiting).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "block_division.cuh"
#include "bounded_wait.cuh"
#include "lynx_common.cuh"
#include "workspace_layout.cuh"

namespace lynx {
namespace {

constexpr int kMaxQ = kWsMaxQ;     // query positions per launch
constexpr int kMaxWindow = 64;     // query positions per call (Section 5.1: at most 64 speculative tokens); more than
                                   // kMaxQ positions or kMaxCols columns run as slices, one pass over the planes each
constexpr int kMaxCols = 64;       // n_q * G per launch
constexpr int kPartStride = kWsPartStride;

struct AttnParams {
  const __nv_bfloat16* q;
  const uint8_t *ka, *kr, *va, *vr;
  const float *km, *vm;
  const int32_t* block_table;
  const int32_t* seq_lens;
  float* out;
  const float* draft;
  int32_t* first_reject;
  float* dev;
  uint32_t* ws_flags;
  uint32_t* ws_tickets;    // [SMs] tickets of the CTAs that share a (sequence, KV head), at the first one's index
  uint32_t* ws_groups;     // [SMs][2] tickets of groups of such CTAs
  uint32_t* ws_seq_ctr;    // [B] rows of a sequence that have been joined (zeroed by the attention kernel)
  uint32_t* ws_long;       // [SMs / kLongStep] word i: 1 + the long segment that CTA kLongStep i lies inside of, or 0
  float* ws_dev;           // [B*Hkv][kMaxQ]
  float* ws_lse;           // [B][nq_stride][Hq] natural-log log-sum-exp of every output row's scores
  float* ws_part;          // [B*Hkv + CTAs][ncols_pad][kPartStride], slot = segment + CTA index (and see seg_word)
  float atol, rtol;
  float sm_log2;           // softmax_scale * log2(e)
  int B, nq, causal, Hq, Hkv, G, bt, num_blocks, max_blocks, ncols;
  // A call may be one slice [j0, j0 + nq) of the caller's n_q query positions (q and out then point at
  // position j0): nq_stride = the caller's n_q (positions per sequence in q and out), tail = n_q - j0
  // (the causal limit of position j of the slice is len - tail + j + 1).  Unsliced: both equal nq.
  int nq_stride, tail;
  int draft_vec;   // draft is 16-byte aligned: its rows are read four values at a time
  BlockDiv bt_div;      // for t / bt
  // The aligned cut (see sk_range), where it is possible at all: CTAs per segment (else 0), and for quotients by that and by Hkv
  int per_seg;
  BlockDiv seg_div, hkv_div;
  int combine_single;   // the attention kernel leaves a segment of one CTA in its slot, too
  int inline_merge;     // the last CTA of a segment joins its slots, not attn_combine_kernel
};
// Block of token t of a sequence.  (No division: its code, at four places of the unit loops, costs more in the instruction caches
// than its time.  Together with rolled drains and one copy of the 4-column kernel's restart, us: one layer of 131072 tokens 37.7 ->
// 37.1, two sequences of 16000 at 8 columns 22.1 -> 21.2, 16 ragged sequences with a verification at 16 columns 276 -> 274, one layer
// of 4096 tokens at 16 columns 18.0 -> 17.0.)
__device__ __forceinline__ int block_of(const AttnParams& p, int t) { return quotient(t, p.bt_div); }
// The contributors of a segment, first CTA << 16 | number of CTAs (0: no tokens), for attn_combine_kernel: in the padding of
// the slot of the segment's index, whosever that slot is.
__device__ __forceinline__ uint32_t* seg_word(const AttnParams& p, size_t bh, int part_cols) {
  return reinterpret_cast<uint32_t*>(p.ws_part + bh * (size_t)part_cols * kPartStride + 130);
}

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
// One probe of the barrier.  The hint lets the hardware park the thread (up to ~20 us here)
// until the phase completes instead of returning at once, so a waiting warp does not burn
// issue slots on polling; completion wakes it early.
constexpr uint32_t kMbarHintNs = 20000;
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(kMbarHintNs)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after ~2 s (at once if another thread of the CTA already gave up),
// records it in the CTA's abort word and returns false.  Callers carry on without the data and the host is told through the workspace status word.  The kernel still
// ends: trip counts follow from the pieces alone, and the hand-offs of pieces between the producer and the
// other warps, which need no data to arrive, have an abort word of their own (kItemAbort words behind the
// other): they stay in step after a wait for data has given up.  Nothing in this kernel waits on another CTA.
constexpr int kItemAbort = 9;
template <int WORD>
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_words) {
  return !abort_words[WORD] &&
         bounded_wait([=] { return mbar_try_wait(bar, parity); }, [] { return globaltimer_ns(); }, abort_words + WORD);
}
// One non-blocking probe of an mbarrier phase.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
template <int WORD = 0>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_word) {
  if (mbar_test(bar, parity)) return true;   // (a plain probe is several times quicker than one that may suspend)
  if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow<WORD>(bar, parity, abort_word);
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  return __byte_perm(a, b, sel);
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
  return v;
}


// Full codes of 8 elements from an anchor word and a residual word: ev = codes of elements
// 0,2,4,6 (one per byte), od = codes of elements 1,3,5,7.
// Each is one shift and one bitwise select, (a & mask) | (b & ~mask), in a single LOP3.
__device__ __forceinline__ uint32_t bit_select(uint32_t a, uint32_t b, uint32_t mask) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xE4;" : "=r"(d) : "r"(a), "r"(b), "r"(mask));
  return d;
}
__device__ __forceinline__ void merge_codes(uint32_t xa, uint32_t xr, uint32_t& ev, uint32_t& od) {
  ev = bit_select(xa << 4, xr, 0xF0F0F0F0u);
  od = bit_select(xa, xr >> 4, 0xF0F0F0F0u);
}
// Natural-log log-sum-exp of a row's scores from its running maximum (or reference exponent) M, in log2 units,
// and the sum L of 2^(score - M); -inf for a row that saw no token.
__device__ __forceinline__ float lse_of(float M, float L) {
  return L > 0.0f ? (M + __log2f(L)) * 0.6931471805599453f : -INFINITY;
}

struct Item {  // one piece: a run of stage-units of one (sequence, KV head) given to one CTA
  int b, hkv, len, first_cta, n_contrib, pad0, pad1, pad2;  // pad0 = units, pad1 = first unit
};

__device__ __forceinline__ void named_bar(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// a / b for 0 <= a < 2^22, 0 < b < 2^22: ten instructions, where an integer division takes thirty (64-bit: a hundred) one after
// the other, in the one warp that the first copy of a launch waits for.
__device__ __forceinline__ int small_div(int a, int b) {
  const int q = __float2int_rz(__fdividef((float)a, (float)b));   // (two units of the last place: off by one at most)
  const int r = a - q * b;
  return q + (r >= b) - (r < 0);
}
__device__ __forceinline__ long long sk_div(long long a, long long b) {   // a, b >= 0
  return ((a | b) >> 22) == 0 ? (long long)small_div((int)a, (int)b) : a / b;
}
struct SkRange {
  long long q, lo, hi, off_lo;   // off_lo: offset of `lo` among the Hkv * U units of sequence b_lo
  int b_lo, hkv, u;              // hkv, u: the head and unit of `lo` where the cut gives them, or hkv < 0
};
// What the aligned cut gives a CTA whatever the lengths: its segment, and which part of it.  (Before the lengths are there: behind
// them lies the first copy of a launch, and an instruction that waits for the one before it is 2 to 5 ns.)
struct SkPlace {
  int s, part, b, hkv;
};
__device__ __forceinline__ SkPlace sk_place(const AttnParams& p, int cta) {
  SkPlace a;
  a.s = p.per_seg > 1 ? quotient(cta, p.seg_div) : cta;
  a.part = cta - a.s * max(p.per_seg, 1);
  a.b = p.Hkv > 1 ? quotient(a.s, p.hkv_div) : a.s;
  a.hkv = a.s - a.b * p.Hkv;
  return a;
}
// The lengths as one warp knows them: lane i keeps sequence i's, so that the first 32 are read once (a look-up again is a
// round trip to the L2 on the way to a launch's first copy).
struct SeqLens {
  const int32_t* lens;
  int cap, len0;
  SeqLens() = default;
  __device__ __forceinline__ SeqLens(const AttnParams& p, int lane) : lens(p.seq_lens), cap(p.max_blocks * p.bt) {
    len0 = lane < p.B ? load(lane) : 0;
  }
  __device__ __forceinline__ int load(int b) const {
    const int len = ld_dep(lens + b);
    return len < 0 ? 0 : (len > cap ? cap : len);
  }
  // by the whole warp, of one sequence
  __device__ __forceinline__ int of(int b) const { return b < 32 ? __shfl_sync(0xFFFFFFFFu, len0, b) : load(b); }
  // by a lane, of sequence b0 + lane
  __device__ __forceinline__ int at(int b0, int lane) const { return b0 == 0 ? len0 : load(b0 + lane); }
};
// The stream-K cut of the work list (units of ST tokens in (sequence, KV head, position) order) for
// CTA `cta` of `n_cta`, derived by one warp from the sequence lengths on the device.  Normally every
// CTA takes q = ceil(total / n_cta) consecutive units, wherever the (sequence, head) boundaries fall.
// When all sequences have the same number of units U and the B * Hkv segments are few enough to give
// each of them c >= 1 CTAs of its own (one layer of a long context per launch), the cut is aligned
// instead: q = ceil(U / c), and CTA i takes part i % c of segment i / c.  No CTA then pays for the
// end of one piece and the start of another, at the cost of n_cta - c * segments idle CTAs (accepted
// up to 15 %).  lo, hi index a list in which every segment occupies c * q entries, so that the
// contributors of a segment and their partial slots follow from lo and q as in the plain cut.
template <int ST>
__device__ __forceinline__ SkRange sk_range(const AttnParams& p, int n_cta, int cta, int lane, const SeqLens& sl, const SkPlace& at) {
  SkRange r;
  r.hkv = r.u = -1;
  long long tot = 0;
  int umin = 0x7FFFFFFF, umax = 0;
  for (int b0 = 0; b0 < p.B; b0 += 32) {
    const bool in = b0 + lane < p.B;
    const int u = in ? (sl.at(b0, lane) + ST - 1) / ST : 0;   // (at most 2^24)
    tot += __reduce_add_sync(0xFFFFFFFFu, (unsigned)u);
    if (in) { umin = min(umin, u); umax = max(umax, u); }
  }
  umin = __reduce_min_sync(0xFFFFFFFFu, umin);
  umax = __reduce_max_sync(0xFFFFFFFFu, umax);
  if (p.per_seg > 0 && umin == umax && umax > 0) {
    const int c = p.per_seg, U = umax;                    // (U at most 2^24)
    const int q = c > 1 ? quotient(U + c - 1, p.seg_div) : U;
    r.q = q;
    r.lo = r.hi = 0; r.b_lo = 0; r.off_lo = 0;
    r.u = at.part * q;
    if (at.b < p.B && r.u < U) {
      r.b_lo = at.b;
      r.hkv = at.hkv;
      r.off_lo = (long long)at.hkv * U + r.u;
      r.lo = (long long)cta * q;                          // (part of segment s: (s c + part) q)
      r.hi = r.lo + min(q, U - r.u);
    }
    return r;
  }
  const long long T = tot * p.Hkv;
  r.q = sk_div(T + n_cta - 1, n_cta);
  r.lo = (long long)cta * r.q;
  r.hi = (r.lo + r.q < T) ? r.lo + r.q : T;
  r.b_lo = 0;
  r.off_lo = 0;
  if (r.lo < r.hi) {
    long long running = 0;
    for (int b0 = 0; b0 < p.B; b0 += 32) {
      const int b = b0 + lane;
      const long long u = b < p.B ? (long long)p.Hkv * ((sl.at(b0, lane) + ST - 1) / ST) : 0;
      long long incl = u;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
      }
      const long long excl = running + incl - u;
      const bool hit = u > 0 && r.lo >= excl && r.lo < excl + u;
      const unsigned mk = __ballot_sync(0xFFFFFFFFu, hit);
      if (mk) {
        const int src = __ffs(mk) - 1;
        r.b_lo = b0 + src;
        r.off_lo = r.lo - __shfl_sync(0xFFFFFFFFu, excl, src);
        break;
      }
      running += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
  }
  return r;
}

// A segment of this many CTAs or more is long: there is a multiple of kLongStep among those that lie inside of it, with nothing
// else to do.  Such a CTA tells attn_combine_kernel, and every other multiple that it does not.
constexpr int kLongSegment = 24, kLongStep = 16;
static_assert(kLongSegment >= kLongStep + 2, "a multiple between the first and the last");
__device__ __forceinline__ void tell_long(const AttnParams& p, int cta, const Item* it) {   // it: a piece of this CTA, or none
  if (cta % kLongStep) return;
  uint32_t seg = 0;
  if (it && it->n_contrib >= kLongSegment && cta > it->first_cta && cta < it->first_cta + it->n_contrib - 1)   // (then the only one)
    seg = 1u + (uint32_t)(it->b * p.Hkv + it->hkv);
  p.ws_long[cta / kLongStep] = seg;
}

// What is left to do for a sequence, by one warp of one CTA each: the count of finished rows that attn_combine_kernel decides by
// starts at zero; where there is no token, outputs are zero and nothing is rejected unless the draft is not zero.
// (Off the path of the sequences' tokens: called behind a CTA's last copy.)
template <bool FULL, int kPartCols>
__device__ __forceinline__ void per_sequence(const AttnParams& p, int cta, int n_cta, int lane, const SeqLens& sl, const Item* it) {
  if (FULL && lane == 0) tell_long(p, cta, it);
  for (int b = cta; b < p.B; b += n_cta) {
    if (FULL && lane == 0) p.ws_seq_ctr[b] = 0u;
    if (sl.of(b) != 0) continue;
    for (int h = lane; h < p.Hkv; h += 32) *seg_word(p, (size_t)b * p.Hkv + h, kPartCols) = 0;
    const size_t n = (size_t)p.nq * p.Hq * LYNX_D;
    for (size_t i = lane; i < n; i += 32) p.out[(size_t)b * p.nq_stride * p.Hq * LYNX_D + i] = 0.0f;
    for (int i = lane; i < p.nq * p.Hq; i += 32) p.ws_lse[(size_t)b * p.nq_stride * p.Hq + i] = -INFINITY;
    if (FULL && p.draft != nullptr) {
      int fr = p.nq;
      for (int j = p.nq - 1; j >= 0; --j) {
        float worst = 0.0f;
        for (int i = lane; i < p.Hq * LYNX_D; i += 32)
          worst = fmaxf(worst, fabsf(ld_dep(p.draft + ((size_t)b * p.nq_stride + j) * p.Hq * LYNX_D + i)) / p.atol);
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) worst = fmaxf(worst, __shfl_xor_sync(0xFFFFFFFFu, worst, off));
        if (lane == 0) p.dev[(size_t)b * p.nq_stride + j] = worst;
        if (worst > 1.0f) fr = j;
      }
      if (lane == 0) p.first_reject[b] = fr;
    }
  }
}

// Joins the partial results of the CTAs that share a (sequence, KV head) and takes the accept / reject decision: W warps per
// output row, its slots (m, l, O) dealt to them, five in flight each, the warps' sums joined in order.
// A programmatic dependent behind every verification and behind anchor calls with few heads, unless no sequence can have more than
// a unit and nothing is to be decided; anchor calls with many heads join in the attention kernel (see launch_combine).
// Latency bounds it -- the look-up of the segment, a round of slots, for verification a ticket and one more round -- and the
// instructions of a thread in a row, so that a row is cut over many threads where it has many slots.  (Before, the last CTA of
// a head joined all its columns behind a ticket and took the decision, and the other SMs had nothing to do.  us, by this step alone:
// one layer of 4096 tokens, 16 columns 27.8 -> 17.6, 4 columns 13.2 -> 11.6, of 131072 tokens, 32 columns, 96.4 -> 87.4, replayed
// from a graph -- 16.5, 9.9 and 80 with the steps since --; two sequences of 131072, 64 columns, 243 -> 236 among other passes; two
// of 16000, 8 columns, 25.7 -> 23.8.)
//
// Where there are many heads a segment has a slot or two on average, and a row is one warp's (four warps for every row: 16
// sequences of 500 tokens, 16 columns, 20.1 -> 21.8 us, 64 of 200, 32 columns, 47 -> 60 us).  But one long sequence among many short
// ones with few heads has up to a slot per SM, 148 of them behind one another in one warp: the rows of long segments (see
// tell_long) go to CTAs of their own in front of the others, four warps a row, eight slots in flight each.  (us, one sequence of 32768 tokens
// among 39 of 64, one KV head, 4 / 16 / 32 columns: 36.6 / 43.2 / 53.4 by a warp per row, 16.8 / 25.3 / 26.8 this way.)
constexpr int kCombineWarps = 4, kCombineFly = 5, kLongFly = 8;
// The sums of slots warp, warp + W, ... of n at `col`, relative to their running maximum M; a lane has four dims.
template <int FLY>
__device__ __forceinline__ void join_slots(const float* col, size_t sstride, int n, int warp, int W, int lane, float4& acc, float& M, float& L) {
  for (int i0 = warp; i0 < n; i0 += W * FLY) {
    float4 o[FLY];
    float2 ml[FLY];
#pragma unroll
    for (int u = 0; u < FLY; ++u) {
      const int i = i0 + u * W;
      ml[u] = make_float2(-INFINITY, 0.0f);
      o[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < n) {
        const float* s = col + (size_t)i * sstride;
        ml[u] = ld_dep(reinterpret_cast<const float2*>(s + 128));
        o[u] = ld_dep(reinterpret_cast<const float4*>(s) + lane);
      }
    }
    const float m0 = M;
#pragma unroll
    for (int u = 0; u < FLY; ++u) M = fmaxf(M, ml[u].x);
    const float f0 = m0 == -INFINITY ? 0.0f : ex2(m0 - M);
    L *= f0;
    acc.x *= f0; acc.y *= f0; acc.z *= f0; acc.w *= f0;
#pragma unroll
    for (int u = 0; u < FLY; ++u) {
      const float f = ml[u].x == -INFINITY ? 0.0f : ex2(ml[u].x - M);
      L = fmaf(ml[u].y, f, L);
      acc.x = fmaf(o[u].x, f, acc.x);
      acc.y = fmaf(o[u].y, f, acc.y);
      acc.z = fmaf(o[u].z, f, acc.z);
      acc.w = fmaf(o[u].w, f, acc.w);
    }
  }
}
// A row per CTA (kWide), or four, and with kWithLong in front of them n_long CTAs for the rows of long segments.
enum CombineMode { kWide, kNarrow, kWithLong };
template <CombineMode MODE>
__global__ void __launch_bounds__(kCombineWarps * 32) attn_combine_kernel(const AttnParams p, int part_cols, int n_slots, int n_long) {
  pdl_trigger();
  const bool for_long = MODE == kWithLong && (int)blockIdx.x < n_long;
  const int W = MODE == kWide || for_long ? kCombineWarps : 1;
  const int warp = W == 1 ? 0 : threadIdx.x >> 5, lane = threadIdx.x & 31;   // warp of the row
  __shared__ float4 o_s[kCombineWarps][32];
  __shared__ float2 ml_s[kCombineWarps];
  int b, j, hq;
  if (for_long) {
    pdl_wait();
    const int i = (int)blockIdx.x / p.ncols, c = (int)blockIdx.x - i * p.ncols;
    const uint32_t bh1 = ld_dep(p.ws_long + i);
    if (bh1 == 0 || bh1 > (uint32_t)(p.B * p.Hkv)) return;
    const int hkv = (int)((bh1 - 1) % p.Hkv);
    b = (int)((bh1 - 1) / p.Hkv);
    j = c / p.G;
    hq = hkv * p.G + (c - j * p.G);
  } else {
    const unsigned r = MODE == kWide ? blockIdx.x : (blockIdx.x - n_long) * kCombineWarps + (threadIdx.x >> 5);
    const unsigned bj = r / p.Hq;
    hq = r % p.Hq;
    j = bj % p.nq;
    b = bj / p.nq;
    if (MODE != kWide && b >= p.B) return;
    pdl_wait();
  }
  const int hkv = hq / p.G, g = hq - hkv * p.G;
  const size_t bh = (size_t)b * p.Hkv + hkv, row = ((size_t)b * p.nq_stride + j) * p.Hq + hq;
  const bool decide = p.draft != nullptr;
  const uint32_t seg = ld_dep(seg_word(p, bh, part_cols));
  float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
  if (decide && warp == 0) {
    const float* dp = p.draft + row * LYNX_D + 4 * lane;   // (no more than the alignment of a float is asked of the draft)
    if (p.draft_vec) d = ld_dep(reinterpret_cast<const float4*>(dp));
    else d = make_float4(ld_dep(dp), ld_dep(dp + 1), ld_dep(dp + 2), ld_dep(dp + 3));
  }
  const int first = min((int)(seg >> 16), n_slots - 1), n = min((int)(seg & 0xFFFFu), n_slots - first);
  if (MODE == kWithLong) {
    // a long segment's rows belong to the first of the multiples inside of it
    if (for_long ? (int)blockIdx.x / p.ncols != first / kLongStep + 1 : n >= kLongSegment) return;
  }
  const bool direct = n == 1 && !p.combine_single;   // written by the attention kernel
  if (n == 0 || (direct && !decide)) return;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float lse = 0.0f;
  if (!direct) {
    const size_t sstride = (size_t)part_cols * kPartStride;
    const float* col = p.ws_part + (bh + first) * sstride + (size_t)(j * p.G + g) * kPartStride;
    float M = -INFINITY, L = 0.0f;
    if (for_long) join_slots<kLongFly>(col, sstride, n, warp, W, lane, acc, M, L);
    else join_slots<kCombineFly>(col, sstride, n, warp, W, lane, acc, M, L);
    if (W > 1) {
      if (warp > 0) o_s[warp][lane] = acc;
      if (lane == 0) ml_s[warp] = make_float2(M, L);
      __syncthreads();
      if (warp > 0) return;
      float mx = M;
#pragma unroll
      for (int k = 1; k < kCombineWarps; ++k) mx = fmaxf(mx, ml_s[k].x);
      const float f0 = M == -INFINITY ? 0.0f : ex2(M - mx);
      L *= f0;
      M = mx;
      acc.x *= f0; acc.y *= f0; acc.z *= f0; acc.w *= f0;
#pragma unroll
      for (int k = 1; k < kCombineWarps; ++k) {
        const float2 ml = ml_s[k];
        const float4 o = o_s[k][lane];
        const float f = ml.x == -INFINITY ? 0.0f : ex2(ml.x - mx);
        L = fmaf(ml.y, f, L);
        acc.x = fmaf(o.x, f, acc.x);
        acc.y = fmaf(o.y, f, acc.y);
        acc.z = fmaf(o.z, f, acc.z);
        acc.w = fmaf(o.w, f, acc.w);
      }
    }
    const float inv = L > 0.0f ? 1.0f / L : 0.0f;
    acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    lse = lse_of(M, L);
  } else {
    if (warp > 0) return;
    acc = ld_dep(reinterpret_cast<const float4*>(p.out + row * LYNX_D) + lane);
  }
  auto store = [&]() {
    if (direct) return;
    reinterpret_cast<float4*>(p.out + row * LYNX_D)[lane] = acc;
    if (lane == 0) p.ws_lse[row] = lse;
  };
  if (!decide) {
    store();
    return;
  }
  // the largest |f - d| / (atol + rtol |f|) of the position (Section 4.3), at first per KV head
  float worst = 0.0f;
  const float fv[4] = {acc.x, acc.y, acc.z, acc.w}, dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) worst = fmaxf(worst, fabsf(fv[i] - dv[i]) / (p.atol + p.rtol * fabsf(fv[i])));
  const int m = __reduce_max_sync(0xFFFFFFFFu, __float_as_int(worst));   // worst >= 0: integer order = float order
  const uint32_t all = (uint32_t)(p.Hq * p.nq);
  uint32_t last = 0;
  if (lane == 0) {
    atomicMax(reinterpret_cast<int*>(p.ws_dev) + bh * kMaxQ + j, m);   // (zeroed by the attention kernel)
    __threadfence();
    last = atomicAdd(p.ws_seq_ctr + b, 1u) == all - 1;        // (likewise)
  }
  store();   // (behind the ticket: its fence has nothing else to wait for)
  // the last row of the sequence decides: a lane per position, the heads' deviations eight loads at a time
  if (__shfl_sync(0xFFFFFFFFu, last, 0)) {
    __threadfence();
    float dev = 0.0f;
    const float* hd = p.ws_dev + (size_t)b * p.Hkv * kMaxQ + lane;
    if (lane < p.nq) {
#pragma unroll 8
      for (int h = 0; h < p.Hkv; ++h) dev = fmaxf(dev, __ldcg(hd + (size_t)h * kMaxQ));
      p.dev[(size_t)b * p.nq_stride + lane] = dev;
    }
    const unsigned rej = __ballot_sync(0xFFFFFFFFu, lane < p.nq && dev > 1.0f);
    if (lane == 0) p.first_reject[b] = rej ? __ffs(rej) - 1 : p.nq;
  }
}

// CTAs of an attention launch with units of st tokens: one per SM, but min_units units each where a sequence has as many.
inline int attention_grid(const AttnParams& p, int st_tokens, int min_units) {
  const long long per = (long long)min_units * st_tokens;
  const long long grid = (long long)p.B * p.Hkv * (((long long)p.max_blocks * p.bt + per - 1) / per);
  const int full = sm_count();
  return grid < 1 ? 1 : grid > full ? full : (int)grid;
}
// The aligned cut of such a launch: each of the B * Hkv segments has CTAs of its own, and 85 % of the grid at least have one.
inline void plan_cut(AttnParams* p, int n_cta) {
  const long long segs = (long long)p->B * p->Hkv;
  p->per_seg = segs <= n_cta && n_cta / segs * segs * 100 >= 85ll * n_cta ? (int)(n_cta / segs) : 0;
  p->seg_div = p->per_seg > 1 ? block_div(p->per_seg) : BlockDiv{0, 0};
  p->hkv_div = p->Hkv > 1 ? block_div(p->Hkv) : BlockDiv{0, 0};
}

// (Nothing to join where every segment is one unit and nothing to decide; anchor calls with many heads join in the attention
// kernel.  bench.py counts kernels by this rule.)
inline lynx_status launch_combine(const AttnParams& p, int part_cols, int st_tokens, int min_units, cudaStream_t st) {
  const long long cap_units = ((long long)p.max_blocks * p.bt + st_tokens - 1) / st_tokens;
  if (p.inline_merge || (!p.draft && !p.combine_single && cap_units <= 1)) return LYNX_OK;
  // a warp per row where a head has no more than a few CTAs on average (one layer: 18; 16 layers of two sequences: 0.6)
  const unsigned rows = (unsigned)(p.B * p.nq * p.Hq);
  if (p.B * p.Hkv * 4 < sm_count())
    return launch_pdl(attn_combine_kernel<kWide>, rows, kCombineWarps * 32, 0, st, p, part_cols, sm_count(), 0);
  const unsigned fours = (rows + kCombineWarps - 1) / kCombineWarps;
  if (cap_units < kLongSegment)   // (no segment has more CTAs than units)
    return launch_pdl(attn_combine_kernel<kNarrow>, fours, kCombineWarps * 32, 0, st, p, part_cols, sm_count(), 0);
  const int n_long = (attention_grid(p, st_tokens, min_units) + kLongStep - 1) / kLongStep * p.ncols;
  return launch_pdl(attn_combine_kernel<kWithLong>, n_long + fours, kCombineWarps * 32, 0, st, p, part_cols, sm_count(), n_long);
}

#include "tc_common.cuh"
#include "attention_i8.cuh"
#include "attention_f16.cuh"
#include "attention_pipe.cuh"

// ------------------------------------------------------------------ host side
// Query positions per launch of a verification call: all of them up to kMaxQ positions and kMaxCols
// columns, else as many whole positions as fit both.
inline int verify_slice(int nq, int G) {
  if (nq <= kMaxQ && nq * G <= kMaxCols) return nq;
  const int by_cols = kMaxCols / G > 0 ? kMaxCols / G : 1;
  return by_cols < kMaxQ ? by_cols : kMaxQ;
}

struct Plan {
  int per;             // query positions per verification launch
  int ncols;           // columns of the widest launch
  WsLayout ws;
};

bool make_plan(const lynx_shape* s, int B, int nq, Plan* pl) {
  if (!s || s->head_dim != LYNX_D || s->num_kv_heads <= 0 || s->num_q_heads <= 0 ||
      s->num_q_heads % s->num_kv_heads != 0 || s->block_tokens <= 0 || s->block_tokens % 16 != 0 ||
      s->num_blocks <= 0 || s->max_blocks_per_seq <= 0 || B <= 0 || nq <= 0 || nq > kMaxWindow)
    return false;
  const int G = s->num_q_heads / s->num_kv_heads;
  if (G > 16) return false;
  // positions per launch of a verification call (anchor calls slice further, to 32 columns); the scratch is
  // sized for the widest launch
  pl->per = verify_slice(nq, G);
  const int ncols = pl->per * G;
  const int64_t cap = (int64_t)s->max_blocks_per_seq * s->block_tokens;
  if (cap >= (1ll << 31)) return false;
  if ((int64_t)s->num_blocks * s->num_kv_heads * s->block_tokens >= (1ll << 32)) return false;
  pl->ncols = ncols;
  // (the partial slots also serve anchor calls on the same workspace, which take up to 32 columns per launch)
  const int cols_anchor = nq * G <= 32 ? nq * G : (32 / G > 0 ? 32 / G : 1) * G;
  const int cols_max = ncols > cols_anchor ? ncols : cols_anchor;
  const int cols_pad = cols_max <= 8 ? 8 : cols_max <= 16 ? 16 : cols_max <= 32 ? 32 : 64;
  pl->ws = ws_layout(sm_count(), B, nq, s->num_q_heads, s->num_kv_heads, cols_pad);
  return true;
}

// Section 4.3's longest agreeing prefix over a window that was verified in slices: the smallest position
// whose deviation exceeds 1, or the number of positions.
__global__ void first_reject_kernel(const float* dev, int B, int nq, int32_t* __restrict__ first_reject) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  int fr = nq;
  for (int j = nq - 1; j >= 0; --j)
    if (dev[(size_t)b * nq + j] > 1.0f) fr = j;
  first_reject[b] = fr;
}

// Section 4.3's agreement test on outputs that are already in memory (a verification pass whose result was joined
// with a BF16 tail first): dev[b][j] = max over heads and dims of |f - d| / (atol + rtol |f|), the arithmetic of
// the decision fused into the verification kernels.  One CTA per (sequence, position).
__global__ void __launch_bounds__(256) deviation_kernel(const float4* out_full, const float4* draft,
                                                        int row_f4, float atol, float rtol, float* __restrict__ dev) {
  const float4* f = out_full + (size_t)blockIdx.x * row_f4;
  const float4* d = draft + (size_t)blockIdx.x * row_f4;
  float worst = 0.0f;
  for (int i = threadIdx.x; i < row_f4; i += 256) {
    const float4 a = f[i], b = ld_dep(d + i);
    worst = fmaxf(worst, fabsf(a.x - b.x) / (atol + rtol * fabsf(a.x)));
    worst = fmaxf(worst, fabsf(a.y - b.y) / (atol + rtol * fabsf(a.y)));
    worst = fmaxf(worst, fabsf(a.z - b.z) / (atol + rtol * fabsf(a.z)));
    worst = fmaxf(worst, fabsf(a.w - b.w) / (atol + rtol * fabsf(a.w)));
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) worst = fmaxf(worst, __shfl_xor_sync(0xFFFFFFFFu, worst, off));
  __shared__ float red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = worst;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) worst = fmaxf(worst, red[w]);
    dev[blockIdx.x] = worst;
  }
}

lynx_status run_attention(bool full, const lynx_shape* shape, const void* q, int B, int nq, int causal,
                          lynx_plane K, lynx_plane V, const int32_t* block_table,
                          const int32_t* seq_lens, float softmax_scale, const float* draft,
                          float atol, float rtol, float* out, int32_t* first_reject, float* dev,
                          void* workspace, size_t workspace_bytes, void* stream, bool fixed_scratch = false) {
  if (B == 0) return LYNX_OK;
  if (!shape) return LYNX_ERR_NULL;
  if (B < 0 || nq <= 0) return LYNX_ERR_SHAPE;
  if (shape->head_dim != LYNX_D || shape->block_tokens <= 0 || shape->block_tokens % 16 != 0)
    return LYNX_ERR_UNSUPPORTED;
  Plan pl;
  if (!make_plan(shape, B, nq, &pl)) return LYNX_ERR_UNSUPPORTED;
  if (!q || !K.anchor || !K.meta || !V.anchor || !V.meta || !block_table || !seq_lens || !out || !workspace)
    return LYNX_ERR_NULL;
  if (full && (!K.residual || !V.residual)) return LYNX_ERR_NULL;
  if (full && draft && (!first_reject || !dev)) return LYNX_ERR_NULL;
  if (!aligned16(q) || !aligned16(K.anchor) || !aligned16(V.anchor) || !aligned16(K.meta) ||
      !aligned16(V.meta) || !aligned16(workspace) || !aligned16(out) ||
      (full && (!aligned16(K.residual) || !aligned16(V.residual))))
    return LYNX_ERR_ALIGN;
  if (workspace_bytes < pl.ws.bytes) return LYNX_ERR_WORKSPACE;
  if (full && draft && !(atol > 0.0f && rtol >= 0.0f)) return LYNX_ERR_SHAPE;

  unsigned char* ws = static_cast<unsigned char*>(workspace);
  AttnParams p;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.ka = K.anchor; p.kr = K.residual; p.km = K.meta;
  p.va = V.anchor; p.vr = V.residual; p.vm = V.meta;
  p.block_table = block_table; p.seq_lens = seq_lens;
  p.out = out; p.draft = full ? draft : nullptr; p.first_reject = first_reject; p.dev = dev;
  p.combine_single = 0;
  // Who joins the partial results: attn_combine_kernel where few heads share the grid (and for verification, which needs it for
  // the decision), the last CTA of a head where a head has a CTA or two on average and its merge overlaps other heads' work (16
  // layers of two sequences of 131072 tokens, 8 columns: 1025 us, 1040 us by a kernel of its own; one layer of 4096 tokens, 4
  // columns: 13.2 us by the last CTA, 11.5 us by the kernel).
  p.inline_merge = !full && (long long)B * shape->num_kv_heads * 4 >= sm_count();
  p.draft_vec = p.draft && aligned16(p.draft);   // (a slice starts whole rows of 512 bytes further on)
  p.ws_flags = reinterpret_cast<uint32_t*>(ws);
  p.ws_tickets = reinterpret_cast<uint32_t*>(ws + pl.ws.off_tickets);
  p.ws_groups = reinterpret_cast<uint32_t*>(ws + pl.ws.off_groups);
  p.ws_seq_ctr = reinterpret_cast<uint32_t*>(ws + pl.ws.off_seq_ctr);
  p.ws_long = reinterpret_cast<uint32_t*>(ws + pl.ws.off_long);
  p.ws_dev = reinterpret_cast<float*>(ws + pl.ws.off_dev);
  p.ws_lse = reinterpret_cast<float*>(ws + pl.ws.off_lse);
  p.ws_part = reinterpret_cast<float*>(ws + pl.ws.off_part);
  p.atol = atol; p.rtol = rtol;
  const float sc = softmax_scale == 0.0f ? 0.08838834764831845f : softmax_scale;
  p.sm_log2 = sc * 1.4426950408889634f;
  p.B = B; p.nq = nq; p.nq_stride = nq; p.tail = nq; p.causal = causal ? 1 : 0;
  p.Hq = shape->num_q_heads; p.Hkv = shape->num_kv_heads; p.G = p.Hq / p.Hkv;
  p.bt = shape->block_tokens; p.num_blocks = shape->num_blocks; p.max_blocks = shape->max_blocks_per_seq;
  p.ncols = pl.ncols;
  p.bt_div = block_div(p.bt);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the fixed array keeps what the previous call left: the status word and the tickets must be zero
  if (fixed_scratch && cudaMemsetAsync(workspace, 0, pl.ws.end_kept, st) != cudaSuccess) return LYNX_ERR_CUDA;
  if (!full) {
    // Anchor attention: the integer tcgen05 kernels take up to 32 columns, 16 as a pipeline of stages, above in teams.  A call with more (33..64) is
    // run as slices of whole query positions, each a pass of its own over the planes, one after the
    // other on the stream (they share the workspace).
    const int per = nq * p.G <= 32 ? nq : (32 / p.G > 0 ? 32 / p.G : 1);
    for (int j0 = 0; j0 < nq; j0 += per) {
      AttnParams ps = p;
      ps.nq = nq - j0 < per ? nq - j0 : per;
      ps.ncols = ps.nq * p.G;
      ps.tail = nq - j0;
      ps.q = p.q + (size_t)j0 * p.Hq * LYNX_D;
      ps.out = p.out + (size_t)j0 * p.Hq * LYNX_D;
      ps.ws_lse = p.ws_lse + (size_t)j0 * p.Hq;
      const lynx_status rc = ps.ncols <= 4 ? launch_pipe<false, 4>(ps, st) : ps.ncols <= 8 ? launch_pipe<false, 8>(ps, st)
                           : ps.ncols <= 16 ? launch_pipe<false, 16>(ps, st) : launch_i8(ps, st);
      if (rc != LYNX_OK) return rc;
    }
    return LYNX_OK;
  }
  // verification: the integer kernels up to 16 columns, tcgen05 with FP16 operands (attention_f16.cuh) above (one layer of
  // 131072 tokens, 32 columns, the attention kernels alone: 83 us by the FP16 one, 174 us as two passes of the integer one at 16;
  // the whole call takes 91 us among other passes).
  // A window of more than kMaxQ positions or kMaxCols columns runs as slices of whole positions, each a pass
  // of its own over the planes that writes its outputs and deviations; the index of the first rejected
  // position over the whole window then follows from the deviations.
  for (int j0 = 0; j0 < nq; j0 += pl.per) {
    AttnParams ps = p;
    ps.nq = nq - j0 < pl.per ? nq - j0 : pl.per;
    ps.ncols = ps.nq * p.G;
    ps.tail = nq - j0;
    ps.q = p.q + (size_t)j0 * p.Hq * LYNX_D;
    ps.out = p.out + (size_t)j0 * p.Hq * LYNX_D;
    ps.ws_lse = p.ws_lse + (size_t)j0 * p.Hq;
    if (p.draft) { ps.draft = p.draft + (size_t)j0 * p.Hq * LYNX_D; ps.dev = p.dev + j0; }
    const lynx_status rc = ps.ncols <= 4 ? launch_pipe<true, 4>(ps, st) : ps.ncols <= 8 ? launch_pipe<true, 8>(ps, st)
                         : ps.ncols <= 16 ? launch_pipe<true, 16>(ps, st) : ps.ncols > 32 ? launch_f16<64, false>(ps, st)
                         : f16_int_pv(ps) ? launch_f16<32, true>(ps, st) : launch_f16<32, false>(ps, st);
    if (rc != LYNX_OK) return rc;
  }
  if (p.draft && pl.per < nq) {
    first_reject_kernel<<<(unsigned)((B + 127) / 128), 128, 0, st>>>(p.dev, B, nq, p.first_reject);
    return launch_status();
  }
  return LYNX_OK;
}

}  // namespace
}  // namespace lynx

extern "C" size_t lynx_workspace_bytes(const lynx_shape* shape, int32_t batch, int32_t n_cols_q) {
  lynx::Plan pl;
  if (!lynx::make_plan(shape, batch, n_cols_q, &pl)) return 0;
  return pl.ws.bytes;
}

extern "C" lynx_status lynx_verify_decision(const float* out_full, const float* draft_out, int32_t batch, int32_t k,
                                            int32_t num_q_heads, float atol, float rtol, int32_t* first_reject,
                                            float* dev, void* stream) {
  using namespace lynx;
  if (batch == 0) return LYNX_OK;
  if (batch < 0 || k <= 0 || k > kMaxWindow || num_q_heads <= 0 || (int64_t)batch * k >= (1ll << 31)) return LYNX_ERR_SHAPE;
  if (!out_full || !draft_out || !first_reject || !dev) return LYNX_ERR_NULL;
  if (!aligned16(out_full) || !aligned16(draft_out)) return LYNX_ERR_ALIGN;
  if (!(atol > 0.0f && rtol >= 0.0f)) return LYNX_ERR_SHAPE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  deviation_kernel<<<(unsigned)(batch * k), 256, 0, st>>>(reinterpret_cast<const float4*>(out_full),
                                                         reinterpret_cast<const float4*>(draft_out),
                                                         num_q_heads * (LYNX_D / 4), atol, rtol, dev);
  lynx_status rc = launch_status();
  if (rc != LYNX_OK) return rc;
  first_reject_kernel<<<(unsigned)((batch + 127) / 128), 128, 0, st>>>(dev, batch, k, first_reject);
  return launch_status();
}

extern "C" const float* lynx_workspace_lse(const lynx_shape* shape, int32_t batch, int32_t n_q, const void* workspace) {
  lynx::Plan pl;
  if (!workspace || !lynx::make_plan(shape, batch, n_q, &pl)) return nullptr;
  return reinterpret_cast<const float*>(static_cast<const unsigned char*>(workspace) + pl.ws.off_lse);
}

extern "C" lynx_status lynx_anchor_attention(const lynx_shape* shape, const void* q_bf16, int32_t batch,
                                             int32_t n_q, int32_t causal, lynx_plane K, lynx_plane V,
                                             const int32_t* block_table, const int32_t* seq_lens,
                                             float softmax_scale, float* out, void* workspace,
                                             size_t workspace_bytes, void* stream) {
  return lynx::run_attention(false, shape, q_bf16, batch, n_q, causal, K, V, block_table, seq_lens,
                             softmax_scale, nullptr, 0.f, 0.f, out, nullptr, nullptr, workspace,
                             workspace_bytes, stream);
}

extern "C" lynx_status lynx_merge_verify_attention(const lynx_shape* shape, const void* q_bf16,
                                                   int32_t batch, int32_t k, int32_t causal,
                                                   lynx_plane K, lynx_plane V,
                                                   const int32_t* block_table, const int32_t* seq_lens,
                                                   float softmax_scale, const float* draft_out,
                                                   float atol, float rtol, float* out_full,
                                                   int32_t* first_reject, float* dev, void* workspace,
                                                   size_t workspace_bytes, void* stream) {
  return lynx::run_attention(true, shape, q_bf16, batch, k, causal, K, V, block_table, seq_lens,
                             softmax_scale, draft_out, atol, rtol, out_full, first_reject, dev,
                             workspace, workspace_bytes, stream);
}

// ---------------------------------------------------------------------------------------------
// Anchor attention for callers that cannot hand over a workspace (no paper counterpart).
//
// The split-K partials, tickets and status word live in one fixed array in device memory that
// is part of the loaded library image: nothing is allocated, by this call or by any routine it
// uses.  Host code cannot use the array's name as an address (on the host the name is only a
// handle for the runtime), so the device address is looked up once per device with
// cudaGetSymbolAddress, while that device is current, and the kernels are given that address.
namespace lynx {
namespace {

constexpr size_t kStaticScratchBytes = 8u << 20;  // 8 MiB held by every GPU that loads the library
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

lynx_status static_scratch_address(void** out) {
  static void* resolved[64] = {nullptr};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LYNX_ERR_CUDA;
  if (resolved[dev] == nullptr) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || ptr == nullptr) return LYNX_ERR_CUDA;
    resolved[dev] = ptr;
  }
  *out = resolved[dev];
  return LYNX_OK;
}

}  // namespace
}  // namespace lynx

extern "C" lynx_status lynx_anchor_attention_static(const lynx_shape* shape, const void* q_bf16,
                                                    int32_t batch, int32_t n_q, int32_t causal,
                                                    lynx_plane K, lynx_plane V,
                                                    const int32_t* block_table, const int32_t* seq_lens,
                                                    float softmax_scale, float* out, void* stream) {
  using namespace lynx;
  if (batch == 0) return LYNX_OK;
  if (!shape) return LYNX_ERR_NULL;
  if (batch < 0 || n_q <= 0) return LYNX_ERR_SHAPE;
  Plan pl;
  if (!make_plan(shape, batch, n_q, &pl)) return LYNX_ERR_UNSUPPORTED;
  if (pl.ws.bytes > kStaticScratchBytes) return LYNX_ERR_WORKSPACE;  // problem too large for the fixed array
  void* scratch = nullptr;
  const lynx_status st = static_scratch_address(&scratch);
  if (st != LYNX_OK) return st;
  // (validated there before anything is enqueued; the words that must start at zero are cleared on
  // `stream` only once the call is known to launch)
  return run_attention(false, shape, q_bf16, batch, n_q, causal, K, V, block_table, seq_lens,
                       softmax_scale, nullptr, 0.f, 0.f, out, nullptr, nullptr, scratch,
                       pl.ws.bytes, stream, true);
}
