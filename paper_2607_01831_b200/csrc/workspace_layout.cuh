// Where the parts of an attention call's workspace lie.  Plain C++, so that it can be checked on the host.
#pragma once
#include <cstddef>
#include <cstdint>

namespace lynx {

constexpr int kWsHeaderBytes = 256;      // word 0: status flags set by kernels
constexpr int kWsMaxQ = 16;              // query positions per launch
constexpr int kWsPartStride = 132;       // floats per (CTA, column) partial: O[128], m, l, segment word, pad
// The scratch has room for this many CTAs per SM, although every kernel runs one: lynx_workspace_bytes and the limit of
// lynx_anchor_attention_static are figures that callers hold (8 bytes to 33 KB per CTA and column count).
constexpr int kWsMaxCtasPerSm = 4;

// What outlives a call -- the status word and the tickets, which every call finds and leaves at zero -- lies in front, at places
// that follow from the number of SMs alone: a workspace serves calls of any batch, heads and positions that it is large enough
// for, and the results of one never lie on the tickets of another.  All that follows is written by a call before it is read.
struct WsLayout {
  size_t off_tickets;   // one per SM: of the segment shared by several CTAs whose first is this one (no CTA is first of two)
  size_t off_groups;    // two per SM: of groups of such CTAs (see slot_group)
  size_t end_kept;
  size_t off_long;      // one per eight SMs at most: what attn_combine_kernel is told of long segments
  size_t off_seq_ctr;   // [B] counts of a sequence's finished rows
  size_t off_dev;       // [B * Hkv][kWsMaxQ] deviations
  size_t off_lse;       // [B][nq][Hq] log-sum-exps
  size_t off_part;      // [B * Hkv + CTAs][cols_pad][kWsPartStride] partial results
  size_t bytes;
};
inline WsLayout ws_layout(int sms, int B, int nq, int Hq, int Hkv, int cols_pad) {
  const auto up = [](size_t x, size_t n) { return (x + n - 1) / n * n; };
  WsLayout w;
  w.off_tickets = kWsHeaderBytes;
  w.off_groups = w.off_tickets + (size_t)sms * 4;
  w.end_kept = w.off_groups + (size_t)2 * sms * 4;
  w.off_long = up(w.end_kept, 128);
  w.off_seq_ctr = up(w.off_long + (size_t)(sms / 8 + 1) * 4, 128);
  // (the room between counts and deviations is not used; the size is a figure that callers hold)
  w.off_dev = up(kWsHeaderBytes + (size_t)2 * sms * kWsMaxCtasPerSm * 4 + (size_t)B * 4 + (size_t)B * Hkv * 4, 256);
  w.off_lse = up(w.off_dev + (size_t)B * Hkv * kWsMaxQ * 4, 256);
  w.off_part = up(w.off_lse + (size_t)B * nq * Hq * 4, 256);
  w.bytes = up(w.off_part + ((size_t)B * Hkv + (size_t)sms * kWsMaxCtasPerSm) * cols_pad * kWsPartStride * 4, 256);
  return w;
}

}  // namespace lynx
