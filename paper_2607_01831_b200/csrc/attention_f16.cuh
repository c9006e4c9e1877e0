// Merge-verify attention for 17..64 columns on the fifth-generation tensor cores: scores as FP16 products, values as FP16 or integer
// ones.  Included by attention.cu inside its namespace.
//
// A unit is 128 tokens.  Both contractions take the 8-bit codes centred, c - 128, which FP16 represents exactly:
//   S^T[128 tokens x NC]      = (codes(K) - 128) . Q^T       A = K in tensor memory (a thread owns a token = a lane),
//                                                            B = Q, FP16 after a power-of-two scale (exact for BF16
//                                                                entries down to 2^-32 of the largest); up to 32 columns
//                                                                in two parts side by side in N (f16_split_q)
//   O^T[128 dims x 2 x 32]   += (codes(V) - 128)^T . [h | r] A = V tile (MN-major), B = the weights as two FP16 terms,
//                                                                w = h + r (22 bits), side by side in N
// or, up to 32 columns where a CTA has many units (f16_int_pv), with kind::i8:
//   O^T[128 dims x 4 x 32]   += (codes(V) - 128)^T . Wd      A = V tile (s8), B = the four bytes of weights scaled to u32
// Centring costs one packed addition per two codes and is what keeps FP32 sufficient: the zero points, 128 steps below
// the centre of a row, would otherwise be added and taken off again around results a hundred times smaller.
// x = s log2(e) + log2(scale_v), w = 2^(x - ref[c]); ref[c] is set so that the largest weight of a column's first unit is
// 2^8 (integers: 1, scaled to 2^26) and raised (accumulators drained or rescaled, rare) before a weight would leave FP16 or u32.  The
// tensor core's FP32 accumulation truncates (0.46 ulp of the running sum per product).  Scores: the high part of a query is a
// multiple of 2^-10 of the largest entry, so that its products with the codes sum up exactly, and the truncation acts on the low
// part, a thousand times smaller.  Values: every kDrainUnits units the accumulators move into an FP32 copy; the integer sums are exact.
//
// Error against 64 bits (2-norm; 34 cases of 17..32 and 26 of 33..64 columns, 64 to 131072 tokens, log-normal, heavy-tailed
// and outlier values).  17..32 columns, against the exact integer products of attention_i8.cuh in two passes: 0.29 times on
// the geometric mean, at most 0.97 times, largest 1.4e-6 (7.5e-6); log-sum-exps 0.54 times, largest 9e-6 (4.4e-5).  With
// whole queries and a drain per 8 units it was 0.42 times on the mean but up to 2.0 times on heavy-tailed keys and long
// contexts.  33..64 columns, against the uncentred kernel before it: 0.09 times, largest 1.2e-5 (3.4e-4).  Values on integers against
// values in FP16, 32 columns, means of six draws: 131072 tokens log-normal 3.6e-7 (6.6e-7), 2 of 30000 heavy-tailed 7.1e-7 (8.6e-7).
//
// Warp roles, one CTA per SM; every hand-off is an mbarrier with a bounded wait, nothing waits on another CTA:
//   warps 0-7    two softmax warpgroups of 32 columns each: scores -> weights -> P tile
//   warps 8-11   K codes into tensor memory, and a piece's queries into the Q tile
//   warps 12-15  V codes into the V tile
//   warps 16-19  producers (tensor-map copies of 16-token sub-blocks): two warps for the K ring, one for the V ring
//   warp 20      issues every tcgen05.mma
//   warps 21, 22 the per-token scalars of the scores and weights at 32 columns (the rest completes the warpgroup, for the
//                register split)
// With 64 columns the groups take one half of the columns each of every unit; with 32 they alternate over the units
// (separate accumulators, merged at the end of a piece), which spares the per-token work of a second group.
// Why specialised warps here and teams in attention_i8.cuh: at these widths the accumulators of teams do not fit tensor
// memory (integer digit planes: 224 columns per team at 32), while the expansions and the softmax of a unit are long
// enough to overlap as pipeline stages with double-buffered S, K and V.
//
// What bounds it: instruction issue and the instruction caches.  A unit takes 4800 warp instructions at 32 columns with integer
// values (6200 with FP16 ones) and 7200 at 64, at 2.3 and 2.6 per cycle; heavy FMA pipe 34 and 46 %, ALU 35 and 39 %, tensor
// pipe 25 and 27 %.  With 64 columns the softmax groups are never idle, with 32 (FP16) they wait a fifth of the time.  What mattered on
// the way: no register spills in the softmax loop (little L1 is left beside 227 KB of shared memory: 400 bytes of spills
// per thread cost a factor of two; hence scores in the 16-lane layout, where a thread sums 8 columns over 4 tokens instead
// of 32 columns over one), rolled loops in the expansions and the producers (118 -> 98 us at 32 columns; unrolled copies of
// a producer: +5 %), products issued by an elected lane (93 -> 30 cycles each), expansions without a register rotation and drains in
// packed additions without selects, behind the scores instead of in front of them (32 columns 88.4 -> 83.0 us).  Twice the softmax warps with
// half of a unit's tokens each and 80 registers: 64 columns +15 %, 32 +4 %.  One layer of 131072 tokens: 174 us as two passes
// of the 16-column integer kernel -> 83 us (32 columns); two sequences, 64 columns: 293 us by the previous kernel (M = columns, codes
// not centred) -> 207 us; the kernel alone, back to back, before the power cap sets in (the calls among other passes: 91 and 227 us).
// Since then both barriers of a stage are probed at once (64 columns 200 -> 197 us), and values go through integer products at 32
// columns: half of the work on V codes, no drains, two instructions a weight instead of five (80 -> 72 us).  At 64 columns the
// conversions to u32, which share their unit with the exponentials, cost what that saves (200 -> 215 us).  Tried and left: K and V codes
// by the same warpgroup, units in turn (72 -> 73), in that order or K a unit ahead (75), a look-ahead by more than one unit (75).

template <int NC, bool INT>
struct F16Cfg {
  static_assert(NC == 32 || (NC == 64 && !INT), "padded column counts");
  static constexpr bool kFull = true, kMetaRing = false;
  static constexpr bool kSplit = NC == 64;          // both groups score every unit (else they alternate)
  static constexpr int kST = 128, kCG = 32, kNG = kCG / 8;
  static constexpr int kPartCols = NC;
  static constexpr int kStageBytes = kST * 128;     // Anchor and Residual of one tensor: [2][128 tokens][64 B]
  static constexpr bool kIntPV = INT;               // P.V on integers: codes less 128 as s8, weights as u32
  static constexpr int kVTile = kIntPV ? 16384 : 32768;   // [128 tokens][128 B], or [2 dim blocks][128 tokens][128 B]
  static constexpr int kPTile = 16384;              // [128 tokens][32 columns x 4 bytes], or [128 tokens][32 h | 32 r]
  static constexpr int kNPV = kIntPV ? 128 : 64;    // N of a group's P.V
  static constexpr int kQP = NC == 32 ? 2 : 1;      // parts of the queries (see f16_split_q)
  static constexpr int kSCols = kQP * NC;           // columns of Q.K^T: the queries' high parts, then the low ones
  static constexpr int kQTile = kSCols * 256;       // [2 dim blocks][kSCols][128 B]
  static constexpr int kRingK = 3, kRingV = 3;
  static constexpr int kOFBytes = kIntPV ? 2 * kCG * 512 : 0;   // FP32 copy of O where tensor memory has no room for it: [group][column][128]
  static constexpr int kOffV = 0, kOffP = 2 * kVTile, kOffOF = kOffP + 2 * kPTile, kOffQ = kOffOF + kOFBytes, kOffRK = kOffQ + kQTile,
                       kOffRV = kOffRK + kRingK * kStageBytes, kOffScal = kOffRV + kRingV * kStageBytes;
  // floats: qs[2][NC], limits[2][NC], exponents[2] (+ 2); per group: ref[32], fac[32], red[4][64], lz[64]
  static constexpr int kGrpScal = 2 * 32 + 256 + 64;
  static constexpr int kOffGrp = kOffScal + (4 * NC + 4) * 4;
  // (Scalars stored as the packed pairs that the softmax takes, in two slots, spare it a tenth of its instructions and cost more in
  // shared memory: 64 columns 197 -> 205 us.)
  static constexpr int kSlots = 4;                                  // units whose per-token scalars are kept: [4][128] float4, [4][128] float
  static constexpr int kOffTok = kOffGrp + 2 * kGrpScal * 4;
  static constexpr int kOffBlk = kOffTok + 4 * 128 * 20;        // [4 producer warps][4 sub-blocks][kI8PieceUnits]
  static constexpr int kOffItems = kOffBlk + 16 * kI8PieceUnits * 4;
  static constexpr int kOffBars = kOffItems + 2 * 32;
  static constexpr int kOffMisc = kOffBars + 44 * 8;
  static constexpr int kSmem = kOffMisc + 256 + 1024;               // + alignment slack
  static_assert(kSmem <= 227 * 1024, "shared memory");
  static_assert(kOffScal % 16 == 0 && kOffGrp % 16 == 0 && kOffBars % 8 == 0, "alignment");
  static constexpr int kTmS = 0, kTmK = 2 * kSCols, kTmO = kTmK + 128, kTmOF = kTmO + 2 * kNPV;   // [2][kSCols], [2][64], [2][kNPV], [2][32]
  static_assert(kTmOF + (kIntPV ? 0 : 64) <= 512, "tensor memory");
  static constexpr int kThreads = 768, kDoneThreads = 256 + 128 + 32;   // softmax warpgroups, producers, products
  // units between drains: each adds 8 truncating products to a sum.  32 columns, one layer of 131072 tokens: a drain per 8
  // units has a largest error of 3.4e-6, per 4 units 2.2e-6, per 2 units 1.4e-6, by when it is below the integer kernel's in
  // every case (4 % of the time between 8 and 2 when it was measured); 64 columns: 3 % of the time for a drain per 16 units, 6 % per 8
  static constexpr int kDrainUnits = kIntPV ? 256 : NC == 64 ? 16 : 2;
  // log2 of the largest weight of a column's first unit, of a weight that raises the references, and of one whose column's is raised
  // with it.  On integers weights are formed relative to that and scaled by kScale afterwards (up to 2^31.5): an exponent of 26 would
  // carry four times the rounding.
  // Integers as a weight of 2^-27 of the largest and less would vanish, and where one token outweighs the others they are what the rest
  // of the context consists of.  So they are rounded up as often as their fraction says (see weight_offset), which leaves the sums
  // without a bias.  Error against 64 bits, 1e-6 of the 2-norm, 32 columns, a token over the rest by 2^20 / 2^26.6 / 2^30: one
  // sequence of 131072 tokens, weights as two FP16 terms 3.1 / 2.7 / 0.46, as integers to nearest at 2^25 1.1 / 58 / 6.6, as here 0.58 / 1.4 / 0.22;
  // 16 of 65536 3.0 / 11.0 / 2.8, 3.6 / 500 / 58, 1.8 / 11.3 / 1.7 (11: of the 32-bit sums of the weights, in all three).  At 2^25 with
  // fractions 1.06 / 1.5 / 0.29 and 3.4 / 11.4 / 1.9; at 2^27 the references are raised so often that log-normal values cost 5 % more.
  // Raising with them only the columns that are 2 over theirs spares 1 % with outliers and 4 % where pieces are short.
  static constexpr float kTop = kIntPV ? 0.0f : 8.0f, kRaise = kIntPV ? 5.5f : 15.0f, kRaiseToo = kIntPV ? 2.0f : 15.0f;
  static constexpr float kScale = 0x1p26f;
  // who computes the per-token scalars: with 64 columns the K warps have the time (261 -> 256 us), with 32 they are the
  // slower stage and two spare warps do it (96.1 us, 97.4 us in the K warps)
  static constexpr bool kMetaK = kSplit;
  // registers per thread after the split (launched with 80 each): 256 * 128 + 256 * 64 + 128 * 56 + 128 * 40 = 768 * 80
  static constexpr int kRegSoft = 128, kRegExp = 64, kRegProd = 56, kRegMma = 40;
};
template <int N>
__device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

// The bounded wait of mbar_wait without a call: ptxas cannot split the registers of a kernel that has calls.
template <class Probe>
__device__ __forceinline__ bool wait_in(Probe probe, volatile int* abort_word) {
  return bounded_wait(probe, [] { return globaltimer_ns(); }, abort_word);
}
__device__ __forceinline__ bool mbar_wait_in(uint32_t bar, uint32_t parity, volatile int* abort_word) {
  if (mbar_test(bar, parity)) return true;
  return wait_in([=] { return mbar_try_wait(bar, parity); }, abort_word);
}

// Two waits whose first probes are under way at the same time.
__device__ __forceinline__ void mbar_wait2_in(uint32_t bar0, uint32_t parity0, uint32_t bar1, uint32_t parity1, volatile int* abort_word) {
  const bool a = mbar_test(bar0, parity0), b = mbar_test(bar1, parity1);
  if (a && b) return;
  mbar_wait_in(bar0, parity0, abort_word);
  mbar_wait_in(bar1, parity1, abort_word);
}

// position -> element within a group of 8: {0,4,2,6,1,5,3,7} (what the nibble expansion yields), its own inverse
__host__ __device__ constexpr int f16_perm(int pos) { return ((pos & 1) << 2) | (pos & 2) | ((pos >> 2) & 1); }

// Four centred FP16 pairs from a word of eight Anchor and a word of eight Residual nibbles: 0x64cc is 1024 + code.
__device__ __forceinline__ uint32_t f16_centre(uint32_t x) {
  uint32_t d;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(x), "r"(0xE480E480u));   // - 1152
  return d;
}
__device__ __forceinline__ void f16_codes(uint32_t xa, uint32_t xr, uint32_t* o) {
  uint32_t ev, od;
  merge_codes(xa, xr, ev, od);
  o[0] = f16_centre((ev & 0x00FF00FFu) | 0x64006400u);
  o[1] = f16_centre(prmt(ev, 0x64646464u, 0x4341));
  o[2] = f16_centre((od & 0x00FF00FFu) | 0x64006400u);
  o[3] = f16_centre(prmt(od, 0x64646464u, 0x4341));
}
// A scaled query entry, |f| < 2^15, in two parts: f becomes a multiple of 32, lo what is left, |lo| <= 16.  The sum of 128
// products of codes (|c - 128| <= 128) with multiples of 32 up to 2^15 stays below 2^24 times 32: exact in FP32 in any order.
// Both parts are exact in FP16: an entry has eight bits, and those above 2^12 are multiples of 32 themselves.  (Against whole
// queries, 32 columns: 92.2 -> 93.5 us for one layer of 131072 tokens.)
__device__ __forceinline__ void f16_split_q(float& f, float& lo) {
  constexpr float kRound = 402653184.0f;   // 1.5 * 2^23 * 32
  const float hi = (f + kRound) - kRound;
  lo = f - hi;
  f = hi;
}
__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// K codes of a token (thread r of 128 = TMEM lane r) into 64 columns of tensor memory.
__device__ __forceinline__ void f16_expand_k(uint32_t raw, int r, uint32_t tm_k) {
  // (a rolled loop: five roles share an instruction cache of some 12 KB per scheduler.  No loads ahead: these warps have time to
  // wait for shared memory, and moving the next chunk into place costs eight instructions a step)
#pragma unroll 1
  for (int h = 0; h < 4; ++h) {
    const uint32_t row = raw + k_chunk((uint32_t)r, (uint32_t)h);
    const uint4 xa = lds128(row), xr = lds128(row + 8192u);
    uint32_t regs[16];
    f16_codes(xa.x, xr.x, regs);
    f16_codes(xa.y, xr.y, regs + 4);
    f16_codes(xa.z, xr.z, regs + 8);
    f16_codes(xa.w, xr.w, regs + 12);
    TmemRegs<16>::st(tm_k + h * 16, regs);
  }
}
// V codes of a unit into the V tile by 128 threads: thread i takes the 16-byte chunk i & 3 (32 elements) of rows i >> 2 + 32 j.
// Half of the threads take the two 8-byte halves of a chunk in the other order: the four threads of a row then store to
// four chunk positions per instruction, and rows r and r + 2, which share their banks in the raw stage, read different halves.
__device__ __forceinline__ void f16_expand_v(uint32_t raw, uint32_t tile, int i) {
  const int cc = i & 3, row0 = i >> 2;
  const uint32_t sw = (uint32_t)(((cc >> 1) ^ (row0 >> 1)) & 1) * 2u;
  const uint32_t base = tile + (uint32_t)(cc >> 1) * 16384u + (uint32_t)row0 * 128u;
  const uint32_t swz = (uint32_t)(((cc & 1) * 4) ^ (row0 & 7) ^ (int)sw) * 16u;
  uint32_t a = raw + (uint32_t)(row0 * 64 + cc * 16), dst = base + swz;
#pragma unroll 1
  for (int j = 0; j < 4; ++j, a += 2048u, dst += 4096u) {   // (rolled: see f16_expand_k)
    const uint2 xa[2] = {lds64(a + sw * 4u), lds64(a + (sw ^ 2u) * 4u)}, xr[2] = {lds64(a + 8192u + sw * 4u), lds64(a + 8192u + (sw ^ 2u) * 4u)};
    const uint32_t wa[4] = {xa[0].x, xa[0].y, xa[1].x, xa[1].y}, wr[4] = {xr[0].x, xr[0].y, xr[1].x, xr[1].y};
#pragma unroll
    for (int k = 0; k < 4; ++k) {   // register k holds word k ^ sw of the chunk
      uint32_t o[4];
      f16_codes(wa[k], wr[k], o);
      sts128(dst ^ (uint32_t)(k * 16), o[0], o[1], o[2], o[3]);
    }
  }
}

// V codes of a unit, less 128, as bytes into the V tile by four warps: i8_expand with the top bit of every code flipped (and rolled:
// see f16_expand_k).
__device__ __forceinline__ void f16_expand_v8(uint32_t raw, uint32_t tile, int w4, int lane) {
  const int row8 = lane >> 2, j = lane & 3;
  uint32_t a = raw + (uint32_t)((w4 * 8 + row8) * 64 + j * 16), dst = tile + (uint32_t)(w4 * 8 + row8) * 128u;
  const uint32_t c0 = (uint32_t)((2 * j) ^ row8) << 4, c1 = (uint32_t)((2 * j + 1) ^ row8) << 4;
#pragma unroll 1
  for (int s = 0; s < 4; ++s, a += 2048u, dst += 4096u) {
    const uint4 xa = lds128(a), xr = lds128(a + 8192u);
    const uint32_t wa[4] = {xa.x, xa.y, xa.z, xa.w}, wr[4] = {xr.x, xr.y, xr.z, xr.w};
    uint32_t ev[4], od[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) merge_codes(wa[k] ^ 0x88888888u, wr[k], ev[k], od[k]);
    sts128(dst + c0, ev[0], ev[1], ev[2], ev[3]);
    sts128(dst + c1, od[0], od[1], od[2], od[3]);
  }
}
// Column of a group whose weights' bytes are word k of 16-byte chunk c of a row of the P tile (stmatrix deals a thread's columns
// 8 j + 2 i and 8 j + 2 i + 1 to chunks j and 4 + j).
__host__ __device__ constexpr int f16_col(int c, int k) { return 8 * (c & 3) + 2 * k + (c >> 2); }
// What is added to a weight on its way to the nearest integer: -1/2 to 1/2, spread evenly over any run of tokens (the multiples of the
// golden section, modulo one), so that of many like weights the share that their fraction says is rounded up.
__device__ __forceinline__ float weight_offset(int tok) {
  return __uint_as_float(0x3F800000u | ((uint32_t)tok * 2654435769u >> 9)) - 1.5f;
}
// The sum of a column from its four byte planes.
__device__ __forceinline__ float f16_planes(const uint32_t* a) {
  return fmaf(fmaf(fmaf((float)(int)a[3], 256.0f, (float)(int)a[2]), 256.0f, (float)(int)a[1]), 256.0f, (float)(int)a[0]);
}

// A producer warp: derives the CTA's range like the others.  The V warp publishes the pieces and does what is left to do for a
// sequence: its copies are the last to be waited for.
// Warps 0, 1 copy one half of the K sub-blocks each, warp 2 the V sub-blocks, warp 3 the metadata of both (where kMetaRing).  full0,
// empty0, stages: of the warp's own ring.
// What bounds a producer is the latency of its instructions in a row: some 55 cycles per copy, 300 per unit.  Hence gathers of four
// sub-blocks per copy for V and the metadata (the 128-byte swizzle of K does not go with them), and always all eight sub-blocks of a
// unit, whether or not the sequence has them.
constexpr int kPublisher = 2;
template <class C, class MAPS>
__device__ __forceinline__ void plane_producer(const AttnParams& p, const SkRange& rng, const SeqLens& sl, int pw, int lane, uint32_t sbase, uint32_t full0,
                                               uint32_t empty0, int stages, uint32_t qfull0, uint32_t qempty0, uint32_t* blk_s, Item* items,
                                               volatile int* abort_word, const MAPS* maps, int bar_done) {
  constexpr int ST = C::kST;
  const int lg = pw < 2 ? 2 : 3;                 // log2 of the sub-blocks of a unit that are this warp's
  const int sub0 = pw == 1 ? 4 : 0;
  uint32_t* my_blk = blk_s + (pw < 2 ? 4 * pw : 8 * (pw - 1)) * kI8PieceUnits;
  int b = rng.b_lo, len = sl.of(b), U = (len + ST - 1) / ST;
  int hkv = rng.hkv, u = rng.u;
  if (hkv < 0) {
    hkv = (int)sk_div(rng.off_lo, U);
    u = (int)(rng.off_lo - (long long)hkv * U);
  }
  const int n_units = (int)(rng.hi - rng.lo);
  int remaining = n_units, slot = 0, ic = 0;
  uint32_t phase = 1;   // (a fresh barrier passes a wait for the phase before its first)
  while (remaining > 0) {
    const int n = min(remaining, U - u);
    if (pw == kPublisher) {
      const int qi = ic & 1;
      if (ic >= 2) mbar_wait_in(qempty0 + qi * 8, ((ic >> 1) - 1) & 1, abort_word + kItemAbort);
      const long long seg0 = rng.lo + (n_units - remaining) - u;  // first unit of this segment
      if (lane == 0) {
        Item it;
        it.b = b; it.hkv = hkv; it.len = len;
        it.first_cta = (int)sk_div(seg0, rng.q);
        it.n_contrib = (int)sk_div(seg0 + U - 1, rng.q) - it.first_cta + 1;
        it.pad0 = n; it.pad1 = u; it.pad2 = 0;
        items[qi] = it;
        if (u == 0) *seg_word(p, (size_t)b * p.Hkv + hkv, C::kPartCols) = (uint32_t)it.first_cta << 16 | (uint32_t)it.n_contrib;
        mbar_arrive(qfull0 + qi * 8);
      }
      __syncwarp();
      if (C::kFull && u == 0 && lane < kMaxQ) p.ws_dev[((size_t)b * p.Hkv + hkv) * kMaxQ + lane] = 0.0f;   // (see attn_combine_kernel)
    }
    for (int c0 = 0; c0 < n; c0 += kI8PieceUnits) {
      const int cn = min(kI8PieceUnits, n - c0);
      for (int i = lane; i < cn << lg; i += 32) {
        const int t0 = (u + c0 + (i >> lg)) * ST + (sub0 + (i & ((1 << lg) - 1))) * 16;
        uint32_t row = 0;  // sub-block beyond the end of the sequence: any that exists, its levels meet weights of zero
        if (t0 < len) {
          const int bi = block_of(p, t0);
          int blk = ld_dep(p.block_table + (size_t)b * p.max_blocks + bi);
          if (blk < 0 || blk >= p.num_blocks) {
            atomicOr(p.ws_flags, kFlagBadBlock);
            blk = blk < 0 ? 0 : p.num_blocks - 1;
          }
          row = (uint32_t)(((size_t)blk * p.Hkv + hkv) * p.bt + (t0 - bi * p.bt));
        }
        my_blk[i] = map_row(row, pw < 2);
      }
      __syncwarp();
      for (int k = 0; k < cn; ++k) {
        mbar_wait_in(empty0 + slot * 8, phase, abort_word);
        const uint4* rows = reinterpret_cast<const uint4*>(my_blk) + (k << (lg - 2));
        // (one elected lane: with a copy per lane the compiler walks through the lanes, operands to the uniform datapath and back)
        if (tc_elect()) {
          const uint32_t bar = full0 + slot * 8;
          const uint4 r0 = rows[0];
          if (pw < 2) {
            const uint32_t dst = sbase + C::kOffRK + (uint32_t)(slot * C::kStageBytes + sub0 * 1024), r[4] = {r0.x, r0.y, r0.z, r0.w};
            mbar_expect_tx(bar, C::kFull ? 8192u : 4096u);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              tma_box(dst + i * 1024, &maps->m[0], r[i], bar);
              if (C::kFull) tma_box(dst + 8192 + i * 1024, &maps->m[2], r[i], bar);
            }
          } else {
            const uint4 r1 = rows[1];
            if (pw == 2) {
              const uint32_t dst = sbase + C::kOffRV + (uint32_t)(slot * C::kStageBytes);
              mbar_expect_tx(bar, C::kFull ? 16384u : 8192u);
              tma_gather4(dst, &maps->m[1], r0, bar);
              tma_gather4(dst + 4096, &maps->m[1], r1, bar);
              if (C::kFull) {
                tma_gather4(dst + 8192, &maps->m[3], r0, bar);
                tma_gather4(dst + 12288, &maps->m[3], r1, bar);
              }
            } else if constexpr (C::kMetaRing) {
              const uint32_t dst = sbase + C::kOffMeta + (uint32_t)(slot * 2048);
              mbar_expect_tx(bar, 2048u);
              tma_gather4(dst, &maps->meta[0], r0, bar);
              tma_gather4(dst + 512, &maps->meta[0], r1, bar);
              tma_gather4(dst + 1024, &maps->meta[1], r0, bar);
              tma_gather4(dst + 1536, &maps->meta[1], r1, bar);
            }
          }
        }
        __syncwarp();
        if (++slot == stages) { slot = 0; phase ^= 1; }
      }
      __syncwarp();  // my_blk is rewritten by the next round
    }
    remaining -= n;
    u += n;
    ++ic;
    if (u == U && remaining > 0) {
      u = 0;
      if (++hkv == p.Hkv) {
        hkv = 0;
        do {
          ++b;
          len = b < p.B ? sl.of(b) : 0;
          U = (len + ST - 1) / ST;
        } while (b < p.B && U == 0);
        if (b >= p.B) break;  // cannot happen: the range ends inside the list
      }
    }
  }
  __syncwarp();
  bar_arrive(bar_done, C::kDoneThreads);
}

// The per-token scalars of a unit, for N tokens (32 apart) of a thread: scale and offset of the scores, log2 of the value
// scale, its reciprocal and the zero point in units of it.  Metadata is read two steps ahead: the block id of the unit after
// next, the (scale, zero) pairs of the next unit.
template <class C, int N>
struct F16Meta {
  float4* tok4;
  float* tok1;
  const int32_t* table;
  int i0, ih, len, n_piece, u0;
  int blk_n[N];
  float2 km[N], vm[N];
  __device__ __forceinline__ void init(const AttnParams& p, unsigned char* smem, int first) {
    i0 = first;
    tok4 = reinterpret_cast<float4*>(smem + C::kOffTok) + i0;
    tok1 = reinterpret_cast<float*>(smem + C::kOffTok + 4 * 128 * 16) + i0;
  }
  __device__ __forceinline__ int blk_of(const AttnParams& p, int uu, int i) const {
    const int t = (u0 + uu) * C::kST + i0 + 32 * i;
    if (uu >= n_piece || t >= len) return 0;
    return ld_dep(table + block_of(p, t));
  }
  __device__ __forceinline__ void meta_of(const AttnParams& p, int uu, int i, int blk) {
    const int t = (u0 + uu) * C::kST + i0 + 32 * i;
    km[i] = make_float2(0.f, 0.f); vm[i] = km[i];
    if (uu >= n_piece || t >= len) return;
    const int in_blk = t - block_of(p, t) * p.bt;
    blk = min(max(blk, 0), p.num_blocks - 1);     // (out-of-range ids are reported by the producer)
    const uint32_t row = (uint32_t)(((size_t)blk * p.Hkv + ih) * p.bt + in_blk);
    km[i] = ld_dep(reinterpret_cast<const float2*>(p.km) + row);
    vm[i] = ld_dep(reinterpret_cast<const float2*>(p.vm) + row);
  }
  __device__ __forceinline__ void piece(const AttnParams& p, const Item& it) {
    ih = it.hkv; len = it.len; n_piece = it.pad0; u0 = it.pad1;
    table = p.block_table + (size_t)it.b * p.max_blocks;
    int blk0[N];
#pragma unroll
    for (int i = 0; i < N; ++i) { blk0[i] = blk_of(p, 0, i); blk_n[i] = blk_of(p, 1, i); }
#pragma unroll
    for (int i = 0; i < N; ++i) meta_of(p, 0, i, blk0[i]);
  }
  __device__ __forceinline__ void unit(const AttnParams& p, int u, int gs, float ca) const {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const bool valid = (u0 + u) * C::kST + i0 + 32 * i < len;
      if (C::kSplit && valid && !(vm[i].x < 16.0f)) atomicOr(p.ws_flags, kFlagRange);   // beyond the stated range of this width
      const float sve = fmaxf(vm[i].x, 9.094947e-13f);   // floor 2^-40
      const float ia = valid ? rcp_approx(sve) : 0.0f;
      const int at = gs % C::kSlots * 128 + 32 * i;
      tok4[at] = make_float4(km[i].x * ca, fmaf(km[i].x, 128.0f, km[i].y) * p.sm_log2, lg2_approx(sve), ia);
      tok1[at] = fmaf(sve, 128.0f, vm[i].y) * ia;
    }
  }
  __device__ __forceinline__ void next(const AttnParams& p, int u) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      meta_of(p, u + 1, i, blk_n[i]);
      blk_n[i] = blk_of(p, u + 2, i);
    }
  }
};

template <int NC, bool INT>
__global__ void __launch_bounds__(F16Cfg<NC, INT>::kThreads, 1) attn_f16_kernel(const AttnParams p,
                                                                           const __grid_constant__ PlaneMaps maps) {
  using C = F16Cfg<NC, INT>;
  constexpr bool SPLIT = C::kSplit;
  constexpr int CG = C::kCG, NG = C::kNG, STEP = SPLIT ? 1 : 2, kDW = 8;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  float* scal = reinterpret_cast<float*>(smem + C::kOffScal);
  Item* items = reinterpret_cast<Item*>(smem + C::kOffItems);
  int* misc = reinterpret_cast<int*>(smem + C::kOffMisc);   // [0], [kItemAbort] abort, [7] units, [8] tensor memory base, [40 + g] accumulate
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);   // (known to be uniform)
  const uint32_t kfull = sbase + C::kOffBars, kempty = kfull + 32, vfull = kempty + 32, vempty = vfull + 24;
  const uint32_t qfull = vempty + 24, qempty = qfull + 16, qready = qempty + 16;   // [2]: piece published / left / queries in place
  const uint32_t kready = qready + 16, sfull = kready + 16, sfree = sfull + 16;    // [2]: K in TMEM / scores valid / scores read
  const uint32_t vready = sfree + 16, vfree = vready + 16;                         // [2]: V tile written / read
  const uint32_t pready = vfree + 16, pvdone = pready + 16;                        // [group]: weights written / P.V complete
  const uint32_t mready = pvdone + 16, mfree = mready + 32;                        // [4]: per-token scalars written / read
  volatile int* abort_word = misc;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 16 && lane < 4) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.m[lane])) : "memory");
  if (tid == 0) {
    for (int i = 0; i < C::kRingK; ++i) { mbar_init(kfull + i * 8, 2); mbar_init(kempty + i * 8, 4); }
    for (int i = 0; i < C::kRingV; ++i) { mbar_init(vfull + i * 8, 1); mbar_init(vempty + i * 8, 4); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(qfull + i * 8, 1);
      mbar_init(qempty + i * 8, C::kMetaK ? 12 : 14);
      mbar_init(qready + i * 8, 4);
      mbar_init(kready + i * 8, 4);
      mbar_init(sfull + i * 8, 1);
      mbar_init(sfree + i * 8, SPLIT ? 8 : 4);
      mbar_init(vready + i * 8, 4);
      mbar_init(vfree + i * 8, SPLIT ? 2 : 1);
      mbar_init(pready + i * 8, 4);
      mbar_init(pvdone + i * 8, 1);
    }
    for (int i = 0; i < 4; ++i) { mbar_init(mready + i * 8, C::kMetaK ? 4 : 2); mbar_init(mfree + i * 8, SPLIT ? 8 : 4); }
    for (int i = 0; i < 64; ++i) misc[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < 2 * C::kGrpScal; i += C::kThreads) reinterpret_cast<float*>(smem + C::kOffGrp)[i] = 0.0f;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(misc + 8)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem0 = __shfl_sync(0xFFFFFFFFu, *reinterpret_cast<volatile uint32_t*>(misc + 8), 0);
  // nothing in global memory has been touched so far: wait for the grids this one depends on (the producers by themselves)
  int n_units = 0;
  if (warp < 16 || warp >= 20) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    named_bar(7, C::kThreads);
    n_units = misc[7];
  }

  // ================================================================================== softmax warpgroups
  if (warp < 8) {
    reg_inc<C::kRegSoft>();
    const int g = warp >> 2, w4 = warp & 3, r = tid & 127;
    const uint32_t lane_sel = (uint32_t)(w4 * 32) << 16;
    const uint32_t tm_o = tmem0 + C::kTmO + g * C::kNPV + lane_sel, tm_of = tmem0 + C::kTmOF + g * 32 + lane_sel;
    float* of_s = reinterpret_cast<float*>(smem + C::kOffOF) + g * CG * 128 + r;   // (kIntPV)
    // this thread's tokens of a unit: t0 + 8 k, k = 0..3; its columns 8 j + c2, + 1
    const int t0 = w4 * 32 + (lane >> 2), c2 = (lane & 3) * 2;
    // row lane & 7 of block lane >> 3 of a warp's first eight tokens in the P tile (the remainders or odd columns: 64 bytes on, swizzled)
    const uint32_t p_addr = sbase + C::kOffP + g * C::kPTile + (uint32_t)(w4 * 32 + (lane & 7)) * 128u +
                            (uint32_t)((lane >> 3) ^ (lane & 7)) * 16u;
    float* grp = reinterpret_cast<float*>(smem + C::kOffGrp) + g * C::kGrpScal;
    float *ref_s = grp, *fac_s = grp + 32, *red_s = grp + 64, *lz_s = grp + 320;
    const int bar_g = 1 + g;
    const int col0 = SPLIT ? g * CG : 0;            // first column of this group
    const int dim_out = C::kIntPV ? 32 * (r >> 5) + 8 * ((r >> 2) & 3) + 2 * (r & 3) + ((r >> 4) & 1) : (r & ~7) + f16_perm(r & 7);
    const float4* tok4 = reinterpret_cast<const float4*>(smem + C::kOffTok) + t0;
    const float* tok1 = reinterpret_cast<const float*>(smem + C::kOffTok + 4 * 128 * 16) + t0;
    uint32_t n_own = 0;                             // units of this group so far
    int gs_base = 0, ic = 0;
    while (gs_base < n_units) {
      const int qi = ic & 1;
      mbar_wait_in(qfull + qi * 8, (ic >> 1) & 1, abort_word + kItemAbort);
      const Item item = items[qi];
      const int len = item.len, n_piece = item.pad0;
      const int u_first = SPLIT ? 0 : (g ^ gs_base) & 1;
      const bool have = u_first < n_piece;
      uint64_t l2[NG], zs2[NG];                     // softmax sums of this thread's tokens, two columns per register pair
      uint64_t qs2[NG], ref2[NG];                   // the columns' sums of q and reference exponents
#pragma unroll
      for (int j = 0; j < NG; ++j) { l2[j] = 0ull; zs2[j] = 0ull; ref2[j] = 0ull; }
      bool have_of = false;
      int units_in_acc = 0;
      // Moves the accumulators (the group's last P.V is complete) into the FP32 copy, scaled by fac_s[] if asked.
      auto drain = [&](bool scale) {
        tc_fence_after();
        // (loops: the caller's values, scores among them, fill the registers)
        if constexpr (C::kIntPV) {
#pragma unroll 1
          for (int c = 0; c < CG / 4; ++c) {
            uint32_t a[16];
            TmemRegs<16>::ld(tm_o + c * 16, a);
            tc_wait_ld();
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              float* o = of_s + f16_col(c, k) * 128;
              const float v = f16_planes(a + 4 * k);
              *o = have_of ? *o + v : v;
            }
          }
          have_of = true;
          units_in_acc = 0;
          return;
        }
#pragma unroll 1
        for (int c = 0; c < CG; c += kDW) {
          uint32_t h[kDW], q[kDW], of[kDW];
          TmemRegs<kDW>::ld(tm_o + c, h);
          TmemRegs<kDW>::ld(tm_o + 32 + c, q);
          TmemRegs<kDW>::ld(tm_of + c, of);
          tc_wait_ld();
          if (!have_of) {   // (a piece's first drain finds the previous piece's copy)
#pragma unroll
            for (int k = 0; k < kDW; ++k) of[k] = 0u;
          }
          if (units_in_acc > 0) {   // (else the accumulators have not been restarted since the last drain)
#pragma unroll
            for (int k = 0; k < kDW; k += 2) {
              const uint64_t v = f2_add(f2_add(f2_pack(__uint_as_float(h[k]), __uint_as_float(h[k + 1])),
                                               f2_pack(__uint_as_float(q[k]), __uint_as_float(q[k + 1]))),
                                        f2_pack(__uint_as_float(of[k]), __uint_as_float(of[k + 1])));
              float a, b;
              f2_unpack(v, a, b);
              of[k] = __float_as_uint(a);
              of[k + 1] = __float_as_uint(b);
            }
          }
          if (scale) {
#pragma unroll
            for (int k = 0; k < kDW; ++k) of[k] = __float_as_uint(__uint_as_float(of[k]) * fac_s[c + k]);
          }
          TmemRegs<kDW>::st(tm_of + c, of);
        }
        tc_wait_st();
        have_of = true;
        units_in_acc = 0;
      };
      // (kIntPV) After a change of the references: the sums of the columns that it concerns, scaled where they are and taken apart into
      // byte planes again.  Rarely more than one column of 32, which is why the others are left alone: with a drain of all columns
      // raises took a fifth of the time where outliers make them frequent.  (Known by one vote of the group's first warp, not from 32
      // factors: with outliers one sequence of 131072 tokens 78.3 -> 77.5 us, 4 of 32768 84.1 -> 83.0, 16 of 2000 38.5 -> 37.9.)
      auto rescale = [&](uint32_t raised) {
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < CG / 4; ++c) {
          const uint32_t cols = raised >> f16_col(c, 0);   // (its columns are 2 apart)
          if (!(cols & 0x55u)) continue;
          uint32_t a[16];
          TmemRegs<16>::ld(tm_o + c * 16, a);
          tc_wait_ld();
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (!(cols >> (2 * k) & 1u)) continue;
            const float f = fac_s[f16_col(c, k)];
            float v = f16_planes(a + 4 * k) * f;
            const int p3 = __float2int_rn(v * 0x1p-24f);
            v = fmaf((float)p3, -0x1p24f, v);
            const int p2 = __float2int_rn(v * 0x1p-16f);
            v = fmaf((float)p2, -0x1p16f, v);
            const int p1 = __float2int_rn(v * 0x1p-8f);
            v = fmaf((float)p1, -0x1p8f, v);
            a[4 * k] = (uint32_t)__float2int_rn(v);
            a[4 * k + 1] = (uint32_t)p1;
            a[4 * k + 2] = (uint32_t)p2;
            a[4 * k + 3] = (uint32_t)p3;
            if (have_of) of_s[f16_col(c, k) * 128] *= f;
          }
          TmemRegs<16>::st(tm_o + c * 16, a);
        }
        tc_wait_st();
        tc_fence_before();
      };
      if (have) {
        const int full_lim = p.causal ? len - p.tail + 1 : len;
        const int* lim_s = reinterpret_cast<const int*>(scal + 2 * NC + qi * NC) + col0;
        bool fresh = true;
        mbar_wait_in(qready + qi * 8, (ic >> 1) & 1, abort_word);
#pragma unroll
        for (int j = 0; j < NG; ++j) qs2[j] = *reinterpret_cast<const uint64_t*>(scal + qi * NC + col0 + 8 * j + c2);
        for (int u = u_first; u < n_piece; u += STEP, ++n_own) {
          const int gs = gs_base + u, sl = gs & 1;
          const int unit_t0 = (item.pad1 + u) * C::kST;
          // ---- scores: log2 of the weights relative to the columns' references ------------------------------
          const int ms = gs % C::kSlots;
          mbar_wait2_in(mready + ms * 8, (gs / C::kSlots) & 1, sfull + sl * 8, (gs >> 1) & 1, abort_word);
          tc_fence_after();
          uint64_t y2[4][NG];
          bool scale = false;
          uint32_t raised = 0;   // (kIntPV) the columns whose references changed
#pragma unroll 1
          for (int pass = 0; pass < 2; ++pass) {   // (a second time, from tensor memory, after a change of the references)
          const uint32_t tm_s = tmem0 + C::kTmS + sl * C::kSCols + col0 + lane_sel;
          uint32_t s[2][4 * NG];   // one part: tokens t0, t0 + 8 | t0 + 16, t0 + 24; two parts: the parts of one half
          if (C::kQP == 1) {
            tc_ld_16x256(tm_s, s[0]);
            tc_ld_16x256(tm_s + (16u << 16), s[1]);
            tc_wait_ld();
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (C::kQP == 2 && (k & 1) == 0) {
              tc_ld_16x256(tm_s + ((uint32_t)(8 * k) << 16), s[0]);
              tc_ld_16x256(tm_s + NC + ((uint32_t)(8 * k) << 16), s[1]);
              tc_wait_ld();
            }
            const float4 ts = tok4[ms * 128 + 8 * k];
            const uint64_t al2 = f2_pack(ts.x, ts.x), be2 = f2_pack(ts.y, ts.y), lsv2 = f2_pack(ts.z, ts.z);
#pragma unroll
            for (int j = 0; j < NG; ++j) {
              const uint32_t* sv = s[C::kQP == 2 ? 0 : k >> 1] + 4 * j + 2 * (k & 1);
              uint64_t rest = f2_fma(be2, qs2[j], f2_sub(lsv2, ref2[j]));
              if (C::kQP == 2) {
                const uint32_t* lv = s[1] + 4 * j + 2 * (k & 1);
                rest = f2_fma(f2_pack(__uint_as_float(lv[0]), __uint_as_float(lv[1])), al2, rest);
              }
              y2[k][j] = f2_fma(f2_pack(__uint_as_float(sv[0]), __uint_as_float(sv[1])), al2, rest);
            }
          }
          if (unit_t0 + C::kST > full_lim) {
#pragma unroll
            for (int j = 0; j < NG; ++j) {
              const int la = lim_s[8 * j + c2] - unit_t0 - t0, lb = lim_s[8 * j + c2 + 1] - unit_t0 - t0;
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                float a, b;
                f2_unpack(y2[k][j], a, b);
                if (8 * k >= la) a = -INFINITY;
                if (8 * k >= lb) b = -INFINITY;
                y2[k][j] = f2_pack(a, b);
              }
            }
          }
          float ymax = -INFINITY;
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < NG; ++j) {
              float a, b;
              f2_unpack(y2[k][j], a, b);
              ymax = max3(ymax, a, b);
            }
          if (n_own > 0) mbar_wait_in(pvdone + g * 8, (n_own - 1) & 1, abort_word);   // P free, accumulators current
          // (behind the scores: the product that is waited for here has had their time to complete)
          if constexpr (C::kIntPV) {
            if (scale) rescale(raised);
            if (units_in_acc >= C::kDrainUnits) drain(false);
          } else {
            if (scale || units_in_acc >= C::kDrainUnits) drain(scale);
          }
          // ---- a piece's first unit, or a weight that would leave FP16: new reference exponents ----------
          if (!bar_or(bar_g, 128, fresh || ymax > C::kRaise)) break;
#pragma unroll
            for (int j = 0; j < NG; ++j) {
              float ma = -INFINITY, mb = -INFINITY;
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                float a, b;
                f2_unpack(y2[k][j], a, b);
                ma = fmaxf(ma, a);
                mb = fmaxf(mb, b);
              }
#pragma unroll
              for (int off = 4; off <= 16; off <<= 1) {
                ma = fmaxf(ma, __shfl_xor_sync(0xFFFFFFFFu, ma, off));
                mb = fmaxf(mb, __shfl_xor_sync(0xFFFFFFFFu, mb, off));
              }
              if (lane < 4) { red_s[w4 * CG + 8 * j + c2] = ma; red_s[w4 * CG + 8 * j + c2 + 1] = mb; }
            }
            named_bar(bar_g, 128);
            if (r < CG) {
              const float old = fresh ? 0.0f : ref_s[r];
              const float mx = fmaxf(fmaxf(red_s[r], red_s[CG + r]), fmaxf(red_s[2 * CG + r], red_s[3 * CG + r])) + old;
              float nw = old, f = 1.0f;
              if (fresh) { nw = fmaxf(mx, -1.0e4f) - C::kTop; f = 0.0f; }
              else if (mx - old > C::kRaiseToo) { nw = mx - C::kTop; f = ex2_full(old - nw); }
              ref_s[r] = nw;
              fac_s[r] = f;
              if (C::kIntPV) {   // (the group's first warp)
                const uint32_t columns = __ballot_sync(0xFFFFFFFFu, f != 1.0f);
                if (r == 0) red_s[255] = __uint_as_float(columns);
              }
            }
            named_bar(bar_g, 128);
            if (C::kIntPV) raised = __float_as_uint(red_s[255]);
#pragma unroll
            for (int j = 0; j < NG; ++j) {
              const uint64_t f2 = *reinterpret_cast<const uint64_t*>(fac_s + 8 * j + c2);
              const uint64_t nw2 = *reinterpret_cast<const uint64_t*>(ref_s + 8 * j + c2);
              l2[j] = f2_mul(l2[j], f2);
              zs2[j] = f2_mul(zs2[j], f2);
              ref2[j] = nw2;
            }
            scale = !fresh;
            fresh = false;
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(sfree + sl * 8);   // the scores have been read: the unit after next may have their place
          // ---- weights of this thread's tokens into the P tile --------------------------------------------------
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float ia = tok4[ms * 128 + 8 * k].w, ib = tok1[ms * 128 + 8 * k];
            const uint64_t ia2 = f2_pack(ia, ia), ib2 = f2_pack(ib, ib);
            const float off = C::kIntPV ? weight_offset(unit_t0 + t0 + 8 * k) : 0.0f;
            uint32_t h[4], q[4];
#pragma unroll
            for (int j = 0; j < NG; ++j) {
              float a, b, ha, hb;
              f2_unpack(y2[k][j], a, b);
              const float wa = ex2_ftz(a), wb = ex2_ftz(b);
              const uint64_t w2 = f2_pack(wa, wb);
              l2[j] = f2_fma(w2, ia2, l2[j]);
              zs2[j] = f2_fma(w2, ib2, zs2[j]);
              if constexpr (C::kIntPV) {   // even and odd columns
                f2_unpack(f2_fma(w2, f2_pack(C::kScale, C::kScale), f2_pack(off, off)), a, b);
                asm("cvt.rni.u32.f32 %0, %1;" : "=r"(h[j]) : "f"(a));
                asm("cvt.rni.u32.f32 %0, %1;" : "=r"(q[j]) : "f"(b));
                continue;
              }
              h[j] = pack_f16x2(wa, wb);
              asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tcvt.f32.f16 %0, lo;\n\tcvt.f32.f16 %1, hi;\n\t}"
                  : "=f"(ha), "=f"(hb) : "r"(h[j]));
              f2_unpack(f2_sub(w2, f2_pack(ha, hb)), a, b);
              q[j] = pack_f16x2(a, b);
            }
            stm_x4(p_addr + k * 1024, h[0], h[1], h[2], h[3]);
            stm_x4((p_addr ^ 64u) + k * 1024, q[0], q[1], q[2], q[3]);
          }
          if (r == 0) misc[40 + g] = units_in_acc > 0 ? 1 : 0;
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          tc_fence_before();
          __syncwarp();
          if (lane == 0) { mbar_arrive(mfree + ms * 8); mbar_arrive(pready + g * 8); }
          ++units_in_acc;
        }
        mbar_wait_in(pvdone + g * 8, (n_own - 1) & 1, abort_word);   // the last P.V
        drain(false);
      }
      // ---- end of the piece: totals over the 128 tokens of a unit, then the result -------------------------
      if (have) {
#pragma unroll
        for (int j = 0; j < NG; ++j) {
          float v[4];
          f2_unpack(l2[j], v[0], v[1]);
          f2_unpack(zs2[j], v[2], v[3]);
#pragma unroll
          for (int off = 4; off <= 16; off <<= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] += __shfl_xor_sync(0xFFFFFFFFu, v[i], off);
          if (lane < 4) {
            float* d = red_s + w4 * 64 + 8 * j + c2;
            d[0] = v[0]; d[1] = v[1]; d[32] = v[2]; d[33] = v[3];
          }
        }
        named_bar(bar_g, 128);
        if (r < 64) lz_s[r] = (red_s[r] + red_s[64 + r]) + (red_s[128 + r] + red_s[192 + r]);
        named_bar(bar_g, 128);
      } else {
        if (r < 64) lz_s[r] = 0.0f;
        if (r < CG) ref_s[r] = -INFINITY;
        named_bar(bar_g, 128);
      }
      const size_t bh = (size_t)item.b * p.Hkv + item.hkv;
      float* part = p.ws_part + (bh + (size_t)blockIdx.x) * (size_t)C::kPartCols * kPartStride;
      auto put = [&](int c, float v, float m, float l) {   // column c, this lane's dim
        if (c >= p.ncols) return;
        part[(size_t)c * kPartStride + dim_out] = v;
        if (r == 0) *reinterpret_cast<float2*>(part + (size_t)c * kPartStride + 128) = make_float2(m, l);
      };
      // (rolled loops, eight columns of tensor memory at a time: this code runs once per piece)
      auto o_cols = [&](int c, float* o) {
        uint32_t t[8];
        TmemRegs<8>::ld(tm_of + c, t);
        tc_wait_ld();
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k] = have ? __uint_as_float(t[k]) : 0.0f;
      };
      if (SPLIT) {
#pragma unroll 1
        for (int c = 0; c < CG; c += 8) {
          float o[8];
          o_cols(c, o);
#pragma unroll
          for (int k = 0; k < 8; ++k) put(col0 + c + k, o[k] + lz_s[32 + c + k], ref_s[c + k], lz_s[c + k]);
        }
      } else if constexpr (C::kIntPV) {
        // each group merges and writes one half of the columns
        named_bar(3, 256);   // (the other group's copy and totals are in place)
        const float* of_o = of_s + (g ? -CG * 128 : CG * 128);
        const float* ogrp = reinterpret_cast<const float*>(smem + C::kOffGrp) + (g ^ 1) * C::kGrpScal;
        const bool have_o = ((g ^ 1 ^ gs_base) & 1) < n_piece;
#pragma unroll 4
        for (int cc = 16 * g; cc < 16 * g + 16; ++cc) {
          const float m1 = ref_s[cc], m2 = ogrp[cc], M = fmaxf(m1, m2);
          const float f1 = ex2_full(m1 - M), f2 = ex2_full(m2 - M);
          const float l = lz_s[cc] * f1 + ogrp[320 + cc] * f2;
          const float z = lz_s[32 + cc] * f1 + ogrp[320 + 32 + cc] * f2;
          const float o = ((have ? of_s[cc * 128] * f1 : 0.0f) + (have_o ? of_o[cc * 128] * f2 : 0.0f)) * (1.0f / C::kScale);
          put(cc, o + z, M, l);
        }
      } else {
        // each group hands the other one half of its columns through its idle P tile, and merges and writes the other half
        float* mail = reinterpret_cast<float*>(smem + C::kOffP + g * C::kPTile);
        const int g0 = 16 * g;   // first column of this group's half
#pragma unroll 1
        for (int c = 0; c < 16; c += 8) {
          float o[8];
          o_cols(16 - g0 + c, o);
#pragma unroll
          for (int k = 0; k < 8; ++k) mail[(c + k) * 128 + r] = o[k];
        }
        named_bar(3, 256);
        const float* omail = reinterpret_cast<const float*>(smem + C::kOffP + (g ^ 1) * C::kPTile);
        const float* ogrp = reinterpret_cast<const float*>(smem + C::kOffGrp) + (g ^ 1) * C::kGrpScal;
#pragma unroll 1
        for (int c = 0; c < 16; c += 8) {
          float o[8];
          o_cols(g0 + c, o);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int cc = g0 + c + k;
            const float m1 = ref_s[cc], m2 = ogrp[cc], M = fmaxf(m1, m2);
            const float f1 = ex2_full(m1 - M), f2 = ex2_full(m2 - M);
            const float l = lz_s[cc] * f1 + ogrp[320 + cc] * f2;
            const float z = lz_s[32 + cc] * f1 + ogrp[320 + 32 + cc] * f2;
            put(cc, (o[k] * f1 + omail[(c + k) * 128 + r] * f2) + z, M, l);
          }
        }
      }
      tc_fence_before();
      named_bar(3, 256);   // (the other group's sums and totals have been read)
      if (lane == 0) mbar_arrive(qempty + qi * 8);
      gs_base += n_piece;
      ++ic;
    }
    // ---- release the tensor memory: every product has been waited for, and the warps that issue copies and products are done
    tc_fence_before();
    named_bar(5, C::kDoneThreads);
    if (warp == 0) {
      land_after_abort([] { return globaltimer_ns(); }, abort_word);
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem0), "r"(512u) : "memory");
    }
    if (tid == 0 && (misc[0] || misc[kItemAbort])) atomicOr(p.ws_flags, kFlagTimeout);
    return;
  }
  // ================================================================================== K codes and queries
  if (warp < 12) {
    reg_dec<C::kRegExp>();
    const int kt = tid - 256, w4 = warp & 3;
    const uint32_t tm_k = tmem0 + C::kTmK + ((uint32_t)(w4 * 32) << 16);
    float* amax_s = reinterpret_cast<float*>(misc + 48);
    F16Meta<C, 1> meta;
    float ca = 0.0f;
    if (C::kMetaK) meta.init(p, smem, kt);
    int gs = 0, ic = 0, slot = 0;
    uint32_t phase = 0;
    while (gs < n_units) {
      const int qi = ic & 1;
      mbar_wait_in(qfull + qi * 8, (ic >> 1) & 1, abort_word + kItemAbort);
      const int ib = items[qi].b, ih = items[qi].hkv, len = items[qi].len, n_piece = items[qi].pad0;
      // ---- the piece's queries: thread = 16-byte chunk kt & 15 of columns kt >> 4, + 8, ... ---------------------
      {
        // (read once and kept, maxima on packed pairs, sums by exchanging halves, no division per chunk: with the
        // results written eight columns at a time, 64 columns of 85 tokens 18.8 -> 15.0 us, 32 columns of 4 x 7056 34.8 -> 32.6 us.
        // At 64 columns they spill 72 bytes of these warps' registers, once per piece.)
        constexpr int NI = NC / 8;
        const uint32_t g_inv = 65536u / (uint32_t)p.G + 1u;   // c / G = c * g_inv >> 16 for c < 64, G <= 16
        uint4 qv[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const uint32_t c = (uint32_t)(i * 8 + (kt >> 4)), j = c * g_inv >> 16, hh = c - j * (uint32_t)p.G;
          qv[i] = make_uint4(0u, 0u, 0u, 0u);
          if ((int)c < p.ncols)
            qv[i] = ld_dep(reinterpret_cast<const uint4*>(p.q + (((size_t)ib * p.nq_stride + j) * p.Hq + (size_t)ih * p.G + hh) * LYNX_D) + (kt & 15));
        }
        uint32_t amax2 = 0u;
        float sums[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const uint32_t w[4] = {qv[i].x, qv[i].y, qv[i].z, qv[i].w};
          uint64_t s2 = 0ull;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            asm("max.bf16x2 %0, %0, %1;" : "+r"(amax2) : "r"(w[k] & 0x7FFF7FFFu));
            s2 = f2_add(s2, f2_pack(__uint_as_float(w[k] << 16), __uint_as_float(w[k] & 0xFFFF0000u)));
          }
          float lo, hi;
          f2_unpack(s2, lo, hi);
          sums[i] = lo + hi;
        }
        float amax = fmaxf(__uint_as_float(amax2 << 16), __uint_as_float(amax2 & 0xFFFF0000u));
        {   // the sums of the 16 lanes of a column: lane i of them returns that of chunk i / (16 / NI)
          int off = 8;
#pragma unroll
          for (int m = NI / 2; m >= 1; m >>= 1, off >>= 1)
#pragma unroll
            for (int i = 0; i < m; ++i) {
              const bool up = (lane & off) != 0;
              const float give = up ? sums[i] : sums[i + m], keep = up ? sums[i + m] : sums[i];
              sums[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, off);
            }
#pragma unroll
          for (; off >= 1; off >>= 1) sums[0] += __shfl_xor_sync(0xFFFFFFFFu, sums[0], off);
          if ((lane & (16 / NI - 1)) == 0) scal[qi * NC + ((kt & 15) / (16 / NI)) * 8 + (kt >> 4)] = sums[0];
        }
        amax = warp_max(amax);
        if (lane == 0) amax_s[w4] = amax;
        named_bar(4, 128);
        amax = fmaxf(fmaxf(amax_s[0], amax_s[1]), fmaxf(amax_s[2], amax_s[3]));
        // |q 2^e| in [2^14, 2^15) for the largest entry
        int e = 0;
        if (amax > 0.0f && amax < INFINITY) e = 14 - (((__float_as_int(amax) >> 23) & 0xFF) - 127);
        e = max(-100, min(100, e));
        const float up = __int_as_float((127 + e) << 23);
        if (C::kMetaK) ca = p.sm_log2 * __int_as_float((127 - e) << 23);
        else if (kt == 0) reinterpret_cast<int*>(scal)[4 * NC + qi] = e;
        if (kt < NC) reinterpret_cast<int*>(scal)[2 * NC + qi * NC + kt] =
            kt < p.ncols ? (p.causal ? len - p.tail + kt / p.G + 1 : len) : 0;
        if (gs > 0) mbar_wait_in(sfull + ((gs - 1) & 1) * 8, ((gs - 1) >> 1) & 1, abort_word);   // the previous piece's last Q.K^T
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int c = i * 8 + (kt >> 4), ch = kt & 15;
          const uint32_t w[4] = {qv[i].x, qv[i].y, qv[i].z, qv[i].w};
          float f[8];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            f[2 * k] = __uint_as_float(w[k] << 16) * up;
            f[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u) * up;
          }
          const uint32_t dst = sbase + C::kOffQ + (uint32_t)(ch >> 3) * (C::kSCols * 128u) + (uint32_t)c * 128u +
                               (uint32_t)((ch & 7) ^ (c & 7)) * 16u;
          if (C::kQP == 2) {
            float lo[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) f16_split_q(f[k], lo[k]);
            sts128(dst + NC * 128u, pack_f16x2(lo[0], lo[4]), pack_f16x2(lo[2], lo[6]), pack_f16x2(lo[1], lo[5]), pack_f16x2(lo[3], lo[7]));
          }
          sts128(dst, pack_f16x2(f[0], f[4]), pack_f16x2(f[2], f[6]), pack_f16x2(f[1], f[5]), pack_f16x2(f[3], f[7]));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        named_bar(4, 128);
        if (lane == 0) { mbar_arrive(qready + qi * 8); mbar_arrive(qempty + qi * 8); }
      }
      // (the item is still there: the softmax groups have not left the piece)
      if (C::kMetaK) meta.piece(p, items[qi]);
      for (int u = 0; u < n_piece; ++u, ++gs) {
        if (C::kMetaK) {
          const int ms = gs % C::kSlots;
          mbar_wait_in(mfree + ms * 8, ((gs / C::kSlots) - 1) & 1, abort_word);
          meta.unit(p, u, gs, ca);
          __syncwarp();
          if (lane == 0) mbar_arrive(mready + ms * 8);
          meta.next(p, u);
        }
        mbar_wait2_in(kfull + slot * 8, phase, sfull + (gs & 1) * 8, ((gs >> 1) - 1) & 1, abort_word);   // and Q.K^T of the unit before last
        tc_fence_after();
        f16_expand_k(sbase + C::kOffRK + (uint32_t)slot * C::kStageBytes, kt, tm_k + (uint32_t)(gs & 1) * 64u);
        __syncwarp();
        if (lane == 0) mbar_arrive(kempty + slot * 8);
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(kready + (gs & 1) * 8);
        if (++slot == C::kRingK) { slot = 0; phase ^= 1; }
      }
      ++ic;
    }
    return;
  }
  // ================================================================================== V codes
  if (warp < 16) {
    reg_dec<C::kRegExp>();
    const int vt = tid - 384;
    int slot = 0;
    uint32_t phase = 0;
    for (int gs = 0; gs < n_units; ++gs) {
      mbar_wait2_in(vfull + slot * 8, phase, vfree + (gs & 1) * 8, ((gs >> 1) - 1) & 1, abort_word);
      const uint32_t raw = sbase + C::kOffRV + (uint32_t)slot * C::kStageBytes, tile = sbase + C::kOffV + (uint32_t)(gs & 1) * C::kVTile;
      if constexpr (C::kIntPV) f16_expand_v8(raw, tile, warp & 3, lane);
      else f16_expand_v(raw, tile, vt);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) { mbar_arrive(vempty + slot * 8); mbar_arrive(vready + (gs & 1) * 8); }
      if (++slot == C::kRingV) { slot = 0; phase ^= 1; }
    }
    return;
  }
  // ================================================================================== producers
  // (Behind the roles above and not in front of them: the instruction caches again.  us, 32 columns, in front / behind: 16 sequences of
  // 2000 tokens 35.4 / 34.6, 4 of 7056 31.8 / 31.2, 16 ragged ones 95.2 / 92.6, one of 131072 72.7 / 71.9.)
  if (warp < 20) {
    reg_dec<C::kRegProd>();
    const int pw = warp - 16;
    const SkPlace at = sk_place(p, blockIdx.x);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const SeqLens sl(p, lane);
    const SkRange rng = sk_range<C::kST>(p, gridDim.x, blockIdx.x, lane, sl, at);
    n_units = rng.lo < rng.hi ? (int)(rng.hi - rng.lo) : 0;
    if (pw == 0 && lane == 0) misc[7] = n_units;
    __syncwarp();
    bar_arrive(7, C::kThreads);   // the range is published (the producers know it and do not wait)
    if (n_units == 0 || pw == 3) bar_arrive(5, C::kDoneThreads);
    else
      plane_producer<C>(p, rng, sl, pw, lane, sbase, pw < 2 ? kfull : vfull, pw < 2 ? kempty : vempty, pw < 2 ? C::kRingK : C::kRingV, qfull,
                        qempty, reinterpret_cast<uint32_t*>(smem + C::kOffBlk), items, abort_word, &maps, 5);
    if (pw == kPublisher) per_sequence<true, C::kPartCols>(p, blockIdx.x, gridDim.x, lane, sl, n_units ? items : nullptr);
    return;
  }
  // ================================================================================== products
  reg_dec<C::kRegMma>();
  // ---- per-token scalars of the scores and weights (warps 21, 22: a lane has tokens 64 w + lane and 32 further on) ----
  if (!C::kMetaK && (warp == 21 || warp == 22)) {
    F16Meta<C, 2> meta;
    meta.init(p, smem, (warp - 21) * 64 + lane);
    int gs = 0, ic = 0;
    while (gs < n_units) {
      const int qi = ic & 1;
      mbar_wait_in(qfull + qi * 8, (ic >> 1) & 1, abort_word + kItemAbort);
      meta.piece(p, items[qi]);
      const int n_piece = items[qi].pad0;
      mbar_wait_in(qready + qi * 8, (ic >> 1) & 1, abort_word);
      const float ca = p.sm_log2 * __int_as_float((127 - reinterpret_cast<const int*>(scal)[4 * NC + qi]) << 23);
      for (int u = 0; u < n_piece; ++u, ++gs) {
        const int ms = gs % C::kSlots;
        mbar_wait_in(mfree + ms * 8, ((gs / C::kSlots) - 1) & 1, abort_word);
        meta.unit(p, u, gs, ca);
        __syncwarp();
        if (lane == 0) mbar_arrive(mready + ms * 8);
        meta.next(p, u);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(qempty + qi * 8);
      ++ic;
    }
    return;
  }
  if (warp == 20) {
    constexpr uint32_t kIdescS = tc_idesc(C::kSCols, false),
                       kIdescO = C::kIntPV ? i8_idesc(C::kNPV, true, false) | (1u << 7) : tc_idesc(64, true) | (1u << 15);   // (A: signed bytes)
    // (low words of the operand descriptors; the issuing thread keeps them in registers)
    constexpr uint32_t kHi = i8_desc_hi(1024u, 2u);
    const uint32_t q_lo = i8_desc_lo(sbase + C::kOffQ, 16u), v_lo = i8_desc_lo(sbase + C::kOffV, 16384u),
                   p_lo = i8_desc_lo(sbase + C::kOffP, 16384u);
    auto qk = [&](int gs) {
      const int sl = gs & 1;
      mbar_wait2_in(kready + sl * 8, (gs >> 1) & 1, sfree + sl * 8, ((gs >> 1) - 1) & 1, abort_word);
      tc_fence_after();
      if (tc_elect()) {
        const uint32_t d = tmem0 + C::kTmS + sl * C::kSCols, a = tmem0 + C::kTmK + sl * 64;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          tc_mma_ts(d, a + ks * 8u, i8_pack(q_lo + (uint32_t)(((ks >> 2) * C::kSCols * 128 + (ks & 3) * 32) >> 4), kHi), kIdescS, ks > 0 ? 1u : 0u);
        tc_commit(sfull + sl * 8);
      }
      __syncwarp();
    };
    auto pv = [&](int gs) {
      const int sl = gs & 1;
      mbar_wait_in(vready + sl * 8, (gs >> 1) & 1, abort_word);
#pragma unroll 1
      for (int g = SPLIT ? 0 : sl; g < (SPLIT ? 2 : sl + 1); ++g) {
        mbar_wait_in(pready + g * 8, (SPLIT ? gs : gs >> 1) & 1, abort_word);
        tc_fence_after();
        const uint32_t acc = *reinterpret_cast<volatile int*>(misc + 40 + g) ? 1u : 0u;
        if (tc_elect()) {
          const uint32_t d = tmem0 + C::kTmO + g * C::kNPV, vl = v_lo + sl * (C::kVTile >> 4), pl = p_lo + g * (C::kPTile >> 4);
#pragma unroll
          for (int ks = 0; ks < (C::kIntPV ? 4 : 8); ++ks) {
            if constexpr (C::kIntPV) i8_mma_ss(d, i8_pack(vl + ks * 256u, kHi), i8_pack(pl + ks * 256u, kHi), kIdescO, ks > 0 ? 1u : acc);
            else tc_mma_ss(d, i8_pack(vl + ks * 128u, kHi), i8_pack(pl + ks * 128u, kHi), kIdescO, ks > 0 ? 1u : acc);
          }
          tc_commit(pvdone + g * 8);
          tc_commit(vfree + sl * 8);
        }
        __syncwarp();
      }
    };
    // Q.K^T runs a unit ahead of P.V.  With 32 columns, where a group has one place for its scores, two units where it can: the
    // scores of unit gs are given up before its weights are complete.  It must not insist on unit gs + 2: where pieces are short
    // its queries may belong to a piece that is published only once unit gs has been left.  (One layer of 131072 tokens 89.2 ->
    // 88.4 us; with 64 columns, which have two places, looking ahead costs 2 %.)
    int next = 0;
#pragma unroll 1
    for (int gs = 0; gs < n_units; ++gs) {
#pragma unroll 1
      while (next < min(gs + 2, n_units)) qk(next++);
      if (!SPLIT && next < n_units) {
        const uint32_t kb = kready + (next & 1) * 8, kp = (next >> 1) & 1, sb = sfree + (next & 1) * 8, sp = kp ^ 1u;
        const uint32_t pb = pready + (gs & 1) * 8, pp = (gs >> 1) & 1;
        // (one answer for the warp: the products are issued by an elected lane, and `next` has to be the same in all)
        if (first_of([&](auto probe) { wait_in(probe, abort_word); }, [&] { return mbar_test(kb, kp) && mbar_test(sb, sp); },
                     [&] { return mbar_test(pb, pp); }, [](bool seen) { return __any_sync(0xFFFFFFFFu, seen) != 0; }))
          qk(next++);
      }
      pv(gs);
    }
    bar_arrive(5, C::kDoneThreads);
  }
}

template <int NC, bool INT>
lynx_status launch_f16(AttnParams p, cudaStream_t st) {
  using C = F16Cfg<NC, INT>;
  p.combine_single = 1;
  constexpr int kMin = 1;
  const lynx_status rc = launch_units<true, PlaneMaps, C::kSmem, C::kThreads, C::kST, kMin, attn_f16_kernel<NC, INT>>(p, st);
  return rc != LYNX_OK ? rc : launch_combine(p, C::kPartCols, C::kST, kMin, st);
}

// P.V on integers where a table gives each CTA 24 units or more and has room for five in a sequence: they take less per unit, 0.3 us more
// at the end of a piece, and some 4000 cycles whenever a reference is raised, which outliers do mostly in a piece's first units.  us, FP16 /
// integers, 32 columns, log-normal and outlier values: one sequence of 16384 (7 units per CTA) 24.0 / 23.1 and 25.2 / 26.1, 4 of 7056 (12) 31.2 /
// 28.6 and 32.3 / 32.7; 24 units and more: 200 of 500 (pieces of 4) 148.7 / 153.2 and 153.1 / 166.6, 160 of 600 (5) 156 / 145 and 158 / 155, 100 of
// 1000 130.5 / 117.0 and 130.5 / 125.2, 24 of 4000 84.5 / 75.4 and 85.7 / 80.8, one of 131072 80.0 / 72.3 and 82.5 / 77.5.  The host does not know the
// lengths: short sequences in a wide table go there, too.  (Both variants in one kernel that decides by the lengths: the instruction caches,
// 72.1 -> 75.1 us for one sequence of 131072, 16.0 -> 16.6 for one of 4096; each role's two codes side by side 73.5 and 18.1.)
inline bool f16_int_pv(const AttnParams& p) {
  const long long tokens = (long long)p.max_blocks * p.bt;
  return tokens > 4 * 128 && tokens * p.B * p.Hkv >= 24ll * 128 * sm_count();
}
