// Attention on the integer path of the fifth-generation tensor cores (tcgen05.mma kind::i8, accumulators in tensor memory), a team
// of warps per unit.  Included by attention.cu inside its namespace: shares AttnParams and the stream-K cut of the work with the
// other kernels.  The kernel here takes anchor calls with 17..32 columns, whose accumulators leave no tensor memory for the buffers of
// attention_pipe.cuh; that one shares the algebra and the expansions and takes up to 16 columns.
//
// With one (scale, zero) per token row the two contractions of Section 2's attention run on the
// integer levels themselves (see attention.cu).  Here both are exact integer tensor-core
// products over a 128-token stage-unit:
//   S^T[128 tokens x 3 * 32] = level(K)[128 x 128 dims] . Qd^T     A = K levels (u8, in tensor memory),
//                                                                   B = three balanced s8 digit planes
//                                                                       of the fixed-point query
//   O^T[128 dims x 4 * 32]  += level(V)^T[128 x 128 tokens] . Wd    A = V tile (u8, MN-major),
//                                                                   B = the four bytes of the u32
//                                                                       fixed-point weights (MN-major)
// Query columns (n_q * G) are padded to 32 (anchor calls with more are run in slices).  The int32 accumulators are exact, so
// there is no rounding in either product: the query is good to 2^-22 of its largest entry and a weight to 2^-28 of the largest
// weight seen so far.
//
// Weights.  For token t and column c,  x = s * log2(e) + log2(scale_v(t))  and  W = 2^(x - ref[c])
// rounded to a u32, with ref[c] chosen so that the largest W of the first unit is 2^28; a later x
// that would push W beyond 2^31.5 raises ref[c] (rare), which ends the current accumulation: the
// int32 accumulators are added, scaled, into an FP32 copy (in registers) and restart
// from zero.  The same happens before they could overflow.  The softmax sums use the unrounded
// W / scale_v, so a single attended token reproduces its value row to FP32 rounding.
//
// Warp roles of a CTA (one CTA per SM):
//   Two teams of eight warps take the units of the CTA's range in turn
//     and do everything for it, so that no hand-off between warps with different jobs lies on the
//     path of a unit and the teams hide one another's latencies:
//       K levels into tensor memory (a thread owns a token = a TMEM lane; Q.K^T takes its A
//         operand from there, so the K levels never pass through shared memory again);
//       Q.K^T (one thread issues four tcgen05.mma and a commit);
//       V level tile into shared memory (128-byte-swizzled canonical layout, MN-major);
//       scores -> weights: S read back (TMEM lane = token), per-token scale / zero point / causal
//         limit applied, weights written to the team's P tile;
//       P.V (one thread issues), accumulators in the team's tensor memory, their FP32 copy in registers.
//     The two warpgroups of a team share the tokens of a unit, each scoring 16 columns, one expanding K, the other V.
//     The team that owns a piece's first unit also writes the piece's query digit planes; at the
//     end of a piece the teams' partial results are merged by the team that owns its last unit.
//   Producer warps stream the raw planes into a shared-memory ring (cp.async.bulk).  The per-token
//     (scale, zero) pairs do not travel with them (the copy engine takes ~35 cycles per copy
//     whatever its size): every thread reads its own, two units ahead.
// All hand-offs are mbarriers or sequence counters with bounded waits; nothing waits on another CTA.
//
// Element order along head_dim inside operand tiles: byte 16 (2 j + parity) + 4 w + i of a row
// holds dim 32 j + 8 w + 2 i + parity (what the nibble expansion yields with two logic
// operations per word); the query planes use the same order and O is un-permuted at write-out.

// Tensor maps of the planes; a box is one 16-token sub-block, 1 KiB contiguous.  K planes as [rows / 2][128 bytes] with the 128-byte
// swizzle: the copy engine stores 16-byte chunk j of a pair of tokens r >> 1 at position j ^ ((r >> 1) & 7), so that the eight
// threads of a quarter-warp that read chunk i of their own rows (64 bytes apart) meet in no bank (see k_chunk).  V planes as
// [rows / 16][1024 bytes] without swizzle, which gathers of four sub-blocks take, too.  (148 CTAs, nothing but copies, TB/s: rows of
// 64 bytes 6.50 by four issuing warps, of 128 and more 6.75; one warp 3.06, two 6.0; gathers by one warp 4.3, by two 6.7.)
struct alignas(64) PlaneMaps {
  static constexpr bool kMeta = false;
  CUtensorMap m[4];   // K Anchor, V Anchor, K Residual, V Residual (the order of the stage's arrays)
};
struct alignas(64) PipeMaps : PlaneMaps {
  static constexpr bool kMeta = true;
  CUtensorMap meta[2];   // (scale, zero) pairs of K, V: [rows / 16][32 floats], for gathers of four sub-blocks
};
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                 const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiled encode_tiled() {
  static EncodeTiled fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiled>(f);
  }();
  return fn;
}
inline bool i8_plane_map(CUtensorMap* m, const uint8_t* base, uint64_t rows, bool k_plane) {
  const EncodeTiled fn = encode_tiled();
  if (!fn || !base || rows == 0) return false;
  const cuuint64_t dims[2] = {k_plane ? 128u : 256u, k_plane ? rows / 2 : rows / 16};   // (bytes, 32-bit words; rows is a multiple of 16)
  const cuuint64_t strides[1] = {k_plane ? 128u : 1024u};
  const cuuint32_t box[2] = {k_plane ? 128u : 256u, k_plane ? 8u : 1u}, es[2] = {1, 1};
  return fn(m, k_plane ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint8_t*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, k_plane ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
inline bool meta_map(CUtensorMap* m, const float* base, uint64_t rows) {
  const EncodeTiled fn = encode_tiled();
  if (!fn || !base || rows == 0) return false;
  const cuuint64_t dims[2] = {32, rows / 16};
  const cuuint64_t strides[1] = {128};
  const cuuint32_t box[2] = {32, 1}, es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// Four rows of a map (of V planes, of metadata) one behind the other into shared memory.
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap* map, uint4 r, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cta.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(r.x), "r"(r.y), "r"(r.z), "r"(r.w), "r"(bar)
      : "memory");
}
// The row of a plane's map at which the sub-block of plane row `row` starts, K or V (and the metadata's).
__device__ __forceinline__ uint32_t map_row(uint32_t row, bool k_plane) { return row >> (k_plane ? 1 : 4); }
// Offset of 16-byte chunk i of token r's 64 bytes in a raw K stage.
__device__ __forceinline__ uint32_t k_chunk(uint32_t r, uint32_t i) {
  return (r >> 1) * 128u + ((((r & 1u) * 4u + i) ^ ((r >> 1) & 7u)) << 4);
}
// the box of a plane that starts at row `row` of its map into shared memory
__device__ __forceinline__ void tma_box(uint32_t dst, const CUtensorMap* map, uint32_t row, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(bar)
      : "memory");
}

constexpr int kI8PieceUnits = 32;  // stage-units whose block ids a producer warp looks up at a time

struct I8Cfg {
  static constexpr int kST = 128;                   // tokens per stage-unit
  static constexpr int kCols = 32, kPartCols = kCols;    // query columns, column stride of the partial slots
  static constexpr int kStageBytes = kST * 128;     // K Anchor, V Anchor (the metadata is read with plain loads: the copy engine takes ~35 cycles per copy)
  static constexpr int kOffKA = 0, kOffVA = kST * 64;
  static constexpr int kNQK = 3 * kCols;            // N of the Q.K^T product (three digit planes)
  static constexpr int kNPV = 4 * kCols;            // N of the P.V product (four bytes of a weight)
  // a team is two warpgroups that share the tokens of a unit, each scoring 16 columns (and one expanding K, the other V)
  static constexpr int kGroups = 2, kCG = kCols / kGroups;
  static constexpr int kTeamWarps = 4 * kGroups, kTeamThreads = 32 * kTeamWarps;
  static constexpr int kTeams = 2, kProdWarps = 2, kProdWarp0 = kTeamWarps * kTeams;
  static constexpr int kThreads = (kProdWarp0 + kProdWarps) * 32;
  // shared memory map (offsets from a 1024-byte aligned base)
  static constexpr int kTile = 16384;                    // V level tile: [128 tokens][128 B]
  static constexpr int kPRow = 4 * kCols, kPTile = 128 * kPRow;   // P tile, a row of 128 bytes per token
  static constexpr int kTeamBytes = kTile + kPTile;      // (the K levels live in tensor memory)
  static constexpr int kQTile = kNQK * 128;
  static_assert(kQTile % 1024 == 0 && kCols * 128 * 4 <= kTile, "the deposit of a team: O in its V tile, (l, zs, ref) in its P tile");
  static constexpr int kOffQT = kTeams * kTeamBytes;
  static constexpr int kOffRing = kOffQT + 2 * kQTile;
  static constexpr int kTeamScal = (8 * kCols + 4 * 2 * kCols + 2 * kCols) * 4;   // qs, ref, factor, limits, maxima; reduce scratch; totals
  static constexpr int kFixedTail = 2 * kCols * 256 + kTeams * kTeamScal + 8 * kI8PieceUnits * 4 + 2 * 32 + 64 * 8 + (1 + kTeams) * 256 + 64;
  static constexpr int kAvail = 227 * 1024 - 1024 - kOffRing - kFixedTail;
  static constexpr int kNStage = kAvail / kStageBytes > 8 ? 8 : kAvail / kStageBytes;
  static_assert(kNStage >= 2, "ring too small");
  static constexpr int kOffQRaw = kOffRing + kNStage * kStageBytes;
  static constexpr int kOffScal = kOffQRaw + 2 * kCols * 256;
  static constexpr int kOffBlk = kOffScal + kTeams * kTeamScal;
  static constexpr int kOffItems = kOffBlk + 8 * kI8PieceUnits * 4;
  static constexpr int kOffBars = kOffItems + 2 * 32;
  static constexpr int kOffMisc = kOffBars + 64 * 8;             // [1 + teams][64] ints
  static constexpr int kSmem = kOffMisc + (1 + kTeams) * 256 + 64 + 1024;   // + alignment slack
  static_assert(kSmem <= 227 * 1024, "shared memory");
  static_assert(kOffScal % 16 == 0 && kTeamScal % 16 == 0 && kOffBars % 8 == 0, "alignment");
  // tensor memory columns of a team: S, O accumulators, K levels (128 bytes per token); the FP32 copy of O stays in registers
  static constexpr int kTmS = 0, kTmO = kNQK, kTmK = kNQK + kNPV, kTmTeam = 256, kTmCols = 512;
  static_assert(kTmK + 32 <= kTmTeam && kTeams * kTmTeam <= kTmCols, "tensor memory");
  static constexpr int kDrainUnits = 4096;  // own units after which the int32 sums could overflow (128 * 15 * 255 each)
};

template <>
struct TmemRegs<4> {
  static __device__ __forceinline__ void ld(uint32_t a, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  }
  static __device__ __forceinline__ void st(uint32_t a, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};"
                 ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
  }
};

// Instruction descriptor of kind::i8: int32 accumulate, u8 A, u8 or s8 B, M = 128.
__host__ __device__ constexpr uint32_t i8_idesc(int n, bool mn_major, bool b_signed) {
  return (2u << 4) | ((b_signed ? 1u : 0u) << 10) | ((mn_major ? 1u : 0u) << 15) | ((mn_major ? 1u : 0u) << 16) |
         ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void i8_mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(0u) : "memory");
}
__device__ __forceinline__ void i8_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, {%5, %5, %5, %5}, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(0u) : "memory");
}
// barrier among `n` threads that also ORs a predicate over them
__device__ __forceinline__ bool bar_or(int id, int n, bool pred) {
  uint32_t res;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(res) : "r"(pred ? 1u : 0u), "r"(id), "r"(n) : "memory");
  return res != 0;
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Packed pairs of FP32 values (one 64-bit register pair, one instruction per pair of operations)
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// (One instruction per maximum and the sums below instead of butterflies in the restart and at the end of a piece, which lie in and
// around the unit loop: fewer steps in a row where a piece starts and ends, and less code in the instruction caches.  us, before the
// power cap sets in: 16 ragged sequences at 16 columns 321 -> 275 (in it 338 -> 307), 16 layers of two sequences of 131072 tokens at 8
// columns 907 -> 878; one layer of 131072 tokens at 4 columns 39.0 -> 37.7, two sequences of 16000 at 8 columns 24.0 -> 21.8.)
__device__ __forceinline__ float warp_max(float x) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
// The sums (or whatever `op` is) of N values per lane over a warp: lane i returns that of value i / (32 / N).  Half of the values change
// places at every step, 2 N - 2 additions in all where N butterflies would take 5 N; each sum in the order of a butterfly.
template <int N, class Op>
__device__ __forceinline__ float warp_halves(float (&v)[N], int lane, Op op) {
  static_assert(N == 4 || N == 8 || N == 16 || N == 32, "lanes share the values evenly");
  int off = 16;
#pragma unroll
  for (int m = N / 2; m >= 1; m >>= 1, off >>= 1)
#pragma unroll
    for (int i = 0; i < m; ++i) {
      const bool up = (lane & off) != 0;
      const float give = up ? v[i] : v[i + m], keep = up ? v[i + m] : v[i];
      v[i] = op(keep, __shfl_xor_sync(0xFFFFFFFFu, give, off));
    }
#pragma unroll
  for (; off >= 1; off >>= 1) v[0] = op(v[0], __shfl_xor_sync(0xFFFFFFFFu, v[0], off));
  return v[0];
}
template <int N>
__device__ __forceinline__ float warp_sums(float (&v)[N], int lane) {
  return warp_halves(v, lane, [](float a, float b) { return a + b; });
}
__device__ __forceinline__ float ex2_full(float x) {   // no flush of small results
  float y;
  asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Expand the nibble planes of one tensor of a 128-token raw stage into its u8 level tile.  A warp
// takes 8 token rows per step (512 contiguous raw bytes): lane = (row & 7) * 4 + 16-byte chunk.  ODD16: the odd elements of an
// Anchor plane as they lie in their bytes, 16 times the level (the caller takes it off the sums).  FLIP: what the Anchor words are
// exclusive-ored with (0x88888888: the codes less 128, as signed bytes).
template <bool FULL, bool ODD16 = false, uint32_t FLIP = 0>
__device__ __forceinline__ void i8_expand(uint32_t raw_a, uint32_t raw_r, uint32_t tile, int w4, int lane) {
  const int row8 = lane >> 2, j = lane & 3;
  uint4 xa[4], xr[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const uint32_t off = (uint32_t)(((w4 + 4 * s) * 8 + row8) * 64 + j * 16);
    xa[s] = lds128(raw_a + off);
    if (FULL) xr[s] = lds128(raw_r + off);
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int row = (w4 + 4 * s) * 8 + row8;
    const uint32_t a[4] = {xa[s].x, xa[s].y, xa[s].z, xa[s].w};
    uint32_t ev[4], od[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (FULL) {
        const uint32_t r[4] = {xr[s].x, xr[s].y, xr[s].z, xr[s].w};
        merge_codes(a[k] ^ FLIP, r[k], ev[k], od[k]);
      } else {
        ev[k] = a[k] & 0x0F0F0F0Fu;
        od[k] = ODD16 ? a[k] & 0xF0F0F0F0u : (a[k] >> 4) & 0x0F0F0F0Fu;
      }
    }
    const uint32_t base = tile + (uint32_t)row * 128u;
    const uint32_t c0 = (uint32_t)((2 * j) ^ (row & 7)) << 4, c1 = (uint32_t)((2 * j + 1) ^ (row & 7)) << 4;
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + c0), "r"(ev[0]), "r"(ev[1]), "r"(ev[2]),
                 "r"(ev[3]) : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + c1), "r"(od[0]), "r"(od[1]), "r"(od[2]),
                 "r"(od[3]) : "memory");
  }
}

// K levels of a 128-token raw stage into tensor memory: thread r owns token r (TMEM lane r) and writes
// its 128 level bytes to 32 columns, byte 4 col + b in the order of the operand tiles (see the header).
template <bool FULL, bool RAW, uint32_t FLIP = 0>
__device__ __forceinline__ void i8_expand_k_tmem(uint32_t raw_a, uint32_t raw_r, int r, uint32_t tm_k) {
  uint4 xa[4], xr[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t off = k_chunk((uint32_t)r, (uint32_t)i);
    xa[i] = lds128(raw_a + off);
    if (FULL) xr[i] = lds128(raw_r + off);
  }
  uint32_t regs[32];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t a[4] = {xa[j].x, xa[j].y, xa[j].z, xa[j].w};
    uint32_t rr[4] = {0, 0, 0, 0};
    if (FULL) { rr[0] = xr[j].x; rr[1] = xr[j].y; rr[2] = xr[j].z; rr[3] = xr[j].w; }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      if (FULL) {
        merge_codes(a[w] ^ FLIP, rr[w], regs[8 * j + w], regs[8 * j + 4 + w]);
      } else if (RAW) {   // bytes 16 j + 4 w .. + 3 of the row as they are, and their low nibbles 64 bytes further on
        regs[4 * j + w] = a[w];
        regs[16 + 4 * j + w] = a[w] & 0x0F0F0F0Fu;
      } else {
        regs[8 * j + w] = a[w] & 0x0F0F0F0Fu;
        regs[8 * j + 4 + w] = (a[w] >> 4) & 0x0F0F0F0Fu;
      }
    }
  }
  TmemRegs<32>::st(tm_k, regs);
}

// One of the producer warps: the stream-K bookkeeping (every warp derives the same range and
// pieces; warp 0 alone publishes them, loads the queries and handles empty sequences) and, per
// unit, its share of the plane copies: 8 sub-blocks of 16 tokens x K and V, four sub-blocks per warp.
__device__ __forceinline__ void i8_producer(const AttnParams& p, int pw, int lane, uint32_t ring_u32,
                                            uint32_t full0, uint32_t empty0, uint32_t qfull0, uint32_t qempty0,
                                            uint32_t qraw_u32, uint32_t* blk_s, Item* items, int* misc,
                                            volatile int* abort_word, const PlaneMaps* maps) {
  using C = I8Cfg;
  constexpr int ST = C::kST, NSTAGE = C::kNStage, NARR = 2;   // (K, V)
  const int n_cta = gridDim.x, cta = blockIdx.x;
  const SeqLens sl(p, lane);
  const SkRange rng = sk_range<ST>(p, n_cta, cta, lane, sl, sk_place(p, cta));
  const long long q = rng.q, lo = rng.lo, hi = rng.hi, off_lo = rng.off_lo;
  const int b_lo = rng.b_lo;
  if (pw == 0 && lane == 0) misc[7] = lo < hi ? (int)(hi - lo) : 0;
  __syncthreads();  // (A) the range is published
  const int n_units = (int)(lo < hi ? hi - lo : 0);
  if (n_units == 0) {
    if (pw == 0) per_sequence<false, C::kPartCols>(p, cta, n_cta, lane, sl, nullptr);
    return;
  }

  constexpr int SPW = 8 / C::kProdWarps;       // 16-token sub-blocks per warp
  constexpr int RP = SPW * NARR;               // roles of this warp: (sub-block, array)
  const int role = pw * RP + (lane < RP ? lane : 0);
  const int sub = role / NARR, arr = role % NARR, sub_first = SPW * pw;
  const uint32_t my_bytes = 1024u;
  const uint32_t my_dst = (uint32_t)(arr == 0 ? C::kOffKA : C::kOffVA) + (uint32_t)sub * my_bytes;
  constexpr uint32_t kBytesSub = 2u * 1024u;   // bytes of one sub-block
  uint32_t* my_blk = blk_s + pw * SPW * kI8PieceUnits;   // [SPW sub-blocks][kI8PieceUnits]
  int b = b_lo, len = sl.of(b), U = (len + ST - 1) / ST;
  int hkv = (int)sk_div(off_lo, U), u = (int)(off_lo - (long long)hkv * U);
  int remaining = n_units, gs = 0, ic = 0;
  while (remaining > 0) {
    const int n = min(remaining, U - u);
    const int qi = ic & 1;
    if (pw == 0) {
      if (ic >= 2) mbar_wait<kItemAbort>(qempty0 + qi * 8, ((ic >> 1) - 1) & 1, abort_word);
      const long long seg0 = lo + (n_units - remaining) - u;  // first unit of this segment
      if (lane == 0) {
        Item it;
        it.b = b; it.hkv = hkv; it.len = len;
        it.first_cta = (int)sk_div(seg0, q);
        it.n_contrib = (int)sk_div(seg0 + U - 1, q) - it.first_cta + 1;
        it.pad0 = n; it.pad1 = u; it.pad2 = 0;
        items[qi] = it;
        if (u == 0) *seg_word(p, (size_t)b * p.Hkv + hkv, C::kPartCols) = (uint32_t)it.first_cta << 16 | (uint32_t)it.n_contrib;
        mbar_expect_tx(qfull0 + qi * 8, (uint32_t)(p.nq * p.G * LYNX_D * 2));
      }
      __syncwarp();
      for (int j = lane; j < p.nq; j += 32)
        bulk_g2s(qraw_u32 + (uint32_t)((qi * C::kCols + j * p.G) * LYNX_D * 2),
                 p.q + (((size_t)b * p.nq_stride + j) * p.Hq + (size_t)hkv * p.G) * LYNX_D,
                 (uint32_t)(p.G * LYNX_D * 2), qfull0 + qi * 8);
    }
    for (int c0 = 0; c0 < n; c0 += kI8PieceUnits) {
      const int cn = min(kI8PieceUnits, n - c0);
      for (int i2 = lane; i2 < SPW * cn; i2 += 32) {
        const int i = i2 / SPW;
        const int t0 = (u + c0 + i) * ST + (sub_first + (i2 % SPW)) * 16;
        uint32_t row = 0xFFFFFFFFu;  // sub-block beyond the end of the sequence: nothing to copy
        if (t0 < len) {
          const int bi = block_of(p, t0);
          int blk = ld_dep(p.block_table + (size_t)b * p.max_blocks + bi);
          if (blk < 0 || blk >= p.num_blocks) {
            atomicOr(p.ws_flags, kFlagBadBlock);
            blk = blk < 0 ? 0 : p.num_blocks - 1;
          }
          row = (uint32_t)(((size_t)blk * p.Hkv + hkv) * p.bt + (t0 - bi * p.bt));
        }
        my_blk[(i2 % SPW) * kI8PieceUnits + i] = row;
      }
      __syncwarp();
      for (int k = 0; k < cn; ++k, ++gs) {
        const int slot = gs % NSTAGE;
        if (gs >= NSTAGE) mbar_wait(empty0 + slot * 8, ((gs / NSTAGE) - 1) & 1, abort_word);
        const uint32_t row = my_blk[(sub - sub_first) * kI8PieceUnits + k];
        const uint32_t bar = full0 + slot * 8;
        if (lane == 0) {
          uint32_t bytes = 0;
#pragma unroll
          for (int i = 0; i < SPW; ++i) bytes += my_blk[i * kI8PieceUnits + k] != 0xFFFFFFFFu ? kBytesSub : 0u;
          if (bytes) mbar_expect_tx(bar, bytes);
          else mbar_arrive(bar);
        }
        __syncwarp();
        if (lane < RP && row != 0xFFFFFFFFu)
          tma_box(ring_u32 + slot * C::kStageBytes + my_dst, &maps->m[arr], map_row(row, arr == 0), bar);
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
  bar_arrive(9, C::kThreads);
  if (pw == 0) per_sequence<false, C::kPartCols>(p, cta, n_cta, lane, sl, items);
}

// Largest |q| of a piece's raw queries, by nthr threads (index i), reduced over the warp; the caller combines the warps.
__device__ __forceinline__ float i8_q_absmax(const unsigned char* qraw, int i, int nthr) {
  float amax = 0.0f;
  for (int k = i; k < I8Cfg::kCols * 16; k += nthr) {
    const uint4 v = reinterpret_cast<const uint4*>(qraw)[k];
    const uint32_t ww[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      amax = fmaxf(amax, fabsf(__uint_as_float(ww[j] << 16)));
      amax = fmaxf(amax, fabsf(__uint_as_float(ww[j] & 0xFFFF0000u)));
    }
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, off));
  return amax;
}
// Fixed-point exponent of a piece's queries: |q * 2^e| < 2^22.
__device__ __forceinline__ int i8_q_exponent(float amax) {
  int e = 0;
  if (amax > 0.0f && amax < INFINITY) e = 21 - (((__float_as_int(amax) >> 23) & 0xFF) - 127);
  return max(-100, min(100, e));
}

// The two halves of a shared-memory matrix descriptor (the MMA-issuing thread keeps the low words of
// its operands in registers and adds the K-step offset: building descriptors is a chain of dependent
// instructions in the one thread everybody waits for).
__host__ __device__ constexpr uint32_t i8_desc_hi(uint32_t sbo_bytes, uint32_t layout) {
  return ((sbo_bytes >> 4) & 0x3FFFu) | (1u << 14) | (layout << 29);
}
__device__ __forceinline__ uint32_t i8_desc_lo(uint32_t addr, uint32_t lbo_bytes) {
  return ((addr >> 4) & 0x3FFFu) | (((lbo_bytes >> 4) & 0x3FFFu) << 16);
}
__device__ __forceinline__ uint64_t i8_pack(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}
// Joining the slots of a segment that several CTAs share, by the last of them (atomic tickets that reset themselves, nobody waits).
// A segment of more than kOneLevel CTAs -- a long sequence among many short ones, with few heads -- is joined in two levels, so
// that no CTA walks through all of its slots: the last CTA of each kGroup neighbouring ones joins theirs into the first of them,
// the last group the groups'.
constexpr int kGroup = 8, kOneLevel = 24;
// The group of this CTA (its first slot, its slots) and the group's ticket, which lies with its first CTA: that one can lead two
// groups, the first of the segment that starts in its range and a later one of the segment that ends there.
struct SlotGroup {
  int first, count;
  uint32_t* ticket;
};
__device__ __forceinline__ SlotGroup slot_group(const AttnParams& p, const Item& item) {
  if (item.n_contrib <= kOneLevel) return {0, item.n_contrib, p.ws_tickets + item.first_cta};
  const int first = ((int)blockIdx.x - item.first_cta) / kGroup * kGroup;
  return {first, min(kGroup, item.n_contrib - first), p.ws_groups + 2 * (item.first_cta + first) + (first == 0 ? 1 : 0)};
}
__device__ __forceinline__ bool last_of(uint32_t* ticket, int n) { return atomicInc(ticket, (uint32_t)n - 1) == (uint32_t)n - 1; }
// `count` slots from `first` on, STRIDE apart, by all teams: a warp per column, a lane four dims, four slots in flight.  Into the
// output, or (`top` false) into the first of them.
template <class C>
__device__ __forceinline__ void i8_join(const AttnParams& p, const Item& item, int first, int count, int stride, bool top, int tid) {
  constexpr size_t kSlot = (size_t)C::kPartCols * kPartStride;
  const int lane = tid & 31;
  float* seg = p.ws_part + ((size_t)item.b * p.Hkv + item.hkv + (size_t)(item.first_cta + first)) * kSlot;
#pragma unroll 1
  for (int c = tid >> 5; c < p.ncols; c += C::kTeams * C::kTeamWarps) {
    float* col = seg + (size_t)c * kPartStride;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float M = -INFINITY, L = 0.0f;
#pragma unroll 1
    for (int i0 = 0; i0 < count; i0 += 4) {
      float4 o[4];
      float2 ml[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float* s = col + (size_t)(min(i0 + u, count - 1) * stride) * kSlot;
        ml[u] = __ldcg(reinterpret_cast<const float2*>(s + 128));
        o[u] = __ldcg(reinterpret_cast<const float4*>(s) + lane);
        if (i0 + u >= count) ml[u].x = -INFINITY;
      }
      const float m0 = M;
      M = fmaxf(fmaxf(fmaxf(M, ml[0].x), ml[1].x), fmaxf(ml[2].x, ml[3].x));   // (finite: every slot's is)
      const float f0 = ex2(m0 - M);
      L *= f0;
      acc.x *= f0; acc.y *= f0; acc.z *= f0; acc.w *= f0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float f = ex2(ml[u].x - M);
        L = fmaf(ml[u].y, f, L);
        acc.x = fmaf(o[u].x, f, acc.x);
        acc.y = fmaf(o[u].y, f, acc.y);
        acc.z = fmaf(o[u].z, f, acc.z);
        acc.w = fmaf(o[u].w, f, acc.w);
      }
    }
    if (!top) {
      __syncwarp();   // (all lanes have read the first slot)
      reinterpret_cast<float4*>(col)[lane] = acc;
      if (lane == 0) *reinterpret_cast<float2*>(col + 128) = make_float2(M, L);
      continue;
    }
    const float inv = L > 0.0f ? 1.0f / L : 0.0f;
    const int j = c / p.G;
    const size_t row = ((size_t)item.b * p.nq_stride + j) * p.Hq + (size_t)item.hkv * p.G + (c - j * p.G);
    reinterpret_cast<float4*>(p.out + row * LYNX_D)[lane] = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
    if (lane == 0) p.ws_lse[row] = lse_of(M, L);
  }
}
// The segments that a CTA shares -- its first with the CTAs before it, its last with those behind -- once all of its slots have been
// written, fenced and passed a barrier.  (At the end of the CTA, not of the piece: within reach of the unit loop this code costs
// registers there.  us, before -> after: one sequence of 32768 tokens among 39 of 64, one KV head, 4 / 16 columns 24.0 / 72.1 ->
// 14.3 / 21.4; 8 of 65536, 8 KV heads, 8 / 16 columns 132.6 / 184.2 -> 131.4 / 180.4; 6 of 9000, 4 / 32 columns 18.4 / 55.2 -> 18.5 / 52.8.)
template <class C>
__device__ __forceinline__ void i8_join_shared(const AttnParams& p, const Item* shared, int tid, int* misc) {
  constexpr int kThreads = C::kTeams * C::kTeamThreads;
  if (tid < 2) {   // (both tickets at once)
    misc[1 + tid] = 0;
    if (shared[tid].n_contrib > 1) {
      const SlotGroup g = slot_group(p, shared[tid]);
      misc[1 + tid] = last_of(g.ticket, g.count);
    }
  }
  named_bar(14, kThreads);
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    if (misc[1 + i] == 0) continue;
    const Item item = shared[i];
    const int n = item.n_contrib;
    bool top = n <= kOneLevel;
    SlotGroup g = slot_group(p, item);
    __threadfence();
#pragma unroll 1
    for (int stride = 1;; stride = kGroup) {
      i8_join<C>(p, item, g.first, g.count, stride, top, tid);
      if (top) break;
      g.first = 0;
      g.count = (n + kGroup - 1) / kGroup;
      __threadfence();
      named_bar(14, kThreads);
      if (tid == 0) misc[3] = last_of(p.ws_tickets + item.first_cta, g.count);
      named_bar(14, kThreads);
      if (misc[3] == 0) break;
      __threadfence();
      top = true;
    }
  }
}
// Bounded wait until a shared-memory sequence counter has reached `need` (a counter, unlike an mbarrier
// phase, cannot be misread by a waiter that is ahead of the writer).  Gives up after ~2 s like mbar_wait.
__device__ __noinline__ bool seq_wait(const volatile int* ctr, int need, volatile int* abort_word) {
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i) {
      if (*ctr >= need) { __threadfence_block(); return true; }
      __nanosleep(40);
    }
    if (*abort_word) return false;
    if (globaltimer_ns() - t0 > 2000000000ull) { *abort_word = 1; return false; }
  }
}

__global__ void __launch_bounds__(I8Cfg::kThreads, 1) attn_i8_kernel(const AttnParams p, const __grid_constant__ PlaneMaps maps) {
  using C = I8Cfg;
  constexpr int NSTAGE = C::kNStage, T = C::kTeams, G = C::kGroups, CP = C::kCols, CG = C::kCG, TT = C::kTeamThreads;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  unsigned char* qraw = smem + C::kOffQRaw;
  uint32_t* blk_s = reinterpret_cast<uint32_t*>(smem + C::kOffBlk);
  Item* items = reinterpret_cast<Item*>(smem + C::kOffItems);
  int* misc = reinterpret_cast<int*>(smem + C::kOffMisc);
  const int tid = threadIdx.x, lane = tid & 31;
  // (broadcast from lane 0 so that the compiler knows the warp index, and all that follows from it -- team, tiles,
  // operand descriptors -- to be the same for every lane: such values can live in uniform registers)
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
  const uint32_t ring_u32 = sbase + C::kOffRing;
  const uint32_t full0 = sbase + C::kOffBars, empty0 = full0 + NSTAGE * 8;
  const uint32_t qfull0 = empty0 + NSTAGE * 8, qempty0 = qfull0 + 16;
  const uint32_t qready0 = qempty0 + 16;          // [query slot]  the digit planes of the piece are written
  const uint32_t sfull0 = qready0 + 16;           // [team]  Q.K^T complete: scores valid, K tile free
  const uint32_t pvdone0 = sfull0 + T * 8;        // [team]  P.V complete: P and V tiles free, accumulators current
  volatile int* abort_word = misc;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // a dependent grid may be scheduled as SMs become free
  // misc[0], misc[kItemAbort]: abort words; misc[8] = tensor memory base; misc[16 + t] = deposits written by team t, misc[24 + t] = deposits of team t read;
  // misc[32 + s] = completed phases of raw stage s

  if (tid == 0) {
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(full0 + i * 8, C::kProdWarps);
      mbar_init(empty0 + i * 8, C::kTeamWarps);   // the warps of the team that owns the unit
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(qfull0 + i * 8, 1);
      mbar_init(qempty0 + i * 8, C::kTeamWarps * T);
      mbar_init(qready0 + i * 8, C::kTeamWarps);
    }
    for (int i = 0; i < T; ++i) {
      mbar_init(sfull0 + i * 8, 1);
      mbar_init(pvdone0 + i * 8, 1);
    }
    for (int i = 0; i < (1 + T) * 64 + 16; ++i) misc[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // raw query slots (their padding columns stay zero) and query digit planes (their padding rows too)
  for (int i = tid; i < 2 * CP * 256 / 16; i += C::kThreads) reinterpret_cast<uint4*>(qraw)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < 2 * C::kQTile / 16; i += C::kThreads)
    reinterpret_cast<uint4*>(smem + C::kOffQT)[i] = make_uint4(0, 0, 0, 0);
  // the teams' scalars (the reference exponents must be finite numbers before their first use)
  for (int i = tid; i < T * C::kTeamScal / 4; i += C::kThreads) reinterpret_cast<float*>(smem + C::kOffScal)[i] = 0.0f;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  // nothing in global memory has been touched so far: wait for the grids this one depends on
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp >= C::kProdWarp0) {
    i8_producer(p, warp - C::kProdWarp0, lane, ring_u32, full0, empty0, qfull0, qempty0,
                         sbase + C::kOffQRaw, blk_s, items, misc, abort_word, &maps);
    return;
  }
  __syncthreads();  // (A)
  const int n_units = misc[7];
  if (n_units == 0) return;

  // ---- tensor memory ---------------------------------------------------------------------------
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(misc + 8)),
                 "r"((uint32_t)C::kTmCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  named_bar(14, T * TT);
  tc_fence_after();
  const uint32_t tmem0 = __shfl_sync(0xFFFFFFFFu, *reinterpret_cast<volatile uint32_t*>(misc + 8), 0);   // (known to be uniform)
  constexpr uint32_t kIdescS = i8_idesc(C::kNQK, false, true), kIdescO = i8_idesc(C::kNPV, true, false);

  // =============================================================================================
  // Teams.  Team t takes the units gs = t, t + T, ... of the CTA's range and does everything for
  // them: K tile, Q.K^T, V tile, scores -> weights, P.V.
  // =============================================================================================
  const int tm = warp / C::kTeamWarps, grp = (warp >> 2) % G, w4 = warp & 3;
  const int r = tid & 127;                        // token of the unit (S), output dim position (O): TMEM lane
  const int tt = r + 128 * grp;                   // thread of the team
  const int c0 = grp * CG;                        // first column of this thread's column group
  const uint32_t lane_sel = (uint32_t)(w4 * 32) << 16;
  const uint32_t tm_s = tmem0 + tm * C::kTmTeam + C::kTmS + c0 + lane_sel;        // + plane * CP
  const uint32_t tm_o = tmem0 + tm * C::kTmTeam + C::kTmO + 4 * c0 + lane_sel;
  float* my_scal = reinterpret_cast<float*>(smem + C::kOffScal + tm * C::kTeamScal);
  float* qs_s = my_scal, *ref_s = my_scal + CP, *fac_s = my_scal + 2 * CP;
  int* lim_s = reinterpret_cast<int*>(my_scal + 3 * CP);
  float* amax_s = my_scal + 4 * CP;               // [team warps]
  const float* zero_s = my_scal + 5 * CP;         // [CP] zeros (never written after the set-up)
  float* my_red = my_scal + 8 * CP;               // [team warps][2 CG]
  float* my_lz = my_scal + 16 * CP;               // [2 CP]
  const int tw = grp * 4 + w4;                    // warp of the team
  Item* shared = reinterpret_cast<Item*>(misc + 64 + 16);   // [2] this CTA's first and last segment where others have part in it (zeroed)
  // named barriers of this team.  On bar_k and bar_p all but the issuing warp only arrive; each has an id of its own, so that
  // between two arrivals of a warp there lies a barrier at which all warps synchronise (the restart question): the phases stay apart
  // even if the waits for products in between have given up.
  static_assert(T <= 4, "barrier ids: 1.. bar_tm, 5.. bar_p, 9 and 14 all teams, 10.. bar_k");
  const int bar_tm = 1 + tm, bar_p = 5 + tm, bar_k = 10 + tm;
  const uint32_t vtile = sbase + tm * C::kTeamBytes, ptile = vtile + C::kTile;
  float* my_hdr = reinterpret_cast<float*>(smem + tm * C::kTeamBytes + C::kTile);   // [3 CP] l, zs, ref of this team's deposit (in its idle P tile)
  const uint32_t tm_k = tmem0 + tm * C::kTmTeam + C::kTmK;
  const int dim_out = 32 * (r >> 5) + 8 * ((r >> 2) & 3) + 2 * (r & 3) + ((r >> 4) & 1);   // head dim of lane r of O
  // this thread's row of the P tile: 16-byte chunk j goes to position j ^ p_swz
  const uint32_t p_swz = (uint32_t)r & 7u;
  const uint32_t p_row = ptile + (uint32_t)r * C::kPRow;
  const float cb = p.sm_log2;
  // descriptor low words of the MMA operands (used by the team's issuing thread)
  const uint32_t qd_lo0 = i8_desc_lo(sbase + C::kOffQT, 16u), vd_lo = i8_desc_lo(vtile, 16384u), pd_lo = i8_desc_lo(ptile, 16384u);
  constexpr uint32_t kQdHi = i8_desc_hi(1024u, 2u), kVdHi = i8_desc_hi(1024u, 2u), kPdHi = i8_desc_hi(8u * C::kPRow, 2u);
  uint32_t dep_cnt[T];                            // deposits made so far, per team (every team keeps the same count)
#pragma unroll
  for (int i = 0; i < T; ++i) dep_cnt[i] = 0;
  uint32_t my_deps = 0;                           // this team's own deposits
  bool ack_pending = false;                       // this team's last deposit (in its V tile) may not have been read yet

  int gs_base = 0, ic = 0;
  while (gs_base < n_units) {
    const int qi = ic & 1;
    mbar_wait<kItemAbort>(qfull0 + qi * 8, (ic >> 1) & 1, abort_word);
    const Item item = items[qi];
    const int len = item.len, n_piece = item.pad0;
    const int team0 = gs_base % T;                        // team of the piece's first unit
    const int u_first = (tm - team0 + T) % T;             // this team's units of the piece: u_first, u_first + T, ...
    const int team_f = (gs_base + n_piece - 1) % T;       // team of the piece's last unit: it writes the piece's result
    if (u_first < n_piece) {
      const bool finisher = tm == team_f;
      if (finisher && tt == 0 && item.n_contrib > 1) shared[gs_base == 0 ? 0 : 1] = item;   // (see behind the loop)
      const int full_lim = p.causal ? len - p.tail + 1 : len;
      // ---- the piece's queries: fixed-point exponent, sum of q per column, causal limits ----------
      const unsigned char* qb = qraw + qi * CP * 256;
      {
        const float am = i8_q_absmax(qb, tt, TT);
        if (lane == 0) amax_s[tw] = am;
        for (int c = tw; c < CP; c += C::kTeamWarps) {
          const uint2 v = *reinterpret_cast<const uint2*>(qb + c * 256 + lane * 8);
          float sum = (__uint_as_float(v.x << 16) + __uint_as_float(v.x & 0xFFFF0000u)) +
                      (__uint_as_float(v.y << 16) + __uint_as_float(v.y & 0xFFFF0000u));
#pragma unroll
          for (int off = 16; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
          if (lane == 0) qs_s[c] = sum;
        }
        if (tt < CP) lim_s[tt] = tt < p.ncols ? (p.causal ? len - p.tail + tt / p.G + 1 : len) : 0;
        named_bar(bar_tm, TT);
      }
      float amax = 0.0f;
#pragma unroll
      for (int i = 0; i < C::kTeamWarps; ++i) amax = fmaxf(amax, amax_s[i]);
      const int e = i8_q_exponent(amax);
      const float ca = p.sm_log2 * __int_as_float((127 - e) << 23) * 16.0f;
      const uint32_t qt = sbase + C::kOffQT + qi * C::kQTile;
      if (u_first == 0) {
        // this team owns the piece's first unit: it writes the three balanced s8 digit planes of
        // q_int = rint(q 2^e), rows plane * CP + column.  (The slot's previous planes belong to the piece
        // before last, which every team has left: the queries of this piece were loaded after that.)
        // Eight entries per thread and step: the first product of a launch waits for this.
        const float up = __int_as_float((127 + e) << 23);
        constexpr int NP = 3;
#pragma unroll 1
        for (int it = tt; it < CP * 16; it += TT) {
          const int c = it >> 4, j = (it >> 2) & 3, w = it & 3;   // column, 32 dims of the row, 8 of them
          const uint4 v = *reinterpret_cast<const uint4*>(qb + it * 16);
          const uint32_t ww[4] = {v.x, v.y, v.z, v.w};
          uint32_t acc[NP][2];
#pragma unroll
          for (int pln = 0; pln < NP; ++pln) { acc[pln][0] = 0; acc[pln][1] = 0; }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            int qv2[2];
#pragma unroll
            for (int par = 0; par < 2; ++par) {
              const float f = par ? __uint_as_float(ww[i] & 0xFFFF0000u) : __uint_as_float(ww[i] << 16);
              const int qv = __float2int_rn(f * up);
              qv2[par] = max(-4194303, min(4194303, qv));
            }
            // half 0 / 1 of the row: even / odd dims
#pragma unroll
            for (int par = 0; par < 2; ++par) {
              int qv = qv2[par];
#pragma unroll
              for (int pln = 0; pln < NP; ++pln) {
                const int dgt = (int)(signed char)(qv & 0xFF);
                acc[pln][par] |= (uint32_t)(dgt & 0xFF) << (8 * i);
                qv = (qv - dgt) >> 8;
              }
            }
          }
#pragma unroll
          for (int pln = 0; pln < NP; ++pln) {
            const int n = pln * CP + c;
#pragma unroll
            for (int par = 0; par < 2; ++par) {
              const int chunk = 2 * j + par;   // 16 bytes of the row's 128
              const uint32_t a = qt + (uint32_t)n * 128u + ((uint32_t)(chunk ^ (n & 7)) << 4) + 4u * w;
              asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(acc[pln][par]) : "memory");
            }
          }
        }
      }
      if (u_first == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(qready0 + qi * 8);
      }

      uint64_t l2[CG / 2], zs2[CG / 2];   // softmax sums, two columns per register pair
      float of_r[CG];                     // FP32 copy of O (tensor memory has no room for it)
#pragma unroll
      for (int c = 0; c < CG / 2; ++c) { l2[c] = 0ull; zs2[c] = 0ull; }
      bool fresh = true, have_of = false;
      int units_in_acc = 0;
      uint32_t n_own = (uint32_t)((gs_base + u_first) / T);   // index of the unit among this team's units

      // Ends the current accumulation (the team's last P.V is complete): the int32 accumulators, four
      // byte planes per column, are added to the FP32 copy and the sum is scaled by fac_s[] (the change
      // of the reference exponents).
      auto drain = [&](bool scale) {
        if (units_in_acc > 0) {
          tc_fence_after();
#pragma unroll
          for (int c4 = 0; c4 < CG / 4; ++c4) {
            uint32_t a[16];
            TmemRegs<16>::ld(tm_o + c4 * 16, a);
            tc_wait_ld();
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float v = fmaf(fmaf(fmaf((float)(int)a[4 * k + 3], 256.0f, (float)(int)a[4 * k + 2]), 256.0f,
                                        (float)(int)a[4 * k + 1]), 256.0f, (float)(int)a[4 * k]);
              const float old = !have_of ? 0.0f : of_r[c4 * 4 + k];
              of_r[c4 * 4 + k] = (old + v) * (scale ? fac_s[c0 + c4 * 4 + k] : 1.0f);
            }
          }
          have_of = true;
          units_in_acc = 0;
        } else if (have_of && scale) {
#pragma unroll
          for (int c = 0; c < CG; ++c) of_r[c] *= fac_s[c0 + c];
        }
      };

      // Metadata of this thread's token, read with plain loads two steps ahead: the block id of the unit
      // after next (a block-table look-up whose result is first touched one step later, so that nothing
      // waits for it), the (scale, zero) pairs of the next unit.
      auto blk_of = [&](int uu) -> int {      // the raw table entry (0 where there is no such token)
        const int t = (item.pad1 + uu) * C::kST + r;
        if (uu >= n_piece || t >= len) return 0;
        return ld_dep(p.block_table + (size_t)item.b * p.max_blocks + block_of(p, t));
      };
      auto row_of = [&](int uu, int blk) -> uint32_t {
        const int t = (item.pad1 + uu) * C::kST + r;
        if (uu >= n_piece || t >= len) return 0xFFFFFFFFu;
        const int in_blk = t - block_of(p, t) * p.bt;
        blk = min(max(blk, 0), p.num_blocks - 1);     // (out-of-range ids are reported by the producer)
        return (uint32_t)(((size_t)blk * p.Hkv + item.hkv) * p.bt + in_blk);
      };
      auto meta_of = [&](uint32_t row, float2& k2, float2& v2) {
        k2 = make_float2(0.f, 0.f); v2 = k2;
        if (row != 0xFFFFFFFFu) {
          k2 = ld_dep(reinterpret_cast<const float2*>(p.km) + row);
          v2 = ld_dep(reinterpret_cast<const float2*>(p.vm) + row);
        }
      };
      int blk_n1 = blk_of(u_first + T), blk_n2 = blk_of(u_first + 2 * T);
      float2 km_c, vm_c;
      meta_of(row_of(u_first, blk_of(u_first)), km_c, vm_c);

      for (int u = u_first; u < n_piece; u += T, ++n_own) {
        const int gs = gs_base + u, slot = gs % NSTAGE;
        const int unit_t0 = (item.pad1 + u) * C::kST;
        const int tok = unit_t0 + r;
        const uint32_t st = ring_u32 + slot * C::kStageBytes;
        // stages are shared between the teams: the wait for this stage's phase gs / NSTAGE is only well
        // defined once the phase before it is known to be complete (its owner says so in misc[32 + slot])
        if (gs >= NSTAGE && *reinterpret_cast<volatile int*>(misc + 32 + slot) < gs / NSTAGE)
          seq_wait(misc + 32 + slot, gs / NSTAGE, abort_word);
        mbar_wait(full0 + slot * 8, (gs / NSTAGE) & 1, abort_word);
        if (tt == 0) *reinterpret_cast<volatile int*>(misc + 32 + slot) = gs / NSTAGE + 1;
        float2 km = km_c, vm = vm_c;
        meta_of(row_of(u + T, blk_n1), km_c, vm_c);   // for this team's next unit
        blk_n1 = blk_n2;
        blk_n2 = blk_of(u + 3 * T);                   // and the block id of the one after the one after
        if (ack_pending) {   // uniform over the team: its last deposit (in the V tile) has been read
          if (tt == 0) seq_wait(misc + 24 + tm, (int)my_deps, abort_word);
          named_bar(bar_tm, TT);
          ack_pending = false;
        }
        // ---- K levels (free: the team's previous Q.K^T has been waited for), then Q.K^T; V tile (free
        // once the team's previous P.V is complete): one group expands K, the other V.
        if (grp == 0) {
          i8_expand_k_tmem<false, false>(st + C::kOffKA, 0u, r, tm_k + lane_sel);
          tc_wait_st();
        } else {
          if (n_own > 0) mbar_wait(pvdone0 + tm * 8, (n_own - 1) & 1, abort_word);
          i8_expand<false>(st + C::kOffVA, 0u, vtile, w4, lane);
        }
        tc_fence_before();
        // (only the issuing warp waits for the others' K levels: they go on to the V tile.  An elected lane issues: the
        // operands stay on the uniform datapath, see tc_elect.)
        if (tw != 0) bar_arrive(bar_k, TT);
        else named_bar(bar_k, TT);
        if (tw == 0) {
          if (u == u_first) mbar_wait(qready0 + qi * 8, (ic >> 1) & 1, abort_word);   // the piece's query planes
          tc_fence_after();
          if (tc_elect()) {
            const uint32_t d = tmem0 + tm * C::kTmTeam + C::kTmS;
            const uint32_t qd_lo = qd_lo0 + (uint32_t)qi * (C::kQTile >> 4);
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4)
              i8_mma_ts(d, tm_k + (uint32_t)k4 * 8u, i8_pack(qd_lo + (uint32_t)k4 * 2u, kQdHi), kIdescS, k4 > 0 ? 1u : 0u);
            tc_commit(sfull0 + tm * 8);
          }
        }
        __syncwarp();
        if (grp == 0 && n_own > 0) mbar_wait(pvdone0 + tm * 8, (n_own - 1) & 1, abort_word);   // (the other group has waited already)
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + slot * 8);
        const bool valid = tok < len;
        if (!valid) { km = make_float2(0.f, 0.f); vm = make_float2(0.f, 0.f); }
        const float sve = fmaxf(16.0f * vm.x, 9.094947e-13f);   // floor 2^-40
        const float al = km.x * ca;
        const float be = fmaf(km.x, 8.0f, km.y) * cb;
        const float lsv = lg2_approx(sve);
        const float ia = valid ? rcp_approx(sve) : 0.0f;
        const float ib = fmaf(vm.x, 8.0f, vm.y) * ia;

        // ---- scores of this thread's token -------------------------------------------------------
        mbar_wait(sfull0 + tm * 8, n_own & 1, abort_word);
        tc_fence_after();
        // y = log2 of the weight relative to the column's reference exponent, two columns per register pair
        uint64_t y2[CG / 2];
        {
          uint32_t s0[CG], s1[CG], s2[CG];
          TmemRegs<CG>::ld(tm_s, s0);
          TmemRegs<CG>::ld(tm_s + CP, s1);
          TmemRegs<CG>::ld(tm_s + 2 * CP, s2);
          tc_wait_ld();
          const uint64_t al2 = f2_pack(al, al), be2 = f2_pack(be, be), lsv2 = f2_pack(lsv, lsv);
          const uint64_t k256 = f2_pack(256.0f, 256.0f);
          const float* ref_r = fresh ? zero_s : ref_s;   // (a piece's first unit: relative to zero)
#pragma unroll
          for (int c = 0; c < CG / 2; ++c) {
            // the digit-plane sums put together: exact in int32 two planes at a time
            const uint64_t hi = f2_pack((float)((int)s2[2 * c] * 256 + (int)s1[2 * c]), (float)((int)s2[2 * c + 1] * 256 + (int)s1[2 * c + 1]));
            const uint64_t lo = f2_pack((float)(int)s0[2 * c], (float)(int)s0[2 * c + 1]);
            const uint64_t qs2 = *reinterpret_cast<const uint64_t*>(qs_s + c0 + 2 * c);
            const uint64_t rf2 = *reinterpret_cast<const uint64_t*>(ref_r + c0 + 2 * c);
            y2[c] = f2_fma(f2_fma(hi, k256, lo), al2, f2_fma(be2, qs2, f2_sub(lsv2, rf2)));
          }
        }
        if (unit_t0 + C::kST > full_lim) {
#pragma unroll
          for (int c = 0; c < CG / 2; ++c) {
            float a, b;
            f2_unpack(y2[c], a, b);
            if (tok >= lim_s[c0 + 2 * c]) a = -INFINITY;
            if (tok >= lim_s[c0 + 2 * c + 1]) b = -INFINITY;
            y2[c] = f2_pack(a, b);
          }
        }
        // ---- reference exponents: raised when a weight would leave the u32 range -----------------------
        float ymax = -INFINITY;
#pragma unroll
        for (int c = 0; c < CG / 2; ++c) {
          float a, b;
          f2_unpack(y2[c], a, b);
          ymax = max3(ymax, a, b);
        }
        // A restart of the accumulation (new reference exponents, the int32 sums drained into the FP32 copy) is a decision of the whole
        // team: one P.V covers all columns.
        const bool forced = fresh || units_in_acc >= C::kDrainUnits;   // uniform over the team
        const bool over = ymax > 31.5f;
        auto restart = [&]() {
#pragma unroll
          for (int c = 0; c < CG; ++c) {   // (rare path: back to absolute exponents x = y + ref)
            float a, b;
            f2_unpack(y2[c >> 1], a, b);
            const float mx = warp_max(((c & 1) ? b : a) + (fresh ? 0.0f : ref_s[c0 + c]));
            if (lane == 0) my_red[tw * CG + c] = mx;
          }
          named_bar(bar_tm, TT);
          if (tt < CP) {
            const float* mr = my_red + (tt / CG) * 4 * CG + (tt % CG);   // the four warps of the column's group
            const float mx = fmaxf(fmaxf(mr[0], mr[CG]), fmaxf(mr[2 * CG], mr[3 * CG]));
            const float old = fresh ? 0.0f : ref_s[tt];
            float nw = old, f = 1.0f;
            if (fresh) { nw = fmaxf(mx, -1.0e4f) - 28.0f; f = 0.0f; }
            else if (mx - old > 31.5f) { nw = mx - 28.0f; f = ex2_full(old - nw); }
            ref_s[tt] = nw;
            fac_s[tt] = f;
            my_red[C::kTeamWarps * CG + tt] = nw - old;   // what the change takes off every exponent of the column
          }
          named_bar(bar_tm, TT);
#pragma unroll
          for (int c = 0; c < CG / 2; ++c) {
            const uint64_t f2 = *reinterpret_cast<const uint64_t*>(fac_s + c0 + 2 * c);
            l2[c] = f2_mul(l2[c], f2);
            zs2[c] = f2_mul(zs2[c], f2);
            // the exponents again, relative to the new references
            const uint64_t od = *reinterpret_cast<const uint64_t*>(my_red + C::kTeamWarps * CG + c0 + 2 * c);
            y2[c] = f2_sub(y2[c], od);
          }
          drain(true);   // (the team's previous P.V has been waited for)
          fresh = false;
        };
        if (bar_or(bar_tm, TT, forced || over)) restart();
        // ---- weights of this thread's token into its row of the P tile -------------------------------------
        {
          uint32_t wi[CG];
          const uint64_t ia2 = f2_pack(ia, ia), ib2 = f2_pack(ib, ib);
#pragma unroll
          for (int c = 0; c < CG / 2; ++c) {
            float a, b;
            f2_unpack(y2[c], a, b);
            const float wa = ex2_ftz(a), wb = ex2_ftz(b);
            asm("cvt.rni.u32.f32 %0, %1;" : "=r"(wi[2 * c]) : "f"(wa));
            asm("cvt.rni.u32.f32 %0, %1;" : "=r"(wi[2 * c + 1]) : "f"(wb));
            const uint64_t w2 = f2_pack(wa, wb);
            l2[c] = f2_fma(w2, ia2, l2[c]);
            zs2[c] = f2_fma(w2, ib2, zs2[c]);
          }
#pragma unroll
          for (int j = 0; j < CG / 4; ++j)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                         ::"r"(p_row + (((uint32_t)(grp * (CG / 4) + j) ^ p_swz) << 4)), "r"(wi[4 * j]), "r"(wi[4 * j + 1]),
                           "r"(wi[4 * j + 2]), "r"(wi[4 * j + 3]) : "memory");
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          tc_fence_before();
          // the P tile and the V tile are complete, S has been read: the issuing warp waits for it
          if (tw != 0) bar_arrive(bar_p, TT);
          else named_bar(bar_p, TT);
        }
        if (tw == 0) {
          tc_fence_after();
          if (tc_elect()) {
            const uint32_t d = tmem0 + tm * C::kTmTeam + C::kTmO;
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4)
              i8_mma_ss(d, i8_pack(vd_lo + (uint32_t)k4 * (4096u >> 4), kVdHi),
                        i8_pack(pd_lo + (uint32_t)k4 * ((32u * C::kPRow) >> 4), kPdHi),
                        kIdescO, (units_in_acc > 0 || k4 > 0) ? 1u : 0u);
            tc_commit(pvdone0 + tm * 8);
          }
        }
        __syncwarp();
        ++units_in_acc;
      }
      // ---- end of the piece for this team -----------------------------------------------------------
      mbar_wait(pvdone0 + tm * 8, (n_own - 1) & 1, abort_word);   // the last P.V
      drain(false);   // the FP32 copy now holds this team's part of O
      float of[CG];
#pragma unroll
      for (int c = 0; c < CG; ++c) of[c] = of_r[c];
      tc_fence_before();
      // totals of l and zs over the 128 token lanes of every column group
      {
        float v[2 * CG];   // l of the group's columns, then zs
#pragma unroll
        for (int c = 0; c < CG / 2; ++c) {
          f2_unpack(l2[c], v[2 * c], v[2 * c + 1]);
          f2_unpack(zs2[c], v[CG + 2 * c], v[CG + 2 * c + 1]);
        }
        const float sum = warp_sums(v, lane);
        if ((lane & (32 / (2 * CG) - 1)) == 0) my_red[tw * 2 * CG + lane / (32 / (2 * CG))] = sum;
      }
      named_bar(bar_tm, TT);
      if (tt < 2 * CP) {   // my_lz: l of the CP columns, then zs
        const int which = tt / CP, c = tt % CP;
        const float* mr = my_red + (c / CG) * 4 * 2 * CG + which * CG + (c % CG);   // the four warps of the column's group
        my_lz[tt] = (mr[0] + mr[2 * CG]) + (mr[4 * CG] + mr[6 * CG]);
      }
      named_bar(bar_tm, TT);
      if (!finisher) {
        // deposit O in this team's V tile and (l, zs, ref) in its P tile (both idle: its last P.V is
        // complete), for the team that owns the piece's last unit
        float* mail = reinterpret_cast<float*>(smem + tm * C::kTeamBytes);
#pragma unroll
        for (int c = 0; c < CG; ++c) mail[(c0 + c) * 128 + r] = of[c];
        if (tt < CP) {
          my_hdr[tt] = my_lz[tt];
          my_hdr[CP + tt] = my_lz[CP + tt];
          my_hdr[2 * CP + tt] = ref_s[tt];
        }
        __threadfence_block();
        named_bar(bar_tm, TT);
        ++my_deps;
        if (tt == 0) *reinterpret_cast<volatile int*>(misc + 16 + tm) = (int)my_deps;
        ack_pending = true;
      } else {
        float lt[CG], zt[CG], mt[CG];
#pragma unroll
        for (int c = 0; c < CG; ++c) { lt[c] = my_lz[c0 + c]; zt[c] = my_lz[CP + c0 + c]; mt[c] = ref_s[c0 + c]; }
        // (one wait for all of them, one barrier before and one behind: team by team cost two barriers each)
        auto deposit = [&](int d) { return d != tm && (d - team0 + T) % T < n_piece; };   // (not itself, nor a team without a unit in the piece)
        if (tt == 0) {
#pragma unroll
          for (int d = 0; d < T; ++d)
            if (deposit(d)) seq_wait(misc + 16 + d, (int)dep_cnt[d] + 1, abort_word);
        }
        named_bar(bar_tm, TT);
#pragma unroll
        for (int d = 0; d < T; ++d) {
          if (!deposit(d)) continue;
          const float* mo = reinterpret_cast<const float*>(smem + d * C::kTeamBytes);
          const float* mh = reinterpret_cast<const float*>(smem + d * C::kTeamBytes + C::kTile);
#pragma unroll
          for (int c = 0; c < CG; ++c) {
            const float o2 = mo[(c0 + c) * 128 + r], l2 = mh[c0 + c];
            const float z2 = mh[CP + c0 + c], m2 = mh[2 * CP + c0 + c];
            const float M = fmaxf(mt[c], m2);
            const float f1 = ex2_full(mt[c] - M), f2 = ex2_full(m2 - M);
            of[c] = of[c] * f1 + o2 * f2;
            lt[c] = lt[c] * f1 + l2 * f2;
            zt[c] = zt[c] * f1 + z2 * f2;
            mt[c] = M;
          }
        }
        __threadfence_block();
        named_bar(bar_tm, TT);
        if (tt == 0) {
#pragma unroll
          for (int d = 0; d < T; ++d)
            if (deposit(d)) *reinterpret_cast<volatile int*>(misc + 24 + d) = (int)dep_cnt[d] + 1;   // it may deposit again
        }
        const bool direct = item.n_contrib == 1;
        const size_t bh = (size_t)item.b * p.Hkv + item.hkv;
        float* part = p.ws_part + (bh + (size_t)blockIdx.x) * (size_t)C::kPartCols * kPartStride;
#pragma unroll
        for (int cc = 0; cc < CG; ++cc) {
          const int c = c0 + cc;
          if (c >= p.ncols) break;
          const float v = of[cc] + zt[cc];
          if (direct) {
            const int j = c / p.G, hh = c % p.G;
            p.out[(((size_t)item.b * p.nq_stride + j) * p.Hq + item.hkv * p.G + hh) * LYNX_D + dim_out] =
                lt[cc] > 0.0f ? v / lt[cc] : 0.0f;
            if (r == 0) p.ws_lse[((size_t)item.b * p.nq_stride + j) * p.Hq + item.hkv * p.G + hh] = lse_of(mt[cc], lt[cc]);
          } else {
            part[(size_t)c * kPartStride + dim_out] = v;
            if (r == 0) *reinterpret_cast<float2*>(part + (size_t)c * kPartStride + 128) = make_float2(mt[cc], lt[cc]);
          }
        }
      }
    }
    // every team keeps count of every team's deposits (the phase of its deposit barrier)
#pragma unroll
    for (int d = 0; d < T; ++d)
      if (d != team_f && (d - team0 + T) % T < n_piece) ++dep_cnt[d];
    __syncwarp();
    if (lane == 0) mbar_arrive(qempty0 + qi * 8);
    gs_base += n_piece;
    ++ic;
  }
  // ---- release the tensor memory ---------------------------------------------------------------
  tc_fence_before();
  // (a thread sees what its own team has noted: whose slots are its own.  Here, not behind a piece, where it holds up the next: 12
  // ragged sequences of up to 9000 tokens, 8 columns, 36.5 -> 35.3 us)
  const auto any_shared = [&]() { return p.inline_merge && (shared[0].n_contrib > 1 || shared[1].n_contrib > 1); };
  if (any_shared()) __threadfence();
  named_bar(9, C::kThreads);   // (the producers have arrived there behind their last copy)
  if (any_shared()) i8_join_shared<C>(p, shared, tid, misc);
  if (warp == 0) {
    land_after_abort([] { return globaltimer_ns(); }, abort_word);
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem0), "r"((uint32_t)C::kTmCols)
                 : "memory");
  }
  if (tid == 0 && (misc[0] || misc[kItemAbort])) atomicOr(p.ws_flags, kFlagTimeout);
}

// Launches one of the persistent attention kernels: SMEM bytes, THREADS per CTA, units of ST tokens, at least MIN of them
// per CTA where a sequence has as many (and no more CTAs than SMs).
// The integer kernels take two: their teams or softmax groups do them side by side (by teams, one layer of 4096 tokens, 4 / 16 columns, us replayed from
// a graph: one unit per CTA 12.9 / 18.2, two 11.6 / 17.7, three 12.9 / 22.5, four 12.7 / 22.4; four by the CTA, whatever the
// sequences, as before: 17.2 / 36.0 for one sequence of 85 tokens, a CTA to itself for each head 8.5 / 17.7).  The FP16
// kernels take one (64 columns, 85 tokens: 18.5, four 90; two sequences of 189 tokens: 18.0, two 19.0, four 48).
template <bool FULL, class MAPS, int SMEM, int THREADS, int ST, int MIN, auto KERN>
lynx_status launch_units(AttnParams p, cudaStream_t st) {
  static bool configured[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    if (cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) != cudaSuccess)
      return LYNX_ERR_CUDA;
    configured[dev] = true;
  }
  // Programmatic dependent launch: when the kernel before this one in the stream is of the same kind (one
  // launch per layer of a decoder), this grid's CTAs may become resident, and set up their shared and tensor
  // memory, while the last CTAs of that kernel are still merging; they read nothing before
  // griddepcontrol.wait, i.e. before that kernel has completed and its memory is visible.
  cudaLaunchConfig_t cfg = {};
  const int grid = attention_grid(p, ST, MIN);
  plan_cut(&p, grid);
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  MAPS maps;
  const uint64_t plane_rows = (uint64_t)p.num_blocks * p.Hkv * p.bt;
  if (!i8_plane_map(&maps.m[0], p.ka, plane_rows, true) || !i8_plane_map(&maps.m[1], p.va, plane_rows, false))
    return LYNX_ERR_CUDA;
  if (FULL) {
    if (!i8_plane_map(&maps.m[2], p.kr, plane_rows, true) || !i8_plane_map(&maps.m[3], p.vr, plane_rows, false))
      return LYNX_ERR_CUDA;
  } else {
    maps.m[2] = maps.m[0];
    maps.m[3] = maps.m[1];
  }
  if constexpr (MAPS::kMeta)
    if (!meta_map(&maps.meta[0], p.km, plane_rows) || !meta_map(&maps.meta[1], p.vm, plane_rows)) return LYNX_ERR_CUDA;
  if (cudaLaunchKernelEx(&cfg, KERN, p, maps) != cudaSuccess) return LYNX_ERR_CUDA;
  return launch_status();
}

inline lynx_status launch_i8(const AttnParams& p, cudaStream_t st) {
  using C = I8Cfg;
  constexpr int kMin = 2;
  const lynx_status rc = launch_units<false, PlaneMaps, C::kSmem, C::kThreads, C::kST, kMin, attn_i8_kernel>(p, st);
  return rc != LYNX_OK ? rc : launch_combine(p, C::kPartCols, C::kST, kMin, st);
}
