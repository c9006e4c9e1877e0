// Anchor and merge-verify attention for up to 16 columns as a pipeline of specialised warps; the products are those of
// attention_i8.cuh (levels and weights as integers, tcgen05.mma kind::i8), see there.  Included by attention.cu inside its namespace.
//
// Warp roles, one CTA per SM; every hand-off is an mbarrier with a bounded wait, nothing waits on another CTA:
//   softmax      three or four warpgroups, a unit of 128 tokens in turn each: scores -> weights -> P tile (a thread owns a token)
//   K            four warps: K levels into tensor memory
//   V            four warps: V levels into a V tile
//   producers    two warps for the K ring, one for the V ring, one for the metadata's (see plane_producer)
//   products     a warp issues Q.K^T, another P.V
//   queries      two warps: a piece's queries as digit planes, a piece ahead
// Why stages and not teams that do everything for a unit (attn_i8_kernel): a team's unit is one chain of dependent steps, some 4500
// cycles, and registers, tensor memory and barriers allow three or four teams; here every stage works on units of its own, and what
// a unit takes is the longest stage, 600 to 1000 cycles.  us, teams -> stages: 16 layers of two sequences of 131072 tokens, 8
// columns, 912 -> 790 (before the power cap sets in; among other passes 1026 -> 963), one layer of 131072 tokens, 4 columns, 37.1 ->
// 35.0, of 4096 10.5 -> 9.4; 16 ragged sequences, 16 columns, 276 -> 243 (303 -> 283), 4 columns with a BF16 tail 166 -> 153; two
// sequences of 16000, 8 columns, 22.2 -> 19.4; verification of one layer of 4096 tokens, 16 columns, 16.8 -> 14.4.
//
// Exponents are relative to the column's largest weight and the weights scaled by 2^28 afterwards: an exponent of 28 would carry
// four times the rounding of one below 8.
//
// What bounds it: memory, 0.90-0.95 of the copy rate on long contexts, and on short ones the latency of the stages in a row.  What
// mattered on the way, us for 16 layers at 8 columns and for 16 ragged sequences at 16:
//   - metadata by gathers into a ring of its own: read by the softmax threads two units ahead, its latency was a third of their
//     time (986, 282 -> 886, 281); read ahead by two warps for all, in registers, 1475.
//   - producers that do little per unit (see plane_producer): 1054 -> 908 with copies in a row instead of a loop, 859 -> 821 and
//     273 -> 258 with gathers for V.
//   - softmax groups: two 886, 281, four and three 859, 273.
//   - both barriers of a stage probed at once, one commit per P.V, V tiles for three units: 821 -> 800, 258 -> 252.
//   - two P tiles per group at 16 columns: with one, the groups' weights and their products came to alternate, all groups waiting
//     for products and then all products for weights: 252 -> 243.  (At 4 and 8 columns groups hardly wait for products.)
template <bool FULL, int CP>
struct PipeCfg {
  static_assert(CP == 4 || CP == 8 || CP == 16, "padded column counts");
  static constexpr bool kFull = FULL;
  static constexpr int kST = 128, kSG = CP == 16 ? 3 : 4;
  static constexpr int kWarpK = 4 * kSG, kWarpV = kWarpK + 4, kWarpProd = kWarpV + 4, kWarpQK = kWarpProd + 4, kWarpPV = kWarpQK + 1, kWarpQ = kWarpPV + 1;
  static constexpr int kPartCols = CP < 8 ? 8 : CP;      // column stride of the partial slots
  // raw K bytes (see I8Cfg): at 8 columns, too, where the fourth digit plane is in the padding of N and K levels are a stage of their own
  static constexpr bool kRawK = !FULL && CP <= 8;
  static constexpr int kQPlanes = kRawK ? 4 : 3;
  static constexpr int kNQK = (kQPlanes * CP + 15) / 16 * 16, kNPV = 4 * CP;   // N of the products
  // Full codes enter less 128, as signed bytes: one operation per eight codes, and the sums of scores and values are no longer the
  // difference of two that are some thirty times larger.  Error against 64 bits, 1e-6 of the 2-norm, means of six draws, teams / stages
  // with whole codes / less 128: 4 ragged sequences of up to 32768, heavy-tailed, 16 columns 1.10 / 1.05 / 0.49; 2 of 20000, outliers, 8
  // columns 2.37 / 2.40 / 0.76; a mean of 132096 normal values 33 / 33 / 0.25.  1 % of the time of 16 ragged sequences.
  static constexpr uint32_t kFlip = FULL ? 0x88888888u : 0u;
  static constexpr uint32_t kSignedA = FULL ? 1u << 7 : 0u;   // of the instruction descriptors
  static constexpr bool kMetaRing = true;
  static constexpr int kNT = FULL && CP == 16 ? 6 : 8;                          // units whose metadata are kept: [kNT][K, V][128 tokens][scale, zero]
  // buffers of the scores and of K levels in tensor memory, V tiles, P tiles of a group, barriers of P.V
  static constexpr int kNB = CP == 16 ? 3 : 4, kNV = 3, kPB = CP == 16 ? 2 : 1, kNP = 4 * kPB;
  static constexpr int kStageBytes = kST * 64 * (FULL ? 2 : 1);   // Anchor (and Residual) of one tensor: [2][128 tokens][64 B]
  static constexpr int kVTile = 16384;                   // [128 tokens][128 B]
  static constexpr int kPRow = 4 * CP < 32 ? 32 : 4 * CP, kPTile = 128 * kPRow;
  static constexpr int kPLayout = kPRow == 32 ? 6 : kPRow == 64 ? 4 : 2;   // descriptor swizzle mode of the P tile
  static constexpr int kQTile = (kNQK * 128 + 1023) / 1024 * 1024;
  static constexpr int kOffV = 0, kOffP = kNV * kVTile, kOffQ = kOffP + kSG * kPB * kPTile, kOffMeta = kOffQ + 2 * kQTile, kOffRK = kOffMeta + kNT * 2048;
  // floats: qs[2][CP], limits[2][CP], exponents[2], maxima[2], zeros[CP]; per group: ref[CP], fac[CP], lz[2 CP], red[4][2 CP]
  static constexpr int kScal = 5 * CP + 4, kGrpScal = 12 * CP;
  static constexpr int kTail = (kScal + kSG * kGrpScal) * 4 + 24 * kI8PieceUnits * 4 + 2 * 32 + 88 * 8 + 256;
  static constexpr int kAvail = 227 * 1024 - 1024 - kOffRK - kTail;
  static constexpr int kStages = kAvail / kStageBytes > 16 ? 16 : kAvail / kStageBytes, kRingK = kStages / 2, kRingV = kStages - kRingK;
  static_assert(kRingK >= 3 && kRingV <= 8, "ring too small");
  static constexpr int kOffRV = kOffRK + kRingK * kStageBytes, kOffScal = kOffRV + kRingV * kStageBytes;
  static constexpr int kOffGrp = kOffScal + kScal * 4, kOffBlk = kOffGrp + kSG * kGrpScal * 4;
  static constexpr int kOffItems = kOffBlk + 24 * kI8PieceUnits * 4;
  static constexpr int kOffBars = kOffItems + 2 * 32, kOffMisc = kOffBars + 88 * 8;
  static constexpr int kSmem = kOffMisc + 256 + 1024;    // + alignment slack
  static_assert(kSmem <= 227 * 1024, "shared memory");
  static_assert(kOffGrp % 16 == 0 && kOffBlk % 16 == 0 && kOffBars % 8 == 0 && (CP % 4) == 0, "alignment");
  static_assert(CP * 512 <= kPTile, "the deposit lives in the group's P tile");
  static constexpr int kTmS = 0, kTmK = kNB * kNQK, kTmO = kTmK + kNB * 32, kTmOF = kTmO + kSG * kNPV;
  static_assert(kTmOF + kSG * CP <= 512, "tensor memory");
  static constexpr int kThreads = 32 * (kWarpQ + 2), kTeams = kSG, kTeamWarps = 4, kTeamThreads = 128;
  static constexpr int kDoneThreads = kSG * 128 + 128 + 64;   // softmax warpgroups, producers, products
  // A group's units between drains: a unit adds up to 128 * 128 * 255 to the sum of a byte plane of full codes, 128 * 240 * 255 of an
  // Anchor's odd dims, so that 514 or 274 could pass int32.
  static constexpr int kDrainUnits = 256;
  static_assert(128ll * (FULL ? 128 : 240) * 255 * kDrainUnits < 1ll << 31, "no sum overflows");
  // registers per thread after the split; launched with 72 or 64 each: 384 * 104 + 512 * 48, 512 * 80 + 512 * 48
  static constexpr int kRegSoft = kSG == 3 ? 104 : 80, kRegRest = 48;
};

template <int N>
struct TmemCols;   // (N consecutive columns of the thread's own lane, N a power of two up to 16)
template <> struct TmemCols<4> : TmemRegs<4> {};
template <> struct TmemCols<8> : TmemRegs<8> {};
template <> struct TmemCols<16> : TmemRegs<16> {};

template <bool FULL, int CP>
__global__ void __launch_bounds__(PipeCfg<FULL, CP>::kThreads, 1) attn_pipe_kernel(const AttnParams p, const __grid_constant__ PipeMaps maps) {
  using C = PipeCfg<FULL, CP>;
  constexpr int SG = C::kSG, NB = C::kNB, NV = C::kNV, NP = C::kNP, PB = C::kPB;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  float* scal = reinterpret_cast<float*>(smem + C::kOffScal);
  Item* items = reinterpret_cast<Item*>(smem + C::kOffItems);
  int* misc = reinterpret_cast<int*>(smem + C::kOffMisc);   // [0], [kItemAbort] abort, [1..3] joining, [7] units, [8] tensor memory base, [40 + ..] accumulate
  Item* shared = reinterpret_cast<Item*>(misc + 16);        // [2] this CTA's first and last segment where others have part in it
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);   // (known to be uniform)
  const uint32_t kfull = sbase + C::kOffBars, kempty = kfull + 64, vfull = kempty + 64, vempty = vfull + 64;   // [ring]
  const uint32_t qfull = vempty + 64, qempty = qfull + 16, qready = qempty + 16;   // [2]: piece published / left / queries in place
  const uint32_t kready = qready + 16, sfull = kready + 8 * NB, sfree = sfull + 8 * NB;   // [NB]: K in TMEM / scores valid / scores read
  const uint32_t vready = sfree + 8 * NB, pready = vready + 8 * NV;                // [NV]: V tile written, [group][PB]: weights written
  const uint32_t pvdone = pready + 8 * SG * PB;                                         // [NP]: P.V of a unit complete, P and V tile free
  static_assert(NP >= SG * PB && NP >= NV, "no unit's phase passes before it has been waited for");
  const uint32_t mfull = pvdone + 8 * NP, mfree = mfull + 8 * C::kNT;              // [kNT]: metadata there / read
  static_assert(4 * 8 + 6 + 3 * NB + NV + SG * PB + NP + 2 * C::kNT <= 88, "barriers");
  volatile int* abort_word = misc;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == C::kWarpProd && lane < 4) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.m[lane])) : "memory");
  if (tid == 0) {
    for (int i = 0; i < C::kRingK; ++i) { mbar_init(kfull + i * 8, 2); mbar_init(kempty + i * 8, 4); }
    for (int i = 0; i < C::kRingV; ++i) { mbar_init(vfull + i * 8, 1); mbar_init(vempty + i * 8, 4); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(qfull + i * 8, 1);
      mbar_init(qempty + i * 8, 4 * SG + 3);
      mbar_init(qready + i * 8, 2);
    }
    for (int i = 0; i < NB; ++i) { mbar_init(kready + i * 8, 4); mbar_init(sfull + i * 8, 1); mbar_init(sfree + i * 8, 4); }
    for (int i = 0; i < NV; ++i) mbar_init(vready + i * 8, 4);
    for (int i = 0; i < SG * PB; ++i) mbar_init(pready + i * 8, 4);
    for (int i = 0; i < NP; ++i) mbar_init(pvdone + i * 8, 1);
    for (int i = 0; i < C::kNT; ++i) { mbar_init(mfull + i * 8, 1); mbar_init(mfree + i * 8, 4); }
    for (int i = 0; i < 64; ++i) misc[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < C::kScal + SG * C::kGrpScal; i += C::kThreads) scal[i] = 0.0f;
  for (int i = tid; i < 2 * C::kQTile / 16; i += C::kThreads)   // (padding rows of the digit planes)
    reinterpret_cast<uint4*>(smem + C::kOffQ)[i] = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(misc + 8)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem0 = __shfl_sync(0xFFFFFFFFu, *reinterpret_cast<volatile uint32_t*>(misc + 8), 0);
  // nothing in global memory has been touched so far: wait for the grids this one depends on
  // ================================================================================== producers
  if (warp >= C::kWarpProd && warp < C::kWarpQK) {
    reg_dec<C::kRegRest>();
    const int pw = warp - C::kWarpProd;
    const SkPlace at = sk_place(p, blockIdx.x);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const SeqLens sl(p, lane);
    const SkRange rng = sk_range<C::kST>(p, gridDim.x, blockIdx.x, lane, sl, at);
    const int n_units = rng.lo < rng.hi ? (int)(rng.hi - rng.lo) : 0;
    if (pw == 0 && lane == 0) misc[7] = n_units;
    __syncwarp();
    bar_arrive(7, C::kThreads);   // the range is published (the producers know it and do not wait)
    if (n_units == 0) bar_arrive(9, C::kDoneThreads);
    else
      plane_producer<C>(p, rng, sl, pw, lane, sbase, pw < 2 ? kfull : pw == 2 ? vfull : mfull, pw < 2 ? kempty : pw == 2 ? vempty : mfree,
                        pw < 2 ? C::kRingK : pw == 2 ? C::kRingV : C::kNT, qfull, qempty,
                        reinterpret_cast<uint32_t*>(smem + C::kOffBlk), items, abort_word, &maps, 9);
    if (pw == kPublisher) per_sequence<FULL, C::kPartCols>(p, blockIdx.x, gridDim.x, lane, sl, n_units ? items : nullptr);
    return;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  named_bar(7, C::kThreads);
  const int n_units = misc[7];

  // ================================================================================== softmax warpgroups
  if (warp < C::kWarpK) {
    reg_inc<C::kRegSoft>();
    const int g = warp >> 2, w4 = warp & 3, r = tid & 127;   // r: token of the unit (S), dim position (O): TMEM lane
    const uint32_t lane_sel = (uint32_t)(w4 * 32) << 16;
    const uint32_t tm_s = tmem0 + C::kTmS + lane_sel, tm_o = tmem0 + C::kTmO + g * C::kNPV + lane_sel,
                   tm_of = tmem0 + C::kTmOF + g * CP + lane_sel;
    float* grp = reinterpret_cast<float*>(smem + C::kOffGrp) + g * C::kGrpScal;
    float *ref_s = grp, *fac_s = grp + CP, *lz_s = grp + 2 * CP, *red_s = grp + 4 * CP;
    const float* zero_s = scal + 4 * CP + 4;        // [CP] zeros (never written after the set-up)
    const int bar_g = 1 + g;
    const uint32_t p_swz = C::kPRow == 32 ? ((uint32_t)r >> 2) & 1u : C::kPRow == 64 ? ((uint32_t)r >> 1) & 3u : (uint32_t)r & 7u;
    const uint32_t p_row = sbase + C::kOffP + g * PB * C::kPTile + (uint32_t)r * C::kPRow;   // 16-byte chunk j goes to position j ^ p_swz
    const int dim_out = 32 * (r >> 5) + 8 * ((r >> 2) & 3) + 2 * (r & 3) + ((r >> 4) & 1);   // head dim of lane r of O
    const float cb = p.sm_log2, unit = !FULL && ((r >> 4) & 1) ? 0x1p-32f : 0x1p-28f;   // of the sums (odd dims of the Anchor: 16 times their levels)
    const float2* meta = reinterpret_cast<const float2*>(smem + C::kOffMeta) + r;   // [unit][K, V][128]
    int gs_base = 0, ic = 0;
    while (gs_base < n_units) {
      const int qi = ic & 1;
      mbar_wait_in(qfull + qi * 8, (ic >> 1) & 1, abort_word + kItemAbort);
      const Item item = items[qi];
      const int len = item.len, n_piece = item.pad0;
      const int u_first = (g + SG - gs_base % SG) % SG;
      const bool have = u_first < n_piece;
      if (!FULL && tid == 0 && item.n_contrib > 1) shared[gs_base == 0 ? 0 : 1] = item;   // (see behind the loop)
      uint64_t l2[CP / 2], zs2[CP / 2];             // softmax sums of this thread's tokens, two columns per register pair
#pragma unroll
      for (int c = 0; c < CP / 2; ++c) { l2[c] = 0ull; zs2[c] = 0ull; }
      bool have_of = false;
      int units_in_acc = 0;
      // Ends the current accumulation (the group's last P.V is complete): the int32 accumulators, four byte planes per column,
      // are added to the FP32 copy, scaled by fac_s[] (the change of the reference exponents).
      auto sums = [&](int c4, float* o) {   // columns 4 c4 .. + 3
        uint32_t a[16], of[4];
        TmemRegs<16>::ld(tm_o + c4 * 16, a);
        TmemRegs<4>::ld(tm_of + c4 * 4, of);
        tc_wait_ld();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float v = fmaf(fmaf(fmaf((float)(int)a[4 * k + 3], 256.0f, (float)(int)a[4 * k + 2]), 256.0f,
                              (float)(int)a[4 * k + 1]), 256.0f, (float)(int)a[4 * k]);
          v *= unit;
          if (units_in_acc == 0) v = 0.0f;   // (the accumulators have not been restarted since the last drain)
          o[k] = have_of ? v + __uint_as_float(of[k]) : v;
        }
      };
      auto drain = [&]() {
        tc_fence_after();
#pragma unroll 1
        for (int c4 = 0; c4 < CP / 4; ++c4) {
          float o[4];
          uint32_t of[4];
          sums(c4, o);
#pragma unroll
          for (int k = 0; k < 4; ++k) of[k] = __float_as_uint(o[k] * fac_s[c4 * 4 + k]);
          TmemRegs<4>::st(tm_of + c4 * 4, of);
        }
        tc_wait_st();
        have_of = true;
        units_in_acc = 0;
      };
      if (have) {
        const int full_lim = p.causal ? len - p.tail + 1 : len;
        const float* qs_s = scal + qi * CP;
        const int* lim_s = reinterpret_cast<const int*>(scal + 2 * CP + qi * CP);
        bool fresh = true;
        mbar_wait_in(qready + qi * 8, (ic >> 1) & 1, abort_word);
        const int e = reinterpret_cast<const int*>(scal)[4 * CP + qi];
        const float ca = p.sm_log2 * __int_as_float((127 - e) << 23) * ((FULL || C::kRawK) ? 1.0f : 16.0f);
        int last = 0;
        for (int u = u_first; u < n_piece; u += SG) {
          const int gs = gs_base + u, sb = gs % NB;
          last = gs;
          const int unit_t0 = (item.pad1 + u) * C::kST, tok = unit_t0 + r;
          // ---- scores: y = log2 of the weight relative to the column's reference exponent --------------
          const int mt = gs % C::kNT;
          mbar_wait2_in(mfull + mt * 8, (gs / C::kNT) & 1, sfull + sb * 8, (gs / NB) & 1, abort_word);
          tc_fence_after();
          float2 km = meta[mt * 256], vm = meta[mt * 256 + 128];
          const bool valid = tok < len;
          if (!valid) { km = make_float2(0.f, 0.f); vm = make_float2(0.f, 0.f); }
          const float sve = fmaxf(FULL ? vm.x : 16.0f * vm.x, 9.094947e-13f);   // floor 2^-40
          const float al = km.x * ca;
          const float be = fmaf(km.x, FULL ? 128.0f : 8.0f, km.y) * cb;
          const float lsv = lg2_approx(sve);
          const float ia = valid ? rcp_approx(sve) : 0.0f;
          const float ib = (FULL ? fmaf(sve, 128.0f, vm.y) : fmaf(vm.x, 8.0f, vm.y)) * ia;
          uint64_t y2[CP / 2];
          {
            uint32_t s0[CP], s1[CP], s2[CP], s3[C::kRawK ? CP : 1];
            const uint32_t a = tm_s + sb * C::kNQK;
            TmemCols<CP>::ld(a, s0);
            TmemCols<CP>::ld(a + CP, s1);
            TmemCols<CP>::ld(a + 2 * CP, s2);
            if (C::kRawK) TmemCols<CP>::ld(a + 3 * CP, s3);
            tc_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { mbar_arrive(sfree + sb * 8); mbar_arrive(mfree + mt * 8); }   // the scores have been read, and the metadata
            const uint64_t al2 = f2_pack(al, al), be2 = f2_pack(be, be), lsv2 = f2_pack(lsv, lsv);
            const uint64_t k256 = C::kRawK ? f2_pack(65536.0f, 65536.0f) : f2_pack(256.0f, 256.0f);
            const float* ref_r = fresh ? zero_s : ref_s;   // (a piece's first unit: relative to zero)
#pragma unroll
            for (int c = 0; c < CP / 2; ++c) {
              uint64_t hi, lo;   // the digit-plane sums put together: exact in int32 two planes at a time
              if (C::kRawK) {
                hi = f2_pack((float)((int)s3[2 * c] * 256 + (int)s2[2 * c]), (float)((int)s3[2 * c + 1] * 256 + (int)s2[2 * c + 1]));
                lo = f2_pack((float)((int)s1[2 * c] * 256 + (int)s0[2 * c]), (float)((int)s1[2 * c + 1] * 256 + (int)s0[2 * c + 1]));
              } else {
                hi = f2_pack((float)((int)s2[2 * c] * 256 + (int)s1[2 * c]), (float)((int)s2[2 * c + 1] * 256 + (int)s1[2 * c + 1]));
                lo = f2_pack((float)(int)s0[2 * c], (float)(int)s0[2 * c + 1]);
              }
              const uint64_t qs2 = *reinterpret_cast<const uint64_t*>(qs_s + 2 * c);
              const uint64_t rf2 = *reinterpret_cast<const uint64_t*>(ref_r + 2 * c);
              y2[c] = f2_fma(f2_fma(hi, k256, lo), al2, f2_fma(be2, qs2, f2_sub(lsv2, rf2)));
            }
          }
          if (unit_t0 + C::kST > full_lim) {
#pragma unroll
            for (int c = 0; c < CP / 2; ++c) {
              float a, b;
              f2_unpack(y2[c], a, b);
              if (tok >= lim_s[2 * c]) a = -INFINITY;
              if (tok >= lim_s[2 * c + 1]) b = -INFINITY;
              y2[c] = f2_pack(a, b);
            }
          }
          float ymax = -INFINITY;
#pragma unroll
          for (int c = 0; c < CP / 2; ++c) {
            float a, b;
            f2_unpack(y2[c], a, b);
            ymax = max3(ymax, a, b);
          }
          const int pb = gs / SG % PB;
          if (gs >= SG * PB) mbar_wait_in(pvdone + ((gs - SG * PB) % NP) * 8, ((gs - SG * PB) / NP) & 1, abort_word);   // P free
          // ---- a piece's first unit, a weight that would leave the u32 range, sums about to overflow: new references ----
          if (bar_or(bar_g, 128, fresh || units_in_acc >= C::kDrainUnits || ymax > 3.5f)) {
            // (By exchanging halves, as the sums: a maximum per column and instruction took 2 us of a piece at 16 columns, now 0.9; 64
            // sequences of 16 tokens 27.2 -> 24.1 us, 16 ragged long ones 242 -> 241; verification at 8 columns 23.6 -> 22.7.  At 4 columns 1 %
            // slower, Anchor at 8 0.5 % on long contexts.)
            if constexpr (CP == 16 || (FULL && CP == 8)) {
              float x[CP];   // (back to absolute exponents x = y + ref)
#pragma unroll
              for (int c = 0; c < CP / 2; ++c) {
                f2_unpack(y2[c], x[2 * c], x[2 * c + 1]);
                if (!fresh) { x[2 * c] += ref_s[2 * c]; x[2 * c + 1] += ref_s[2 * c + 1]; }
              }
              const float top = warp_halves(x, lane, [](float u, float v) { return fmaxf(u, v); });
              if ((lane & (32 / CP - 1)) == 0) red_s[w4 * CP + lane / (32 / CP)] = top;
            } else {
#pragma unroll
              for (int c = 0; c < CP; ++c) {
                float a, b;
                f2_unpack(y2[c >> 1], a, b);
                const float top = warp_max(((c & 1) ? b : a) + (fresh ? 0.0f : ref_s[c]));
                if (lane == 0) red_s[w4 * CP + c] = top;
              }
            }
            named_bar(bar_g, 128);
            if (r < CP) {
              const float mx = fmaxf(fmaxf(red_s[r], red_s[CP + r]), fmaxf(red_s[2 * CP + r], red_s[3 * CP + r]));
              const float old = fresh ? 0.0f : ref_s[r];
              float nw = old, f = 1.0f;
              if (fresh) { nw = fmaxf(mx, -1.0e4f); f = 0.0f; }
              else if (mx > old) { nw = mx; f = ex2_full(old - nw); }
              ref_s[r] = nw;
              fac_s[r] = f;
              red_s[4 * CP + r] = nw - old;   // what the change takes off every exponent of the column
            }
            named_bar(bar_g, 128);
#pragma unroll
            for (int c = 0; c < CP / 2; ++c) {
              const uint64_t f2 = *reinterpret_cast<const uint64_t*>(fac_s + 2 * c);
              l2[c] = f2_mul(l2[c], f2);
              zs2[c] = f2_mul(zs2[c], f2);
              y2[c] = f2_sub(y2[c], *reinterpret_cast<const uint64_t*>(red_s + 4 * CP + 2 * c));
            }
            if (!fresh) {
              if (PB > 1) mbar_wait_in(pvdone + ((gs - SG) % NP) * 8, ((gs - SG) / NP) & 1, abort_word);   // accumulators current
              drain();
            }
            fresh = false;
          }
          // ---- weights of this thread's token into its row of the P tile ----------------------------------
          {
            uint32_t wi[CP];
            const uint64_t ia2 = f2_pack(ia, ia), ib2 = f2_pack(ib, ib);
#pragma unroll
            for (int c = 0; c < CP / 2; ++c) {
              float a, b;
              f2_unpack(y2[c], a, b);
              const float wa = ex2_ftz(a), wb = ex2_ftz(b);
              const uint64_t w2 = f2_pack(wa, wb);
              f2_unpack(f2_mul(w2, f2_pack(0x1p28f, 0x1p28f)), a, b);
              asm("cvt.rni.u32.f32 %0, %1;" : "=r"(wi[2 * c]) : "f"(a));
              asm("cvt.rni.u32.f32 %0, %1;" : "=r"(wi[2 * c + 1]) : "f"(b));
              l2[c] = f2_fma(w2, ia2, l2[c]);
              zs2[c] = f2_fma(w2, ib2, zs2[c]);
            }
#pragma unroll
            for (int j = 0; j < CP / 4; ++j)
              sts128(p_row + pb * C::kPTile + (((uint32_t)j ^ p_swz) << 4), wi[4 * j], wi[4 * j + 1], wi[4 * j + 2], wi[4 * j + 3]);
          }
          if (r == 0) misc[40 + g * PB + pb] = units_in_acc > 0 ? 1 : 0;
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(pready + (g * PB + pb) * 8);
          ++units_in_acc;
        }
        mbar_wait_in(pvdone + (last % NP) * 8, (last / NP) & 1, abort_word);   // the last P.V
        tc_fence_after();
      }
      // ---- end of the piece: totals over the 128 tokens of a unit, then the result -------------------------
      float of[CP];
      if (have) {
#pragma unroll
        for (int c4 = 0; c4 < CP / 4; ++c4) sums(c4, of + 4 * c4);
        float v[2 * CP];   // l of the columns, then zs
#pragma unroll
        for (int c = 0; c < CP / 2; ++c) {
          f2_unpack(l2[c], v[2 * c], v[2 * c + 1]);
          f2_unpack(zs2[c], v[CP + 2 * c], v[CP + 2 * c + 1]);
        }
        const float sum = warp_sums(v, lane);
        if ((lane & (32 / (2 * CP) - 1)) == 0) red_s[w4 * 2 * CP + lane / (32 / (2 * CP))] = sum;
        named_bar(bar_g, 128);
        if (r < 2 * CP) lz_s[r] = (red_s[r] + red_s[2 * CP + r]) + (red_s[4 * CP + r] + red_s[6 * CP + r]);
      } else {
#pragma unroll
        for (int c = 0; c < CP; ++c) of[c] = 0.0f;
        if (r < 2 * CP) lz_s[r] = 0.0f;
        if (r < CP) ref_s[r] = -INFINITY;
      }
      // every group leaves its sums in its idle P tile, and joins and writes a share of the columns
      {
        constexpr int H = (CP + SG - 1) / SG;
        float* mail = reinterpret_cast<float*>(smem + C::kOffP + g * PB * C::kPTile);
#pragma unroll
        for (int c = 0; c < CP; ++c) mail[c * 128 + r] = of[c];
        named_bar(5, SG * 128);
        const bool direct = item.n_contrib == 1;
        float* part = p.ws_part + ((size_t)item.b * p.Hkv + item.hkv + (size_t)blockIdx.x) * (size_t)C::kPartCols * kPartStride;
        const float* grps = reinterpret_cast<const float*>(smem + C::kOffGrp);
        const float* mails = reinterpret_cast<const float*>(smem + C::kOffP) + r;
        const int c0 = g * H, nc = min(H, p.ncols - c0);
        // what is the same for all 128 dims of column c: the groups' factors, its sums, its row
        struct { float f[SG], z, l; uint32_t row; } t;
        const auto look = [&](int c, bool leads) {
          float M = grps[c];
#pragma unroll
          for (int i = 1; i < SG; ++i) M = fmaxf(M, grps[i * C::kGrpScal + c]);
          t.l = t.z = 0.0f;
#pragma unroll
          for (int i = 0; i < SG; ++i) {
            const float* gi = grps + i * C::kGrpScal + c;
            t.f[i] = ex2_full(gi[0] - M);
            t.l = fmaf(gi[2 * CP], t.f[i], t.l);
            t.z = fmaf(gi[3 * CP], t.f[i], t.z);
          }
          t.row = 0;
          if (direct) {
            const int j = c / p.G, hh = c - j * p.G;
            t.row = (uint32_t)((item.b * p.nq_stride + j) * p.Hq + item.hkv * p.G + hh);
            if (leads) p.ws_lse[t.row] = lse_of(M, t.l);
          } else if (leads) {
            *reinterpret_cast<float2*>(part + (size_t)c * kPartStride + 128) = make_float2(M, t.l);
          }
        };
        const auto put = [&](int c) {
          float o = 0.0f;
#pragma unroll
          for (int i = 0; i < SG; ++i) o = fmaf(mails[i * (PB * C::kPTile / 4) + c * 128], t.f[i], o);
          const float v = o + t.z;
          if (direct) p.out[(size_t)t.row * LYNX_D + dim_out] = t.l > 0.0f ? v / t.l : 0.0f;
          else part[(size_t)c * kPartStride + dim_out] = v;
        };
        if constexpr (H > 1) {
          // By a thread per column: the instructions of a piece's end share the schedulers with 27 other warps, and every thread for itself
          // took 2.1 us at 16 columns, of the 6.7 for a piece of one unit (64 sequences of 16 tokens 27.2 us, 31.5 by every thread).
          static_assert(8 * H <= 8 * CP && SG <= 4, "room for the columns' scalars");
          if (r < nc) {
            look(c0 + r, true);
#pragma unroll
            for (int i = 0; i < SG; ++i) red_s[8 * r + i] = t.f[i];
            *reinterpret_cast<float4*>(red_s + 8 * r + 4) = make_float4(t.z, t.l, __uint_as_float(t.row), 0.0f);
          }
          named_bar(bar_g, 128);
          // (rolled: three columns at a time 231 -> 238 us for 16 ragged sequences at 16 columns, for the instruction caches)
#pragma unroll 1
          for (int i = 0; i < nc; ++i) {
            const float4 f = *reinterpret_cast<const float4*>(red_s + 8 * i), zl = *reinterpret_cast<const float4*>(red_s + 8 * i + 4);
            const float fs[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int k = 0; k < SG; ++k) t.f[k] = fs[k];
            t.z = zl.x;
            t.l = zl.y;
            t.row = __float_as_uint(zl.z);
            put(c0 + i);
          }
        } else if (nc > 0) {   // (a group's only column: not worth a barrier, 77.4 -> 74.6 us for 512 sequences of 16 tokens at 4 columns)
          look(c0, r == 0);
          put(c0);
        }
      }
      tc_fence_before();
      named_bar(5, SG * 128);   // (the mail and the groups' totals have been read)
      if (lane == 0) mbar_arrive(qempty + qi * 8);
      gs_base += n_piece;
      ++ic;
    }
    // ---- release the tensor memory: every product has been waited for, and the warps that issue copies and products are done
    tc_fence_before();
    const auto any_shared = [&]() { return !FULL && p.inline_merge && (shared[0].n_contrib > 1 || shared[1].n_contrib > 1); };
    if (n_units > 0 && any_shared()) __threadfence();
    named_bar(9, C::kDoneThreads);
    if (n_units > 0 && any_shared()) i8_join_shared<C>(p, shared, tid, misc);
    if (warp == 0) {
      land_after_abort([] { return globaltimer_ns(); }, abort_word);
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem0), "r"(512u) : "memory");
    }
    if (tid == 0 && (misc[0] || misc[kItemAbort])) atomicOr(p.ws_flags, kFlagTimeout);
    return;
  }
  // ================================================================================== K levels
  if (warp < C::kWarpV) {
    reg_dec<C::kRegRest>();
    const int kt = tid - C::kWarpK * 32, w4 = warp & 3;
    const uint32_t tm_k = tmem0 + C::kTmK + ((uint32_t)(w4 * 32) << 16);
    int slot = 0;
    uint32_t phase = 0;
    for (int gs = 0; gs < n_units; ++gs) {
      const int sb = gs % NB;
      mbar_wait2_in(kfull + slot * 8, phase, sfull + sb * 8, ((gs / NB) - 1) & 1, abort_word);   // and Q.K^T of the unit that was here before
      tc_fence_after();
      const uint32_t raw = sbase + C::kOffRK + (uint32_t)slot * C::kStageBytes;
      i8_expand_k_tmem<FULL, C::kRawK, C::kFlip>(raw, raw + 8192u, kt, tm_k + (uint32_t)sb * 32u);
      __syncwarp();
      if (lane == 0) mbar_arrive(kempty + slot * 8);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(kready + sb * 8);
      if (++slot == C::kRingK) { slot = 0; phase ^= 1; }
    }
    return;
  }
  // ================================================================================== V levels
  if (warp < C::kWarpProd) {
    reg_dec<C::kRegRest>();
    int slot = 0;
    uint32_t phase = 0;
    for (int gs = 0; gs < n_units; ++gs) {
      const int vb = gs % NV;
      // (the tile's previous product; before there was one: of a phase that a fresh barrier passes)
      mbar_wait2_in(vfull + slot * 8, phase, pvdone + ((gs + NP - NV) % NP) * 8, ((gs + NP - NV) / NP - 1) & 1, abort_word);
      const uint32_t raw = sbase + C::kOffRV + (uint32_t)slot * C::kStageBytes;
      i8_expand<FULL, !FULL, C::kFlip>(raw, raw + 8192u, sbase + C::kOffV + (uint32_t)vb * C::kVTile, warp & 3, lane);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) { mbar_arrive(vempty + slot * 8); mbar_arrive(vready + vb * 8); }
      if (++slot == C::kRingV) { slot = 0; phase ^= 1; }
    }
    return;
  }
  reg_dec<C::kRegRest>();
  // ================================================================================== Q.K^T
  constexpr uint32_t kHi = i8_desc_hi(1024u, 2u), kPdHi = i8_desc_hi(8u * C::kPRow, (uint32_t)C::kPLayout);
  if (warp == C::kWarpQK) {
    constexpr uint32_t kIdescS = i8_idesc(C::kNQK, false, true) | C::kSignedA;
    const uint32_t q_lo = i8_desc_lo(sbase + C::kOffQ, 16u);
    int gs = 0, ic = 0;
    while (gs < n_units) {
      const int qi = ic & 1;
      mbar_wait_in(qfull + qi * 8, (ic >> 1) & 1, abort_word + kItemAbort);
      const int n_piece = items[qi].pad0;
      mbar_wait_in(qready + qi * 8, (ic >> 1) & 1, abort_word);
#pragma unroll 1
      for (int u = 0; u < n_piece; ++u, ++gs) {
        const int sb = gs % NB;
        mbar_wait2_in(kready + sb * 8, (gs / NB) & 1, sfree + sb * 8, ((gs / NB) - 1) & 1, abort_word);
        tc_fence_after();
        if (tc_elect()) {
          const uint32_t d = tmem0 + C::kTmS + sb * C::kNQK, a = tmem0 + C::kTmK + sb * 32, q = q_lo + (uint32_t)qi * (C::kQTile >> 4);
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4) i8_mma_ts(d, a + k4 * 8u, i8_pack(q + k4 * 2u, kHi), kIdescS, k4 > 0 ? 1u : 0u);
          tc_commit(sfull + sb * 8);
        }
        __syncwarp();
      }
      if (lane == 0) mbar_arrive(qempty + qi * 8);
      ++ic;
    }
    bar_arrive(9, C::kDoneThreads);
    return;
  }
  // ================================================================================== P.V
  if (warp == C::kWarpPV) {
    constexpr uint32_t kIdescO = i8_idesc(C::kNPV, true, false) | C::kSignedA;
    const uint32_t v_lo = i8_desc_lo(sbase + C::kOffV, 16384u), p_lo = i8_desc_lo(sbase + C::kOffP, 16384u);
#pragma unroll 1
    for (int gs = 0; gs < n_units; ++gs) {
      const int vb = gs % NV, g = gs % SG, gb = g * PB + gs / SG % PB;
      mbar_wait2_in(vready + vb * 8, (gs / NV) & 1, pready + gb * 8, (gs / (SG * PB)) & 1, abort_word);
      tc_fence_after();
      const uint32_t acc = *reinterpret_cast<volatile int*>(misc + 40 + gb) ? 1u : 0u;
      if (tc_elect()) {
        const uint32_t d = tmem0 + C::kTmO + g * C::kNPV, vl = v_lo + vb * (C::kVTile >> 4), pl = p_lo + gb * (C::kPTile >> 4);
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4)
          i8_mma_ss(d, i8_pack(vl + k4 * (4096u >> 4), kHi), i8_pack(pl + k4 * ((32u * C::kPRow) >> 4), kPdHi), kIdescO, k4 > 0 ? 1u : acc);
        tc_commit(pvdone + (gs % NP) * 8);
      }
      __syncwarp();
    }
    bar_arrive(9, C::kDoneThreads);
    return;
  }
  // ================================================================================== queries
  // Thread qt of 64 has the 16-byte chunks qt & 15 of columns qt >> 4, + 4, ...: 8 entries each
  {
    constexpr int NI = CP / 4, NP = C::kQPlanes;
    const int qt = tid - C::kWarpQ * 32;
    const uint32_t g_inv = 65536u / (uint32_t)p.G + 1u;   // c / G = c * g_inv >> 16 for c < 64, G <= 16
    int gs = 0, ic = 0;
    while (gs < n_units) {
      const int qi = ic & 1;
      mbar_wait_in(qfull + qi * 8, (ic >> 1) & 1, abort_word + kItemAbort);
      const int ib = items[qi].b, ih = items[qi].hkv, len = items[qi].len;
      gs += items[qi].pad0;
      uint4 qv[NI];
      uint32_t amax2 = 0u;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const uint32_t c = (uint32_t)(i * 4 + (qt >> 4)), j = c * g_inv >> 16, hh = c - j * (uint32_t)p.G;
        qv[i] = make_uint4(0u, 0u, 0u, 0u);
        if ((int)c < p.ncols)
          qv[i] = ld_dep(reinterpret_cast<const uint4*>(p.q + (((size_t)ib * p.nq_stride + j) * p.Hq + (size_t)ih * p.G + hh) * LYNX_D) + (qt & 15));
      }
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const uint32_t w[4] = {qv[i].x, qv[i].y, qv[i].z, qv[i].w};
        float sum = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          asm("max.bf16x2 %0, %0, %1;" : "+r"(amax2) : "r"(w[k] & 0x7FFF7FFFu));
          sum += __uint_as_float(w[k] << 16) + __uint_as_float(w[k] & 0xFFFF0000u);
        }
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
        if ((qt & 15) == 0) scal[qi * CP + i * 4 + (qt >> 4)] = sum;
      }
      const float am = warp_max(fmaxf(__uint_as_float(amax2 << 16), __uint_as_float(amax2 & 0xFFFF0000u)));
      if (lane == 0) scal[4 * CP + 2 + (warp & 1)] = am;
      named_bar(6, 64);
      const int e = i8_q_exponent(fmaxf(scal[4 * CP + 2], scal[4 * CP + 3]));
      const float up = __int_as_float((127 + e) << 23);
      if (qt == 0) reinterpret_cast<int*>(scal)[4 * CP + qi] = e;
      if (qt < CP) reinterpret_cast<int*>(scal)[2 * CP + qi * CP + qt] = qt < p.ncols ? (p.causal ? len - p.tail + qt / p.G + 1 : len) : 0;
      // three balanced s8 digit planes of q_int = rint(q 2^e), rows plane * CP + column (four where K goes in as raw bytes)
      const uint32_t qtile = sbase + C::kOffQ + qi * C::kQTile;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const int c = i * 4 + (qt >> 4), j = (qt >> 2) & 3, w = qt & 3;   // column, 32 dims of the row, 8 of them
        const uint32_t ww[4] = {qv[i].x, qv[i].y, qv[i].z, qv[i].w};
        // A balanced digit is a byte of the value plus 128 in every digit, less 128 again: the top bit flipped.  (Taken off digit by
        // digit it was 200 instructions for eight entries, and a launch's first product waits for it: verification of 4096 tokens at 16
        // columns 15.3 -> 14.8 us.)
        constexpr int kBias = NP == 4 ? (int)0x80808080u : 0x808080;
        uint32_t val[2][4];   // [even, odd dims][pair]
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int even = max(-4194303, min(4194303, __float2int_rn(__uint_as_float(ww[k] << 16) * up)));
          const int odd = max(-4194303, min(4194303, __float2int_rn(__uint_as_float(ww[k] & 0xFFFF0000u) * up)));
          // what multiplies the byte pair (odd value) and its low nibble (16 x even value - odd value), where K goes in as raw bytes
          val[0][k] = (uint32_t)((C::kRawK ? odd : even) + kBias);
          val[1][k] = (uint32_t)((C::kRawK ? 16 * even - odd : odd) + kBias);
        }
        uint32_t acc[NP][2];
#pragma unroll
        for (int par = 0; par < 2; ++par) {
          const uint32_t l01 = prmt(val[par][0], val[par][1], 0x5140u), l23 = prmt(val[par][2], val[par][3], 0x5140u);
          const uint32_t h01 = prmt(val[par][0], val[par][1], 0x7362u), h23 = prmt(val[par][2], val[par][3], 0x7362u);
          acc[0][par] = prmt(l01, l23, 0x5410u) ^ 0x80808080u;
          acc[1][par] = prmt(l01, l23, 0x7632u) ^ 0x80808080u;
          acc[2][par] = prmt(h01, h23, 0x5410u) ^ 0x80808080u;
          if (NP == 4) acc[NP - 1][par] = prmt(h01, h23, 0x7632u) ^ 0x80808080u;
        }
#pragma unroll
        for (int pln = 0; pln < NP; ++pln) {
          const int n = pln * CP + c;
#pragma unroll
          for (int par = 0; par < 2; ++par) {
            const int chunk = C::kRawK ? 4 * par + j : 2 * j + par;   // 16 bytes of the row's 128
            const uint32_t a = qtile + (uint32_t)n * 128u + ((uint32_t)(chunk ^ (n & 7)) << 4) + 4u * w;
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(acc[pln][par]) : "memory");
          }
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      named_bar(6, 64);   // (the maxima have been read, too)
      if (lane == 0) { mbar_arrive(qready + qi * 8); mbar_arrive(qempty + qi * 8); }
      ++ic;
    }
  }
}

template <bool FULL, int CP>
lynx_status launch_pipe(const AttnParams& p, cudaStream_t st) {
  using C = PipeCfg<FULL, CP>;
  constexpr int kMin = 2;
  const lynx_status rc = launch_units<FULL, PipeMaps, C::kSmem, C::kThreads, C::kST, kMin, attn_pipe_kernel<FULL, CP>>(p, st);
  return rc != LYNX_OK ? rc : launch_combine(p, C::kPartCols, C::kST, kMin, st);
}
