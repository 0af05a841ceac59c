// Fused split-K GQA decode attention over the mixed-precision cache (Eq. 1 with Eq. 3 applied on the fly),
// warp-specialised form.
//
// Work unit = 32 tokens of one stream, taken two at a time (a step of 64 tokens; blocks hold an even number of units).  All
// units of all streams are split evenly over the CTAs; inside a CTA they are split over TEAMS of warps.  A team shares one
// ring of staged steps (1-D bulk copies signalled on mbarriers):
//
//   a logits warp     expands the step's 2-bit key codes into tensor-core A fragments (one logic op and one fp16 FMA
//                     per pair of codes: A = c*s, exact in fp16) and runs q.K^T on mma.sync m16n8k16 tiles with the g
//                     query heads of the KV head as the N dimension.  The zero-point term q.z of the key groups is one
//                     more tile chain per step (rows 0..7 the first unit's group, rows 8..15 the second's); the promoted
//                     (BF16) channels and the UINT4 high plane are further tiles.  The step's 64 x 8 logits go to the
//                     partner through shared memory, in the place of the key codes and scales they were made from.
//   the values warp   keeps the online softmax, builds the value-scale tables,
//                     folds the value scales into the probabilities and runs P.V with the raw value codes as fp16
//                     subnormals in the A operand (one logic op per pair of codes); value zero-points and the softmax
//                     denominator ride on one extra tile.  It owns the output accumulators and refills the ring.
//
// Neither warp holds the other's state, so both need far fewer registers than a warp that does everything, more warps
// fit an SM, and the logits of one step overlap the values of the one before.  The packed layout stores the codes in
// A-fragment order: a lane's 16-byte shared-memory load is exactly its registers; nothing dequantized is ever written back
// to shared memory.  Unquantized units (residual window, sink) are read straight from global memory in bf16 and are taken
// first, while the first staged copies are in flight.
//
// What bounds it: instruction issue and the latency of each warp's chain of dependent work, with three or four warps per
// scheduler.  Two units per step instead of one (attention_single.cu) give every chain an independent twin, halve the
// waits, hand-overs and zero-point tiles per unit (690 -> 598 warp instructions per unit) and need no hand-over buffers; the
// promoted channels and the UINT4 plane, read from global memory a unit ahead there, come through shared memory ahead of time
// (without that the longer steps were slower than single units: 39.0 us at the 7b shape).  Clocks around the waits: with
// two tiers the logits warp is the longer role by a quarter, with a 4-bit base by a factor of two, hence two logits warps
// per values warp there.  us per launch, one unit / two units per step / with two logits warps: 7b shape (B = 8, T = 32768) 36.7 /
// 35.3; three tiers 54.4 / 48.7 / 46.2; 4-bit base (8b shape, B = 16, T = 16384) 110.7 / 109.5 / 101.7; 4-bit values 88.4 / 82;
// 32b shape (B = 64, T = 32768, G = 128) 463 / 433 = 3.1 TB/s.  (Those five were taken side by side with a reference maximum raised only
// by factors of 8; as the kernel is now: 34.3, 46.4, 95.5, 80.6, 421.)
#include "warp_ops.cuh"

namespace mixkvq {

cudaError_t launch_combine(const float* ws, float* out, int g, int Hkv, int Hq, int mode, int n,
                           long long units_per_stream, int S, cudaStream_t stream, const int4* seq = nullptr,
                           const int* seq_prefix = nullptr, float* lse_out = nullptr, bool early = false, void* rope_q = nullptr, void* rope_k = nullptr,
                           const float* rope_cos = nullptr, const float* rope_sin = nullptr);
// the same split, one unit at a time (attention_single.cu)
cudaError_t launch_attention_single(const LayerView& lv, const void* q, float scale, float* ws, int grid, float* out, float* lse, bool wide,
                                    cudaStream_t stream);
cudaError_t attention_single_setup();

namespace {

// A team: one values warp and its logits warps, which take the steps in turn.  Two tiers: one logits warp, four teams per CTA
// (three where 4-bit values need the shared memory); a UINT4 tier or a 4-bit base makes the logits about twice the values'
// work, so two logits warps, two teams per CTA.  Two CTAs per SM: 16 warps at 128 registers or 12 at 168.
__host__ __device__ constexpr int logits_warps_of(int u4) { return u4 != 0 ? 2 : 1; }
__host__ __device__ constexpr int teams_of(int u4, bool v4) { return u4 != 0 ? 2 : (v4 ? 3 : 4); }
__host__ __device__ constexpr int threads_of(int u4, bool v4) { return teams_of(u4, v4) * (logits_warps_of(u4) + 1) * 32; }
constexpr int kCtasPerSm = 2;
__host__ __device__ constexpr int stages_of(int u4) { return u4 != 0 ? 4 : 3; }            // ring stages per team
constexpr int kMaxStages = 4;
__host__ __device__ constexpr int unit_bytes_of(int G, bool v4) { return 2048 + 128 * (kD / G) + (v4 ? 1024 : 0); }
// one ring stage: the two units of a step with their key-meta groups (512 B each) in the block's own order: a group before
// each unit (G = 32), or one group before both
__host__ __device__ constexpr int stage_bytes(int G, bool v4) { return (G == 32 ? 1024 : 512) + 2 * unit_bytes_of(G, v4); }
// Tables of a team: per logits warp the key scales {s, -4s} of two groups (2 x 576) and the key zero-point tiles (576), then
// the value scales of two units (2 x 320) and the value zero-point tiles of two units (2 x 544).
constexpr int kZprepOff = 1152, kKeyPrepBytes = 1728;
__host__ __device__ constexpr int svp_off(int u4) { return logits_warps_of(u4) * kKeyPrepBytes; }
__host__ __device__ constexpr int zvp_off(int u4) { return svp_off(u4) + 640; }
__host__ __device__ constexpr int prep_bytes(int u4) { return zvp_off(u4) + 1088; }
constexpr int kKprepGroup = 576, kSvpUnit = 320, kZvpUnit = 544;
constexpr int kRBufBytes = 1024;             // hand-over of an unquantized unit's logits: 32 bytes per lane
// A step's extras (the promoted channels and the UINT4 high plane), copied a step or two ahead by each logits warp for its own steps
// (three slots, two where two logits warps take turns; the values warp is no place for this although it has more time: it
// refills the ring, and with the extras its wait for the copies made the 7b shape 38.9 us instead of 35.3):
// the block's channel lists (in a step that begins a block, and where something does not fit) | where the step's extras lie in
// the stream's arena (only then) | rows of the first kRowPairs pairs of promoted channels of both units (128 B each) | three tiers:
// the first kPlanePairs pairs of UINT4 channels of both units (16 B each); 4-bit base: both units' dense planes.  What does not
// fit is read from global memory in the step itself, requested into the L2 cache with the slot.  (us per launch with the lists and the
// table entry read in the step and nothing requested / so / one unit at a time: 8b shape, 16384 tokens, 32 promoted channels 133 /
// 111 / 112, 32 and 32 UINT4 channels 170 / 140 / 140; 32b shape, G = 128, 8192 tokens, 32 promoted 235 / 187 / 188, 12 and 22 221 / 203 / 193;
// three tiers with 34 and 94 channels, 7b shape 41.6 / 33.2 / 47.6.  8 or 16 pairs in the slots: up to 15 % faster beyond 8 channels,
// but 4 % slower with the usual 4, the L1 cache being what the slots take.)
constexpr int kRowPairs = 4, kPlanePairs = 16;
__host__ __device__ constexpr int slots_of(int u4) { return u4 != 0 ? 2 : 3; }
constexpr int kListBytes = 144, kWhereOff = kListBytes, kRowsOff = 160, kPlaneOff = kRowsOff + 2 * kRowPairs * 128;
__host__ __device__ constexpr int slot_bytes(int u4) { return kPlaneOff + (u4 == 1 ? 2 * kPlanePairs * 16 : u4 == 2 ? 2048 : 0); }
__host__ __device__ constexpr int team_bytes(int G, int u4, bool v4) {
  return stages_of(u4) * stage_bytes(G, v4) + logits_warps_of(u4) * (slots_of(u4) * slot_bytes(u4) + kRBufBytes) + prep_bytes(u4);
}
// mbarriers of a team: staged copy landed [stages], logits ready [stages], then per logits warp for unquantized units: ready, taken
constexpr int kBarsPerTeam = 2 * kMaxStages + 4;
constexpr int kQS = 136;                     // halves per row of the query tables (272 bytes: rows fall on different banks)
constexpr int kPrefixBytes = ((kMaxRaggedBatch + 1) * 4 + 15) / 16 * 16;     // a ragged batch's prefix sums
__host__ __device__ constexpr int bar_bytes(int teams) { return (teams * kBarsPerTeam * 8 + 127) / 128 * 128; }
__host__ __device__ constexpr int smem_bytes(int G, int u4, bool v4) {
  return teams_of(u4, v4) * (team_bytes(G, u4, v4) + 64) + bar_bytes(teams_of(u4, v4)) + (u4 == 1 ? 2 : 1) * 8 * kQS * 2 + kPrefixBytes;
}
constexpr int kResidualWeight = 3;           // an unquantized 32-token unit counts as this many packed units in the split
constexpr int kMergeStride = 132;            // floats per head row of a pair's output in the merge
// A wait on a barrier polls at most this many times; a poll suspends the thread for up to about a microsecond, so
// the wait gives up after about two seconds at the latest (a few milliseconds if the polls return at once).
constexpr uint32_t kWaitPolls = 1u << 21;

// Byte offset of (k-tile kt, lane column t) in the key-scale table: 16 bytes {s_a, -4 s_a, s_b, -4 s_b} (half2 each: the
// lane's channel pairs 16kt + 2t, +1 and 16kt + 8 + 2t, +1); 16 bytes of padding after every second k-tile keep the
// preparation's stores free of bank conflicts.  The zero-point table has the same shape: {z_a of unit 0, of unit 1, z_b of
// unit 0, of unit 1}, times 2^(pos - 8): the A fragment of a tile whose rows 0..7 are unit 0's group, rows 8..15 unit 1's.
__device__ __forceinline__ constexpr int kprep_off(int kt, int t) { return 144 * (kt >> 1) + 64 * (kt & 1) + 16 * t; }
// Bit position (inside each 16-bit half, after the shift below) of k-tile kt's 2-bit field.
__device__ __forceinline__ constexpr int key_pos(int kt) { return (0x86486464u >> (4 * kt)) & 0xF; }
// k-tiles 0,1 are read from (w << 4), 2..4 from w, 5..7 from (w >> 6)
__device__ __forceinline__ uint32_t key_shift(uint32_t w, int kt) { return kt < 2 ? (w << 4) : (kt < 5 ? w : (w >> 6)); }

// warp w of the CTA with one logits warp per team: team w / 2; the logits warps are spread evenly over the four schedulers of
// the SM (w mod 4)
__device__ __forceinline__ bool is_logits_warp(int warp) { return ((warp ^ (warp >> 2)) & 1) == 0; }

// kU4: how the configuration can use the UINT4 tier: 0 = never (tau_u4 >= tau_bf16), 1 = some channels (high plane stored
// per channel pair, gathered), 2 = 4-bit base (dense high plane)
// kV4: 4-bit values (a second plane of 2-bit value codes per unit, scale 4 s_v)
// kDirect: one CTA per stream, which writes the output (and the log-denominators) instead of a partial
// (q without __restrict__: a direct call that rotates writes the rows that it reads)
template <int G, int kU4, bool kV4, bool kDirect>
__global__ void __launch_bounds__(threads_of(kU4, kV4), kCtasPerSm)
attention_ws_kernel(LayerView lv, const __nv_bfloat16* q, float scale_log2e, uint32_t four2, float* __restrict__ ws,
                    float* __restrict__ out, float* __restrict__ lse_out) {
  constexpr int VG = kD / G;              // value groups per token
  constexpr int TPG = 8 / VG;             // 16-channel tiles per value group
  constexpr int UPG = G / 32;             // units per key group
  constexpr int kGroups = UPG == 1 ? 2 : 1;                    // key groups of a step
  constexpr int kTeams = teams_of(kU4, kV4), kL = logits_warps_of(kU4), kThreads = threads_of(kU4, kV4);
  constexpr int kStages = stages_of(kU4), kSlotCount = slots_of(kU4), kSlotBytes = slot_bytes(kU4);
  static_assert(smem_bytes(G, kU4, kV4) <= 113 * 1024, "two CTAs per SM");
  constexpr int kStageBytes = stage_bytes(G, kV4);
  constexpr int kTeamBytes = team_bytes(G, kU4, kV4);
  // a unit: key codes 1024, value codes 1024, value scales (and the values' high plane 1024)
  constexpr uint32_t kUnitBytes = unit_bytes_of(G, kV4);
  constexpr uint32_t kUnitStep = kUnitBytes + (UPG == 1 ? 512u : 0u);      // from a step's first unit to its second, staged
  constexpr int kSlotBase = kStages * kStageBytes;             // offsets inside a team's shared memory
  constexpr int kPrepBase = kSlotBase + kL * kSlotCount * kSlotBytes;
  constexpr int kRBufBase = kPrepBase + prep_bytes(kU4);
  constexpr int kQBytes = (kU4 == 1 ? 2 : 1) * 8 * kQS * 2;
  constexpr int kSpillUnroll = kU4 == 0 ? 2 : 4;               // (128 registers / 168)
  extern __shared__ __align__(128) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane >> 2, t = lane & 3;
  const int team = kL == 1 ? warp >> 1 : warp / 3;
  const bool logits_role = kL == 1 ? is_logits_warp(warp) : warp % 3 != 2;
  const uint32_t lsub = kL == 1 || !logits_role ? 0u : (uint32_t)(warp % 3);      // which of the team's logits warps

  const uint32_t smem_base = smem_u32(smem);
  const uint32_t ring_u32 = smem_base + team * kTeamBytes;                  // the team's shared memory starts with its ring
  const uint32_t tail_u32 = smem_base + kTeams * kTeamBytes;
  const uint32_t bar_u32 = tail_u32 + team * (kBarsPerTeam * 8);            // staged copy landed [kStages]
  const uint32_t lfull_u32 = bar_u32 + kStages * 8;                         // logits ready [kStages]
  const uint32_t rfull_u32 = bar_u32 + 2 * kStages * 8, rempty_u32 = rfull_u32 + 8 * kL;    // [kL] each
  const uint32_t qb16_u32 = tail_u32 + bar_bytes(kTeams);                           // [8][kQS] q, bf16 bits (0 for heads >= g)
  const uint32_t qf16_u32 = qb16_u32 + 8 * kQS * 2;                         // [8][kQS] q, fp16 (three tiers)
  float* mS = reinterpret_cast<float*>(smem + kTeams * kTeamBytes + bar_bytes(kTeams) + kQBytes);    // [kTeams][8]
  float* lS = mS + kTeams * 8;                                                                       // [kTeams][8]
  int* prefS = reinterpret_cast<int*>(lS + kTeams * 8);                     // ragged batch: seq_prefix[0 .. B]

  if (threadIdx.x < kTeams * kBarsPerTeam) {
    mbar_init(tail_u32 + 8 * threadIdx.x, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (!logits_role) {
    // constant rows of the zero-point / denominator tiles ([2 units][2 ks: 68 words][8 rows][4 t]{k 2t.., k 8 + 2t..}):
    // row 4 is all ones, the other rows >= VG stay zero
    for (int i = lane; i < 2 * kZvpUnit / 4; i += 32)
      sts32(ring_u32 + kPrepBase + zvp_off(kU4) + 4 * i, ((i % 68) >> 3) == 4 ? 0x3C003C00u : 0u);
  }
  __syncthreads();

  const int S = lv.B * lv.Hkv, U = lv.U, g = lv.g;
  // Fill of the stream at hand: the same for every stream, or (ragged batch) taken per sequence from the table in
  // device memory at the start of every segment.
  int f_nb = lv.n_blocks, f_r = lv.r, f_ns = lv.n_sink;
  int packed_units = f_nb * U;
  // unquantized 32-token units: those of the residual window, then those of the sink
  int res_units = (f_r + 31) / 32, bf16_units = res_units + (f_ns + 31) / 32;
  int Us = packed_units + kResidualWeight * bf16_units;             // split positions; an unquantized unit spans several

  // Programmatic dependent launch: the grid may have been started while the kernel before it in the stream was still
  // running.  Nothing above touches global memory.  dep_wait() waits for that kernel's results and lets the kernel after
  // this one be started early in the same way; every thread calls it before its first access to global memory, with one
  // exception: when the host knows that the kernel before this one did not write this layer's packed blocks
  // (stage_early), the first staged copies of the packed units go out before the wait.  That is safe because what may
  // still be running then besides that kernel is the split kernel before it, if it is a merge (see common.cuh).
  bool dep_waited = false;
  auto dep_wait = [&]() {
    if (!dep_waited) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      dep_waited = true;
    }
  };
  if (!lv.stage_early || lv.seq != nullptr) dep_wait();     // the table of a ragged batch is read right below
  if (lv.seq != nullptr) {
    // the prefix sums go to shared memory in one round trip: the segments below search them
    for (int i = threadIdx.x; i <= lv.B; i += kThreads) prefS[i] = lv.seq_prefix[i];
    __syncthreads();
  }
  // the CTA's share of all streams' positions; in a ragged batch it is a part of one stream (below)
  const long long total = (long long)Us * S;
  const long long cb = kDirect ? (long long)Us * blockIdx.x : lv.seq != nullptr ? 0 : split_begin(total, gridDim.x, blockIdx.x);
  const long long ce = kDirect ? cb + Us : lv.seq != nullptr ? 1 : split_begin(total, gridDim.x, blockIdx.x + 1);

  uint32_t ring_stage = 0;        // ring stage of the next step of this warp
  uint32_t ring_parity = 0;       // phase parity of that stage's barriers
  uint32_t rit[kL] = {};          // unquantized units handed over so far, per logits warp of the team
  bool gave_up = false;
  // A wait that runs out sets gave_up; the warp carries on with whatever the shared memory holds (every address it
  // forms stays inside the CTA's shared memory and the stream's arrays), its later waits are skipped, and the team's
  // result is replaced by zeros at the end.  Straight-line code: no exit in the middle of a step.
  auto wait_or_give_up = [&](uint32_t bar, uint32_t parity) {
    if (!gave_up && !mbar_wait_polls(bar, parity, lv.wait_polls ? lv.wait_polls : kWaitPolls)) gave_up = true;
  };
  auto next_stage = [&](uint32_t sg) { return sg + 1u == (uint32_t)kStages ? 0u : sg + 1u; };
  auto advance_stage = [&]() {
    ring_stage = next_stage(ring_stage);
    ring_parity ^= (ring_stage == 0u) ? 1u : 0u;
  };

  for (long long seg = cb; seg < ce;) {
    int s, ub, ue;
    // A whole stream is its CTA's only segment.  Said so, no register is kept for a next one: two tiers spilled 56 to 80 bytes in their main
    // loops, 0 to 4 so; 32b shape, 32 x 2000 tokens, G = 128, 8 layers 174 / 166 us per step.
    if (kDirect) {
      s = blockIdx.x;
      ub = 0;
      ue = Us;
      seg = ce;
    } else if (lv.seq != nullptr) {
      // ragged batch: the sequence whose CTAs this one is among (empty sequences have none), the stream and the part of it
      int b = 0;
      while (b + 1 < lv.B && prefS[b + 1] <= (int)blockIdx.x) ++b;
      const int4 f = lv.seq[b];
      f_nb = f.x; f_r = f.y; f_ns = f.z; Us = f.w;
      packed_units = f_nb * U;
      res_units = (f_r + 31) / 32;
      bf16_units = res_units + (f_ns + 31) / 32;
      const int parts = (prefS[b + 1] - prefS[b]) / lv.Hkv, rel = (int)blockIdx.x - prefS[b], hk = rel / parts;
      s = b * lv.Hkv + hk;
      ub = (int)split_begin(Us, parts, rel - hk * parts);
      ue = (int)split_begin(Us, parts, rel - hk * parts + 1);
      seg = ce;
    } else {
      s = (int)(seg / Us);
      ub = (int)(seg - (long long)s * Us);
      ue = (int)min((long long)Us, ce - (long long)s * Us);
      seg += ue - ub;
    }
    // ---- this team's share of the segment.  The unquantized units of the segment go to different teams (unit i to
    // team kTeams - 1 - i % kTeams); the packed units are split in order, in steps of two, so that every team carries about
    // the same weight.  (A stream's packed units are even in number; a boundary at an odd one moves up, on both sides.)
    const int pk_b = (min(ub, packed_units) + 1) & ~1, pk_e = (min(ue, packed_units) + 1) & ~1;
    const int res_b = (max(ub, packed_units) - packed_units + kResidualWeight - 1) / kResidualWeight;
    const int res_e = ue > packed_units ? (ue - packed_units + kResidualWeight - 1) / kResidualWeight : res_b;
    const int n_res = res_e - res_b;
    int wb = pk_b, we = pk_b;
    {
      const int n_packed = pk_e - pk_b, weight = n_packed + kResidualWeight * n_res;
      int given = 0, res_given = 0;              // packed and unquantized units of the teams before
#pragma unroll
      for (int w = 0; w < kTeams; ++w) {
        const int first_i = kTeams - 1 - w;      // unquantized units first_i, first_i + kTeams, ...
        res_given += n_res > first_i ? (n_res - first_i + kTeams - 1) / kTeams : 0;
        // everything up to this team against its exact share (weight < 2^24: 32-bit arithmetic)
        const int upto = w == kTeams - 1
                             ? n_packed
                             : min(n_packed, max(given, (weight * (w + 1) / kTeams - kResidualWeight * res_given + 1) & ~1));
        if (w == team) {
          wb = pk_b + given;
          we = pk_b + upto;
        }
        given = upto;
      }
    }
    const int n_steps = (we - wb) >> 1;

    // ---- the first copies of this segment go out before anything else (values warp): they do not depend on the query.
    // The packed units of a stream are one uniform sequence (a group's scales, then its units), whatever the block size,
    // so the copy source only ever moves forward: `isrc` is the next step to stage.
    int issued = 0;
    const char* isrc = lv.base + (size_t)s * lv.base_stride + (size_t)wb * kUnitBytes + 512u * (size_t)((wb + UPG - 1) / UPG);
    // G = 128: a group's scales lie before its first half; a step that is the second half brings them along where its logits
    // warp did not have the first half
    constexpr bool kMetaAlways = kL > 1;
    uint32_t ihalf = UPG == 4 ? (uint32_t)(wb >> 1) & 1u : 0u;      // G = 128: the step is its group's second half
    // stages the next step (if there is one left) in ring stage sg; all lanes keep the position
    auto issue = [&](uint32_t sg, bool first) {
      const uint32_t dst = ring_u32 + sg * kStageBytes, bar = bar_u32 + sg * 8u;
      // Nothing more after a wait that ran out: its stage's barrier is still armed, and what is under way is awaited at the end.
      // (The lanes may differ in that: the copying lane's own view decides, so it never arms a barrier that it has not seen free.)
      const uint32_t enabled = issued < n_steps && !gave_up ? 1u : 0u;
      if (UPG != 4 || ihalf == 0u) {
        stage_copy(dst, isrc, (uint32_t)kStageBytes, bar, first ? lv.debug_extra_tx : 0u, enabled);
        isrc += kStageBytes;
      } else {
        if (first || kMetaAlways)
          stage_copy2(dst + 512, isrc, 2 * kUnitBytes, dst, isrc - 2 * kUnitBytes - 512, 512u, bar, first ? lv.debug_extra_tx : 0u, enabled);
        else stage_copy(dst + 512, isrc, 2 * kUnitBytes, bar, 0u, enabled);
        isrc += 2 * kUnitBytes;
      }
      if (UPG == 4) ihalf ^= 1u;
      issued += (int)enabled;
    };
    const uint32_t stage0 = ring_stage, parity0 = ring_parity;
    // The extras of a step are copied kSlotCount - 1 of the warp's own steps ahead.  The copies' cursor: block cbi and unit cu
    // in it, the block's table entry and the entry of the next block or (two logits warps) of the next copy, under way.
    const char* extras = lv.extras + (size_t)s * lv.extras_stride;
    const uint2* table = reinterpret_cast<const uint2*>(lv.table + (size_t)s * lv.table_stride);
    constexpr int kOwnUnits = 2 * kL;                             // from a warp's step to its next one
    const uint32_t slot0_u32 = ring_u32 + kSlotBase + lsub * (kSlotCount * kSlotBytes);
    int cbi = 0, cu = 0, last_bi = -1, to_request = logits_role ? (n_steps - (int)lsub + kL - 1) / kL : 0;
    uint2 c_entry = make_uint2(0u, 0u), c_next = make_uint2(0u, 0u);
    auto next_position = [&](int& b, int& v) {
      v += kOwnUnits;
      if constexpr (kL == 1) {
        if (v == U) {
          v = 0;
          ++b;
        }
      } else {
        while (v >= U) {
          v -= U;
          ++b;
        }
      }
    };
    auto request_entry = [&]() {
      int b = cbi + 1, v = 0;
      if constexpr (kL != 1) {
        b = cbi;
        v = cu;
        next_position(b, v);
      }
      if (b < f_nb) c_next = table[b];
    };
    // requests the next own step's extras (nothing past the last step); returns its block's counts: pairs of promoted channels,
    // UINT4 channels << 8, and bit 16 in a step that begins a block (or is the first one)
    auto request_extras = [&](uint32_t slot) -> uint32_t {
      uint32_t counts = 0u;
      if (to_request > 0) {
        const int n16 = c_entry.y & 0xFF, n4 = (c_entry.y >> 8) & 0xFF, n16p = (n16 + 1) >> 1;
        const bool begins = kL == 1 ? last_bi < 0 || cu == 0 : cbi != last_bi;
        counts = (uint32_t)n16p | ((uint32_t)n4 << 8) | (begins ? 0x10000u : 0u);
        const uint32_t hdr = extras_header_bytes(n16, n4), unit = extras_unit_bytes(n16, n4, kU4 == 2);
        const char* ex = extras + (size_t)c_entry.x * 16;
        const char* exu = ex + hdr + (size_t)cu * unit;
        const uint32_t dst = slot0_u32 + slot * kSlotBytes;
        const bool spills = n16p > kRowPairs || (kU4 == 1 && n4 > 2 * kPlanePairs);
        if ((begins || spills) && 16u * lane < hdr) cp_async16(dst + 16 * lane, ex + 16 * lane);          // (hdr <= kListBytes)
        if (spills) {
          if (lane == 0) sts32(dst + kWhereOff, c_entry.x + ((hdr + (uint32_t)cu * unit) >> 4));
          if (kRowPairs + lane < n16p) {
            prefetch_l2(exu + 128 * (kRowPairs + lane));
            prefetch_l2(exu + unit + 128 * (kRowPairs + lane));
          }
          if (kU4 == 1 && lane < 16 && 16 * (lane & 7) < n4) prefetch_l2(exu + (lane >> 3) * unit + 128 * n16p + 128 * (lane & 7));
        }
        // rows: lane = (pair, 16-byte piece); the pieces of a row are swizzled by the pair so that the tile's reads fall on
        // different banks
        if ((lane >> 3) < n16p) {
          const uint32_t rd = dst + kRowsOff + (lane >> 3) * 128 + (((lane & 7) ^ (2 * (lane >> 3))) << 4);
          cp_async16(rd, exu + 16 * lane);
          cp_async16(rd + kRowPairs * 128, exu + unit + 16 * lane);
        }
        if constexpr (kU4 == 1) {
          if ((lane & 15) < (n4 + 1) >> 1) cp_async16(dst + kPlaneOff + 16 * lane, exu + (lane >> 4) * unit + 128 * n16p + 16 * (lane & 15));
        }
        if constexpr (kU4 == 2) {
          if (n16 + n4 > 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              cp_async16(dst + kPlaneOff + 512 * k + 16 * lane, exu + (k >> 1) * unit + 128 * n16p + 512 * (k & 1) + 16 * lane);
          }
        }
        --to_request;
        last_bi = cbi;
        next_position(cbi, cu);
        if (kL != 1 || cbi != last_bi) {
          c_entry = c_next;
          request_entry();
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      return counts;
    };
    uint32_t counts[kSlotCount];              // of the current own step and those ahead
#pragma unroll
    for (int i = 0; i < kSlotCount; ++i) counts[i] = 0u;
    auto request_first = [&]() {
      cbi = (wb + 2 * (int)lsub) / U;
      cu = wb + 2 * (int)lsub - cbi * U;
      c_entry = table[cbi];
      request_entry();
#pragma unroll
      for (int i = 0; i < kSlotCount - 1; ++i) counts[i] = request_extras(i);
    };
    uint32_t slot = 0;                        // of the current own step
    if (!logits_role) {
#pragma unroll 1
      for (uint32_t i = 0, sg = ring_stage; i < (uint32_t)kStages; ++i, sg = next_stage(sg)) issue(sg, i == 0);
    }
    if (to_request > 0 && lv.stage_early) request_first();
    // Two tiers, G = 32, split streams: the query rows, the step's token and the segment's unquantized units are requested into the L2 cache
    // before the wait (a request has no other effect, whatever the kernel before this one still writes): of a model's many layers they have
    // left it since the step before.  Only ahead of a wait: not for a CTA's later segments, nor in a ragged batch, whose table is read behind it.
    // us per decode step, without / with: 7b shape, 8 x 32768 tokens, 28 layers 1062 / 1047, 4 x 120000, 8 layers 503 / 493, 32b shape, 64 x
    // 8000, 6 layers 779 / 771, 64 x 1500 250 / 253.  (Not all of it is the requests': a ragged batch, which makes none, takes 799 / 791 in the
    // two builds of the kernel.)  Elsewhere it delays what goes out first or gives nothing: three tiers, 7b shape, 8 x 32768, 14 layers 700 / 709; 4-bit
    // base, G = 128, 8 x 38643, 4 layers 220.6 / 221.4; two tiers, G = 128, 32b shape, 64 x 32768, 3 layers 1266 / 1287, G = 64, 7b shape, 16 x 12000,
    // 14 layers 427 / 430; one CTA per stream, 32b shape, 32 x 2000, 8 layers 176 / 180; one unit per step, 4-bit values, 24 x 1147, 28 layers 364 /
    // 370, 4 x 6001, 16 layers 251.2 / 250.1.
    if (kU4 == 0 && G == 32 && !kDirect && !dep_waited) {
      const int b = s / lv.Hkv, hk = s % lv.Hkv, h = threadIdx.x >> 1;
      if (h < g) prefetch_l2(reinterpret_cast<const char*>(q + ((size_t)b * lv.Hq + hk * g + h) * kD) + 128 * (threadIdx.x & 1));
      else if (lv.new_k != nullptr && h < g + 2) prefetch_l2(reinterpret_cast<const char*>((h == g ? lv.new_k : lv.new_v) + (size_t)s * kD) + 128 * (threadIdx.x & 1));
      for (int i = threadIdx.x; i < n_res * 128; i += kThreads) {          // per unit 64 lines of keys, 64 of values
        const int bu = res_b + (i >> 7);
        const bool in_sink = bu >= res_units, values = (i & 64) != 0;
        const char* rows = in_sink ? lv.sink + (size_t)s * lv.sink_stride + (values ? (size_t)lv.sink_len * 256 : 0)
                                   : (values ? lv.resv + (size_t)s * lv.resv_stride : lv.resk + (size_t)s * lv.resk_stride);
        prefetch_l2(rows + (size_t)(bu - (in_sink ? res_units : 0)) * 8192 + 128 * (i & 63));
      }
    }
    dep_wait();
    if (to_request > 0 && !lv.stage_early) request_first();

    // fused decode step: the newest token (slot r - 1) is not in the residual store yet; the warps that take its unit read it from
    // the step's tensors, store its rows and update the importance accumulator
    const int jn = f_r - 1;
    // ---- query of this stream: bf16 and fp16 tables (heads >= g are zero rows)
    {
      uint4 q_regs = make_uint4(0u, 0u, 0u, 0u);      // thread (h, c) of the first 128: head h, channels 8c .. 8c+7
      const size_t row0 = (size_t)s * g;              // (b Hkv + hk) g = b Hq + hk g
      const int h = threadIdx.x >> 4, c = threadIdx.x & 15;
      if (h < g) q_regs = reinterpret_cast<const uint4*>(q + (row0 + h) * kD)[c];
      RopeInput rope_in{};
      if (lv.rope_cos != nullptr) rope_in = rope_request<kThreads>(lv, s);
      __syncthreads();          // the previous segment's readers of the tables are done
      if (h < 8) {
        sts128(qb16_u32 + (h * kQS + 8 * c) * 2, q_regs.x, q_regs.y, q_regs.z, q_regs.w);
        if (kU4 == 1)      // the fp16 table is for the gathered UINT4 channels
          sts128(qf16_u32 + (h * kQS + 8 * c) * 2, bf16x2_to_f16x2(q_regs.x), bf16x2_to_f16x2(q_regs.y),
                 bf16x2_to_f16x2(q_regs.z), bf16x2_to_f16x2(q_regs.w));
      }
      if (lv.rope_cos != nullptr) {
        __syncthreads();
        // the CTA with the new key's unit reads the rotated key from the window; where the CTA has the whole stream nobody else reads
        // the caller's rows, and it leaves them rotated
        rope_rotate<kThreads, kQS, kU4 == 1>(
            lv, s, g, rope_in, qb16_u32, qf16_u32,
            jn >= 32 * res_b && jn < 32 * res_e ? reinterpret_cast<uint16_t*>(lv.resk + (size_t)s * lv.resk_stride + (size_t)jn * 256) : nullptr,
            kDirect ? reinterpret_cast<uint16_t*>(const_cast<__nv_bfloat16*>(q)) + row0 * kD : nullptr);
      }
      __syncthreads();
    }

    // unquantized units of this team: first_res, first_res + kTeams, ... < n_res
    const int first_res = kTeams - 1 - team;

    const uint32_t qrow_u32 = qb16_u32 + r * (kQS * 2), qfrow_u32 = qf16_u32 + r * (kQS * 2);

    if (logits_role) {
      // =====================================================================================================
      // logits warp
      // =====================================================================================================
      // ---- unquantized units: bf16 keys straight from global memory.  The channel a k-slot stands for is free as long as
      // both operands agree: lane column t of k-tile 2j (2j+1) takes channels 32j + 8t + 0..3 (4..7), so that a lane's
      // four k-tiles' worth of a token row is one 16-byte load.
      bool takes_new = false;         // this warp took the step's token
      for (int ri = first_res + (int)lsub * kTeams; ri < n_res; ri += kL * kTeams) {
        const int bu = res_b + ri;                        // unquantized unit: residual window first, then the sink
        const bool in_sink = bu >= res_units;
        const int wu = in_sink ? bu - res_units : bu;     // unit inside its window
        const int rt = in_sink ? f_ns : f_r;        // tokens in that window
        const int j0 = wu * 32;
        const char* resk = in_sink ? lv.sink + (size_t)s * lv.sink_stride : lv.resk + (size_t)s * lv.resk_stride;
        const bool holds_new = !in_sink && lv.new_k != nullptr && jn >= j0 && jn < j0 + 32;
        float Sx[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          const int ta = j0 + mt * 16 + r, tb = ta + 8;
          const uint4* rowa = reinterpret_cast<const uint4*>(resk + (size_t)ta * 256);
          const uint4* rowb = reinterpret_cast<const uint4*>(resk + (size_t)tb * 256);
          if (holds_new && lv.rope_cos == nullptr && ta == jn) rowa = reinterpret_cast<const uint4*>(lv.new_k + (size_t)s * kD);
          if (holds_new && lv.rope_cos == nullptr && tb == jn) rowb = reinterpret_cast<const uint4*>(lv.new_k + (size_t)s * kD);
          uint4 ka[4], kb[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            ka[j] = ta < rt ? rowa[4 * j + t] : make_uint4(0u, 0u, 0u, 0u);
            kb[j] = tb < rt ? rowb[4 * j + t] : make_uint4(0u, 0u, 0u, 0u);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint4 qq = lds128(qrow_u32 + (32 * j + 8 * t) * 2);
            mma_bf16(Sx[mt], ka[j].x, kb[j].x, ka[j].y, kb[j].y, qq.x, qq.y);
            mma_bf16(Sx[mt], ka[j].z, kb[j].z, ka[j].w, kb[j].w, qq.z, qq.w);
          }
        }
        takes_new = takes_new || holds_new;
        // hand over (the buffer is free once the partner has taken the previous unquantized unit)
        wait_or_give_up(rempty_u32 + 8 * lsub, (rit[0] & 1u) ^ 1u);
        const uint32_t rb = ring_u32 + kRBufBase + kRBufBytes * lsub + lane * 32;
        sts128(rb, __float_as_uint(Sx[0][0]), __float_as_uint(Sx[0][1]), __float_as_uint(Sx[0][2]), __float_as_uint(Sx[0][3]));
        sts128(rb + 16, __float_as_uint(Sx[1][0]), __float_as_uint(Sx[1][1]), __float_as_uint(Sx[1][2]), __float_as_uint(Sx[1][3]));
        __syncwarp();
        mbar_arrive_one(rfull_u32 + 8 * lsub);
        ++rit[0];
      }

      // ---- packed units
      // B fragments of q for the base key tiles: head r, channels 16kt + {2t, 2t+1} and {2t+8, 2t+9}, times mult(kt)
      uint32_t bq[8][2];
#pragma unroll
      for (int kt = 0; kt < 8; ++kt) {
        const float mult = (float)(1 << (8 - key_pos(kt)));
#pragma unroll
        for (int hch = 0; hch < 2; ++hch) {
          const uint32_t w = lds32(qrow_u32 + (16 * kt + 8 * hch + 2 * t) * 2);
          bq[kt][hch] = pack_half2(bf_lo(w) * mult, bf_hi(w) * mult);
        }
      }
      // per-lane constants of the key-group preparation: the lane converts channels 4*lane .. 4*lane+3 (k-tile lane / 4)
      const float pk_zs = __uint_as_float((119u + (uint32_t)key_pos(lane >> 2)) << 23);        // 2^(pos - 8)
      const uint32_t kprep_u32 = ring_u32 + kPrepBase + lsub * kKeyPrepBytes;
      const uint32_t kp_wr = kprep_u32 + kprep_off(lane >> 2, 2 * (lane & 1)) + 8 * ((lane >> 1) & 1);
      const uint32_t zp_wr = kp_wr + kZprepOff;
      const uint32_t kp_rd = kprep_u32 + 16 * t;
      const uint32_t zp_rd = kprep_u32 + kZprepOff + 16 * t;
      const uint32_t lane16 = ring_u32 + lane * 16;
      // byte offset inside the scale table of channel c's scale (half)
      auto scale_byte = [&](uint32_t c) -> uint32_t {
        const int kt = c >> 4, col = c & 15;
        return c < 128 ? (uint32_t)(kprep_off(kt, (col & 7) >> 1) + 8 * (col >> 3) + 2 * (col & 1)) : 0xFFFFu;
      };
      float zc[4] = {0.f, 0.f, 0.f, 0.f};   // zero-point terms q . z: [0..1] of unit 0's key group, [2..3] of unit 1's
      // three tiers: the block's first 2 kPlanePairs UINT4 channels (two tiles of eight pairs): B fragments (gathered fp16
      // query pairs) and, per pair, where the two channels' scales sit in the scale table (0xFFFF: no channel)
      uint32_t u4q[2][2] = {{0u, 0u}, {0u, 0u}}, u4s[2][2] = {{~0u, ~0u}, {~0u, ~0u}};
      // B fragment of the block's first 2 kRowPairs promoted channels (gathered query entries; 0 past the count)
      uint32_t xb = 0u;
      // query entries of a pair of channel numbers (0xFF: no channel)
      auto query_pair = [&](uint32_t row, uint32_t two) -> uint32_t {
        const uint32_t c0 = two & 0xFFu, c1 = (two >> 8) & 0xFFu;
        return (c0 < 128 ? lds16(row + 2 * c0) : 0u) | ((c1 < 128 ? lds16(row + 2 * c1) : 0u) << 16);
      };
      if (lsub == 1u) advance_stage();
#pragma unroll 1
      for (int i = (int)lsub; i < n_steps; i += kL) {
        wait_or_give_up(bar_u32 + ring_stage * 8u, ring_parity);
        const uint32_t stg = lane16 + ring_stage * kStageBytes;         // this lane's 16 bytes of the stage's first section
        // G = 128: the group's second half finds the tables as the first left them
        const bool has_meta = UPG != 4 || kMetaAlways || i == 0 || (((wb >> 1) + i) & 1) == 0;
        // the extras of a later step are requested into the slot that was read in the step before; this step's have arrived
        const uint32_t later = request_extras(slot == 0 ? kSlotCount - 1 : slot - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(kSlotCount - 1) : "memory");
        // the key codes: two 16-byte loads per lane and unit are the A fragments of all its sixteen key tiles
        uint4 kw[2][2];
#pragma unroll
        for (int un = 0; un < 2; ++un) {
          kw[un][0] = lds128(stg + 512 + un * kUnitStep);
          kw[un][1] = lds128(stg + 512 + un * kUnitStep + 512);
        }
        // ---- key-group preparation: fp16 scale pairs {s, -4s} in fragment order, zero-point tile.  The tables of the
        // previous step were last read by this warp alone.
        if (has_meta) {
          __syncwarp();
          uint32_t za[2], zb[2];
#pragma unroll
          for (int gi = 0; gi < kGroups; ++gi) {
            const uint4 mz = lds128(stg + gi * (512 + kUnitBytes));   // channels 4*lane .. 4*lane+3
            const uint32_t neg4 = 0xC400C400u;   // half2(-4, -4)
            const uint32_t ma = pack_half2(bf_lo(mz.x), bf_lo(mz.y)), mb = pack_half2(bf_lo(mz.z), bf_lo(mz.w));
            sts64(kp_wr + kKprepGroup * gi, ma, hmul2_u(ma, neg4));
            sts64(kp_wr + kKprepGroup * gi + 16, mb, hmul2_u(mb, neg4));
            za[gi] = pack_half2(bf_hi(mz.x) * pk_zs, bf_hi(mz.y) * pk_zs);
            zb[gi] = pack_half2(bf_hi(mz.z) * pk_zs, bf_hi(mz.w) * pk_zs);
          }
          sts64(zp_wr, za[0], za[kGroups - 1]);
          sts64(zp_wr + 16, zb[0], zb[kGroups - 1]);
        }
        __syncwarp();      // tables and extras are read by other lanes below, and the key codes' place is written at the end

        float Sx[2][2][4];
#pragma unroll
        for (int un = 0; un < 2; ++un)
#pragma unroll
          for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int k = 0; k < 4; ++k) Sx[un][mt][k] = 0.f;
        const uint32_t slot_u32 = slot0_u32 + slot * kSlotBytes;
        const int n16p = counts[0] & 0xFF, n4pairs = (((counts[0] >> 8) & 0xFF) + 1) >> 1;
        if (counts[0] & 0x10000u) {
          // a block begins: its channel lists
          xb = t < n16p ? query_pair(qrow_u32, lds16(slot_u32 + 2 * t)) : 0u;
          if constexpr (kU4 == 1) {
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
#pragma unroll
              for (int hp = 0; hp < 2; ++hp) {
                const int p = 8 * kk + 4 * hp + t;
                const uint32_t two = p < n4pairs ? lds16(slot_u32 + 2 * n16p + 2 * p) : 0xFFFFu;
                u4q[kk][hp] = query_pair(qfrow_u32, two);
                u4s[kk][hp] = scale_byte(two & 0xFFu) | (scale_byte(two >> 8) << 16);
              }
          }
        }
        // where the step's extras lie in global memory, for what the slot does not hold
        const bool spill16 = n16p > kRowPairs, spill4 = kU4 == 1 && n4pairs > kPlanePairs;
        const char* exu = nullptr;
        uint32_t ex_unit = 0u;
        if (spill16 || spill4) {
          ex_unit = extras_unit_bytes(2 * n16p, 2 * n4pairs, kU4 == 2);
          exu = extras + (size_t)lds32(slot_u32 + kWhereOff) * 16;
        }
        // ---- promoted channels: raw bf16 keys (A fragments with k = 8: lane (r, t) holds channel pair t for tokens r, r + 8 of
        // both m-tiles), a gathered q.  Pairs past the count read the last pair (their query entries are 0).
        if (n16p > 0) {
          const uint32_t row = slot_u32 + kRowsOff + 128 * min(t, n16p - 1) + 4 * r, sw = 32 * min(t, n16p - 1);
#pragma unroll
          for (int un = 0; un < 2; ++un)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
              mma_bf16_k8(Sx[un][mt], lds32(row + un * (kRowPairs * 128) + (sw ^ (64 * mt))), lds32(row + un * (kRowPairs * 128) + (sw ^ (64 * mt + 32))), xb);
          if (spill16) {
#pragma unroll kSpillUnroll
            for (int p0 = kRowPairs; p0 < n16p; p0 += 4) {
              const int p = min(p0 + t, n16p - 1);
              const uint32_t b = p0 + t < n16p ? query_pair(qrow_u32, lds16(slot_u32 + 2 * p)) : 0u;
              const char* e = exu + (p * 32 + r) * 4;
#pragma unroll
              for (int un = 0; un < 2; ++un)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
                  mma_bf16_k8(Sx[un][mt], *reinterpret_cast<const uint32_t*>(e + un * ex_unit + 64 * mt),
                              *reinterpret_cast<const uint32_t*>(e + un * ex_unit + 64 * mt + 32), b);
            }
          }
        }
        // ---- UINT4 high plane (three tiers): c_hi * 4s, gathered q in fp16.  The first two tiles (32 channels) use the
        // block's gathered query pairs and scale positions; further tiles look their channels up per step.
        if constexpr (kU4 == 1) {
          if (n4pairs > 0) {
            const uint32_t kpb = kprep_u32;
            auto plane_tile = [&](int un, const uint32_t (&words)[2], const uint32_t (&sidx)[2], const uint32_t (&qb)[2]) {
              uint32_t a[2][4];
#pragma unroll
              for (int hp = 0; hp < 2; ++hp) {
                const uint32_t w = words[hp] >> (8 * (r >> 2));
                const uint32_t i0 = sidx[hp] & 0xFFFFu, i1 = sidx[hp] >> 16;
                const uint32_t tb = kpb + (UPG == 1 ? kKprepGroup * un : 0);
                const uint32_t s0 = i0 != 0xFFFFu ? lds16(tb + i0) : 0u;
                const uint32_t s1 = i1 != 0xFFFFu ? lds16(tb + i1) : 0u;
                const uint32_t sc = s0 | (s1 << 16);
                const uint32_t m4 = hmul2_u(sc, four2);                // 4s
                const uint32_t o4 = hmul2_u(sc, 0xCC00CC00u);          // -16s
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                  for (int rh = 0; rh < 2; ++rh) {
                    const int f = 2 * mt + rh;
                    const uint32_t code = ((w << (8 - 2 * f)) & 0x03000300u) | four2;          // 4 + c_hi
                    a[mt][2 * hp + rh] = hfma2_u(code, m4, o4);                                // c_hi * 4s
                  }
              }
#pragma unroll
              for (int mt = 0; mt < 2; ++mt) mma_f16(Sx[un][mt], a[mt][0], a[mt][1], a[mt][2], a[mt][3], qb[0], qb[1]);
            };
            {
              const uint32_t pl = slot_u32 + kPlaneOff + 16 * t + 4 * (r & 3);
#pragma unroll
              for (int kk = 0; kk < 2; ++kk) {
                if (kk * 8 < n4pairs) {
#pragma unroll
                  for (int un = 0; un < 2; ++un) {
                    // (pairs past the count have zero scales and query entries)
                    const uint32_t words[2] = {lds32(pl + un * (16 * kPlanePairs) + 128 * kk), lds32(pl + un * (16 * kPlanePairs) + 128 * kk + 64)};
                    plane_tile(un, words, u4s[kk], u4q[kk]);
                  }
                }
              }
            }
            if (spill4) {
              for (int p0 = kPlanePairs; p0 < n4pairs; p0 += 8) {
                uint32_t sidx[2], qb[2], words[2][2] = {{0u, 0u}, {0u, 0u}};
#pragma unroll
                for (int hp = 0; hp < 2; ++hp) {
                  const int p = p0 + 4 * hp + t;
                  uint32_t two = 0xFFFFu;
                  if (p < n4pairs) {
                    two = lds16(slot_u32 + 2 * n16p + 2 * p);
#pragma unroll
                    for (int un = 0; un < 2; ++un)
                      words[un][hp] = reinterpret_cast<const uint32_t*>(exu + un * ex_unit + 128 * n16p)[p * 4 + (r & 3)];
                  }
                  qb[hp] = query_pair(qfrow_u32, two);
                  sidx[hp] = scale_byte(two & 0xFFu) | (scale_byte(two >> 8) << 16);
                }
#pragma unroll
                for (int un = 0; un < 2; ++un) plane_tile(un, words[un], sidx, qb);
              }
            }
          }
        }
        // ---- q.K^T on the key tiles.  One pass over a plane of 2-bit codes: the base (low) plane with the scales s, and,
        // with a 4-bit base, first the dense high plane (codes c >> 2, laid out like the low plane) with the scales 4s.
        auto key_pass = [&](const uint4 (&w)[2][2], bool high) {
#pragma unroll
          for (int kt = 0; kt < 8; ++kt) {
            // scales of the lane's channel pairs (16kt + 2t, +1) and (16kt + 8 + 2t, +1); code bias 4 -> offset -4 s
            uint4 kp[2];
#pragma unroll
            for (int gi = 0; gi < kGroups; ++gi) {
              kp[gi] = lds128(kp_rd + kKprepGroup * gi + kprep_off(kt, 0));
              if (high) kp[gi] = make_uint4(hmul2_u(kp[gi].x, four2), hmul2_u(kp[gi].y, four2), hmul2_u(kp[gi].z, four2), hmul2_u(kp[gi].w, four2));
            }
            const uint32_t mask = 0x00030003u << key_pos(kt);
#pragma unroll
            for (int un = 0; un < 2; ++un) {
              const uint4& k4 = kp[un & (kGroups - 1)];
#pragma unroll
              for (int mt = 0; mt < 2; ++mt) {
                const uint32_t kwd[4] = {w[un][mt].x, w[un][mt].y, w[un][mt].z, w[un][mt].w};
                uint32_t a[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const uint32_t code = (key_shift(kwd[j], kt) & mask) | four2;              // 4 + c * 2^(pos-8)
                  a[j] = hfma2_u(code, j < 2 ? k4.x : k4.z, j < 2 ? k4.y : k4.w);            // c * s * 2^(pos-8)
                }
                mma_f16(Sx[un][mt], a[0], a[1], a[2], a[3], bq[kt][0], bq[kt][1]);
              }
            }
          }
        };
        if constexpr (kU4 == 2) {
          if (n16p + n4pairs > 0) {          // (a block whose extras did not fit the arena has no high plane)
            const uint32_t pl = slot_u32 + kPlaneOff + 16 * lane;
            const uint4 hw[2][2] = {{lds128(pl), lds128(pl + 512)}, {lds128(pl + 1024), lds128(pl + 1536)}};
            key_pass(hw, true);
          }
        }
        if (has_meta) {
          // the zero-point terms q . z: a tile chain of its own; the partner adds them to the logits
#pragma unroll
          for (int kt = 0; kt < 8; ++kt) {
            const uint4 zz = lds128(zp_rd + kprep_off(kt, 0));
            if (kt == 0) mma_f16_to(zc, zz.x, zz.y, zz.z, zz.w, bq[0][0], bq[0][1], 0.f, 0.f, 0.f, 0.f);
            else mma_f16(zc, zz.x, zz.y, zz.z, zz.w, bq[kt][0], bq[kt][1]);
          }
        }
        key_pass(kw, false);

        // ---- hand the logits over: [m-tile][tokens r / r + 8] x heads 2t, 2t+1, where the units' key codes were, and the
        // zero-point terms where the first group's scales were (every lane has read both, see the barrier above)
        {
          const uint32_t lb = stg + 512 + lane * 16;
#pragma unroll
          for (int un = 0; un < 2; ++un)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
              sts128(lb + un * kUnitStep + 16 * mt, __float_as_uint(Sx[un][mt][0]), __float_as_uint(Sx[un][mt][1]),
                     __float_as_uint(Sx[un][mt][2]), __float_as_uint(Sx[un][mt][3]));
          sts128(stg, __float_as_uint(zc[0]), __float_as_uint(zc[1]), __float_as_uint(zc[2]), __float_as_uint(zc[3]));
          __syncwarp();
          mbar_arrive_one(lfull_u32 + ring_stage * 8u);
        }
#pragma unroll
        for (int k = 0; k + 2 < kSlotCount; ++k) counts[k] = counts[k + 1];
        counts[kSlotCount - 2] = later;
        slot = slot + 1 == kSlotCount ? 0u : slot + 1;
        if constexpr (kL == 2) advance_stage();
        advance_stage();
      }
      // The step's bookkeeping comes last: the partner's chain hangs on the logits, nothing in this launch on these stores.
      // Four channels' sums run side by side.  Decode steps, 7b shape, batch 8: 32768 tokens, 28 layers 1134.6 -> 1126.0 us;
      // three tiers, 20011 tokens, 14 layers 524.3 -> 517.7.
      if (takes_new) {
        // store the new key row and add |q| to the importance accumulator (channels 4*lane .. 4*lane+3, heads
        // ascending: the order of the plain append)
        if (lv.rope_cos == nullptr) {
          const uint2 kn = reinterpret_cast<const uint2*>(lv.new_k + (size_t)s * kD)[lane];
          reinterpret_cast<uint2*>(lv.resk + (size_t)s * lv.resk_stride + (size_t)jn * 256)[lane] = kn;
        }
        double2* acc = reinterpret_cast<double2*>(lv.state + (size_t)s * lv.state_stride) + 2 * lane;
        double2 a0 = acc[0], a1 = acc[1];
        for (int h = 0; h < g; ++h) {
          const uint2 qh = lds64(qb16_u32 + (h * kQS + 4 * lane) * 2);
          a0.x = __dadd_rn(a0.x, (double)fabsf(bf_lo(qh.x)));
          a0.y = __dadd_rn(a0.y, (double)fabsf(bf_hi(qh.x)));
          a1.x = __dadd_rn(a1.x, (double)fabsf(bf_lo(qh.y)));
          a1.y = __dadd_rn(a1.y, (double)fabsf(bf_hi(qh.y)));
        }
        acc[0] = a0;
        acc[1] = a1;
        if (lane == 0) *reinterpret_cast<uint32_t*>(lv.state + (size_t)s * lv.state_stride + 1024) += (uint32_t)g;
      }
      if (gave_up && lane == 0) atomicOr(lv.status, (uint32_t)MIXKVQ_DEV_COPY_TIMEOUT);
    } else {
      // =====================================================================================================
      // values warp
      // =====================================================================================================
      float O[8][4];       // O^T tiles: [channel tile] x (channels r, r+8) x (heads 2t, 2t+1), scaled 2^-20
      float Zc[4] = {0.f, 0.f, 0.f, 0.f};   // rows 0..VG-1: sum p * z_v per value group; row 4: sum p
      float m0 = -INFINITY, m1 = -INFINITY; // running reference maximum (log2 domain) of heads 2t, 2t+1
#pragma unroll
      for (int ct = 0; ct < 8; ++ct)
#pragma unroll
        for (int i = 0; i < 4; ++i) O[ct][i] = 0.f;
      // raises the reference maximum to max(reference, u) and rescales what has been accumulated
      auto raise_reference = [&](float u0, float u1) {
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
          u0 = fmaxf(u0, __shfl_xor_sync(0xffffffffu, u0, off));
          u1 = fmaxf(u1, __shfl_xor_sync(0xffffffffu, u1, off));
        }
        const float n0 = fmaxf(m0, u0), n1 = fmaxf(m1, u1);
        const float a0 = exp2f(m0 - n0), a1 = exp2f(m1 - n1);    // exp2(-inf) = 0 on the first unit
#pragma unroll
        for (int ct = 0; ct < 8; ++ct) {
          O[ct][0] *= a0; O[ct][1] *= a1; O[ct][2] *= a0; O[ct][3] *= a1;
        }
        Zc[0] *= a0; Zc[1] *= a1; Zc[2] *= a0; Zc[3] *= a1;
        m0 = n0;
        m1 = n1;
      };

      // ---- unquantized units: bf16 values straight from global memory, 8x8 tiles transposed in registers
      uint32_t rsub = 0;                    // the logits warp that has the unit
      for (int ri = first_res; ri < n_res; ri += kTeams) {
        const int bu = res_b + ri;
        const bool in_sink = bu >= res_units;
        const int wu = in_sink ? bu - res_units : bu;
        const int rt = in_sink ? f_ns : f_r;
        const int j0 = wu * 32;
        const char* resv = in_sink ? lv.sink + (size_t)s * lv.sink_stride + (size_t)lv.sink_len * 256
                                   : lv.resv + (size_t)s * lv.resv_stride;
        const bool holds_new = !in_sink && lv.new_v != nullptr && jn >= j0 && jn < j0 + 32;
        // rows of this lane: tokens j0 + 8i + r, i = 0..3; word 2t.. of a 16-channel tile
        const uint32_t* rowp[4];
        bool rowv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tok = j0 + 8 * i + r;
          rowv[i] = tok < rt;
          rowp[i] = reinterpret_cast<const uint32_t*>(resv + (size_t)tok * 256) + t;
          if (holds_new && tok == jn) rowp[i] = reinterpret_cast<const uint32_t*>(lv.new_v + (size_t)s * kD) + t;
        }
        if (holds_new) {
          const uint2 vn = reinterpret_cast<const uint2*>(lv.new_v + (size_t)s * kD)[lane];
          reinterpret_cast<uint2*>(lv.resv + (size_t)s * lv.resv_stride + (size_t)jn * 256)[lane] = vn;
        }
        // the first tile's loads go out before the wait for the logits
        uint32_t x[2][4];      // [ks][{tokens r, channels lo}, {tokens r, channels hi}, {tokens r + 8, lo}, {tokens r + 8, hi}]
        auto load_tile = [&](int ct) {
#pragma unroll
          for (int ks = 0; ks < 2; ++ks)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              x[ks][2 * hh] = rowv[2 * ks + hh] ? rowp[2 * ks + hh][8 * ct] : 0u;
              x[ks][2 * hh + 1] = rowv[2 * ks + hh] ? rowp[2 * ks + hh][8 * ct + 4] : 0u;
            }
        };
        load_tile(0);
        wait_or_give_up(rfull_u32 + 8 * rsub, (rsub ? rit[kL - 1] : rit[0]) & 1u);
        const uint32_t rb = ring_u32 + kRBufBase + kRBufBytes * rsub + lane * 32;
        const uint4 s0 = lds128(rb), s1 = lds128(rb + 16);
        __syncwarp();
        mbar_arrive_one(rempty_u32 + 8 * rsub);
        if (rsub) ++rit[kL - 1];
        else ++rit[0];
        if constexpr (kL == 2) rsub ^= 1u;
        // logits (log2 domain) of tokens j0 + 16 mt + r (+ 8), heads 2t, 2t+1; tokens past the window count for nothing
        float xl[2][4];
        {
          const float sx[2][4] = {{__uint_as_float(s0.x), __uint_as_float(s0.y), __uint_as_float(s0.z), __uint_as_float(s0.w)},
                                  {__uint_as_float(s1.x), __uint_as_float(s1.y), __uint_as_float(s1.z), __uint_as_float(s1.w)}};
#pragma unroll
          for (int mt = 0; mt < 2; ++mt) {
            const bool va = (j0 + mt * 16 + r) < rt, vb = (j0 + mt * 16 + 8 + r) < rt;
            xl[mt][0] = va ? sx[mt][0] * scale_log2e : -INFINITY;
            xl[mt][1] = va ? sx[mt][1] * scale_log2e : -INFINITY;
            xl[mt][2] = vb ? sx[mt][2] * scale_log2e : -INFINITY;
            xl[mt][3] = vb ? sx[mt][3] * scale_log2e : -INFINITY;
          }
        }
        raise_reference(fmaxf(fmaxf(xl[0][0], xl[0][2]), fmaxf(xl[1][0], xl[1][2])),
                        fmaxf(fmaxf(xl[0][1], xl[0][3]), fmaxf(xl[1][1], xl[1][3])));
        // probabilities scaled 2^-20 (the scale of the accumulators), as an exact bf16 pair (high part, remainder);
        // B fragments [k-step][tokens 2t.. / 2t+8..] of head r
        uint32_t Bh[2][2], Bl[2][2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const float p0 = exp2f(xl[mt][2 * hh] - m0) * 9.5367431640625e-07f;
            const float p1 = exp2f(xl[mt][2 * hh + 1] - m1) * 9.5367431640625e-07f;
            const uint32_t hi = pack_bf162(p0, p1);
            Bh[mt][hh] = movmatrix_trans(hi);
            Bl[mt][hh] = movmatrix_trans(pack_bf162(p0 - bf_lo(hi), p1 - bf_hi(hi)));
          }
        // denominator: row 4 of the extra tile is 2^20, which undoes the scale of the probabilities
        const uint32_t ones = (r == 4) ? 0x49804980u : 0u;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          mma_bf16(Zc, ones, 0u, ones, 0u, Bh[ks][0], Bh[ks][1]);
          mma_bf16(Zc, ones, 0u, ones, 0u, Bl[ks][0], Bl[ks][1]);
        }
        // tile (ct, ks): A = V^T, 16 channels x 16 tokens: a0 = (channels r, tokens 2t..), a1 = (channels r + 8, tokens 2t..),
        // a2 = (channels r, tokens 8 + 2t..), a3 = (channels r + 8, tokens 8 + 2t..)
#pragma unroll
        for (int ct = 0; ct < 8; ++ct) {
          uint32_t a[2][4];
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            a[ks][0] = movmatrix_trans(x[ks][0]);
            a[ks][1] = movmatrix_trans(x[ks][1]);
            a[ks][2] = movmatrix_trans(x[ks][2]);
            a[ks][3] = movmatrix_trans(x[ks][3]);
          }
          if (ct + 1 < 8) load_tile(ct + 1);
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            mma_bf16(O[ct], a[ks][0], a[ks][1], a[ks][2], a[ks][3], Bh[ks][0], Bh[ks][1]);
            mma_bf16(O[ct], a[ks][0], a[ks][1], a[ks][2], a[ks][3], Bl[ks][0], Bl[ks][1]);
          }
        }
      }

      // ---- packed units
      // per-lane constants of the value-group preparation: the lane converts the scales and zero-points of tokens 2 pi,
      // 2 pi + 1 of a unit, VG / 2 groups of them (VG = 1: of unit lane / 16)
      // value scales: [4 t: 20 words][4 vg][2 ks][2 ch] half2 s_v'; zero-point tile: [2 ks: 68 words][8 rows][4 t][2 ch] half2
      // (rows < VG z_v, row 4 ones)
      const int pi = VG == 1 ? lane & 15 : lane >> 1, vg0 = VG == 1 ? 0 : (lane & 1) * (VG / 2);
      const int p_ks = pi >> 3, p_ch = (pi >> 2) & 1, p_t = pi & 3;
      const float pv_up = __uint_as_float((131u - 2u * (uint32_t)(2 * p_ks + p_ch)) << 23);          // 2^(4 - 2 * (2 ks + ch))
      const uint32_t sv_wr = ring_u32 + kPrepBase + svp_off(kU4) + (VG == 1 ? (uint32_t)(lane >> 4) * kSvpUnit : 0u) +
                             4 * (p_t * 20 + vg0 * 4 + p_ks * 2 + p_ch);
      const uint32_t zv_wr = ring_u32 + kPrepBase + zvp_off(kU4) + (VG == 1 ? (uint32_t)(lane >> 4) * kZvpUnit : 0u) +
                             4 * (p_ks * 68 + vg0 * 8 + p_t * 2 + p_ch);
      const uint32_t sv_rd = ring_u32 + kPrepBase + svp_off(kU4) + t * 80;
      const uint32_t zv_rd = ring_u32 + kPrepBase + zvp_off(kU4) + lane * 8;
      const uint32_t lane16 = ring_u32 + lane * 16;
      const uint32_t vm_rd = ring_u32 + 512 + 2048 + (2 * pi) * (4 * VG) + 4 * vg0 + (VG == 1 ? (uint32_t)(lane >> 4) * kUnitStep : 0u);
#pragma unroll 1
      for (int i = 0; i < n_steps; ++i) {
        wait_or_give_up(bar_u32 + ring_stage * 8u, ring_parity);
        const uint32_t st = lane16 + ring_stage * kStageBytes + 512;      // this lane's 16 bytes of the first unit's first section
        // ---- value-group preparation.  The tables of the previous step were last read before the warp barrier that closed
        // it.
        {
          const uint32_t vm = vm_rd + ring_stage * kStageBytes;
          auto convert = [&](uint32_t m0, uint32_t m1, int un, int k) {          // {s, z} of the pair's two tokens, group vg0 + k
            sts32(sv_wr + un * kSvpUnit + 16 * k, pack_half2(bf_lo(m0) * pv_up, bf_lo(m1) * pv_up));
            sts32(zv_wr + un * kZvpUnit + 32 * k, pack_half2(bf_hi(m0), bf_hi(m1)));
          };
          if constexpr (VG == 4) {
#pragma unroll
            for (int un = 0; un < 2; ++un) {
              const uint2 a = lds64(vm + un * kUnitStep), b = lds64(vm + un * kUnitStep + 16);
              convert(a.x, b.x, un, 0);
              convert(a.y, b.y, un, 1);
            }
          } else if constexpr (VG == 2) {
#pragma unroll
            for (int un = 0; un < 2; ++un) convert(lds32(vm + un * kUnitStep), lds32(vm + un * kUnitStep + 8), un, 0);
          } else {
            const uint2 a = lds64(vm);
            convert(a.x, a.y, 0, 0);
          }
        }
        uint4 vw[2][2];
#pragma unroll
        for (int un = 0; un < 2; ++un) {
          vw[un][0] = lds128(st + un * kUnitStep + 1024);
          vw[un][1] = lds128(st + un * kUnitStep + 1536);
        }
        __syncwarp();      // the tables written above are read by other lanes below
        wait_or_give_up(lfull_u32 + ring_stage * 8u, ring_parity);
        float sx[2][2][4];
        {
          const uint32_t lb = st + lane * 16;
#pragma unroll
          for (int un = 0; un < 2; ++un)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
              const uint4 x = lds128(lb + un * kUnitStep + 16 * mt);
              sx[un][mt][0] = __uint_as_float(x.x); sx[un][mt][1] = __uint_as_float(x.y);
              sx[un][mt][2] = __uint_as_float(x.z); sx[un][mt][3] = __uint_as_float(x.w);
            }
        }
        const uint4 zq = lds128(st - 512);
        // logit = (sx + q . z) * scale: the zero-point term of the key group is the same for every token of the unit
        const float zl[2][2] = {{__uint_as_float(zq.x) * scale_log2e, __uint_as_float(zq.y) * scale_log2e},
                                {__uint_as_float(UPG == 1 ? zq.z : zq.x) * scale_log2e, __uint_as_float(UPG == 1 ? zq.w : zq.y) * scale_log2e}};
        // ---- online softmax (log2 domain); heads 2t, 2t+1; tokens r, r+8 of each m-tile.
        // The reference is the largest logit so far: a probability is exact in fp16 only where it is the reference, and the
        // largest matter most.  (Raising it only when it is exceeded by 3 or more keeps the probabilities inside the fp16 range as well
        // and is 0.5 to 1 % faster; relative error then against now: three tiers, 7b shape, 32768 tokens 1.25e-4 / 0.75e-4, 4-bit base, 8b
        // shape, 16384 tokens 1.96e-4 / 1.10e-4, two tiers, 32b shape, 8000 tokens 1.83e-4 / 1.10e-4.)
        {
          float uu[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float a = fmaf(fmaxf(fmaxf(sx[0][0][h], sx[0][0][2 + h]), fmaxf(sx[0][1][h], sx[0][1][2 + h])), scale_log2e, zl[0][h]);
            const float b = fmaf(fmaxf(fmaxf(sx[1][0][h], sx[1][0][2 + h]), fmaxf(sx[1][1][h], sx[1][1][2 + h])), scale_log2e, zl[1][h]);
            uu[h] = fmaxf(a, b);
          }
          if (__any_sync(0xffffffffu, uu[0] > m0 || uu[1] > m1)) raise_reference(uu[0], uu[1]);
        }
        // P^T B fragments: [unit][k-step][tokens 2t.. / 2t+8..], head r
        uint32_t Pt[2][2][2];
#pragma unroll
        for (int un = 0; un < 2; ++un) {
          const float c0 = zl[un][0] - m0, c1 = zl[un][1] - m1;
#pragma unroll
          for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh)
              Pt[un][mt][hh] = movmatrix_trans(pack_half2(ex2_approx(fmaf(sx[un][mt][2 * hh], scale_log2e, c0)),
                                                          ex2_approx(fmaf(sx[un][mt][2 * hh + 1], scale_log2e, c1))));
        }
        // ---- zero-point and denominator tile: rows 0..VG-1 = z_v of the group, row 4 = ones, the rest zero
#pragma unroll
        for (int un = 0; un < 2; ++un)
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            const uint2 zz = lds64(zv_rd + un * kZvpUnit + ks * 272);
            mma_f16(Zc, zz.x, 0u, zz.y, 0u, Pt[un][ks][0], Pt[un][ks][1]);
          }
        // ---- P.V: codes as fp16 subnormals, scales folded into P; with 4-bit values then the high plane (codes >> 2, the
        // low plane's bit order) with four times the scale
        auto value_pass = [&](const uint4 (&w)[2][2], bool high) {
#pragma unroll
          for (int vg = 0; vg < VG; ++vg) {
            uint32_t Bp[2][2][2];
#pragma unroll
            for (int un = 0; un < 2; ++un) {
              const uint4 sv = lds128(sv_rd + un * kSvpUnit + vg * 16);
              Bp[un][0][0] = hmul2_u(Pt[un][0][0], sv.x); Bp[un][0][1] = hmul2_u(Pt[un][0][1], sv.y);
              Bp[un][1][0] = hmul2_u(Pt[un][1][0], sv.z); Bp[un][1][1] = hmul2_u(Pt[un][1][1], sv.w);
              if (high) {
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                  Bp[un][ks][0] = hmul2_u(Bp[un][ks][0], four2);
                  Bp[un][ks][1] = hmul2_u(Bp[un][ks][1], four2);
                }
              }
            }
#pragma unroll
            for (int un = 0; un < 2; ++un) {
              const uint32_t vwd[8] = {w[un][0].x, w[un][0].y, w[un][0].z, w[un][0].w, w[un][1].x, w[un][1].y, w[un][1].z, w[un][1].w};
#pragma unroll
              for (int ks = 0; ks < 2; ++ks) {
                const uint32_t mk0 = 0x00030003u << (4 * ks), mk1 = 0x00030003u << (4 * ks + 2);
#pragma unroll
                for (int c = 0; c < TPG; ++c) {
                  const int ct = vg * TPG + c;
                  const uint32_t x0 = vwd[ct], x1 = vwd[ct] >> 8;
                  mma_f16(O[ct], x0 & mk0, x1 & mk0, x0 & mk1, x1 & mk1, Bp[un][ks][0], Bp[un][ks][1]);
                }
              }
            }
          }
        };
        value_pass(vw, false);
        if constexpr (kV4) {
#pragma unroll
          for (int un = 0; un < 2; ++un) {
            vw[un][0] = lds128(st + un * kUnitStep + 2048 + 128 * VG);
            vw[un][1] = lds128(st + un * kUnitStep + 2048 + 128 * VG + 512);
          }
          value_pass(vw, true);
        }
        // ---- both warps are done with the step: refill the stage (the logits were written to it by ordinary stores)
        __syncwarp();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(ring_stage, false);
        advance_stage();
      }
      if (__any_sync(0xffffffffu, gave_up)) {
        gave_up = true;
        if (lane == 0) atomicOr(lv.status, (uint32_t)MIXKVQ_DEV_COPY_TIMEOUT);
        // after the wait that ran out no wait was made and no stage refilled, so the last copies may still be on their way, and
        // they write to the ring: wait for them (bounded) before the ring is reused below or the CTA ends
        for (int i = max(0, issued - kStages); i < issued; ++i) {
          const uint32_t pos = stage0 + (uint32_t)i;
          mbar_wait_polls(bar_u32 + (pos % (uint32_t)kStages) * 8u, parity0 ^ ((pos / (uint32_t)kStages) & 1u), lv.wait_polls ? lv.wait_polls : kWaitPolls);
        }
        // what this warp accumulated is not a result: the team contributes nothing
#pragma unroll
        for (int ct = 0; ct < 8; ++ct)
#pragma unroll
          for (int i = 0; i < 4; ++i) O[ct][i] = 0.f;
        Zc[0] = Zc[1] = Zc[2] = Zc[3] = 0.f;
        m0 = m1 = -INFINITY;
      }

      // ---- finish this team's split: true scale, zero-point terms, denominator
#pragma unroll
      for (int ct = 0; ct < 8; ++ct) {
        const int vg = ct / TPG;
        const float z0 = __shfl_sync(0xffffffffu, Zc[0], vg * 4 + t), z1 = __shfl_sync(0xffffffffu, Zc[1], vg * 4 + t);
        O[ct][0] = fmaf(O[ct][0], 1048576.0f, z0);
        O[ct][1] = fmaf(O[ct][1], 1048576.0f, z1);
        O[ct][2] = fmaf(O[ct][2], 1048576.0f, z0);
        O[ct][3] = fmaf(O[ct][3], 1048576.0f, z1);
      }
      const float l0 = __shfl_sync(0xffffffffu, Zc[0], 16 + t), l1 = __shfl_sync(0xffffffffu, Zc[1], 16 + t);
      if (r == 0) {
        mS[team * 8 + 2 * t] = m0;
        mS[team * 8 + 2 * t + 1] = m1;
        lS[team * 8 + 2 * t] = l0;
        lS[team * 8 + 2 * t + 1] = l1;
      }
      // the team's unnormalized output goes to its own, now idle, ring as [8 heads][132] floats
      float* mine = reinterpret_cast<float*>(smem + team * kTeamBytes);
#pragma unroll
      for (int ct = 0; ct < 8; ++ct) {
        mine[(2 * t) * kMergeStride + 16 * ct + r] = O[ct][0];
        mine[(2 * t + 1) * kMergeStride + 16 * ct + r] = O[ct][1];
        mine[(2 * t) * kMergeStride + 16 * ct + 8 + r] = O[ct][2];
        mine[(2 * t + 1) * kMergeStride + 16 * ct + 8 + r] = O[ct][3];
      }
    }

    // the next segment goes on where this one's steps end
    {
      const uint32_t pos = stage0 + (uint32_t)n_steps;
      ring_stage = pos % (uint32_t)kStages;
      ring_parity = (parity0 ^ (pos / (uint32_t)kStages)) & 1u;
    }
    // ---- merge the teams of the CTA, write the partial of (CTA, stream): the 16 threads that own a head add the teams'
    // rows with the factors 2^(m_p - M).
    __syncthreads();
    for (int idx = threadIdx.x; idx < 256; idx += kThreads) {
      const int h = idx >> 5, c = 4 * (idx & 31);          // head, first of the thread's four channels
      float M = -INFINITY, L = 0.f, f[kTeams];
#pragma unroll
      for (int w = 0; w < kTeams; ++w) M = fmaxf(M, mS[w * 8 + h]);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < kTeams; ++w) {
        const float mw = mS[w * 8 + h];
        f[w] = (mw == -INFINITY) ? 0.f : ex2_approx(mw - M);
        L += f[w] * lS[w * 8 + h];
        const float4 o = *reinterpret_cast<const float4*>(smem + w * kTeamBytes + (h * kMergeStride + c) * 4);
        acc.x += f[w] * o.x; acc.y += f[w] * o.y; acc.z += f[w] * o.z; acc.w += f[w] * o.w;
      }
      if constexpr (kDirect) {
        // (l == 0: the teams gave up, the status word says so)
        if (h < g) {
          const float inv = L > 0.f ? 1.f / L : 0.f;
          const size_t row = (size_t)s * g + h;           // (b Hkv + hk) g + h = b Hq + hk g + h
          *reinterpret_cast<float4*>(out + row * kD + c) = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
          // natural logarithm of the softmax denominator (the maximum is kept in the base-2 domain)
          if (lse_out != nullptr && c == 0) lse_out[row] = L > 0.f ? (M + log2f(L)) * 0.6931471805599453f : -INFINITY;
        }
      } else {
        float* part = ws + (size_t)(blockIdx.x + s) * kPartialFloats + h * 130;
        *reinterpret_cast<float2*>(part + 2 + c) = make_float2(acc.x, acc.y);
        *reinterpret_cast<float2*>(part + 4 + c) = make_float2(acc.z, acc.w);
        if (c == 0) *reinterpret_cast<float2*>(part) = make_float2(M, L);
      }
    }
    if (seg < ce) {
      // another segment follows: its copies are staged into the rings that were just read
      __syncthreads();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
  }
}

template <int G, int kU4, bool kV4, bool kDirect>
cudaError_t launch_d(const LayerView& lv, const __nv_bfloat16* qb, float sl, float* ws, int grid, float* out, float* lse, cudaStream_t stream) {
  return launch_dependent(attention_ws_kernel<G, kU4, kV4, kDirect>, dim3((unsigned)grid), threads_of(kU4, kV4), smem_bytes(G, kU4, kV4), stream, lv, qb, sl, 0x44004400u, ws, out, lse);
}
template <int G, int kU4, bool kV4>
cudaError_t launch_v(const LayerView& lv, const __nv_bfloat16* qb, float sl, float* ws, int grid, float* out, float* lse, cudaStream_t stream) {
  return out != nullptr ? launch_d<G, kU4, kV4, true>(lv, qb, sl, ws, grid, out, lse, stream)
                        : launch_d<G, kU4, kV4, false>(lv, qb, sl, ws, grid, out, lse, stream);
}
template <int G, int kU4>
cudaError_t launch_one(const LayerView& lv, const __nv_bfloat16* qb, float sl, float* ws, int grid, float* out, float* lse, cudaStream_t stream) {
  return lv.v_bits == 4 ? launch_v<G, kU4, true>(lv, qb, sl, ws, grid, out, lse, stream)
                        : launch_v<G, kU4, false>(lv, qb, sl, ws, grid, out, lse, stream);
}

template <int G>
cudaError_t launch_g(const LayerView& lv, const void* q, float scale, float* ws, int grid, float* out, float* lse,
                     cudaStream_t stream) {
  const __nv_bfloat16* qb = static_cast<const __nv_bfloat16*>(q);
  const float sl = scale * 1.4426950408889634f;
  if (lv.dense_hi) return launch_one<G, 2>(lv, qb, sl, ws, grid, out, lse, stream);
  const bool uses_u4 = (lv.budget_bf16 + lv.budget_u4 > 0) ? lv.budget_u4 > 0 : lv.tau_u4 < lv.tau_bf16;
  if (uses_u4) return launch_one<G, 1>(lv, qb, sl, ws, grid, out, lse, stream);
  return launch_one<G, 0>(lv, qb, sl, ws, grid, out, lse, stream);
}

}  // namespace

template <int G, int kU4, bool kV4, bool kDirect>
static cudaError_t setup_d() {
  cudaError_t e = cudaFuncSetAttribute(attention_ws_kernel<G, kU4, kV4, kDirect>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       smem_bytes(G, kU4, kV4));
  if (e != cudaSuccess) return e;
  // the CTAs of an SM only fit with the largest shared-memory carve-out; ask for it explicitly
  return cudaFuncSetAttribute(attention_ws_kernel<G, kU4, kV4, kDirect>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)cudaSharedmemCarveoutMaxShared);
}
template <int G, int kU4, bool kV4>
static cudaError_t setup_v() {
  cudaError_t e = setup_d<G, kU4, kV4, false>();
  return e != cudaSuccess ? e : setup_d<G, kU4, kV4, true>();
}
template <int G, int kU4>
static cudaError_t setup_one() {
  cudaError_t e = setup_v<G, kU4, false>();
  return e != cudaSuccess ? e : setup_v<G, kU4, true>();
}
template <int G>
static cudaError_t setup_g() {
  cudaError_t e = setup_one<G, 0>();
  if (e != cudaSuccess) return e;
  e = setup_one<G, 1>();
  return e != cudaSuccess ? e : setup_one<G, 2>();
}

cudaError_t attention_ws_setup() {
  cudaError_t e = setup_g<32>();
  if (e != cudaSuccess) return e;
  e = setup_g<64>();
  if (e != cudaSuccess) return e;
  e = setup_g<128>();
  return e != cudaSuccess ? e : attention_single_setup();
}

// Split positions per stream: packed units plus the weighted units of the residual window and the sink.
long long attention_ws_positions(const LayerView& lv) {
  return (long long)lv.n_blocks * lv.U + (long long)kResidualWeight * ((lv.r + 31) / 32 + (lv.n_sink + 31) / 32);
}

// Split positions of one stream with the given fill (the entry w of a ragged batch's table)
int attention_ws_positions_of(int n_blocks, int r, int n_sink, int U) {
  return n_blocks * U + kResidualWeight * ((r + 31) / 32 + (n_sink + 31) / 32);
}

// Ragged batch: every stream gets CTAs of its own, as many as make the longest share as short as it can be with about two CTAs
// per SM.  (An even split of all positions, wherever the boundaries fall, gave CTAs that straddle two or three streams and
// drain, reload and merge for each: eight sequences of 640 to 32768 tokens, 31.6 us for the split kernel, 24.8 us so.)
int attention_ws_ragged_split(const int* w, int B, int Hkv, int n_sms, int* ctas) {
  long long total = 0, streams = 0;
  int longest = 1;
  for (int b = 0; b < B; ++b) {
    total += (long long)Hkv * w[b];
    streams += w[b] > 0 ? Hkv : 0;
    longest = max(longest, w[b]);
  }
  const long long even = min((long long)min(n_sms * kCtasPerSm, kMaxCtas / 2), min((total + 1) / 2, max((long long)n_sms, (total + 3) / 4)));
  // with more streams than that, room to split the longest ones
  const long long cap = min(max(even, streams > even / 2 ? streams + even / 2 : even), (long long)kMaxCtas + streams);
  auto count = [&](int share) {
    long long n = 0;
    for (int b = 0; b < B; ++b) n += (long long)Hkv * ((w[b] + share - 1) / share);
    return n;
  };
  int lo = 1, hi = longest;                 // the smallest share per CTA with which the CTAs stay within the cap
  while (lo < hi) {
    const int mid = (lo + hi) / 2;
    if (count(mid) <= cap) hi = mid;
    else lo = mid + 1;
  }
  for (int b = 0; b < B; ++b) ctas[b] = (w[b] + lo - 1) / lo;
  return (int)count(lo);
}

static bool three_tiers(const LayerView& lv) {
  return !lv.dense_hi && ((lv.budget_bf16 + lv.budget_u4 > 0) ? lv.budget_u4 > 0 : lv.tau_u4 < lv.tau_bf16);
}

// A few positions per team: one CTA per stream, which needs no merge.
// Where every stream has an SM to itself (eight pairs of warps) it is the faster up to a number of positions that grows with the
// streams, as their split gets the less out of the rest of the SMs.  us per layer, one CTA per stream / split: two tiers, 16 streams, 24 positions
// 5.96 / 6.02, 28 6.63 / 6.48, 64 streams, 40 8.85 / 9.05, 42 10.3 / 9.6, 128 streams, 42 11.7 / 13.1; three tiers, 4 streams, 14 positions 6.34 / 6.67,
// 18 7.5 / 6.7, 64 streams, 28 9.25 / 10.8, 32 10.3 / 10.1, 128 streams, 40 14.1 / 14.3, 42 15.8 / 15.5; 4-bit base, 4 streams, 14 5.75 / 5.87, 18 6.8 / 5.9,
// 128 streams, 40 13.0 / 14.6; 4-bit values, 16 streams, 18 6.1 / 6.7, 32 streams, 28 7.1 / 7.5, 32 8.1 / 7.5.  With few streams it is the launch
// saved that counts: 4 streams, two tiers, as calls / from a graph, 17 positions 4.7 / 6.3, 4.9 / 5.0, 20 5.75 / 6.3, 5.5 / 5.1, 26 6.6 / 6.3, 6.6 / 5.0.
// With more streams (four pairs, two CTAs per SM): never slower than the split up to 20 positions with two tiers and 2-bit values
// (one CTA per stream / split, 16 streams of the 8b shape 6.4 / 7.9); otherwise a unit takes longer, and beyond 12 positions
// the split is faster as long as it gets by with one CTA per SM (64 streams, 390 tokens, three tiers 6.9 / 8.8; 4-bit base
// 6.8 / 8.6; 4-bit values 6.3 / 7.9; three tiers with 4-bit values 7.6 / 9.2).
static bool one_cta_per_stream(const LayerView& lv, int n_sms) {
  const long long p = attention_ws_positions(lv);
  const int S = lv.B * lv.Hkv;
  const bool plain = !lv.dense_hi && !three_tiers(lv) && lv.v_bits == 2;
  if (S <= n_sms) return p <= (plain ? min(20 + S / 5, 42) : min(13 + S / 4, 40));
  return p <= (plain ? 20 : 12) || (p <= 20 && p * S > 4 * n_sms);
}

// Number of CTAs the split kernel runs for this layer state (also the number of partial-slot owners).  With fewer streams than CTA slots
// a grid that is a multiple of the stream count has no CTA that straddles two streams (a second segment costs a pipeline drain, a
// query load and a second partial), and with one CTA per stream no merge.  All slots are used where that leaves a CTA fewer positions by more
// than the straddling costs: 26 positions against one CTA per stream, 17 against several, 10 with two tiers and 4-bit values, whose
// positions take longer.  Time with a multiple over time with all slots, behind the positions saved.  One CTA per stream: two tiers, 160
// streams 19 .89, 26 1.01, 32 1.03, 224 streams 16 .89, 23 .99, 27 1.015, 37 1.08; three tiers, 224 streams 23 .993, 27 1.05; 4-bit base 23 .973, 27
// 1.04; 4-bit values 23 .993, 27 1.045.  Two to four per stream: two tiers, 112 streams 11 .92, 15 .95, 19 1.01, 64 streams 9 .91, 17 .998, 60
// streams 24 1.045; three tiers 15 .97 to .98, 19 1.01 to 1.02; 4-bit base 15 .985, 19 1.014, 36 (128 streams, 16384 tokens) 105.4 / 98.4 us; two tiers
// with 4-bit values 8 .996, 11 1.01, 19 1.07.
int attention_ws_grid(const LayerView& lv, int n_sms) {
  const int S = lv.B * lv.Hkv;
  if (lv.seq != nullptr) return lv.seq_ctas;
  const long long total = attention_ws_positions(lv) * S;
  // Small caches: two positions per CTA while that leaves one CTA per SM, then more (up to four) before a second CTA per SM:
  // a CTA has four teams, and every CTA of a stream is a partial to merge (one position per CTA / two / four, us per layer with the
  // merge: one sequence of 400 tokens 5.6 / 5.5 / 6.0, 4000 tokens 9.6 / 7.1 / 6.3, eight of 333 8.2 / 7.9 / 6.6).
  const long long wanted = min((total + 1) / 2, max((long long)n_sms, (total + 3) / 4));
  int grid = (int)min((long long)min(n_sms * kCtasPerSm, kMaxCtas / 2), wanted);
  if (one_cta_per_stream(lv, n_sms)) grid = min(grid, S);
  if (grid > S) {
    const int per_stream = grid / S;
    const int straddle = per_stream == 1 ? 26 : (lv.v_bits == 4 && !three_tiers(lv) && !lv.dense_hi ? 10 : 17);
    if ((attention_ws_positions(lv) + per_stream - 1) / per_stream <= (total + grid - 1) / grid + straddle) grid = per_stream * S;
  }
  return grid < 1 ? 1 : grid;
}

cudaError_t launch_attention_ws(const LayerView& lv, const void* q, float* out, float scale, float* ws, int n_sms,
                                cudaStream_t stream, int* launches, float* lse_out, int* form, int* ctas) {
  const int S = lv.B * lv.Hkv;
  const long long Us = attention_ws_positions(lv);
  const int grid = attention_ws_grid(lv, n_sms);
  // Steps of two units need blocks with an even number of them, and pay from a number of units per CTA on: with fewer the
  // coarser split and the longer first step cost more.  us per launch, one unit / two units per step: two tiers, G = 32 (7b
  // shape, batch 8) 8000 tokens, 27 units per CTA, 12.6 / 13.1, 16000 21.5 / 20.5; G = 128 (32b shape, batch 16) 2000 tokens,
  // 31 units, 13.5 / 13.0, 600 tokens, 10 units, 8.3 / 8.15; three tiers (7b shape) 600 tokens, 3 units, 6.4 / 6.7, 2000 tokens,
  // 7.6 units, 9.3 / 7.8 (8b shape, R = 64, 700 tokens, 6.5 units, 9.3 / 8.5, but an error of 0.86e-4 / 1.12e-4); 4-bit base (8b shape, batch 16) 600 tokens, 12 units, 8.9 / 9.3, 2000 tokens, 31 units, 18.7 / 17.7.
  const int from_units = three_tiers(lv) ? 7 : lv.dense_hi ? 20 : lv.G == 128 ? 10 : 40;
  bool by_two = !(lv.U & 1) && (lv.seq != nullptr ? lv.seq_total : Us * S) >= (long long)from_units * grid;
  // A fixed budget of more promoted channels than a step's slot holds: us per launch, one unit / two units per step, 12 channels, 8b
  // shape, 16384 tokens 83 / 87, 32b shape, G = 128, 8192 tokens 141 / 144; 128 channels, 7b shape, G = 128 48.7 / 53; 32 channels, 8b
  // shape 112 / 111.  (Three tiers: two units are the faster.)
  if (lv.budget_bf16 > 2 * kRowPairs && lv.budget_u4 == 0) by_two = false;
  // A short stream with a CTA of its own takes one unit at a time, for the precision: a probability is exact where it is the
  // maximum of its unit.
  if (lv.seq == nullptr && grid == S && one_cta_per_stream(lv, n_sms)) by_two = false;
  // 4-bit values: with more streams than CTAs every CTA begins two or three streams, and the longer steps make each beginning longer.
  // us per launch, one unit / two units per step, 512 streams: three tiers, G = 32 1000 tokens 45 / 49, 1700 58 / 60, 3000 87 / 84,
  // G = 128 1000 tokens 45 / 46, 1700 57 / 56; 4-bit base, G = 64 1700 tokens 61 / 63, 3000 94 / 91, G = 32 1700 64 / 73, 16000
  // 422 / 434; two tiers, G = 32 1000 tokens 39 / 44, 3000 75 / 73.
  if (lv.v_bits == 4 && lv.seq == nullptr && grid < S && (Us < (lv.G == 32 || lv.dense_hi ? 72 : 48) || (lv.dense_hi && lv.G == 32))) by_two = false;
  // With one CTA per stream the split kernel writes the output itself (32b shape, 32 sequences of 900 tokens: 17.9 -> 12.4 us per
  // layer).  Merging several partials in the kernel, by the CTA that finds all of a stream's written, was slower than a merge
  // kernel: a fence, a look at the other CTAs' marks and a serial merge against a dependent launch (one sequence of 400
  // tokens 7.3 us against 5.6; 7b shape 41.1 against 40.7).
  const bool whole = out != nullptr && lv.seq == nullptr && grid == S;
  float* const kernel_out = whole ? out : nullptr;
  // ... with eight pairs of warps where every stream has an SM to itself and four pairs would take several units each.  us per layer, four /
  // eight pairs: 4 streams of the 7b shape, 13 positions (4 packed, 3 unquantized units) 4.6 / 4.3, three tiers 5.7 / 4.6, 20 positions 6.0 / 5.5; 144 streams
  // of the 8b shape, 13 6.4 / 6.3, three tiers 9.2 / 7.4, 4-bit base 7.9 / 6.9, 20 8.2 / 8.2, 10.1 / 9.5, 10.0 / 9.1.  At most 12 positions are at most one unit per pair
  // beside the unquantized ones, and the larger CTA costs more: 9 positions, 4 streams 3.9 / 4.2, 144 streams 5.0 / 5.9.  So it is with most SMs in use
  // and two tiers up to one packed and one unquantized unit per pair (144 streams, 16 positions 7.2 / 7.7; 64 streams 5.5 / 5.3).
  const bool one_each = lv.n_blocks * lv.U <= 4 && Us <= 16;
  const bool wide = whole && grid <= n_sms && Us > 12 && !(one_each && 2 * grid > n_sms && !lv.dense_hi && !three_tiers(lv));
  if (form)
    *form = (by_two ? MIXKVQ_ATTN_TWO_UNITS : MIXKVQ_ATTN_ONE_UNIT) | (whole ? MIXKVQ_ATTN_DIRECT : 0) | (lv.stage_early ? MIXKVQ_ATTN_EARLY : 0) |
            (wide && !by_two ? MIXKVQ_ATTN_EIGHT_PAIRS : 0);
  if (ctas) *ctas = grid;
  cudaError_t e;
  if (!by_two) e = launch_attention_single(lv, q, scale, ws, grid, kernel_out, lse_out, wide, stream);
  else if (lv.G == 32) e = launch_g<32>(lv, q, scale, ws, grid, kernel_out, lse_out, stream);
  else if (lv.G == 64) e = launch_g<64>(lv, q, scale, ws, grid, kernel_out, lse_out, stream);
  else e = launch_g<128>(lv, q, scale, ws, grid, kernel_out, lse_out, stream);
  *launches = 1;
  if (e != cudaSuccess || out == nullptr || whole) return e;     // out == nullptr: split kernel only (timing)
  // The merge lets the next kernel start early (combine.cu) where the CTAs have enough to do that they finish one by one.  us per layer,
  // not early / early, 32 streams (288 CTAs), two tiers 1000 tokens 8.0 / 8.2, 6000 (22 positions per CTA) 14.15 / 14.15, 12000 21.0 / 20.0, three
  // tiers 1000 10.2 / 10.8, 4000 (16) 13.1 / 13.2, 14000 26.6 / 26.2; 64 streams, two tiers 2500 (21) 13.7 / 12.7, three tiers 16.5 / 15.0, 4-bit values 1000
  // (10) 9.5 / 13.7, 1500 (14) 12.0 / 13.8, 2500 15.9 / 14.8; 128 streams, 2500 20.7 / 18.1, three tiers 25.2 / 24.0.  With three tiers or a 4-bit base
  // later where a stream is split over many CTAs, and not where a CTA takes several streams: 8 streams, 28000 tokens (25) 16.9 / 17.4, 4-bit base
  // 17.3 / 18.0 (two tiers 14.9 / 14.8), 16 streams, 13000 (23) 16.7 / 17.2, 17.0 / 17.6, 20000 (36) 21.2 / 21.4, 21.5 / 21.65, 24 streams, 20000 (53) 27.95 / 27.6,
  // 28.4 / 27.9, 8 streams, 70000 (61) 30.1 / 29.9, 30.7 / 30.1; 320 streams, 900 28.7 / 28.9, 27.6 / 28.0.  Two tiers with several streams per CTA: 320
  // streams, 700 tokens (26 positions per stream) 19.9 / 20.1, G = 128 20.7 / 21.2, 1100 (41) 27.4 / 26.6, 25.9 / 25.8.
  const bool two_tiers = !three_tiers(lv) && !lv.dense_hi, may = two_tiers ? S <= grid || lv.seq != nullptr || Us >= 32 : S <= grid;
  const int from_positions = two_tiers || S >= 32 ? 20 : 50;
  const bool early = grid > n_sms && may && (lv.seq != nullptr ? lv.seq_total : Us * S) >= (long long)from_positions * grid;
  e = launch_combine(ws, out, lv.g, lv.Hkv, lv.Hq, 1, grid, Us, S, stream, lv.seq, lv.seq_prefix, lse_out, early,
                     lv.rope_cos != nullptr ? const_cast<void*>(q) : nullptr, const_cast<uint16_t*>(lv.new_k), lv.rope_cos, lv.rope_sin);
  *launches = 2;
  return e;
}

}  // namespace mixkvq
