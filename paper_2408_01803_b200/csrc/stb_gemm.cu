// stb_gemm: prefill GEMM  Y[t][i] = sum_j W^[i][j] X[t][j]  on the 5th-generation tensor cores
// (tcgen05.mma, fp32 accumulators in tensor memory).  The compute-bound prefilling stage of
// Appendix C.2: N = sequence length x batch tokens against one packed layer.
//
// One CTA computes a tile of the output of 128 rows of W^ x up to 256 kAcc tokens, D = A B^T with
//   A = 128 x 64 bf16 slice of W^, decoded from the packed tiles into shared memory in the
//       K-major 128-byte-swizzled layout the tensor core reads,
//   B = kAcc slices of bn x 64 bf16 of X (bn <= 256, a multiple of 16, chosen per call: see gemm_plan), brought in by TMA
//       with the same swizzle; every decoded A stage is multiplied with all of them (kAcc accumulators), which
//       divides the decode work per flop by kAcc,
// in rings over K (kStagesA decoded A stages, up to eight X boxes: the decode warps run ahead of the tensor core).  Warp roles:
//   warps 0..15 decode: see below
//   warp 16, 19 TMA producers (one lane each): X slices, one accumulator's or every other stage's
//   warp 17, 18 MMA issuers (one lane each, on two schedulers): with two accumulators each takes one (4 x tcgen05.mma,
//               K = 16, per stage); with one, each takes every other stage into an accumulator of its own and the
//               epilogue adds the two.  tcgen05.commit frees the boxes and stages; warp 17 allocates / frees TMEM
//   decode:     warp w works on rows 32 (w % 4) .. +31 of the tile = one packed row tile; four warps share a row
//               tile, each taking every fourth block: it loads the block's words with vector loads (its next block ahead),
//               converts the scales to bf16 (RN-even), decodes 64 columns of its four rows per lane into registers,
//               waits for the stage and writes them.  (Four warps sharing every block, one row of a lane each, paid the
//               loads, the waits and the address arithmetic four times: 370 clocks per 32 x 128 tile and SM, now about 220.)
//               Afterwards the same warps read the accumulator (TMEM lanes 32 (w % 4) ..) and store Y.
// The residual term of the salient columns (Eq. 4) is more K: a small kernel first gathers the activations of
// every residual slot (four per residual word, in word order) into Xs[token][slot]; after the blocks of its K
// range a CTA runs the residual slots of those blocks as further stages, A = +-bf16(a_sal2) or 0 by the two-bit
// residual codes, B = Xs through a second tensor map.  The main stages give a salient weight s1 bf16(a_sal1).
// One CTA fits an SM, so the grid runs in waves of 148 output tiles; tiles of a small last wave
// (and all tiles when there are few) are split along K into fp32 partial tiles in the caller's
// workspace and summed by a second kernel.
// Every wait on an mbarrier is bounded; a wait that runs out sets an abort flag (all roles then
// leave their loops), reports STB_ERR_TIMEOUT through dev_status and the CTA still frees TMEM.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/stb.h"
#include "stb_decode.cuh"
#include "stb_layout.cuh"
#include "stb_ptx.cuh"

namespace stb {

constexpr int kBM = 128;          // rows of W^ per CTA (UMMA M)
// Token side of the CTA tile: kAcc accumulators of bn tokens (UMMA N, a run-time value).  An MMA of 128 rows takes about 105
// clocks even where N is below 210 (832 clocks per stage of 8 MMAs at N = 64), so two accumulators are for tiles of more
// than 256 tokens (all 512 TMEM columns; a decoded A stage is used twice); up to 256 tokens are one accumulator per issuer,
// the issuers taking turns by the stage.
// kStagesA: ring of decoded A stages (16 KB each): eight beside narrow X boxes (a stage's way round -- written, multiplied,
// freed, seen -- takes about 2000 clocks, four decodes of a decode batch's stage), four beside wide ones.
template <int kAcc_, int kMaxBN_, int kStagesA_>
struct TokCfg { static constexpr int kAcc = kAcc_, kMaxBN = kMaxBN_, kTok = kAcc_ * kMaxBN_, kStagesA = kStagesA_; };
using BatchCfg = TokCfg<1, 64, 8>;
using MidCfg = TokCfg<1, 256, 4>;
using PrefillCfg = TokCfg<2, 256, 4>;
constexpr int kBK = 64;           // K per stage: one 128-byte swizzle row of bf16
constexpr int kMaxStagesB = 8;    // ring of X boxes: as many as fit, up to eight (five of 256 tokens x 64 of K = 32 KB): what is in
                                  // flight from L2 is what hides its latency; a stage of K takes kAcc of them
constexpr int kGroups = 4;                              // decode warps per 32-row quarter: each takes every fourth block
constexpr int kIssuers = 2;                             // MMA-issuing lanes (in two warps, on two schedulers)
constexpr int kDecodeWarps = 4 * kGroups;               // warps 0 .. 15; then the copies (16, 19) and the issuers (17, 18)
constexpr int kTmaWarpA = kDecodeWarps, kIssuerWarpA = kDecodeWarps + 1, kIssuerWarpB = kDecodeWarps + 2, kTmaWarpB = kDecodeWarps + 3;
constexpr int kGemmThreads = 32 * kDecodeWarps + 128;
// registers: 640 x 96 at launch, of which the fifth warpgroup gives some to the decode warps
constexpr int kGemmDecodeRegs = 104, kGemmIssueRegs = 64;
static_assert(32 * kDecodeWarps * kGemmDecodeRegs + 128 * kGemmIssueRegs <= kGemmThreads * 96, "register split within the launch's total");
constexpr uint32_t kStageA = kBM * kBK * 2;      // 16 KB
// "A stage empty" has eight barriers however many stages there are: a decode warp writes the stages it = 2 w, 2 w + 1 (mod 8),
// so it meets every phase of the barriers (it - kStagesA) mod 8 that it waits on, one after the other.
constexpr int kEmptyA = 8;
static_assert(kEmptyA == 2 * kGroups, "the warp of a stage is (stage / 2) mod kGroups");
constexpr uint32_t kGemmBars = 0;                                  // fullA, emptyA, fullB, emptyB, accum, tmem slot, abort
constexpr uint32_t kGemmTab = 512;                                 // position table, 8 bytes per entry and copy
static_assert(8 * (2 * kEmptyA + 4 * kMaxStagesB + 1) + 16 <= kGemmTab, "barrier area");
constexpr uint32_t kSmemMax = 232448;
constexpr double kDecodeClocks = 440.0;    // decode of a stage (gemm_plan)
// X boxes have twice as many barriers as there are boxes, for the same reason: box number hb (two accumulators: 2 stage + a,
// one: the stage) goes to place hb mod nbox, where (nbox odd) the boxes of the two producers alternate; the producer and the
// issuer of box hb meet every phase of the barriers hb mod 2 nbox, but only every second one of a barrier per place, and a
// parity cannot tell the phase before from the phase after.
// What depends on bn: copies of the position table (16, lane-minor: look-ups nearly free of bank conflicts; one where bn = 256
// leaves no room), where the stages and the boxes lie, and how many boxes there are.
// `pairs`: the table is the joint one of 6:8 (decode_tiles).
constexpr uint32_t kPairTabBytes = kMasks6 * kMasks6 * 16;
static_assert(8u * kStageA >= 0x10000u, "whatever a pair field says, its look-up ends in the eight A stages behind the table at the latest");
struct GemmSmem { uint32_t copies, a, b, box, nbox, total; };
__host__ __device__ inline GemmSmem gemm_smem(int kAcc, int stages_a, int bn, bool pairs) {
  GemmSmem g;
  g.box = (uint32_t)bn * kBK * 2;
  for (g.copies = 16;; g.copies = 1) {
    g.a = (kGemmTab + (pairs ? kPairTabBytes : 8u * kPosTableEntries * g.copies) + 1023u) & ~1023u;
    g.b = g.a + (uint32_t)stages_a * kStageA;
    g.nbox = (kSmemMax - g.b) / g.box;
    if (g.nbox >= 5u || g.copies == 1u) break;
  }
  if (g.nbox > (uint32_t)kMaxStagesB) g.nbox = kMaxStagesB;
  g.total = g.b + g.nbox * g.box;
  // a 16-bit output tile is staged where the boxes were
  const uint32_t out = (uint32_t)(kAcc * bn) * kBM * 2u;
  if (g.total < g.b + out) g.total = g.b + out;
  return g;
}
constexpr long long kGemmWaitLimit = 2000000000ll;

// ---- tcgen05 / TMA wrappers ---------------------------------------------------------------
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The descriptors come as their low words (start address / 16; the high word is the same for every operand tile of
// this kernel) and the accumulate flag as a template argument: what an issuing lane runs per stage of K (waits,
// descriptors, MMAs, commits) must stay shorter than the tensor core needs for the stage.
template <bool kAccumulate>
__device__ __forceinline__ void umma_16(uint32_t d_tmem, uint32_t adesc_lo, uint32_t bdesc_lo, uint32_t desc_hi, uint32_t idesc) {
  if (kAccumulate)
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.eq.b32 p, 0, 0;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(adesc_lo), "r"(bdesc_lo), "r"(desc_hi), "r"(idesc) : "memory");
  else
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, 0, 0;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(adesc_lo), "r"(bdesc_lo), "r"(desc_hi), "r"(idesc) : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 r;\n\telect.sync r|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
               "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                 "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                 "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
               : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor of a K-major, 128-byte-swizzled operand tile (rows of 128
// bytes, groups of 8 rows 1024 bytes apart): start address, stride byte offset 1024,
// descriptor version 1, layout type 2 (128-byte swizzle).
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset
  d |= (uint64_t)1 << 46;                  // version
  d |= (uint64_t)2 << 61;                  // SWIZZLE_128B
  return d;
}
// Instruction descriptor: D = f32, A and B both bf16 (format 1) or both fp16 (format 0), both K-major, N = bn, M = 128.
__device__ __forceinline__ uint32_t gemm_idesc(bool f16, int bn) {
  return (1u << 4) | ((f16 ? 0u : 1u) << 7) | ((f16 ? 0u : 1u) << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

// Bounded mbarrier wait with a CTA-wide abort flag (a volatile int in shared memory).  The two
// single-lane roles back off between polls so that their spinning does not take issue slots from
// the decode warps that share their schedulers.
template <bool kBackoff = false>
__device__ __forceinline__ bool gemm_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (kBackoff) __nanosleep(32);
    if (*abort_flag) return false;
    if (clock64() - t0 > kGemmWaitLimit) { *abort_flag = 1; return false; }
  }
  return true;
}

__device__ __forceinline__ uint32_t bf16_bits(uint32_t h16) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(__half2float(__ushort_as_half((unsigned short)h16))));
}

// The byte planes of a row's four main scales (A low, B high bytes, fp16) as bf16.
__device__ __forceinline__ void scales_to_bf16(uint32_t& A, uint32_t& B) {
  const uint32_t h01 = prmt(A, B, 0x5140u), h23 = prmt(A, B, 0x7362u);
  const float2 f01 = __half22float2(*reinterpret_cast<const __half2*>(&h01)), f23 = __half22float2(*reinterpret_cast<const __half2*>(&h23));
  const __nv_bfloat162 b01 = __floats2bfloat162_rn(f01.x, f01.y), b23 = __floats2bfloat162_rn(f23.x, f23.y);
  const uint32_t u01 = *reinterpret_cast<const uint32_t*>(&b01), u23 = *reinterpret_cast<const uint32_t*>(&b23);
  A = prmt(u01, u23, 0x6420u);
  B = prmt(u01, u23, 0x7531u);
}

__device__ __forceinline__ void sts_v4(uint32_t a, const uint32_t (&v)[4]) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ uint2 lds_v2(uint32_t a) {            // (of the position table: written before the roles part, never changed)
  uint2 v;
  asm("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}

// What a decode warp needs to know.
struct DecodeArgs {
  const uint8_t* packed; volatile int* abort_flag;
  uint32_t ptab, entry, stages;              // shared-memory addresses of the position table (bytes per entry of it) and the A stages
  uint32_t bar_full, bar_empty;              // of the A ring
  int mt, b0, b1, nblk, ntile, q, w, lane;   // q: row tile of the CTA's four, w: which of the row tile's four warps
  uint32_t nrw, rw0, rw1;   // residual words of a row tile, and of the blocks [b0, b1)
  int nres;                 // residual stages (64 slots = 16 words each, the first one starts at word rw0 & ~1)
};

// The words of a tile that a lane decodes: load_lane_tile's, with N = 6's pair fields as they are (word 4 mt + s).
template <int N>
struct GemmTile { LaneTile<N> lt; uint32_t fld[8]; };
template <int N>
__device__ __forceinline__ void load_gemm_tile(const uint8_t* tile, int lane, GemmTile<N>& d) {
  if constexpr (mask_pairs(N)) {
    load_planes<N>(tile, off_region(N), d.lt.R, lane);
    load_planes<LaneTile<N>::kFull>(tile, off_sign(N), d.lt.S, lane);
    d.lt.half = 0;
    const uint4 s0 = *reinterpret_cast<const uint4*>(tile + scale_off(N, lane >> 2, 0)), s1 = *reinterpret_cast<const uint4*>(tile + scale_off(N, lane >> 2, 2));
    d.lt.A[0] = s0.x; d.lt.B[0] = s0.y; d.lt.A[1] = s0.z; d.lt.B[1] = s0.w;
    d.lt.A[2] = s1.x; d.lt.B[2] = s1.y; d.lt.A[3] = s1.z; d.lt.B[3] = s1.w;
#pragma unroll
    for (int k = 0; k < 8; ++k) d.fld[k] = *reinterpret_cast<const uint16_t*>(tile + pair_field_off(lane >> 2, k >> 2, k & 3, lane & 3));
  } else {
    load_lane_tile<N>(tile, lane, d.lt);
  }
}

// Decode role of one warp: packed row tile 4 mt + q, every fourth block of the CTA's K range, written into the A stages.
// kF16: the stages hold fp16 (the scales as stored); otherwise bf16 (the scales rounded to nearest even).
// kPairs (6:8): the position selectors of two rows by one look-up with the tile's pair field, whose upper twelve bits are the address of
// their entry: 32 bits of selectors per row, two copies of every entry for even and odd lanes.  Splitting the field into two mask
// indices and looking each up took 60 of the 760 instructions of a tile (28672 x 8192 at 64 tokens 96.5 -> 94.1 us, 11008 x 4096 27.6 ->
// 27.1).  For calls of up to 64 tokens, where the decode is what takes the time and the boxes leave room for the table's 12 KB.
template <int N, bool kF16, int kStagesA, bool kPairs>
__device__ __forceinline__ void decode_tiles(const DecodeArgs& da) {
  const int nblk = da.nblk, q = da.q, b0 = da.b0, b1 = da.b1, w = da.w;
  // The lane plays the part of packed-layout lane 4 g + t with g = lane % 8, t = lane / 8: the eight
  // lanes of a quarter-warp then hold eight different rows g and their 16-byte stores into the
  // swizzled stage fall on eight different 16-byte bank groups (no conflict); loads of the
  // lane-major planes stay coalesced, they are only permuted inside the warp.
  const int g = da.lane & 7, t = da.lane >> 3;
  const int lane = 4 * g + t;
  const int rtile = da.mt * 4 + q;                 // packed row tile
  constexpr uint32_t tbytes = tile_bytes(N);
  const int nmain = 2 * (b1 - b0), nstage = nmain + da.nres;
  // Stage `it` belongs to warp (it / 2) mod 4: the stages 2 w + h (mod 8) with h = 0, 1, so that slot, barriers and the place
  // of the lane's two 16-byte chunks (4 sl + t of its row g) in the slot are the same every time; only the parity changes.
  const uint32_t row_at = da.stages + (uint32_t)((2 * w) % kStagesA) * kStageA + (uint32_t)q * 4096u + (uint32_t)g * 128u;
  const uint32_t at0 = row_at + (uint32_t)((t ^ g) << 4), at1 = row_at + (uint32_t)(((4 + t) ^ g) << 4);
  const uint32_t full = da.bar_full + 8u * (uint32_t)((2 * w) % kStagesA), empty = da.bar_empty + 8u * (uint32_t)((2 * w + kEmptyA - kStagesA) % kEmptyA);
  // before stage `it` is written, stage it - kStagesA must have been read.  Four stages: use it / 8 of the slot pair waits for
  // phase it / 8 (w >= 2) or it / 8 - 1 (w < 2) of that stage's barrier, eight: for phase it / 8 - 1; there is nothing to
  // wait for before phase 0.  The verdict is made warp-uniform.
  const uint32_t early = kStagesA == 8 || w < 2 ? 1u : 0u;
  auto stage_wait = [&](uint32_t use, int h) -> bool {
    if (use < early) return true;
    const uint32_t parity = (use - early) & 1u;
    return __all_sync(0xFFFFFFFFu, mbar_try_wait(empty + 8u * h, parity)) || __all_sync(0xFFFFFFFFu, gemm_wait(empty + 8u * h, parity, da.abort_flag));
  };
  auto stage_done = [&](int h) {
    fence_async_smem();          // generic-proxy writes -> visible to the tensor core
    __syncwarp();
    if (da.lane == 0) mbar_arrive(full + 8u * h);
  };
  auto next_mine = [&](int it) { while (it < nstage && ((it >> 1) & (kGroups - 1)) != w) ++it; return it; };
  if (rtile >= da.ntile) {       // no such rows: zeros
    const uint32_t z[4] = {0, 0, 0, 0};
#pragma unroll 1
    for (int it = next_mine(0); it < nstage; it = next_mine(it + 1)) {
      if (!stage_wait((uint32_t)it / kEmptyA, it & 1)) return;
#pragma unroll
      for (int j = 0; j < 4; ++j) { sts_v4(at0 + (uint32_t)(it & 1) * kStageA + 1024u * j, z); sts_v4(at1 + (uint32_t)(it & 1) * kStageA + 1024u * j, z); }
      stage_done(it & 1);
    }
    return;
  }
  const uint8_t* rtbase = da.packed + tiles_offset(nblk) + (size_t)rtile * tbytes * nblk;
  const uint8_t* resid_rt = da.packed + tiles_offset(nblk) + (size_t)tbytes * nblk * da.ntile + (size_t)rtile * resid_rt_bytes(nblk, da.nrw);
  // Residual stages come after the blocks: 64 residual slots (16 residual words) of K each.  The lane writes the same
  // two 16-byte chunks of its rows: chunk c holds the words 2 c and 2 c + 1 of the stage, four slots each, as
  // +-bf16(a_sal2) or 0.  What a stage needs sits behind two dependent loads from global memory (the word's table
  // entry, then a_sal2 and the codes from the block's record); the entries of the warp's first one are asked for here.
  const ResidWord* rwt = reinterpret_cast<const ResidWord*>(da.packed + rwtab_offset(nblk));
  const uint32_t wfirst = da.rw0 & ~1u;
  auto res_word = [&](int it, int idx) { return wfirst + 16u * (uint32_t)(it - nmain) + 2u * (uint32_t)(4 * (idx >> 1) + t) + (uint32_t)(idx & 1); };
  uint2 e[4];
  auto res_entries = [&](int it) {
#pragma unroll
    for (int idx = 0; idx < 4; ++idx) {
      const uint32_t wd = res_word(it, idx);
      e[idx] = make_uint2(0xFFFFFFFFu, 0u);
      if (it < nstage && wd >= da.rw0 && wd < da.rw1) e[idx] = __ldg(reinterpret_cast<const uint2*>(rwt + wd));
    }
  };
  int rit = next_mine(nmain);
  GemmTile<N> nxt;
  if (b0 + w < b1) load_gemm_tile<N>(rtbase + (size_t)(b0 + w) * tbytes, lane, nxt);
  res_entries(rit);
  uint32_t use = 0;
#pragma unroll 1
  for (int b = b0 + w; b < b1; b += kGroups, ++use) {
    uint32_t mask[4] = {0, 0, 0, 0};                   // word j, byte s: keep-mask index of slot (j, s)
    uint32_t fld[8];
    if constexpr (kPairs) {
#pragma unroll
      for (int k = 0; k < 8; ++k) fld[k] = nxt.fld[k] & 0xFFF0u;        // (nothing to mask in a layer as packed: what altered it since makes no misaligned load)
    } else if constexpr (mask_pairs(N)) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {                    // rows 2 mt, 2 mt + 1, slot s: k = 4 mt + s (multiply-adds: the integer pipe is the busy one)
        const uint32_t J = nxt.fld[k] >> 4, i1 = (J * 2341u) >> 16, i0 = J - kMasks6 * i1;      // (pair_field_index)
        mask[2 * (k >> 2)] = i0 * (1u << (8 * (k & 3))) + mask[2 * (k >> 2)];
        mask[2 * (k >> 2) + 1] = i1 * (1u << (8 * (k & 3))) + mask[2 * (k >> 2) + 1];
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) mask[j] = nxt.lt.mask[j];
    }
    uint32_t A[4], B[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      A[j] = nxt.lt.A[j]; B[j] = nxt.lt.B[j];
      // (a salient weight gets s1 bf16(a_sal1) here; its residual term comes with the residual stages)
      if (!kF16) scales_to_bf16(A[j], B[j]);
    }
    FastRows<N> fr;
    fr.init(nxt.lt, A, B);
    if (b + kGroups < b1) load_gemm_tile<N>(rtbase + (size_t)(b + kGroups) * tbytes, lane, nxt);
    uint32_t XL[4] = {0, 0, 0, 0}, XH[4] = {0, 0, 0, 0};
    if (N == 5) {
#pragma unroll
      for (int j = 0; j < 4; ++j) fr.high(j, 0, XL[j], XH[j]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint2 P[4][2];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
          if constexpr (!kPairs) P[j][sl] = lds_v2(keep_index_of(mask, j, 2 * h + sl) * da.entry + da.ptab);
          else if ((j & 1) == 0) {
            const uint2 e = lds_v2(fld[2 * j + 2 * h + sl] + da.ptab);
            P[j][sl] = selectors_of(e.x);
            P[j + 1][sl] = selectors_of(e.y);
          }
        }
      uint32_t f[4][2][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (N == 6) fr.high(j, h, XL[j], XH[j]);
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) fr.slot2(j, 2 * h + sl, P[j][sl].x, P[j][sl].y, XL[j], XH[j], f[j][sl]);      // group 4 s + t
      }
      if (!stage_wait(use, h)) return;
#pragma unroll
      for (int j = 0; j < 4; ++j) { sts_v4(at0 + h * kStageA + 1024u * j, f[j][0]); sts_v4(at1 + h * kStageA + 1024u * j, f[j][1]); }
      stage_done(h);
    }
  }
#pragma unroll 1
  while (rit < nstage) {
    uint2 a2[4];
    uint32_t word[4];
#pragma unroll
    for (int idx = 0; idx < 4; ++idx) {
      a2[idx] = make_uint2(0u, 0u); word[idx] = 0x55555555u;               // "no term"
      if (e[idx].x != 0xFFFFFFFFu) {
        const uint8_t* rec = resid_rt + resid_block_off((int)(e[idx].x >> 3), res_word(rit, idx) - (e[idx].x & 7u));
        a2[idx] = __ldg(reinterpret_cast<const uint2*>(rec + resid_a2_off(g, 0)));
        word[idx] = __ldg(reinterpret_cast<const uint32_t*>(rec + resid_code_off(e[idx].x & 7u, g)));
      }
    }
    const int it = rit;
    rit = next_mine(it + 1);
    res_entries(rit);
    if (!stage_wait((uint32_t)it / kEmptyA, it & 1)) return;
    const uint32_t shift = (uint32_t)(it & 1) * kStageA;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t f[2][4];
#pragma unroll
      for (int idx = 0; idx < 4; ++idx) {
        const uint32_t h16 = (((j & 2) ? a2[idx].y : a2[idx].x) >> (16 * (j & 1))) & 0xFFFFu;
        const uint32_t v = kF16 ? h16 : bf16_bits(h16);
        const uint32_t L2 = prmt(v, 0u, 0x4040u);                 // (lo, 0, lo, 0)
        const uint32_t H2 = prmt(v, v ^ 0x8000u, 0x2521u);        // (hi, 0, hi ^ 0x80, 0)
        const uint32_t sel = resid_selector(word[idx], j);
        const uint32_t lo4 = prmt(L2, L2, sel), hi4 = prmt(H2, H2, sel);
        f[idx >> 1][2 * (idx & 1)] = prmt(lo4, hi4, 0x5140u);
        f[idx >> 1][2 * (idx & 1) + 1] = prmt(lo4, hi4, 0x7362u);
      }
      sts_v4(at0 + shift + 1024u * j, f[0]);
      sts_v4(at1 + shift + 1024u * j, f[1]);
    }
    stage_done(it & 1);
  }
}

// Gathers the activations of the residual slots: Xs[t][4 w + k] = X[t][128 block(w) + cols(w)[k]] for every residual
// word w of the layer, and zeros in the 128 columns after the last word (a CTA's last residual stage may reach there).
__global__ void gemm_gather_kernel(const uint8_t* __restrict__ packed, int n, int m, int N, const __nv_bfloat16* __restrict__ X, int T,
                                   size_t ldx, __nv_bfloat16* __restrict__ Xs, int ldxs) {
  begin_after(packed, X);          // (the GEMM may start; it waits for this grid before it reads Xs)
  const Header* hdr = reinterpret_cast<const Header*>(packed);
  if (!header_matches(hdr, n, m, N)) return;
  const int nblk = m / kBlock;
  const ResidWord* rwt = reinterpret_cast<const ResidWord*>(packed + rwtab_offset(nblk));
  const uint32_t nrw = hdr->nrw;
  uint32_t W = nrw + 32u;                                   // words written per token: the layer's and 32 of zeros
  if (W > (uint32_t)ldxs / 4u) W = (uint32_t)ldxs / 4u;
  const size_t total = (size_t)T * W;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t t = i / W;
    const uint32_t w = (uint32_t)(i % W);
    uint2 out = make_uint2(0u, 0u);
    if (w < nrw) {
      const uint2 e = __ldg(reinterpret_cast<const uint2*>(rwt + w));
      const unsigned short* xr = reinterpret_cast<const unsigned short*>(X + t * ldx + (size_t)(e.x >> 3) * kBlock);
      out.x = (uint32_t)xr[e.y & 0xFFu] | ((uint32_t)xr[(e.y >> 8) & 0xFFu] << 16);
      out.y = (uint32_t)xr[(e.y >> 16) & 0xFFu] | ((uint32_t)xr[e.y >> 24] << 16);
    }
    *reinterpret_cast<uint2*>(Xs + t * (size_t)ldxs + 4u * w) = out;
  }
}

// ------------------------------------------------------------------------------------------
// Where a call's output tiles lie (gemm_plan).
struct GemmShape { int full_tiles, ksplit, bps, ttiles, bn; GemmSmem smem; };

// whether the position table is the joint one
template <class Cfg>
STB_HD constexpr bool pair_table(int N) { return mask_pairs(N) && Cfg::kMaxBN == BatchCfg::kMaxBN; }

template <int N, class Cfg, bool kF16>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap xsmap, const uint8_t* __restrict__ packed, int n, int m, int T,
            void* __restrict__ Y, int y_16, size_t ldy, float* __restrict__ ws, const __grid_constant__ GemmShape shape, uint32_t box_bytes, int* dev_status) {
  constexpr int kAcc = Cfg::kAcc, kMaxBN = Cfg::kMaxBN, kStagesA = Cfg::kStagesA;
  constexpr bool kPairs = pair_table<Cfg>(N);
  extern __shared__ __align__(1024) uint8_t smem[];
  const int full_tiles = shape.full_tiles, ksplit = shape.ksplit, bps = shape.bps, ttiles = shape.ttiles, bn = shape.bn;
  const GemmSmem& L = shape.smem;
  const int ktok = kAcc * bn;
  const int nblk = m / kBlock, ntile = (n + kTileRows - 1) / kTileRows;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // CTAs 0 .. full_tiles - 1 compute one output tile each over the whole K; the rest come in groups of `ksplit`
  // per tile, each with `bps` blocks of K, and leave fp32 partial tiles in the workspace
  const int cta = (int)blockIdx.x;
  const bool split = cta >= full_tiles;
  const int tile = split ? full_tiles + (cta - full_tiles) / ksplit : cta;
  const int kz = split ? (cta - full_tiles) % ksplit : 0;
  const int tt = tile % ttiles, mt = tile / ttiles;
  const int b0 = split ? kz * bps : 0, b1 = split ? min(nblk, b0 + bps) : nblk;
  // The header first (a buffer packed for another shape must not be read as this one), then at once what the rest of the
  // prologue needs: the word counts and, into L2, the first block each decode warp will read.
  const Header* hdr = reinterpret_cast<const Header*>(packed);
  const BlockInfo* binfo_k = reinterpret_cast<const BlockInfo*>(packed + sizeof(Header));
  const bool fits = header_matches(hdr, n, m, N);
  if (fits && warp < kDecodeWarps) {
    const int q = warp & 3, b = b0 + (warp >> 2), rtile = mt * 4 + q;
    if (b < b1 && rtile < ntile && lane * 128 < (int)tile_bytes(N))
      asm volatile("prefetch.global.L2 [%0];" ::"l"(packed + tiles_offset(nblk) + ((size_t)rtile * nblk + b) * tile_bytes(N) + lane * 128));
  }
  const uint32_t nrw = hdr->nrw;
  uint32_t rw0 = 0, rw1 = 0;
  if (fits && b0 < b1) { rw0 = __ldg(&binfo_k[b0].rw_off); rw1 = b1 < nblk ? __ldg(&binfo_k[b1].rw_off) : nrw; }

  const uint32_t sbase = smem_u32(smem);
  // A ring: full = the four decode warps of the stage's block have written it, empty = the tensor core has read it;
  // B ring: full = the X boxes have landed, empty = the tensor core has read them
  const uint32_t bar_fullA = sbase + kGemmBars, bar_emptyA = bar_fullA + 8 * kEmptyA;
  const uint32_t bar_fullB = bar_emptyA + 8 * kEmptyA, bar_emptyB = bar_fullB + 16 * kMaxStagesB, bar_accum = bar_emptyB + 16 * kMaxStagesB;
  constexpr uint32_t kBarBytes = 8 * (2 * kEmptyA + 4 * kMaxStagesB + 1);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kGemmBars + kBarBytes);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kGemmBars + kBarBytes + 8);

  if (threadIdx.x == 0) {
    // a stage of A is read by both issuers (with one accumulator by one of them), an X box by the issuer of its accumulator
    for (int i = 0; i < kStagesA; ++i) mbar_init(bar_fullA + 8 * i, 4);
    for (int i = 0; i < kEmptyA; ++i) mbar_init(bar_emptyA + 8 * i, kAcc == 1 ? 1 : kIssuers);
    for (int i = 0; i < 2 * kMaxStagesB; ++i) { mbar_init(bar_fullB + 8 * i, 1); mbar_init(bar_emptyB + 8 * i, 1); }
    mbar_init(bar_accum, kIssuers);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if constexpr (kPairs) {
    for (uint32_t i = threadIdx.x; i < kMasks6 * kMasks6; i += kGemmThreads) {
      const uint2 e = pair_selectors(g_pos_table.v[N][i % kMasks6], g_pos_table.v[N][i / kMasks6]);
      reinterpret_cast<uint4*>(smem + kGemmTab)[i] = make_uint4(e.x, e.y, e.x, e.y);
    }
  } else {
    for (uint32_t i = threadIdx.x; i < kPosTableEntries * L.copies; i += kGemmThreads)
      reinterpret_cast<uint2*>(smem + kGemmTab)[i] = g_pos_table.v[N][L.copies == 1u ? i : i >> 4];
  }
  constexpr uint32_t kTmemCols = kAcc == 1 ? 2 * kMaxBN : kAcc * kMaxBN;      // one accumulator: a second one for the other half of K
  if (warp == kIssuerWarpA) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_d = *tmem_slot;
  if (!fits) {                                         // the same for every thread of the grid
    __syncthreads();
    if (warp == kIssuerWarpA) tmem_dealloc(tmem_d, kTmemCols);
    grid_dependency_wait();                            // (what follows on the stream waits for this grid alone)
    if (threadIdx.x == 0 && dev_status) *dev_status = STB_ERR_CORRUPT;
    return;
  }
  // residual words of the CTA's blocks -> residual stages of 16 words, the first one starting at an even word
  const int nres = rw1 > rw0 ? (int)((rw1 - (rw0 & ~1u) + 15u) / 16u) : 0;
  const int nmain = 2 * max(b1 - b0, 0);               // 64-column stages of the blocks
  const int nstage = nmain + nres;

  if (warp >= kDecodeWarps) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kGemmIssueRegs));
  if (warp == kTmaWarpA || warp == kTmaWarpB) {
    // ---------------- TMA producers ----------------
    // (the whole warp runs the loop, one elected lane issues, for the reason given at the MMA issuers)
    // two accumulators: producer w brings box w of every stage; one accumulator: the box of the stages 2 i + w
    const int w = __shfl_sync(0xFFFFFFFFu, warp == kTmaWarpA ? 0 : 1, 0);
    constexpr int kStep = kAcc == 1 ? kIssuers : 1, kBoxStep = 2;
    const bool leader = elect_one();
    const uint32_t box = L.box, nbox = L.nbox;
    const int stages = __shfl_sync(0xFFFFFFFFu, nstage, 0), y = tt * ktok + (kAcc == 1 ? 0 : w * bn);
    const int rwx = __shfl_sync(0xFFFFFFFFu, (int)(4u * (rw0 & ~1u)), 0);
    // place of the box; its barrier and that of the box that was there before (mod nbar), and the latter's parity
    const uint32_t nbar = 2u * nbox;
    uint32_t s = (uint32_t)w, fb = s, eb = s + nbox, ps = 1;
    bool waited = false;
    for (int it = kAcc == 1 ? w : 0; it < stages; it += kStep) {
      const uint32_t bar_empty = bar_emptyB + 8 * eb, bar_full = bar_fullB + 8 * fb;
      bool ok = mbar_try_wait(bar_empty, ps);
      if (!ok) ok = gemm_wait<true>(bar_empty, ps, abort_flag);
      if (!__all_sync(0xFFFFFFFFu, ok)) break;
      if (it < nmain) {
        if (leader) {
          mbar_expect_tx(bar_full, box_bytes);
          tma_load_2d(sbase + L.b + s * box, &xmap, (b0 * 2 + it) * kBK, y, bar_full);
        }
      } else {
        // Xs comes from the gather kernel, which this grid may have overtaken (programmatic dependent launch)
        if (!waited) { grid_dependency_wait(); waited = true; }
        if (leader) {
          mbar_expect_tx(bar_full, box_bytes);
          tma_load_2d(sbase + L.b + s * box, &xsmap, rwx + (it - nmain) * kBK, y, bar_full);
        }
      }
      __syncwarp();
      s += kBoxStep;
      if (s >= nbox) s -= nbox;
      fb += kBoxStep;
      if (fb >= nbar) fb -= nbar;
      eb += kBoxStep;
      if (eb >= nbar) { eb -= nbar; ps ^= 1u; }
    }
    grid_dependency_wait();  // (every CTA, whether or not it had residual stages)
    if (*abort_flag) {       // let copies in flight land before the CTA gives its shared memory up
      const long long t0 = clock64();
      while (clock64() - t0 < 200000) {}
    }
  } else if (warp == kIssuerWarpA || warp == kIssuerWarpB) {
    // ---------------- MMA issuers ----------------
    // The whole warp runs the loop and one elected lane issues: every operand is then warp-uniform to the compiler and sits in
    // uniform registers, where tcgen05 instructions take them (under `lane == 0` each was moved there one by one: an
    // issuer's stage took 850 clocks at 64 tokens, 600 of them its own instructions; now 170 per two stages).
    const int w = __shfl_sync(0xFFFFFFFFu, warp == kIssuerWarpA ? 0 : 1, 0);
    const uint32_t tmem_u = __shfl_sync(0xFFFFFFFFu, tmem_d, 0);
    const bool leader = elect_one();
    // two accumulators: issuer w takes accumulator w (box w of every stage);
    // one accumulator:  issuer w takes the stages 2 i + w into an accumulator of its own
    constexpr int kStep = kAcc == 1 ? kIssuers : 1;
    const uint32_t desc_hi = (uint32_t)(umma_desc(0u) >> 32);
    const uint32_t a_lo0 = (uint32_t)umma_desc(sbase + L.a), b_lo0 = (uint32_t)umma_desc(sbase + L.b);
    const uint32_t dt = tmem_u + (uint32_t)(w * kMaxBN), idesc = gemm_idesc(kF16, bn), box_lo = L.box >> 4, nbox = L.nbox;
    const uint32_t nbar = 2u * nbox;
    uint32_t sa = kAcc == 1 ? (uint32_t)w : 0u, ea = sa, sb = (uint32_t)w, fb = sb;      // ring places and barriers, advanced without divisions
    uint32_t pa = 0, pb = 0;                                                    // their phase parities
    for (int it = kAcc == 1 ? w : 0; it < nstage; it += kStep) {
      const bool ra = mbar_try_wait(bar_fullA + 8 * sa, pa), rb = mbar_try_wait(bar_fullB + 8 * fb, pb);     // both at once
      bool ok = true;
      if (!ra) ok = gemm_wait<true>(bar_fullA + 8 * sa, pa, abort_flag);
      if (!rb && ok) ok = gemm_wait<true>(bar_fullB + 8 * fb, pb, abort_flag);
      if (!__all_sync(0xFFFFFFFFu, ok)) break;
      tc_fence_after();
      const uint32_t a_lo = a_lo0 + sa * (kStageA >> 4), b_lo = b_lo0 + sb * box_lo;
      if (leader) {
        if (it >= kStep) umma_16<true>(dt, a_lo, b_lo, desc_hi, idesc);
        else umma_16<false>(dt, a_lo, b_lo, desc_hi, idesc);
#pragma unroll
        for (int kk = 1; kk < kBK / 16; ++kk) umma_16<true>(dt, a_lo + 2u * kk, b_lo + 2u * kk, desc_hi, idesc);
        umma_commit(bar_emptyB + 8 * fb);        // the box is free once the MMAs that read it have completed
        umma_commit(bar_emptyA + 8 * ea);
      }
      __syncwarp();
      sa += kStep;
      if (sa >= kStagesA) { sa -= kStagesA; pa ^= 1u; }
      ea += kStep;
      if (ea >= kEmptyA) ea -= kEmptyA;
      sb += 2u;
      if (sb >= nbox) sb -= nbox;
      fb += 2u;
      if (fb >= nbar) { fb -= nbar; pb ^= 1u; }
    }
    if (leader) umma_commit(bar_accum);                        // all MMAs this warp issued have completed
    __syncwarp();
  } else if (warp < kDecodeWarps) {
    // ---------------- decode warps ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kGemmDecodeRegs));
    const int gi = warp >> 2;               // decode group: which of the row tile's four warps this one is
    DecodeArgs da;
    da.packed = packed; da.abort_flag = abort_flag;
    da.entry = 8u * L.copies; da.ptab = sbase + kGemmTab + 8u * ((uint32_t)lane & (kPairs ? 1u : L.copies - 1u)); da.stages = sbase + L.a;
    da.bar_full = bar_fullA; da.bar_empty = bar_emptyA;
    da.mt = mt; da.b0 = b0; da.b1 = max(b1, b0); da.nblk = nblk; da.ntile = ntile; da.q = warp & 3; da.w = gi; da.lane = lane;
    da.nrw = nrw; da.rw0 = rw0; da.rw1 = rw1; da.nres = nres;
    decode_tiles<N, kF16, kStagesA, kPairs>(da);

    // ---------------- epilogue: TMEM -> registers -> Y ----------------
    const int q = warp & 3;                        // TMEM lane quarter of this warp
    // A 16-bit output tile goes through shared memory (the X ring: every box has been consumed by then) so that it
    // leaves in 16-byte pieces along the rows: straight from the registers a warp's store is 32 rows x 2 bytes of
    // one token, and the epilogue took a ninth of the CTA's time.  The same for every thread of the CTA:
    const bool staged = y_16 != 0 && !split && (ldy % 8) == 0 && (reinterpret_cast<uintptr_t>(Y) & 15u) == 0;
    uint16_t* stage = reinterpret_cast<uint16_t*>(smem + L.b);           // [token of the tile][row of the tile]
    const bool have = __all_sync(0xFFFFFFFFu, gemm_wait(bar_accum, 0u, abort_flag)) && nstage > 0;
    if (have) {
      tc_fence_after();
      const int row = mt * kBM + 32 * q + lane;                // output feature (row of W^)
      float* wsz = split ? ws + ((size_t)(tile - full_tiles) * ksplit + kz) * (size_t)(kBM * ktok) : nullptr;
      const int chunks = (bn + 31) >> 5;                        // of 32 tokens, per accumulator
#pragma unroll 1
      for (int cc = gi; cc < kAcc * chunks; cc += kGroups) {    // the groups share the column chunks
        const int acc = kAcc == 1 || cc < chunks ? 0 : 1, c0 = 32 * (cc - acc * chunks), live = bn - c0, tok0 = acc * bn + c0;
        uint32_t r[32];
        tmem_ld32(tmem_d + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * kMaxBN + c0), r);
        if (kAcc == 1) {
          // the other half of K sits in the second accumulator
          uint32_t r2[32];
          tmem_ld32(tmem_d + ((uint32_t)(32 * q) << 16) + (uint32_t)(kMaxBN + c0), r2);
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(r2[i]));
        }
        if (staged) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float v = __uint_as_float(r[i]);
            if (i < live) stage[(tok0 + i) * kBM + 32 * q + lane] = kF16 ? __half_as_ushort(__float2half_rn(v)) : __bfloat16_as_ushort(__float2bfloat16_rn(v));
          }
        } else if (row < n) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int tok = tt * ktok + tok0 + i;
            if (i < live && tok < T) {
              const float v = __uint_as_float(r[i]);
              if (wsz) wsz[(size_t)(tok0 + i) * kBM + 32 * q + lane] = v;
              else if (y_16 && kF16) static_cast<__half*>(Y)[(size_t)tok * ldy + row] = __float2half_rn(v);
              else if (y_16) static_cast<__nv_bfloat16*>(Y)[(size_t)tok * ldy + row] = __float2bfloat16_rn(v);
              else static_cast<float*>(Y)[(size_t)tok * ldy + row] = v;
            }
          }
        }
      }
    }
    if (staged) {
      // every decode warp takes the barrier, whatever its wait said
      asm volatile("bar.sync 1, %0;" ::"n"(128 * kGroups) : "memory");
      if (have) {
        const int d = warp * 32 + lane;                  // 0 .. 511: 16 threads per token, 8 rows each
        const int piece = d & 15, row0 = mt * kBM + 8 * piece;
        uint16_t* Y16 = static_cast<uint16_t*>(Y);
#pragma unroll 4
        for (int tl = d >> 4; tl < ktok; tl += (128 * kGroups) / 16) {
          const int tok = tt * ktok + tl;
          if (tok >= T) break;
          const uint4 v = *reinterpret_cast<const uint4*>(stage + tl * kBM + 8 * piece);
          uint16_t* dst = Y16 + (size_t)tok * ldy + row0;
          if (row0 + 8 <= n) *reinterpret_cast<uint4*>(dst) = v;
          else {
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 8; ++e)
              if (row0 + e < n) dst[e] = (uint16_t)(w[e >> 1] >> (16 * (e & 1)));
          }
        }
      }
    }
  }

  // The MMA thread makes sure the tensor core is done with TMEM before it is freed.  Its commit on bar_accum was
  // issued whether or not the loop above was left early, so this wait ends when the instructions issued so far
  // have completed; it keeps its own bound and ignores the abort flag.
  if (warp == kIssuerWarpA && lane == 0) mbar_wait(bar_accum, 0u, kGemmWaitLimit);
  tc_fence_before();
  __syncthreads();
  if (warp == kIssuerWarpA) tmem_dealloc(tmem_d, kTmemCols);
  if (threadIdx.x == 0 && *abort_flag && dev_status) *dev_status = STB_ERR_TIMEOUT;
}

// Split-K reduction of the tiles that were computed in parts: partial tile z of split tile u is
// ws[(u ksplit + z)][token 0..ktok-1][row 0..kBM-1]; summed in z order.  y_16: 1 = bf16, 2 = fp16 output.
__global__ void gemm_reduce_kernel(const float* __restrict__ ws, int first_tile, int split_tiles, int ksplit, int ttiles, int ktok,
                                   int n, int T, void* __restrict__ Y, int y_16, size_t ldy) {
  // four consecutive rows of one token per thread: 16-byte loads of the parts, one 8- or 16-byte store
  begin_after(ws);                 // (a programmatic dependent of the GEMM: its CTAs are set up while the GEMM drains)
  const size_t per = (size_t)kBM * ktok, per4 = per / 4, total = (size_t)split_tiles * per4;
  const bool vec = (ldy % 4) == 0 && (reinterpret_cast<uintptr_t>(Y) & 15u) == 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t u = i / per4, r = (i % per4) * 4;
    const int tile = first_tile + (int)u, tt = tile % ttiles, mt = tile / ttiles;
    const int tok = tt * ktok + (int)(r / kBM), row = mt * kBM + (int)(r % kBM);
    if (tok >= T || row >= n) continue;
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int z = 0; z < ksplit; ++z) {
      const float4 v = __ldcs(reinterpret_cast<const float4*>(ws + (u * ksplit + z) * per + r));
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    const size_t o = (size_t)tok * ldy + row;
    if (vec && row + 4 <= n) {
      if (y_16 == 2) {
        const __half2 lo = __floats2half2_rn(acc.x, acc.y), hi = __floats2half2_rn(acc.z, acc.w);
        *reinterpret_cast<uint2*>(static_cast<__half*>(Y) + o) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
      } else if (y_16 == 1) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
        *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(Y) + o) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
      } else {
        *reinterpret_cast<float4*>(static_cast<float*>(Y) + o) = acc;
      }
    } else {
      const float a4[4] = {acc.x, acc.y, acc.z, acc.w};
      for (int e = 0; e < 4 && row + e < n; ++e) {
        if (y_16 == 2) static_cast<__half*>(Y)[o + e] = __float2half_rn(a4[e]);
        else if (y_16 == 1) static_cast<__nv_bfloat16*>(Y)[o + e] = __float2bfloat16_rn(a4[e]);
        else static_cast<float*>(Y)[o + e] = a4[e];
      }
    }
  }
}

// What stb_gemm_workspace[_min] promise for a shape, in tiles of 128 rows x `ktok` tokens: few output tiles are split along K
// (mandatory), the tiles of a small last wave too (optional).  A call is laid out by gemm_plan below and never needs more.
struct GemmBytes { size_t mandatory, preferred; };
static GemmBytes gemm_bytes(int n, int m, int T, int ktok) {
  const int nblk = m / kBlock, tiles = ((n + kBM - 1) / kBM) * ((T + ktok - 1) / ktok);
  const size_t per = (size_t)kBM * ktok * sizeof(float);
  auto parts = [&](int ks) { const int bps = (nblk + ks - 1) / ks; return (nblk + bps - 1) / bps; };
  int ks = 1;
  if (ktok < 512) {
    double best = 0.0;
    for (int k = 1; k <= 16 && (k == 1 || nblk / k >= 4); ++k) {
      const double cost = (double)(((long long)tiles * k + 147) / 148) * (7.0 + (double)((nblk + k - 1) / k));
      if (k == 1 || cost < best - 1e-9) { best = cost; ks = k; }
    }
  } else {
    if (tiles < 100) ks = 148 / tiles;
    if (ks > 16) ks = 16;
    while (ks > 1 && nblk / ks < 4) --ks;
  }
  ks = parts(ks);
  GemmBytes b = {0, 0};
  if (ks > 1) { b.mandatory = b.preferred = (size_t)tiles * ks * per; return b; }
  const int tail = tiles % 148;
  if (tiles > 148 && tail > 0 && tail <= 74) {
    int kt = 148 / tail;
    if (kt > 16) kt = 16;
    while (kt > 1 && nblk / kt < 4) --kt;
    if (kt > 1) b.preferred = (size_t)tail * parts(kt) * per;
  }
  return b;
}

// How a call is laid out on the 148 SMs (one CTA per SM at a time): the width of the token tiles (2 x bn or 1 x bn tokens, bn a
// multiple of 16), and which tiles are split along K into how many parts -- all of them, or those of the last wave -- chosen
// as the layout whose estimated time is smallest among those whose partial tiles fit `avail` bytes.  In SM clocks:
//   a stage (64 of K):   the decode of two 32 x 128 tiles' worth of weights per row tile, or the tensor core's time for the
//                        tile's tokens, whichever is longer (measured: about 440, and 4.4 x 105 or bn / 2 + 30 per accumulator)
//                        (a GPU full of wide single accumulators ran 1.4 times that, each decoded stage being used once: 8192 x 28672
//                        at 2048 tokens 1006 us against 888 with two, at 1024 tokens 520 against 439)
//   a CTA besides:       prologue, first loads, drain (10000) and epilogue (15 per token)
//   a split:             the second kernel, and its partial tiles written and read (2500 bytes per clock)
struct GemmPlan {
  int acc, bn, ttiles, tiles, full_tiles, split_tiles, ksplit, bps;
  size_t bytes;
};
static void gemm_plan_for(GemmPlan& best, double& best_cost, int acc, int max_bn, int n, int m, int T, size_t avail) {
  const int nblk = m / kBlock, rtiles = (n + kBM - 1) / kBM, most = acc * max_bn;
  for (int tt = (T + most - 1) / most, end = tt + 8; tt <= end; ++tt) {
    int bn = ((T + tt - 1) / tt + acc - 1) / acc;
    bn = bn < 16 ? 16 : (bn + 15) / 16 * 16;
    const int ktok = acc * bn;
    if (bn > max_bn || (tt - 1) * ktok >= T) continue;
    const long long tiles = (long long)rtiles * tt;
    const double wide = acc == 1 && bn > 128 && tiles > 148 ? 1.4 : 1.0;
    const double mma = acc * 4.0 * (bn > 210 ? 0.5 * bn : 105.0) * 1.1 * wide + 30.0, stage = mma > kDecodeClocks ? mma : kDecodeClocks, fixed = 10000.0 + 15.0 * ktok;
    const size_t per = (size_t)kBM * ktok * sizeof(float);
    auto consider = [&](long long full, int ks) {
      const int bps = (nblk + ks - 1) / ks;
      ks = (nblk + bps - 1) / bps;
      const long long rest = tiles - full;
      const size_t bytes = ks > 1 ? (size_t)rest * ks * per : 0;
      if (bytes > avail) return;
      double cost = (double)((full + 147) / 148) * (fixed + nblk * 2.13 * stage) + (double)((rest * ks + 147) / 148) * (fixed + bps * 2.13 * stage);
      if (ks > 1) cost += 4000.0 + 2.0 * (double)bytes / 2500.0;
      if (best.tiles == 0 || cost < best_cost * 0.999) {
        best_cost = cost;
        best.acc = acc; best.bn = bn; best.ttiles = tt; best.tiles = (int)tiles; best.full_tiles = (int)(ks > 1 ? full : tiles); best.split_tiles = (int)(ks > 1 ? rest : 0);
        best.ksplit = ks; best.bps = bps; best.bytes = bytes;
      }
    };
    consider(tiles, 1);
    for (int ks = 2; ks <= 16 && nblk / ks >= 4; ++ks) {
      if (tiles < 148) consider(0, ks);
      else if (tiles % 148) consider(tiles - tiles % 148, ks);
    }
  }
}
static GemmPlan gemm_plan(int n, int m, int T, size_t avail) {
  GemmPlan best = {};
  double cost = 0.0;
  if (T <= BatchCfg::kTok) gemm_plan_for(best, cost, BatchCfg::kAcc, BatchCfg::kMaxBN, n, m, T, avail);
  else {
    gemm_plan_for(best, cost, MidCfg::kAcc, MidCfg::kMaxBN, n, m, T, avail);
    gemm_plan_for(best, cost, PrefillCfg::kAcc, PrefillCfg::kMaxBN, n, m, T, avail);
  }
  return best;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Bytes of the gathered activations Xs[T][m / 4] (bf16) at the head of the workspace: room for the most residual
// slots a layer can have (32 per block), so that the size depends on the shape alone.
static size_t gemm_xs_bytes(int m, int T) { return (((size_t)T * (size_t)(m / 4) * 2u) + 255u) & ~(size_t)255u; }

// A call's tile width in the promise of gemm_bytes: 512 tokens, 64 for a decode batch of fp16 activations.
static int gemm_promise(bool f16, int T) { return f16 && T <= BatchCfg::kTok ? BatchCfg::kTok : PrefillCfg::kTok; }
// partial tiles a call of this shape would like room for
static size_t gemm_preferred(int n, int m, int T, int ktok) {
  const size_t a = gemm_bytes(n, m, T, ktok).preferred, b = gemm_plan(n, m, T, (size_t)-1).bytes;
  return a > b ? a : b;
}

// y_16: 0 = fp32 output, 1 = the 16-bit type of the activations (bf16, or fp16 with kF16)
template <int N, class Cfg, bool kF16>
static int launch_gemm(const GemmPlan& plan, const uint8_t* packed, int n, int m, const void* X, int T, size_t ldx, void* Y, int y_16,
                       size_t ldy, void* ws, int* dev_status, cudaStream_t s) {
  constexpr int kAcc = Cfg::kAcc;
  float* ws_split = reinterpret_cast<float*>(static_cast<uint8_t*>(ws) + gemm_xs_bytes(m, T));
  GemmShape shape;
  shape.full_tiles = plan.full_tiles; shape.ksplit = plan.ksplit; shape.bps = plan.bps; shape.ttiles = plan.ttiles; shape.bn = plan.bn;
  shape.smem = gemm_smem(kAcc, Cfg::kStagesA, plan.bn, pair_table<Cfg>(N));
  EncodeTiledFn enc = encode_tiled_fn();
  if (!enc) return STB_ERR_CUDA;
  const CUtensorMapDataType dt = kF16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  const cuuint32_t box_rows = (cuuint32_t)(T < plan.bn ? T : plan.bn);
  const cuuint32_t box[2] = {(cuuint32_t)kBK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  CUtensorMap map, xsmap;
  {
    const cuuint64_t dims[2] = {(cuuint64_t)m, (cuuint64_t)T};
    const cuuint64_t strides[1] = {(cuuint64_t)ldx * 2};
    if (enc(&map, dt, 2, const_cast<void*>(X), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return STB_ERR_ARG;
  }
  const int ldxs = m / 4;                     // a multiple of 32 elements: rows of Xs start on 64-byte boundaries
  {
    const cuuint64_t dims[2] = {(cuuint64_t)ldxs, (cuuint64_t)T};
    const cuuint64_t strides[1] = {(cuuint64_t)ldxs * 2};
    if (enc(&xsmap, dt, 2, ws, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return STB_ERR_ARG;
  }
  // the shared-memory limit of a kernel is a per-device setting
  static bool attr_done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return STB_ERR_CUDA;
  if (dev < 0 || dev >= 64 || !attr_done[dev]) {
    if (cudaFuncSetAttribute(gemm_kernel<N, Cfg, kF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess) return STB_ERR_CUDA;
    if (dev >= 0 && dev < 64) attr_done[dev] = true;
  }
  // the gather moves 16-bit values: the same kernel serves bf16 and fp16
  if (launch_after(gemm_gather_kernel, dim3(148 * 4), dim3(256), 0, s, packed, n, m, N, static_cast<const __nv_bfloat16*>(X), T, ldx,
                   static_cast<__nv_bfloat16*>(ws), ldxs) != cudaSuccess)
    return STB_ERR_CUDA;
  // The GEMM is a programmatic dependent of the gather: its CTAs may be scheduled while the gather runs (they need
  // Xs only for the residual stages at the end of their K range) and wait (griddepcontrol.wait) before they read it.
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(plan.full_tiles + plan.split_tiles * plan.ksplit));
  cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = shape.smem.total;
  cfg.stream = s;
  cfg.attrs = pdl; cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, gemm_kernel<N, Cfg, kF16>, map, xsmap, packed, n, m, T, Y, y_16, ldy, ws_split, shape,
                         (uint32_t)(box_rows * kBK * 2), dev_status) != cudaSuccess)
    return STB_ERR_CUDA;
  if (plan.split_tiles > 0) {
    cfg.gridDim = dim3(148 * 4);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 0;
    if (cudaLaunchKernelEx(&cfg, gemm_reduce_kernel, (const float*)ws_split, plan.full_tiles, plan.split_tiles, plan.ksplit, plan.ttiles, kAcc * plan.bn,
                           n, T, Y, y_16 ? (kF16 ? 2 : 1) : 0, ldy) != cudaSuccess)
      return STB_ERR_CUDA;
  }
  return STB_OK;
}

template <bool kF16>
static int launch_gemm_n(int N, const uint8_t* packed, int n, int m, const void* X, int T, size_t ldx, void* Y, int y_16,
                         size_t ldy, void* ws, size_t ws_bytes, int* dev_status, cudaStream_t s) {
  const size_t xs_bytes = gemm_xs_bytes(m, T);
  const int ktok = gemm_promise(kF16, T);
  if (ws && (reinterpret_cast<uintptr_t>(ws) & 255u)) return STB_ERR_ARG;
  if (!ws || ws_bytes < xs_bytes || ws_bytes - xs_bytes < gemm_bytes(n, m, T, ktok).mandatory) return STB_ERR_SIZE;
  const size_t preferred = gemm_preferred(n, m, T, ktok);
  const GemmPlan plan = gemm_plan(n, m, T, ws_bytes - xs_bytes < preferred ? ws_bytes - xs_bytes : preferred);
  auto go = [&](auto cfg) {
    using Cfg = decltype(cfg);
    switch (N) {
      case 4: return launch_gemm<4, Cfg, kF16>(plan, packed, n, m, X, T, ldx, Y, y_16, ldy, ws, dev_status, s);
      case 5: return launch_gemm<5, Cfg, kF16>(plan, packed, n, m, X, T, ldx, Y, y_16, ldy, ws, dev_status, s);
      default: return launch_gemm<6, Cfg, kF16>(plan, packed, n, m, X, T, ldx, Y, y_16, ldy, ws, dev_status, s);
    }
  };
  if (T <= BatchCfg::kTok) return go(BatchCfg{});
  return plan.acc == 1 ? go(MidCfg{}) : go(PrefillCfg{});
}

}  // namespace stb

static int gemm_workspace_impl(int n, int m, int N, int T, int ktok, size_t* bytes, bool minimum) {
  if (!bytes) return STB_ERR_ARG;
  if (n < 1 || m < stb::kBlock || m % stb::kBlock != 0 || T < 1) return STB_ERR_SHAPE;
  if (N < 1 || N > 8) return STB_ERR_NM;
  *bytes = stb::gemm_xs_bytes(m, T) + (minimum ? stb::gemm_bytes(n, m, T, ktok).mandatory : stb::gemm_preferred(n, m, T, ktok));
  return STB_OK;
}

extern "C" int stb_gemm_workspace(int n, int m, int N, int T, size_t* bytes) { return gemm_workspace_impl(n, m, N, T, stb::gemm_promise(false, T), bytes, false); }
extern "C" int stb_gemm_workspace_min(int n, int m, int N, int T, size_t* bytes) { return gemm_workspace_impl(n, m, N, T, stb::gemm_promise(false, T), bytes, true); }
extern "C" int stb_gemm_f16_workspace(int n, int m, int N, int T, size_t* bytes) { return gemm_workspace_impl(n, m, N, T, stb::gemm_promise(true, T), bytes, false); }

static int gemm_check_args(const void* packed, int n, int m, int N, const void* X, int T, size_t ldx, void* Y, size_t ldy) {
  if (!packed || !X || !Y) return STB_ERR_ARG;
  if (n < 1 || m < stb::kBlock || m % stb::kBlock != 0 || T < 1) return STB_ERR_SHAPE;
  if (N < 1 || N > 8) return STB_ERR_NM;
  if (N < 4 || N > 6) return STB_ERR_UNSUPPORTED;          // the tensor-core decode covers N = 4, 5, 6
  if (ldx < (size_t)m || ldy < (size_t)n || (ldx % 8) != 0 || (reinterpret_cast<uintptr_t>(X) & 15u)) return STB_ERR_ARG;
  return STB_OK;
}

extern "C" int stb_gemm(const void* packed, int n, int m, int N, const void* X, int T, size_t ldx,
                        void* Y, stb_dtype ydt, size_t ldy, void* ws, size_t ws_bytes,
                        int* dev_status, void* stream) {
  const int rc = gemm_check_args(packed, n, m, N, X, T, ldx, Y, ldy);
  if (rc != STB_OK) return rc;
  if (ydt != STB_F32 && ydt != STB_BF16) return STB_ERR_UNSUPPORTED;
  return stb::launch_gemm_n<false>(N, static_cast<const uint8_t*>(packed), n, m, X, T, ldx, Y, ydt == STB_BF16, ldy, ws, ws_bytes,
                                   dev_status, static_cast<cudaStream_t>(stream));
}

extern "C" int stb_gemm_f16(const void* packed, int n, int m, int N, const void* X, int T, size_t ldx,
                            void* Y, stb_dtype ydt, size_t ldy, void* ws, size_t ws_bytes,
                            int* dev_status, void* stream) {
  const int rc = gemm_check_args(packed, n, m, N, X, T, ldx, Y, ldy);
  if (rc != STB_OK) return rc;
  if (ydt != STB_F32 && ydt != STB_F16) return STB_ERR_UNSUPPORTED;
  return stb::launch_gemm_n<true>(N, static_cast<const uint8_t*>(packed), n, m, X, T, ldx, Y, ydt == STB_F16, ldy, ws, ws_bytes,
                                  dev_status, static_cast<cudaStream_t>(stream));
}

// ------------------------------------------------------------------------------------------
// stb_gemm_noalloc: stb_gemm for callers that can hand over no workspace.  The gathered residual
// activations and the split-K partial sums live in a fixed array inside the library image instead of
// a caller's buffer.
namespace stb {
constexpr size_t kNoAllocScratchBytes = 8u << 20;                       // 8 MiB per device, resident until exit
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocScratchBytes / sizeof(float)];
}  // namespace stb

extern "C" int stb_gemm_noalloc(const void* packed, int n, int m, int N, const void* X, int T, size_t ldx,
                                void* Y, stb_dtype ydt, size_t ldy, int* dev_status, void* stream) {
  if (!packed || !X || !Y) return STB_ERR_ARG;
  if (n < 1 || m < stb::kBlock || m % stb::kBlock != 0 || T < 1) return STB_ERR_SHAPE;
  if (N < 1 || N > 8) return STB_ERR_NM;
  if (N < 4 || N > 6) return STB_ERR_UNSUPPORTED;
  if (ydt != STB_F32 && ydt != STB_BF16) return STB_ERR_UNSUPPORTED;
  if (ldx < (size_t)m || ldy < (size_t)n || (ldx % 8) != 0 || (reinterpret_cast<uintptr_t>(X) & 15u)) return STB_ERR_ARG;
  // this shape needs the caller-workspace entry point if the scratch it cannot do without does not fit
  if (stb::gemm_xs_bytes(m, T) + stb::gemm_bytes(n, m, T, stb::PrefillCfg::kTok).mandatory > stb::kNoAllocScratchBytes) return STB_ERR_SIZE;
  // The array's name is only a host-side handle: ask the runtime for its address on the current
  // device, once per device, and give the kernels that address.
  static float* scratch_of_device[64] = {nullptr};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return STB_ERR_CUDA;
  if (!scratch_of_device[dev]) {
    float* p = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), stb::g_noalloc_scratch) != cudaSuccess || !p) return STB_ERR_CUDA;
    scratch_of_device[dev] = p;
  }
  return stb::launch_gemm_n<false>(N, static_cast<const uint8_t*>(packed), n, m, X, T, ldx, Y, ydt == STB_BF16, ldy,
                                   scratch_of_device[dev], stb::kNoAllocScratchBytes, dev_status, static_cast<cudaStream_t>(stream));
}
