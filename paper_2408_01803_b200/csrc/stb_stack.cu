// stb_layer_stack_resident: a whole list of decode GEMV steps as ONE resident kernel (batch 1..8, N = 4, 5, 6).
//
// The per-layer launches of stb_layer_stack pay, for every layer, a launch ramp, a copy of the activations per
// CTA, a cluster reduction and a last wave that leaves SMs idle.  Here one CTA of 16 warps per SM stays
// resident for the whole list (cooperative launch: all CTAs are on the machine together):
//   * Consecutive steps that read the same activations (q / k / v, gate / up) form a PHASE.  The 32 x 128 tiles of
//     a phase, in (row tile, block) order, are dealt to the CTAs as contiguous ranges and a CTA's range to its 16
//     warps as equal contiguous runs.  When whole row tiles can be dealt with little imbalance (at least 85 % of
//     the SM time used) every CTA gets whole row tiles and no sum crosses CTAs; otherwise the ranges are equal
//     in tiles and a row tile may straddle CTAs.
//   * Each warp's tiles stream through a private ring in shared memory (two slots of up to two tiles and their
//     residual records, two 1-D bulk copies each, mbarrier completion, bounded waits).  Four more warps issue the
//     copies, one lane per ring, and run ahead into the NEXT phases: packed weights never depend on activations, so the
//     stream does not stop at a phase boundary.  They also work out where a chunk belongs (row tile, first block, residual
//     words, end of a run) and leave that beside the slot, so that the other warps only wait, decode and multiply.
//   * Decode and multiply per tile: 6:8 keeps the weights in rank order and lets mma.sp.m16n8k32 place them
//     (activations from an image of x in operand order in shared memory, built once per phase and CTA); 4:8 and 5:8
//     (and 6:8 when the image does not fit) decode to position order for mma.m16n8k16 with the activations from a
//     plain copy in shared memory, or through L1 where that does not fit or is not read often enough to pay.
//   * A step may take x = silu(in) * in2 (the gated activation between gate / up and down of an MLP): the CTA forms
//     it while it stages the activations.
//   * The residual term of the salient columns (Eq. 4): a block's record of the residual stream comes with its tile,
//     four residual words (16 salient slots) of a chunk per tensor-core step; the activations behind every residual
//     word of the phase are gathered into shared memory once x is staged, or, where they are too many, read by their places.
//   * Partial sums: a warp that covers a whole row tile writes y itself; the others leave their head / tail
//     pieces in shared memory and the CTA adds them in tile order at the end of the phase; of a row tile that
//     straddles CTAs the later ones hand their sums to the first through the caller's workspace, every value beside a tag
//     of the launch and phase (one 8-byte store, no fence, no counter), and the first adds them in CTA order and empties
//     their places, so that no value outlives its phase.  Every sum has a fixed order: results are reproducible.
//   * A phase may read what an earlier phase wrote: a CTA starts a phase's arithmetic only when the count of
//     finished row tiles (one counter in the workspace, bumped once per CTA and phase) has reached the total
//     of all earlier phases.  The poll is bounded; when it or an mbarrier wait runs out, an abort flag makes
//     every CTA leave, STB_ERR_TIMEOUT is reported and the last CTA out restores the workspace to zero.
//
// What bounds it.  In the tile loop the integer ALU (2 warp-instructions per clock and SM; at 6:8 it is busy for about 122 of a tile's 157
// clocks, shared memory for 112): about 165 / 185 / 157 clocks per tile and SM at N = 4 / 5 / 6 with residual words, waits and copies.
// Between the last tile of a phase and the first of the next, latencies, 6.5 to 7.5 thousand clocks: the sums, a release (1,050), the
// count of finished row tiles and the activations (a trip through L2 each); before that the warps' ends are spread by 1.5 thousand.  And
// about 9 us per call (launch, set-up, leaving).
// At one row: 7B MLP at 6:8 44.8 -> 36.9 us, 13B block at 5:8 96.1 -> 87.4, 32 7B layers 1905 -> 1683 against 16-byte metadata entries,
// sums of pieces four at a time, one kernel for everything and slots of 4:8 and 5:8 handed back before the product; eight 7B layers at
// eight rows 692 -> 637.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/stb.h"
#include "stb_decode.cuh"
#include "stb_layout.cuh"
#include "stb_ptx.cuh"
#include "stb_tile.cuh"

namespace stb {

constexpr int kSWarps = 16;
constexpr int kSThreads = kSWarps * 32;       // the decoding warps; the copies are issued by a fifth warpgroup,
constexpr int kSAllThreads = kSThreads + 128; // which gives registers up to the other four: 640 x 96 at launch, then
constexpr int kDecodeRegs = 104, kFeedRegs = 64;   // 512 x 104 + 128 x 64 of them
static_assert(kSThreads * kDecodeRegs + 128 * kFeedRegs <= kSAllThreads * 96, "register split within the launch's total");
constexpr int kMaxPhases = 64;                // per launch; longer lists run as several launches
constexpr int kMaxFusedSteps = 4;
constexpr int kSDepth = 2, kSChunk = 2;       // ring: slots per warp, tiles per slot
// A slot holds the tiles of a chunk (of the launch's largest N) and their records: of any two blocks, or, where shared memory is
// short, of two blocks with at most kFewWords residual words together (blocks with more then come one by one).
constexpr uint32_t kFewWords = 8;
constexpr uint32_t slot_tiles(int N) { return kSChunk * tile_bytes(N); }
constexpr uint32_t slot_records(bool few) { return kSChunk * kResidA2Bytes + (few ? kFewWords : kSChunk * kMaxResidWords) * kResidWordBytes; }
static_assert(kFewWords >= kMaxResidWords && slot_tiles(4) % 128 == 0 && slot_tiles(5) % 128 == 0 && slot_tiles(6) % 128 == 0 &&
              slot_records(true) % 128 == 0 && slot_records(false) % 128 == 0, "a block's records fit; slots stay 128-byte aligned");
constexpr long long kSWaitLimit = 2000000000ll;        // about a second of SM clocks
constexpr long long kSSelftestLimit = 100000ll;

struct StackPhase {
  const uint8_t* packed[kMaxFusedSteps];
  void* y[kMaxFusedSteps];
  uint32_t ldy[kMaxFusedSteps];
  int32_t n[kMaxFusedSteps];
  int32_t tile_start[kMaxFusedSteps + 1];     // row tiles of the phase: step i owns [tile_start[i], tile_start[i + 1])
  const __half* x;
  const __half* x2;                           // second input of STB_IN_SILU_MUL, else null
  uint32_t ldx;
  int32_t m;
  uint8_t N, batch, count, f16_mask;          // f16_mask bit i: step i writes fp16
  uint8_t use_image, aligned, gather, pad;    // use_image: 0 activations from global memory, 1 operand-order image (6:8),
                                              // 2 plain fp16 copy in shared memory; aligned: CTA ranges are whole row tiles;
                                              // gather: 2 the residual words' activations are gathered in shared memory, 1 their
                                              // places are there, 0 neither
  uint32_t done_before;                       // row tiles finished by all earlier phases of this launch
};

struct StackParams {
  StackPhase ph[kMaxPhases];
  int32_t nphase;
  // shared memory plan (byte offsets; see SSmem for what comes before)
  uint32_t pos_off[3];                        // position tables of N = 4, 5, 6, 0 where no phase needs one
  uint32_t use_meta6;
  uint32_t ring_off, pdata_off, xs_off, cols_off, x_off, x_bytes;
  uint32_t slot_tiles, slot_bytes, slot_words;     // a ring slot: where its records begin, its size, the residual words it takes
  uint32_t pos_row;                           // bytes from one entry of a position table to the next
  uint32_t part_floats;                       // floats per partial slot: 32 rows x largest batch
  uint32_t max_share;                         // most CTAs that share one row tile
  uint32_t* sync;                             // [0] finished row tiles, [1] abort flag, [2] CTAs that left, [4] launches so far
  uint2* gpart;                               // sums handed on for row tiles that straddle CTAs: { value, tag }, empty ({ 0, 0 }) between launches
  uint32_t gpart_slots;
  int* dev_status;
  long long wait_limit;
  int32_t copies_off;
  int32_t form, only5;                        // the kernel: ResidForm, and whether every phase is 5:8
};

// shared memory: joint 6:8 metadata table first (784 x 16 B, at offset 0: a pair field of a tile is the shared-memory
// address of its entry), when a phase needs it; then, from `base`:
struct SSmem {
  static constexpr uint32_t full = 0;                                          // ring barriers, 16 warps x 2: copies landed ...
  static constexpr uint32_t empty = full + 8 * kSWarps * kSDepth;              // ... and slot read
  static constexpr uint32_t ctl = empty + 8 * kSWarps * kSDepth;               // control words
  static constexpr uint32_t slots = ctl + 64;                                  // row tiles of the partial slots: 32 x 4 B
  static constexpr uint32_t chunks = slots + 2 * kSWarps * 4;                  // what each ring slot holds: 32 x 16 B
  static constexpr uint32_t zero = chunks + kSWarps * kSDepth * 16;            // 384 bytes of zeros: the activations of lanes beyond the batch
  static constexpr uint32_t range = zero + kZeroBytes;                                // this CTA's tiles of every phase
  static constexpr uint32_t nrw = range + 32 * kMaxPhases;                     // residual words per row tile of every step
  static constexpr uint32_t bytes = nrw + 4 * kMaxPhases * kMaxFusedSteps;
};

// A CTA's share of a phase: tiles [lo, hi), the row tiles that lie inside it as a whole, and the row tile of its first tile.
// Where the first or the last row tile straddles CTAs: the CTA where it begins, and how many share it.
struct CtaRange { int32_t lo, hi, whole, first, head_cta, head_share, tail_cta, tail_share; };

__device__ __forceinline__ void red_release_add(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// a value and its tag in one 8-byte access (a scalar one: of a vector access the elements may be seen one by one): whoever sees
// the tag sees the value
__device__ __forceinline__ void st_tagged(uint2* p, float v, uint32_t tag) {
  asm volatile("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tst.relaxed.gpu.global.u64 [%0], t;\n\t}" ::"l"(p), "r"(__float_as_uint(v)), "r"(tag) : "memory");
}
__device__ __forceinline__ uint2 ld_tagged(const uint2* p) {
  uint2 v;
  asm volatile("{\n\t.reg .b64 t;\n\tld.relaxed.gpu.global.u64 t, [%2];\n\tmov.b64 {%0, %1}, t;\n\t}" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const void* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// Coherent loads of activations (written by this kernel, so never through the read-only path)
__device__ __forceinline__ uint32_t ldg_u16_coherent(const void* p) {
  unsigned short v;
  asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
  return v;
}
// silu(a) b = a b / (1 + exp(-a)) in fp32: one reciprocal and one correction of the quotient (Markstein's: the remainder by a
// fused multiply-add), within an ulp of the divided form without its slow path.  Where the quotient or the divisor is infinite
// the remainder is NaN and the product with the reciprocal is already what the division gives.
__device__ __forceinline__ float silu_mul(float a, float b) {
  const float d = 1.0f + __expf(-a);
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(d));
  const float q = a * r, e = fmaf(-d, q, a);
  return (e == e ? fmaf(e, r, q) : q) * b;
}
// fp16 pair (bits) of silu(a) * b per half, in fp32, rounded to nearest even
__device__ __forceinline__ uint32_t silu_mul_bits(uint32_t a, uint32_t b) {
  const float2 fa = __half22float2(*reinterpret_cast<const __half2*>(&a)), fb = __half22float2(*reinterpret_cast<const __half2*>(&b));
  const __half2 r = __floats2half2_rn(silu_mul(fa.x, fb.x), silu_mul(fa.y, fb.y));
  return *reinterpret_cast<const uint32_t*>(&r);
}
// the activations of a residual word's four columns (the bytes of `cols`), as two fp16 pairs
__device__ __forceinline__ uint2 word_x(const __half* x, const __half* x2, uint32_t cols) {
  uint32_t v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = ldg_u16_coherent(x + ((cols >> (8 * k)) & 0xFFu));
  uint2 r = make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
  if (x2) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = ldg_u16_coherent(x2 + ((cols >> (8 * k)) & 0xFFu));
    r.x = silu_mul_bits(r.x, w[0] | (w[1] << 16)); r.y = silu_mul_bits(r.y, w[2] | (w[3] << 16));
  }
  return r;
}

// Dealing the T = R nb tiles of a phase (R row tiles of nb blocks) to G CTAs.
//   aligned:  the first Ge = min(G, R) CTAs get whole row tiles, CTA c the row tiles [c R / Ge, (c + 1) R / Ge)
//   else:     the first Ge = min(G, T) CTAs get the tiles [c T / Ge, (c + 1) T / Ge)
// (no CTA below Ge is empty); a CTA's range is cut into 16 equal runs for its warps.
__host__ __device__ __forceinline__ int dealt_ctas(int R, int nb, bool aligned, int G) {
  const long long units = aligned ? (long long)R : (long long)R * nb;
  return units < (long long)G ? (int)units : G;
}
__host__ __device__ __forceinline__ void cta_range(int R, int nb, bool aligned, int Ge, int c, int& lo, int& hi) {
  if (aligned) {
    lo = (int)((long long)R * c / Ge) * nb;
    hi = (int)((long long)R * (c + 1) / Ge) * nb;
  } else {
    const long long T = (long long)R * nb;
    lo = (int)(T * c / Ge);
    hi = (int)(T * (c + 1) / Ge);
  }
}
// the CTA that owns tile L (not aligned)
__host__ __device__ __forceinline__ int owner_of(long long L, long long T, int Ge) { return (int)(((L + 1) * Ge - 1) / T); }
// a warp's run of its CTA's range
__device__ __forceinline__ void warp_range(const CtaRange& r, int warp, int& lo, int& hi) {
  const int len = r.hi - r.lo;
  lo = r.lo + (int)(((long long)len * warp) >> 4);
  hi = r.lo + (int)(((long long)len * (warp + 1)) >> 4);
}
static_assert(kSWarps == 16, "warp_range divides by 16 with a shift");

__device__ __forceinline__ int step_of(const StackPhase& q, int R) {
  int i = 0;
#pragma unroll
  for (int k = 1; k < kMaxFusedSteps; ++k)
    if (k < q.count && R >= q.tile_start[k]) i = k;
  return i;
}

// What is in a ring slot: x = tiles (bits 0..1), residual words of the first block (from bit 8) and of all (from bit 16), flags;
// y = first block; z = number of the first residual word (counted through the phase where its activations are gathered);
// w = row tile (numbered through the phase).
constexpr uint32_t kSegEnd = 1u << 24;        // the warp's tiles of this row tile end with the chunk ...
constexpr uint32_t kSegWhole = 1u << 25;      // ... and were all of it
constexpr uint32_t kSegLeads = 1u << 26;      // ... or began with its first block
constexpr uint32_t kRunEnd = 1u << 27;        // the warp's run of the phase ends with the chunk

// The copies of one ring: a walk through the warp's tiles of all phases in chunks of up to kSChunk tiles that never cross a
// row tile.  Between chunks it only bumps pointers; the word counts of the next chunk's blocks (which give the size of
// their residual records) are loaded when the previous chunk is issued.
struct TileWalk {
  int phase;              // current phase (== nphase: finished)
  int left;               // tiles left in the warp's run of this phase
  int step, R;            // step, and row tile (numbered through the phase)
  int blk, first;         // next block of the row tile, and the run's first block of it
  uint32_t tb;            // tile bytes of this phase
  uint32_t words;         // residual words of the phase's earlier steps (0 without gathering)
  const uint8_t* src;     // next tile
  const uint8_t* rec;     // next residual record
  uint4 ba, bb;           // second 16 bytes of the BlockInfo of blocks blk, blk + 1: { nsal, rw_off, nrw, - }

  __device__ __forceinline__ int count(int nb) const { return min(min(kSChunk, left), nb - blk); }
  __device__ __forceinline__ void load_info(const StackPhase& q) {
    const uint4* bi = reinterpret_cast<const uint4*>(q.packed[step] + sizeof(Header)) + 4 * blk + 1;
    ba = __ldg(bi);
    bb = make_uint4(0, 0, 0, 0);
    if (count(q.m / kBlock) > 1) bb = __ldg(bi + 4);
  }
  // row tile R, block blk of step `step`; the residual record's place needs the block's first word number
  __device__ __forceinline__ void locate(const StackPhase& q, const uint32_t* nrw) {
    const int nb = q.m / kBlock, rt = R - q.tile_start[step], ntile = q.tile_start[step + 1] - q.tile_start[step];
    const uint8_t* tiles = q.packed[step] + tiles_offset(nb);
    load_info(q);
    src = tiles + ((size_t)rt * nb + blk) * tb;
    rec = tiles + (size_t)tb * nb * ntile + (size_t)rt * resid_rt_bytes(nb, nrw[step]) + kResidA2Bytes * (uint32_t)blk;
    words = 0;
    if (q.gather)
      for (int k = 0; k < step; ++k) words += nrw[k];
    rec += (size_t)kResidWordBytes * ba.y;
  }
  __device__ __forceinline__ void enter(const StackParams& P, const CtaRange* range, const uint32_t* nrw, int ph, int warp) {
    for (phase = ph; phase < P.nphase; ++phase) {
      const StackPhase& q = P.ph[phase];
      const CtaRange r = range[phase];
      int lo, hi;
      warp_range(r, warp, lo, hi);
      if (lo >= hi) continue;
      const int nb = q.m / kBlock;
      tb = tile_bytes(q.N);
      left = hi - lo;
      R = r.first + (int)((uint32_t)(lo - r.first * nb) / (uint32_t)nb);
      blk = first = lo - R * nb;
      step = step_of(q, R);
      locate(q, nrw + phase * kMaxFusedSteps);
      return;
    }
  }
};

// The copying warps, one per scheduler so that none of them loses more issue slots to copying than the others: lane l of
// the i-th feeds the ring of warp 4 l + i.  A slot is refilled when its reader has arrived on its empty barrier;
// the wait has no limit of its own (a reader may be waiting for other CTAs) but ends with the CTA's failed flag.
__device__ __forceinline__ void feed_rings(const StackParams& P, uint8_t* smem, uint8_t* base, volatile int* ctl) {
  const int w = 4 * (int)(threadIdx.x & 31) + (int)((threadIdx.x >> 5) & 3u);
  const CtaRange* range = reinterpret_cast<const CtaRange*>(base + SSmem::range);
  const uint32_t* nrw = reinterpret_cast<const uint32_t*>(base + SSmem::nrw);
  if (w >= kSWarps) return;
  TileWalk t;
  t.enter(P, range, nrw, 0, w);
  const uint32_t full = smem_u32(base + SSmem::full) + 8u * kSDepth * (uint32_t)w, empty = smem_u32(base + SSmem::empty) + 8u * kSDepth * (uint32_t)w;
  const uint32_t ring = smem_u32(smem + P.ring_off) + (uint32_t)w * kSDepth * P.slot_bytes;
  uint4* chunk = reinterpret_cast<uint4*>(base + SSmem::chunks) + kSDepth * w;
  uint32_t k = 0;                                     // chunks issued
  while (t.phase < P.nphase) {
    const uint32_t slot = k % kSDepth;
    if (k >= kSDepth && !mbar_try_wait(empty + 8u * slot, (k / kSDepth - 1u) & 1u)) {
      if (ctl[0]) return;
      __nanosleep(100);               // (a slot lasts its reader about 3 us)
      continue;
    }
    const StackPhase& q = P.ph[t.phase];
    const int nb = q.m / kBlock;
    const uint32_t na = t.ba.z;
    uint32_t nw = na + t.bb.z;
    int cnt = t.count(nb);
    if (nw > P.slot_words) { cnt = 1; nw = na; }
    const bool seg_end = t.blk + cnt == nb || t.left == cnt;
    uint4 c;
    c.x = (uint32_t)cnt | (na << 8) | (nw << 16);
    if (seg_end) c.x |= kSegEnd | (t.first == 0 ? (t.blk + cnt == nb ? kSegWhole : kSegLeads) : 0u);
    if (t.left == cnt) c.x |= kRunEnd;
    c.y = (uint32_t)t.blk; c.z = t.words + t.ba.y; c.w = (uint32_t)t.R;
    chunk[slot] = c;                                  // (seen by the reader through the full barrier)
    const uint32_t tile_b = (uint32_t)cnt * t.tb, rec_b = (uint32_t)cnt * kResidA2Bytes + nw * kResidWordBytes;
    const uint32_t bar = full + 8u * slot, dst = ring + slot * P.slot_bytes;
    mbar_expect_tx(bar, tile_b + rec_b);
    // copies off (the wait self-test): the barrier is armed but nothing will ever complete it
    if (!P.copies_off) {
      bulk_g2s(dst, t.src, tile_b, bar);
      bulk_g2s(dst + P.slot_tiles, t.rec, rec_b, bar);
    }
    ++k;
    t.left -= cnt; t.blk += cnt;
    if (t.left == 0) t.enter(P, range, nrw, t.phase + 1, w);
    else {
      t.src += tile_b; t.rec += rec_b;
      if (t.blk == nb) {
        t.blk = t.first = 0; ++t.R;
        if (t.R == q.tile_start[t.step + 1]) { ++t.step; t.locate(q, nrw + t.phase * kMaxFusedSteps); }
        else t.load_info(q);
      } else t.load_info(q);
    }
  }
}

// What a decoding warp carries through the whole kernel: the slot it reads next and the phase parity of its barrier.
struct WarpState {
  uint32_t slot, parity;
  bool failed;                        // a wait ran out, or the CTA was told to stop
};
struct WarpEnv {
  const StackParams* P;
  uint8_t* smem;
  uint8_t* base;
  uint8_t* ring;                      // of this warp
  const uint4* chunk;
  uint32_t full, empty;
  int warp, lane, g, t;
};
__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kSThreads) : "memory"); }

// ------------------------------------------------------------------------------------------
// Where the residual term finds the activations of a chunk's words:
//   kGathered  gathered for the whole phase in shared memory ([word][batch row], four fp16 each)
//   kPlaced    in the lane's row of activations, staged or in global memory, at places kept in shared memory (four per word)
//   kListed    in global memory, in the columns that the layer's word table names: two trips, for words too many for the others
enum class ResidForm { kGathered, kPlaced, kListed };
struct ResidX {
  const uint8_t* xw;            // kGathered: of the lane's batch row, at the chunk's first word ...
  uint32_t xw_step;             // ... and bytes per word
  const uint2* places;          // kPlaced: of the chunk's first word
  const uint8_t* row;           // kPlaced: the lane's row of activations, null beyond the batch
  const ResidWord* words;       // kListed: the chunk's first word
  const __half *xg, *xg2;       // kListed: the lane's row of the input (null beyond the batch), and of the second one
};
// Residual term of a chunk: its residual words, four (16 salient slots) per tensor-core step, lane t the t-th.  rec: the
// chunk's records; na / nw: words of its first block / of all.  kShared: kPlaced from staged activations.
template <ResidForm kForm, bool kShared>
__device__ __forceinline__ void resid_mul(const uint8_t* rec, uint32_t na, uint32_t nw, int g, int t, const ResidX& X, float (&acc)[2][1][4]) {
#pragma unroll 1
  for (uint32_t k0 = 0; k0 < nw; k0 += 4u) {
    const uint32_t kk = k0 + (uint32_t)t, k = min(kk, nw - 1u);
    const bool second = k >= na;
    // records: a_sal2 of the 32 rows, then the block's words
    const uint8_t* r = rec + k * kResidWordBytes + (second ? 2u * kResidA2Bytes : kResidA2Bytes);
    uint32_t rw = *reinterpret_cast<const uint32_t*>(r + 4 * g), fa[4][2];
    const uint2 a2 = *reinterpret_cast<const uint2*>(rec + (second ? kResidA2Bytes + na * kResidWordBytes : 0u) + 8 * g);
    if (kk >= nw) rw = kNoTerms;
    resid_operands(rw, a2, fa);
    uint2 xr = make_uint2(0, 0);
    if constexpr (kForm == ResidForm::kGathered) xr = *reinterpret_cast<const uint2*>(X.xw + k * X.xw_step);
    else if constexpr (kForm == ResidForm::kPlaced) {
      if (X.row) {
        const uint2 at = X.places[k];
        const uint16_t* x = reinterpret_cast<const uint16_t*>(X.row);
        if (kShared) {
          xr.x = (uint32_t)x[at.x & 0xFFFFu] | ((uint32_t)x[at.x >> 16] << 16);
          xr.y = (uint32_t)x[at.y & 0xFFFFu] | ((uint32_t)x[at.y >> 16] << 16);
        } else {
          xr.x = ldg_u16_coherent(x + (at.x & 0xFFFFu)) | (ldg_u16_coherent(x + (at.x >> 16)) << 16);
          xr.y = ldg_u16_coherent(x + (at.y & 0xFFFFu)) | (ldg_u16_coherent(x + (at.y >> 16)) << 16);
        }
      }
    } else if (X.xg) {
      const uint2 e = __ldg(reinterpret_cast<const uint2*>(X.words + k));
      const size_t o = (size_t)(e.x >> 3) * kBlock;
      xr = word_x(X.xg + o, X.xg2 ? X.xg2 + o : nullptr, e.y);
    }
    mma16816(acc[0][0], fa[0][0], fa[1][0], fa[0][1], fa[1][1], xr.x, xr.y);
    mma16816(acc[1][0], fa[2][0], fa[3][0], fa[2][1], fa[3][1], xr.x, xr.y);
  }
}

// The warp's run of phase q: chunks of residual words and tiles, partial sums out.
// kImage: 6:8 from the operand-order image; kStaged: position order with the activations in a plain copy in shared memory
// kForm: the residual activations are gathered throughout the launch, or, where a phase's are not, found by places / the layer's word table
template <int N, bool kImage, bool kStaged, ResidForm kForm, bool kDot = false>
__device__ __forceinline__ void run_tiles(const WarpEnv& E, WarpState& W, const StackPhase& q, int* pslot, float* pdata) {
  constexpr bool kPlaces = kForm == ResidForm::kPlaced;
  const StackParams& P = *E.P;
  const int lane = E.lane, g = E.g, t = E.t, warp = E.warp, batch = q.batch;
  constexpr uint32_t tb = tile_bytes(N);
  const bool xlive = g < batch;
  const uint8_t* zero = E.base + SSmem::zero;
  // The lane's activations: base and bytes per block.  Lanes beyond the batch read zeros.
  const uint8_t* xbase;
  uint32_t xstep;
  if (kImage) {
    xbase = xlive ? E.smem + P.x_off + (uint32_t)g * ((uint32_t)(q.m / kBlock) * kImgWordsPerBlock * 4u) + (uint32_t)t * 96u : zero;
    xstep = xlive ? kImgWordsPerBlock * 4u : 0u;
  } else if (kStaged) {
    xbase = xlive ? E.smem + P.x_off + (uint32_t)g * (2u * (uint32_t)q.m + kXPad) + (uint32_t)t * 16u : zero;
    xstep = xlive ? 2u * kBlock : 0u;
  } else {
    xbase = xlive ? reinterpret_cast<const uint8_t*>(q.x + (size_t)g * q.ldx + 8 * t) : nullptr;
    xstep = xlive ? 2u * kBlock : 0u;
  }
  const uint32_t xw_step = xlive ? 8u * (uint32_t)batch : 0u;
  const uint8_t* xs = xlive ? E.smem + P.xs_off + (uint32_t)g * 8u : zero;
  const uint8_t* ptab = kImage ? nullptr : E.smem + P.pos_off[N - 4] + (uint32_t)(lane & (kPosCopies - 1)) * 8u;
  const uint32_t prow = P.pos_row;
  float acc[2][1][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int d = 0; d < 4; ++d) acc[a][0][d] = 0.0f;
  uint4 c;
  do {
    const uint32_t slot = W.slot, bar = E.full + 8u * slot;
    // all lanes poll; the verdict is made warp-uniform
    if (!__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, W.parity)) && !__all_sync(0xFFFFFFFFu, mbar_wait(bar, W.parity, P.wait_limit))) { W.failed = true; return; }
    c = E.chunk[slot];
    const uint8_t* tile = E.ring + slot * P.slot_bytes;
    const uint32_t na = (c.x >> 8) & 0xFFu, nw = (c.x >> 16) & 0xFFu;
    const uint8_t* records = tile + P.slot_tiles;
    auto residual = [&] {
      if (nw == 0u) return;
      ResidX X;
      if (kForm == ResidForm::kGathered || q.gather == 2) {
        X.xw = xs + c.z * xw_step; X.xw_step = xw_step;
        resid_mul<ResidForm::kGathered, true>(records, na, nw, g, t, X, acc);
      } else if constexpr (kPlaces) {
        X.places = reinterpret_cast<const uint2*>(E.smem + P.cols_off) + c.z;
        X.row = xlive ? xbase - (uint32_t)t * (kImage ? 96u : 16u) : nullptr;
        resid_mul<ResidForm::kPlaced, kImage || kStaged>(records, na, nw, g, t, X, acc);
      } else {
        X.words = reinterpret_cast<const ResidWord*>(q.packed[step_of(q, (int)c.w)] + rwtab_offset(q.m / kBlock)) + c.z;
        X.xg = xlive ? q.x + (size_t)g * q.ldx : nullptr;
        X.xg2 = q.x2 ? q.x2 + (size_t)g * q.ldx : nullptr;
        resid_mul<ResidForm::kListed, false>(records, na, nw, g, t, X, acc);
      }
    };
    // The words come before the tiles of their chunk: the tensor core cuts off what it adds to a large sum, so that words added to the
    // sum of one more chunk lose more (drawn 4:8 and 5:8 layers, one row, against float64: 0.4 % more error with them after the tiles).
    // Words whose activations are in global memory come after the tiles, whose lines they find in L1 (before them, 2 % slower at two
    // rows, 4 to 8 % at eight).
    constexpr bool kLate = kPlaces && !kImage && !kStaged;
    // When the slot is handed back: once its last tile is in registers, or, gathered in position order, after the products (handing it
    // back in between keeps the loads of the activations behind it: four 7B layers at 4:8 238 -> 221 us, at 5:8 246 -> 230; at 6:8
    // 189.4 against 197.8).
    constexpr bool kBack = kLate || (kForm == ResidForm::kGathered && !kImage);
    if (!kLate) residual();
    const uint8_t* xb = xbase + (size_t)c.y * xstep;
    const int cnt = (int)(c.x & 3u);
#pragma unroll 1
    for (int k = 0; k < cnt; ++k) {
      const uint8_t* const xp[1] = {xb};
      if constexpr (kImage) {
        Tile6 d;
        load_tile(tile, lane, d);
        if (!kBack && k == cnt - 1) { __syncwarp(); if (lane == 0) mbar_arrive(E.empty + 8u * slot); }
        tile_mul<1>(d, E.smem, xp, acc);
      } else {
        TileD<N> d;
        load_tile<N>(tile, lane, ptab, prow, d);
        if (!kBack && k == cnt - 1) { __syncwarp(); if (lane == 0) mbar_arrive(E.empty + 8u * slot); }
        tile_mul<N, kStaged, 1, kDot>(d, xp, acc);
      }
      tile += tb;
      xb += xstep;
    }
    if (kLate) residual();
    if (kBack) { __syncwarp(); if (lane == 0) mbar_arrive(E.empty + 8u * slot); }
    W.slot ^= 1u;
    W.parity ^= slot;
    if (c.x & kSegEnd) {
      // the warp's tiles of the row tile are summed: a whole row tile goes to y, a piece to shared memory
      if (c.x & kSegWhole) {
        const int si = step_of(q, (int)c.w), rt = (int)c.w - q.tile_start[si];
        const bool f16 = (q.f16_mask >> si) & 1;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int d = 0; d < 4; ++d) {
            const int row = rt * kTileRows + g + 16 * mt + 8 * (d >> 1), bc = 2 * t + (d & 1);
            if (row < q.n[si] && bc < batch) {
              if (f16) static_cast<__half*>(q.y[si])[(size_t)bc * q.ldy[si] + row] = __float2half_rn(acc[mt][0][d]);
              else static_cast<float*>(q.y[si])[(size_t)bc * q.ldy[si] + row] = acc[mt][0][d];
            }
          }
      } else {
        // slot 2 w: the row tile began with another warp (or CTA); slot 2 w + 1: it begins here
        const int ps = 2 * warp + (c.x & kSegLeads ? 1 : 0);
        float* pd = pdata + (size_t)ps * P.part_floats;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int d = 0; d < 4; ++d) {
            const int r = g + 16 * mt + 8 * (d >> 1), bc = 2 * t + (d & 1);
            if (bc < batch) pd[r * batch + bc] = acc[mt][0][d];
          }
        if (lane == 0) pslot[ps] = (int)c.w;
      }
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int d = 0; d < 4; ++d) acc[a][0][d] = 0.0f;
    }
  } while (!(c.x & kRunEnd));
}

// ------------------------------------------------------------------------------------------
// Checks the packed headers of all steps (every CTA reads the same headers and takes the same way out), notes their
// residual word counts, and works out this CTA's tile range of every phase.
__device__ __forceinline__ bool stack_setup(const StackParams& P, uint8_t* base, volatile int* ctl) {
  if (threadIdx.x == 0) ctl[3] = 0;
  if (threadIdx.x < kSWarps * kSDepth) {
    mbar_init(smem_u32(base + SSmem::full) + 8u * threadIdx.x, 1);
    mbar_init(smem_u32(base + SSmem::empty) + 8u * threadIdx.x, 1);
    fence_async_smem();
  }
  __syncthreads();
  for (int i = threadIdx.x; i < P.nphase * kMaxFusedSteps; i += kSAllThreads) {
    const StackPhase& q = P.ph[i / kMaxFusedSteps];
    const int k = i % kMaxFusedSteps;
    uint32_t nrw = 0;
    if (k < q.count) {
      const Header* h = reinterpret_cast<const Header*>(q.packed[k]);
      nrw = h->nrw;
      if (!header_matches(h, q.n[k], q.m, q.N)) ctl[3] = 1;
    }
    reinterpret_cast<uint32_t*>(base + SSmem::nrw)[i] = nrw;
  }
  // from the last thread down: the first ones load headers
  for (int i = kSAllThreads - 1 - (int)threadIdx.x; i < P.nphase; i += kSAllThreads) {
    const StackPhase& q = P.ph[i];
    const int nb = q.m / kBlock, R = q.tile_start[q.count], cta = (int)blockIdx.x, G = (int)gridDim.x;
    const int Ge = dealt_ctas(R, nb, q.aligned != 0, G);
    CtaRange r = {0, 0, 0, 0, 0, 1, 0, 1};
    if (cta < Ge) {
      cta_range(R, nb, q.aligned != 0, Ge, cta, r.lo, r.hi);
      r.first = (int)((uint32_t)r.lo / (uint32_t)nb);
      const int up = (int)(((uint32_t)r.lo + (uint32_t)nb - 1u) / (uint32_t)nb), down = (int)((uint32_t)r.hi / (uint32_t)nb);
      r.whole = down > up ? down - up : 0;
      if (!q.aligned) {
        const long long T = (long long)R * nb;
        const int last = (int)((uint32_t)(r.hi - 1) / (uint32_t)nb);
        r.head_cta = owner_of((long long)r.first * nb, T, Ge);
        r.head_share = owner_of((long long)(r.first + 1) * nb - 1, T, Ge) - r.head_cta + 1;
        r.tail_cta = owner_of((long long)last * nb, T, Ge);
        r.tail_share = owner_of((long long)(last + 1) * nb - 1, T, Ge) - r.tail_cta + 1;
      }
    }
    reinterpret_cast<CtaRange*>(base + SSmem::range)[i] = r;
  }
  __syncthreads();
  return ctl[3] == 0;
}

// The decoding warps: all phases in order.
template <ResidForm kForm, bool kOnly5>
__device__ __forceinline__ void decode_phases(const StackParams& P, uint8_t* smem, uint8_t* base, volatile int* ctl, int* pslot, float* pdata, int cta) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* ximg = reinterpret_cast<uint32_t*>(smem + P.x_off);
  WarpEnv E;
  E.P = &P; E.smem = smem; E.base = base; E.warp = warp; E.lane = lane; E.g = lane >> 2; E.t = lane & 3;
  E.ring = smem + P.ring_off + warp * kSDepth * P.slot_bytes;
  E.chunk = reinterpret_cast<const uint4*>(base + SSmem::chunks) + kSDepth * warp;
  E.full = smem_u32(base + SSmem::full) + 8u * kSDepth * (uint32_t)warp;
  E.empty = smem_u32(base + SSmem::empty) + 8u * kSDepth * (uint32_t)warp;
  WarpState W;
  W.slot = 0; W.parity = 0; W.failed = false;
  const uint32_t epoch = __ldcg(P.sync + 4);          // changed only by the last CTA out
  // tables, while the first copies are under way
  if (P.use_meta6) fill_meta6(smem, (int)threadIdx.x, kSThreads);
#pragma unroll
  for (int N = 4; N <= 6; ++N)
    if (P.pos_off[N - 4])
      for (int i = threadIdx.x; i < kPosTableEntries * (int)kPosCopies; i += kSThreads)
        reinterpret_cast<uint2*>(smem + P.pos_off[N - 4])[i] = g_pos_table.v[N][i / (int)kPosCopies];
  if (threadIdx.x < 384 / 4) reinterpret_cast<uint32_t*>(base + SSmem::zero)[threadIdx.x] = 0u;

  for (int ph = 0; ph < P.nphase; ++ph) {
    const StackPhase& q = P.ph[ph];
    const int nb = q.m / kBlock, batch = q.batch;
    const uint32_t* nrw = reinterpret_cast<const uint32_t*>(base + SSmem::nrw) + ph * kMaxFusedSteps;
    const CtaRange range = reinterpret_cast<const CtaRange*>(base + SSmem::range)[ph];
    int wl, wh;
    warp_range(range, warp, wl, wh);

    // where the activation of every residual slot will stand in the staged x (in halves, batch row 0): known before the wait
    uint16_t* cols = reinterpret_cast<uint16_t*>(smem + P.cols_off);
    uint32_t slots = 0;
    if (q.gather) {
#pragma unroll 1
      for (int k = 0; k < q.count; ++k) {
        const uint2* rwt = reinterpret_cast<const uint2*>(q.packed[k] + rwtab_offset(nb));
        const uint32_t cnt = 4u * nrw[k];
#pragma unroll 1
        for (uint32_t i = threadIdx.x; i < cnt; i += kSThreads) {
          const uint2 e = __ldg(rwt + (i >> 2));
          cols[slots + i] = (uint16_t)staged_index(q.use_image == 1, e.x >> 3, (e.y >> (8u * (i & 3u))) & 0xFFu);
        }
        slots += cnt;
      }
    }
    if (lane < 2) pslot[2 * warp + lane] = -1;

    // ---- wait until every earlier phase has finished, then stage the activations ----
    if (q.done_before > 0) {
      if (threadIdx.x == 0 && !ctl[0]) {
        const long long t0 = clock64();
        for (;;) {
          // one load brings the count of finished row tiles (low word) and the abort flag (high word)
          const unsigned long long v = ld_acquire_u64(P.sync);
          if ((uint32_t)v >= q.done_before) break;
          if ((uint32_t)(v >> 32) != 0u) { ctl[0] = 1; break; }
          if (clock64() - t0 > P.wait_limit) {
            ctl[0] = 1;
            atomicExch(P.sync + 1, 1u);
            if (P.dev_status) *P.dev_status = STB_ERR_TIMEOUT;
            break;
          }
        }
      }
      consumers_sync();
    }
    const bool stop = ctl[0] != 0;
    if (stop) W.failed = true;
    // The code between two phases runs once per phase, much of it out of a cold instruction cache: it is kept short rather
    // than unrolled.  An item = eight activations of a batch row; two or three at a time are on their way.
    if (q.use_image && !stop) {
      const int per_row = q.m / 8, items = batch * per_row;
      constexpr int kAhead = kForm == ResidForm::kGathered ? 3 : 2;      // (with 3 the others spill)
#pragma unroll 1
      for (int first = threadIdx.x; first < items; first += kAhead * kSThreads) {
        uint4 v[kAhead], v2[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
          const int it = first + k * kSThreads, r = batch == 1 ? 0 : it / per_row;
          const size_t o = (size_t)r * q.ldx + (size_t)(it - r * per_row) * 8;
          v[k] = v2[k] = make_uint4(0, 0, 0, 0);
          if (it < items) {
            v[k] = ldg_v4_coherent(q.x + o);
            if (q.x2) v2[k] = ldg_v4_coherent(q.x2 + o);
          }
        }
#pragma unroll 1
        for (int cur = first, k = 0; k < kAhead && cur < items; ++k, cur += kSThreads) {
          uint32_t a[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
          const uint32_t b[4] = {v2[0].x, v2[0].y, v2[0].z, v2[0].w};
#pragma unroll
          for (int u = 0; u + 1 < kAhead; ++u) { v[u] = v[u + 1]; v2[u] = v2[u + 1]; }
          if (q.x2) {
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] = silu_mul_bits(a[u], b[u]);
          }
          const int r = batch == 1 ? 0 : cur / per_row, qq = cur - r * per_row;
          if (q.use_image == 1) {
            image_store(ximg + (uint32_t)r * ((uint32_t)nb * kImgWordsPerBlock), (uint32_t)qq >> 4, (uint32_t)qq & 15u, a);
          } else {
            *reinterpret_cast<uint4*>(smem + P.x_off + (uint32_t)r * (2u * (uint32_t)q.m + kXPad) + (uint32_t)qq * 16u) = make_uint4(a[0], a[1], a[2], a[3]);
          }
        }
      }
    }
    consumers_sync();
    if (q.gather == 2 && !stop) {
      // activations of the residual slots: [word of all steps][batch row], four fp16 each
      uint16_t* xs = reinterpret_cast<uint16_t*>(smem + P.xs_off);
      const uint32_t pitch = q.use_image == 1 ? (uint32_t)nb * kImgWordsPerBlock * 2u : (uint32_t)q.m + kXPad / 2u;
#pragma unroll 1
      for (uint32_t i = threadIdx.x; i < slots; i += kSThreads) {
        const uint16_t* src = reinterpret_cast<const uint16_t*>(smem + P.x_off) + cols[i];
        uint16_t* d = xs + (size_t)(i >> 2) * 4u * (uint32_t)batch + (i & 3u);
#pragma unroll 1
        for (int r = 0; r < batch; ++r) d[4 * r] = src[r * pitch];
      }
      consumers_sync();
    }

    // ---- this warp's tiles ----
    if (!W.failed && wl < wh) {
      if constexpr (kOnly5) run_tiles<5, false, true, kForm, true>(E, W, q, pslot, pdata);
      else if (q.use_image == 1) run_tiles<6, true, false, kForm>(E, W, q, pslot, pdata);
      else if (kForm == ResidForm::kGathered) {
        if (q.N == 5) run_tiles<5, false, true, kForm>(E, W, q, pslot, pdata);
        else run_tiles<4, false, true, kForm>(E, W, q, pslot, pdata);
      } else if (q.use_image == 2) {
        if (q.N == 6) run_tiles<6, false, true, kForm>(E, W, q, pslot, pdata);
        else if (q.N == 5) run_tiles<5, false, true, kForm>(E, W, q, pslot, pdata);
        else run_tiles<4, false, true, kForm>(E, W, q, pslot, pdata);
      } else if (q.N == 6) run_tiles<6, false, false, kForm>(E, W, q, pslot, pdata);
      else if (q.N == 5) run_tiles<5, false, false, kForm>(E, W, q, pslot, pdata);
      else run_tiles<4, false, false, kForm>(E, W, q, pslot, pdata);
    }
    if (W.failed && lane == 0 && !ctl[0]) {
      // this warp's own wait ran out: tell the CTA and the grid
      ctl[0] = 1;
      atomicExch(P.sync + 1, 1u);
      if (P.dev_status) *P.dev_status = STB_ERR_TIMEOUT;
    }
    consumers_sync();

    // ---- pieces of row tiles, added in tile order by the warp where the row tile begins (in this CTA) ----
    if (!ctl[0]) {
      const int cont = lane < kSWarps ? pslot[2 * lane] : -1;           // the row tile each warp continues
      const int nval = 32 * batch;                                      // values of a row tile: [row][batch column]
#pragma unroll 1
      for (int s0 = 2 * warp; s0 < 2 * warp + 2; ++s0) {
        const int R = pslot[s0];
        // slot 2 w leads only where the CTA's range begins inside a row tile and no earlier warp has a piece of it
        const uint32_t others = __ballot_sync(0xFFFFFFFFu, cont == R);
        if (R < 0 || (!(s0 & 1) && ((others & ((1u << warp) - 1u)) != 0u || R != range.first || range.lo == R * nb))) continue;
        const uint32_t members = others & ~((2u << warp) - 1u);        // later warps' pieces, in order
        const int si = step_of(q, R);
        const int rt = R - q.tile_start[si];
        const bool f16 = (q.f16_mask >> si) & 1;
        const bool whole = range.lo <= R * nb && range.hi >= (R + 1) * nb;
        // a straddling row tile: the CTA where it begins gathers the others' sums, in CTA order
        const int c_first = R == range.first ? range.head_cta : range.tail_cta, share = R == range.first ? range.head_share : range.tail_share;
        uint2* gp = P.gpart + (size_t)R * P.max_share * P.part_floats;
        const uint32_t tag = ((epoch + 1u) << 6) | (uint32_t)ph;
        bool lost = false;
        for (int v = lane; v < nval; v += 32) {
          const float* pv = pdata + v;
          float sum = pv[(size_t)s0 * P.part_floats];
          // The pieces are loaded all at once and added in order; by four where the kernel has more forms of the tile loop to hold registers
          // for (all at once, it spilled: 13B block at 5:8, two rows, 106.2 us against 103.8).
          if constexpr (kForm == ResidForm::kGathered) {
            float x[kSWarps];
#pragma unroll
            for (int w = 1; w < kSWarps; ++w) x[w] = (members >> w) & 1u ? pv[(uint32_t)(2 * w) * P.part_floats] : 0.0f;
#pragma unroll
            for (int w = 1; w < kSWarps; ++w) sum += x[w];
          } else {
            constexpr int kLoads = 4;
            const float* pw = pv;
#pragma unroll 1
            for (uint32_t mm = members; mm != 0u; mm >>= kLoads) {
              float x[kLoads];
#pragma unroll
              for (int k = 0; k < kLoads; ++k) { x[k] = (mm >> k) & 1u ? *pw : 0.0f; pw += 2 * P.part_floats; }
#pragma unroll
              for (int k = 0; k < kLoads; ++k) sum += x[k];
            }
          }
          if (!whole && cta != c_first) {
            st_tagged(gp + (size_t)(cta - c_first) * P.part_floats + v, sum, tag);
            continue;
          }
          if (!whole) {
            const long long t0 = clock64();
            for (int k = 1; k < share && !lost; ++k) {
              uint2 x = ld_tagged(gp + (size_t)k * P.part_floats + v);
              while (x.y != tag && !lost) {
                lost = clock64() - t0 > P.wait_limit || *reinterpret_cast<volatile uint32_t*>(P.sync + 1) != 0u;
                x = ld_tagged(gp + (size_t)k * P.part_floats + v);
              }
              sum += __uint_as_float(x.x);
              st_tagged(gp + (size_t)k * P.part_floats + v, 0.0f, 0u);      // empty for whoever uses it next
            }
          }
          const int row = rt * kTileRows + (batch == 1 ? v : v / batch), bc = batch == 1 ? 0 : v % batch;
          if (row < q.n[si]) {
            if (f16) static_cast<__half*>(q.y[si])[(size_t)bc * q.ldy[si] + row] = __float2half_rn(sum);
            else static_cast<float*>(q.y[si])[(size_t)bc * q.ldy[si] + row] = sum;
          }
        }
        if (!whole && cta == c_first && lane == 0) atomicAdd(const_cast<int*>(&ctl[1]), 1);
        if (__any_sync(0xFFFFFFFFu, lost) && lane == 0) {
          ctl[0] = 1;
          atomicExch(P.sync + 1, 1u);
          if (P.dev_status) *P.dev_status = STB_ERR_TIMEOUT;
        }
      }
    }
    consumers_sync();
    if (threadIdx.x == 0) {
      const int fin = range.whole + ctl[1];
      ctl[1] = 0;
      // release at GPU scope: the CTA's stores to y (ordered before this thread by the barrier) are visible to
      // whoever sees the count
      if (fin > 0 && !ctl[0]) red_release_add(P.sync, (uint32_t)fin);
    }
  }
}

template <ResidForm kForm, bool kOnly5>
__global__ void __launch_bounds__(kSAllThreads, 1)
stack_kernel(const __grid_constant__ StackParams P) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int cta = (int)blockIdx.x, G = (int)gridDim.x;
  uint8_t* base = smem + (P.use_meta6 ? kMeta6Bytes : 0u);
  volatile int* ctl = reinterpret_cast<volatile int*>(base + SSmem::ctl);      // [0] failed, [1] straddling row tiles this CTA finished, [2] last CTA out, [3] a packed header does not match
  int* pslot = reinterpret_cast<int*>(base + SSmem::slots);
  float* pdata = reinterpret_cast<float*>(smem + P.pdata_off);

  grid_dependency_wait();          // a programmatic dependent of whatever ran before (see the launch): nothing in memory is touched until that is done
  if (!stack_setup(P, base, ctl)) {          // before anything was streamed or the workspace touched
    if (threadIdx.x == 0 && cta == 0 && P.dev_status) *P.dev_status = STB_ERR_CORRUPT;
    return;
  }
  if (threadIdx.x == 0) { ctl[0] = 0; ctl[1] = 0; ctl[2] = 0; }
  __syncthreads();
  grid_launch_dependents();
  if (threadIdx.x >= kSThreads) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFeedRegs));
    feed_rings(P, smem, base, ctl);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kDecodeRegs));
    decode_phases<kForm, kOnly5>(P, smem, base, ctl, pslot, pdata, cta);
  }

  // ---- leaving: let copies in flight land, then the last CTA out restores the workspace ----
  __syncthreads();
  if (ctl[0]) {
    const long long t0 = clock64();
    while (clock64() - t0 < 200000) {}
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const uint32_t old = atomicAdd(P.sync + 2, 1u);
    ctl[2] = (old == (uint32_t)G - 1u) ? 1 : 0;
  }
  __syncthreads();
  if (ctl[2]) {
    __threadfence();
    // a launch that was given up leaves sums that nobody took
    if (*reinterpret_cast<volatile uint32_t*>(P.sync + 1) != 0u)
      for (uint32_t i = threadIdx.x; i < P.gpart_slots; i += kSAllThreads) P.gpart[i] = make_uint2(0u, 0u);
    __syncthreads();
    if (threadIdx.x == 0) { P.sync[0] = 0u; P.sync[1] = 0u; P.sync[2] = 0u; P.sync[4] += 1u; __threadfence(); }
  }
}

// ------------------------------------------------------------------------------------------
// stb_layer_stack_checksum: XOR of all 32-bit words of the tiles and residual streams of every step's packed layer
// (an integrity check for packed layers that were stored or moved).  It walks the layers exactly as stack_kernel
// does -- same dealing, same per-warp rings and bulk copies -- and folds the words instead of decoding them, so its
// rate is also the rate this way of streaming reaches with no arithmetic behind it.
__global__ void __launch_bounds__(kSAllThreads, 1)
checksum_kernel(const __grid_constant__ StackParams P, unsigned long long* __restrict__ sums, int first_step) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int lane = threadIdx.x & 31;
  uint8_t* base = smem + (P.use_meta6 ? kMeta6Bytes : 0u);
  volatile int* ctl = reinterpret_cast<volatile int*>(base + SSmem::ctl);
  if (!stack_setup(P, base, ctl)) {
    if (threadIdx.x == 0 && blockIdx.x == 0 && P.dev_status) *P.dev_status = STB_ERR_CORRUPT;
    return;
  }
  if (threadIdx.x == 0) ctl[0] = 0;
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  bool failed = false;
  if (warp >= kSWarps) feed_rings(P, smem, base, ctl);
  else {
    const uint8_t* ring = smem + P.ring_off + warp * kSDepth * P.slot_bytes;
    const uint4* chunk = reinterpret_cast<const uint4*>(base + SSmem::chunks) + kSDepth * warp;
    const uint32_t full = smem_u32(base + SSmem::full) + 8u * kSDepth * (uint32_t)warp, empty = smem_u32(base + SSmem::empty) + 8u * kSDepth * (uint32_t)warp;
    uint32_t slot = 0, parity = 0;
    int step_base = first_step;                    // index, in the caller's list, of the phase's first step
    for (int ph = 0; ph < P.nphase && !failed; ++ph) {
      const StackPhase& q = P.ph[ph];
      const uint32_t tb = tile_bytes(q.N);
      int lo, hi;
      warp_range(reinterpret_cast<const CtaRange*>(base + SSmem::range)[ph], warp, lo, hi);
      uint32_t fold = 0;
      for (bool more = lo < hi; more;) {
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(full + 8u * slot, parity, P.wait_limit))) { failed = true; break; }
        const uint4 c = chunk[slot];
        const uint8_t* tile = ring + slot * P.slot_bytes;
        const uint32_t cnt = c.x & 3u, rec_b = cnt * kResidA2Bytes + ((c.x >> 16) & 0xFFu) * kResidWordBytes;
        for (uint32_t o = (uint32_t)lane * 4u; o < cnt * tb; o += 128u) fold ^= *reinterpret_cast<const uint32_t*>(tile + o);
        for (uint32_t o = (uint32_t)lane * 4u; o < rec_b; o += 128u) fold ^= *reinterpret_cast<const uint32_t*>(tile + P.slot_tiles + o);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + 8u * slot);
        parity ^= slot;
        slot ^= 1u;
        more = !(c.x & kRunEnd);
        if (c.x & kSegEnd) {
          // words of one step only ever meet words of the same step
#pragma unroll
          for (int d = 16; d > 0; d >>= 1) fold ^= __shfl_xor_sync(0xFFFFFFFFu, fold, d);
          if (lane == 0) atomicXor(sums + step_base + step_of(q, (int)c.w), (unsigned long long)fold);
          fold = 0;
        }
      }
      step_base += q.count;
    }
    if (failed && lane == 0) ctl[0] = 1;
  }
  if (failed) {
    const long long t0 = clock64();
    while (clock64() - t0 < 200000) {}
    if (lane == 0 && P.dev_status) *P.dev_status = STB_ERR_TIMEOUT;
  }
}

// ------------------------------------------------------------------------------------------
// Host side: steps -> phases -> launches.
static bool same_input(const stb_step& a, const stb_step& b) {
  return a.in == b.in && a.in2 == b.in2 && a.input == b.input && a.ldin == b.ldin && a.batch == b.batch && a.m == b.m &&
         a.N == b.N && b.out != a.in && b.out != a.in2;
}

static int check_step(const stb_step& s) {
  if (!s.packed || !s.in || !s.out) return STB_ERR_ARG;
  if (s.n < 1 || s.m < kBlock || s.m % kBlock != 0) return STB_ERR_SHAPE;
  if (s.N < 1 || s.N > 8) return STB_ERR_NM;
  if (s.N < 4 || s.N > 6) return STB_ERR_UNSUPPORTED;
  if (s.batch < 1 || s.batch > 64) return STB_ERR_SIZE;
  if (s.batch > 8) return STB_ERR_UNSUPPORTED;
  if (s.odt != STB_F32 && s.odt != STB_F16) return STB_ERR_UNSUPPORTED;
  if (s.ldin < (size_t)s.m || s.ldout < (size_t)s.n || (s.ldin % 8) != 0 || (reinterpret_cast<uintptr_t>(s.in) & 15u)) return STB_ERR_ARG;
  if (s.ldin > 0xFFFFFFFFull || s.ldout > 0xFFFFFFFFull) return STB_ERR_ARG;
  if (s.input != STB_IN_PLAIN && s.input != STB_IN_SILU_MUL) return STB_ERR_ARG;
  if (s.input == STB_IN_SILU_MUL && (!s.in2 || (reinterpret_cast<uintptr_t>(s.in2) & 15u))) return STB_ERR_ARG;
  return STB_OK;
}

// Whole row tiles per CTA when that keeps at least 85 % of the SM time busy: R row tiles on G CTAs take
// ceil(R / G) rounds of which R / G are needed.
static bool deal_aligned(long long R, int G) {
  const long long rounds = (R + G - 1) / G;
  return (double)R / (double)G >= 0.85 * (double)rounds;
}

// at most so many CTAs share one row tile of a phase of R row tiles x nb blocks dealt to G CTAs by equal tile counts
static uint32_t max_share_of(long long R, int nb, int G) {
  const long long Ge = dealt_ctas((int)R, nb, false, G);
  const long long s = (Ge + R - 1) / R + 1;
  return (uint32_t)(s < Ge ? s : Ge);
}

static int stack_sm_count(int* out) {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return STB_ERR_CUDA;
  if (dev < 0 || dev >= 64) return STB_ERR_CUDA;
  if (!cached[dev]) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) return STB_ERR_CUDA;
    cached[dev] = v;
  }
  *out = cached[dev];
  return STB_OK;
}

constexpr uint32_t kSmemLimit = 227 * 1024;
constexpr unsigned long long kGatherMax = 16 * 1024;     // shared memory for the residual words' activations, and for their places

// Lays out the shared memory of a launch and chooses each phase's staging; false where not even the rest fits.  image: 6:8 phases may
// take the operand-order image.  gather: the residual words' activations are gathered where they fit (2), or read by their places
// (1), or found by the layer's word table (0).  few: ring slots for few residual words.
static uint32_t up128(uint32_t v) { return (v + 127u) & ~127u; }
struct SmemForm { bool image; int gather; bool few; };
static bool plan_smem(StackParams& sp, const SmemForm& form, int ctas) {
  bool any6 = false, dense[3] = {false, false, false}, bare_phase[kMaxPhases] = {};
  int most_N = 4;
  for (int p = 0; p < sp.nphase; ++p) {
    if (sp.ph[p].N > most_N) most_N = sp.ph[p].N;
    if (sp.ph[p].N == 6 && form.image) any6 = true;
    else dense[sp.ph[p].N - 4] = true;
  }
  sp.slot_tiles = slot_tiles(most_N);
  sp.slot_bytes = sp.slot_tiles + slot_records(form.few);
  sp.slot_words = form.few ? kFewWords : kSChunk * kMaxResidWords;
  // 6:8 phases may fall back to position order; their table is then needed as well.  A phase that stays without staged
  // activations has none to gather either.
  for (int round = 0;; ++round) {
    uint32_t o = 0;
    sp.use_meta6 = any6 ? 1 : 0;
    if (any6) o = kMeta6Bytes;
    o += SSmem::bytes;
    for (int k = 0; k < 3; ++k) {
      sp.pos_off[k] = 0;
      if (dense[k]) { o = up128(o); sp.pos_off[k] = o; o += kPosBytes; }
    }
    sp.pos_row = kPosCopies * 8;
    sp.ring_off = up128(o);
    o = sp.ring_off + kSWarps * kSDepth * sp.slot_bytes;
    sp.pdata_off = o;
    o += 32u * sp.part_floats * 4u;
    // the residual words' places and activations: sized for the most words the phase's layers can have
    sp.xs_off = o;
    uint32_t xs_max = 0, cols_max = 0;
    for (int p = 0; p < sp.nphase; ++p) {
      StackPhase& q = sp.ph[p];
      const unsigned long long need = 8ull * (unsigned long long)kMaxResidWords * (unsigned long long)(q.m / kBlock) * q.count;
      q.gather = form.gather > 0 && need <= kGatherMax && q.m <= 32768 ? 1 : 0;
      if (form.gather == 2 && q.gather && !bare_phase[p] && need * q.batch <= kGatherMax) q.gather = 2;
      if (q.gather == 2 && need * q.batch > xs_max) xs_max = (uint32_t)(need * q.batch);
      if (q.gather && need > cols_max) cols_max = (uint32_t)need;
    }
    sp.cols_off = up128(o + xs_max);
    o = up128(sp.cols_off + cols_max);
    sp.x_off = o;
    sp.x_bytes = 0;
    const long long room = (long long)kSmemLimit - (long long)o;
    if (room < 0) return false;
    bool again = false;
    for (int p = 0; p < sp.nphase; ++p) {
      StackPhase& q = sp.ph[p];
      const unsigned long long img = 4ull * q.batch * (unsigned long long)(q.m / kBlock) * kImgWordsPerBlock;
      const unsigned long long plain = (unsigned long long)q.batch * (2ull * (unsigned long long)q.m + kXPad);
      q.use_image = 0;
      unsigned long long need = 0;
      if (q.N == 6 && any6 && (long long)img <= room) { q.use_image = 1; need = img; }
      else {
        if (!dense[q.N - 4]) { dense[q.N - 4] = true; again = true; }
        // Staging costs a trip to L2 for all of x before the first tile, and pays where the CTA's row tiles read it again: with
        // several rows from 1.5 row tiles per CTA and row on (three 4:8 layers of 4096, 4 rows: 213 us against 226 with every
        // phase staged that fits; 7B gate and up, 4.6 row tiles per CTA, 2 rows: MLP 47.4 against 49.4 without).
        const bool stage = q.x2 || q.batch == 1 || 2 * q.tile_start[q.count] >= 3 * q.batch * ctas;
        if (stage && (long long)plain <= room) { q.use_image = 2; need = plain; }
        else if (q.gather == 2) { bare_phase[p] = true; again = true; }
      }
      if (need > sp.x_bytes) sp.x_bytes = (uint32_t)need;
    }
    if (!again || round > kMaxPhases) return true;
  }
}

// Builds the phases of steps [i0, ...) into `sp` (at most kMaxPhases), returns the index of the first step not taken.
static int build_phases(const stb_step* steps, int count, int i0, int G, StackParams& sp, size_t& sync_need, size_t& gpart_need) {
  sp.nphase = 0;
  sp.part_floats = 32; sp.max_share = 1; sp.gpart_slots = 0;
  uint32_t done = 0;
  long long maxR = 0;
  int i = i0;
  // first pass: phases and the largest batch (the partial slots are sized by it)
  while (i < count && sp.nphase < kMaxPhases) {
    StackPhase& q = sp.ph[sp.nphase];
    const stb_step& st = steps[i];
    int j = i + 1;
    while (j < count && j - i < kMaxFusedSteps && same_input(st, steps[j])) ++j;
    q.count = (uint8_t)(j - i);
    q.tile_start[0] = 0;
    q.f16_mask = 0;
    for (int k = 0; k < kMaxFusedSteps; ++k) { q.packed[k] = nullptr; q.y[k] = nullptr; q.ldy[k] = 0; q.n[k] = 0; q.tile_start[k + 1] = 0; }
    for (int k = i; k < j; ++k) {
      const stb_step& sk = steps[k];
      q.packed[k - i] = static_cast<const uint8_t*>(sk.packed);
      q.y[k - i] = sk.out; q.ldy[k - i] = (uint32_t)sk.ldout; q.n[k - i] = sk.n;
      if (sk.odt == STB_F16) q.f16_mask |= (uint8_t)(1u << (k - i));
      q.tile_start[k - i + 1] = q.tile_start[k - i] + (sk.n + kTileRows - 1) / kTileRows;
    }
    for (int k = q.count; k < kMaxFusedSteps; ++k) q.tile_start[k + 1] = q.tile_start[q.count];
    q.x = static_cast<const __half*>(st.in);
    q.x2 = st.input == STB_IN_SILU_MUL ? static_cast<const __half*>(st.in2) : nullptr;
    q.ldx = (uint32_t)st.ldin; q.m = st.m; q.N = (uint8_t)st.N; q.batch = (uint8_t)st.batch;
    q.use_image = 0; q.gather = 0; q.pad = 0;
    q.done_before = done;
    const long long R = q.tile_start[q.count];
    done += (uint32_t)R;
    if (R > maxR) maxR = R;
    if ((uint32_t)(32 * st.batch) > sp.part_floats) sp.part_floats = (uint32_t)(32 * st.batch);
    q.aligned = deal_aligned(R, G) ? 1 : 0;
    const uint32_t share = q.aligned ? 1u : max_share_of(R, st.m / kBlock, G);
    if (share > sp.max_share) sp.max_share = share;
    ++sp.nphase;
    i = j;
  }
  // second pass: where each phase takes its activations from.  6:8: the operand-order image if it fits, else, as for the
  // others, a plain copy or global memory; a formed input (silu(in) * in2) must be staged.  The image costs the 12 KB of the
  // metadata table for the whole launch, gathering and full slots their room: the first form that fits, has a use for the table and
  // stages what must be.  (Ranked by measurement: 6:8 in position order takes 160 clocks a tile against 100, few words per
  // slot 1 %, places instead of gathering 1 to 3 %.)
  static const SmemForm forms[] = {{true, 2, false}, {true, 2, true}, {true, 1, true}, {false, 2, false}, {false, 2, true}, {false, 1, true}, {true, 0, true}, {false, 0, true}};
  bool found = false;
  for (int k = 0; k < (int)(sizeof(forms) / sizeof(forms[0])) && !found; ++k) {
    found = plan_smem(sp, forms[k], G);
    for (int p = 0; p < sp.nphase; ++p)
      if (sp.ph[p].x2 && sp.ph[p].use_image == 0) found = false;
    if (found && forms[k].image) {                                 // no phase takes the image: without its table
      found = false;
      for (int p = 0; p < sp.nphase; ++p) found = found || sp.ph[p].use_image == 1;
    }
  }
  if (!found) return -1;                                           // a formed input does not fit shared memory
  // The kernel: gathered throughout (every phase is staged then) with 6:8 as an image, by places where not all are gathered or a 6:8 phase
  // is in position order, or by the word tables where one phase has neither; phases that are gathered stay so, but places and tables do
  // not go together.  (One kernel with all seven loops has 165 KB of code, the first of these 84: 9 % of its warps' time went to fetching
  // instructions.  6:8 in position order, gathered, had a place in the first until its loops were thinned out; such lists are faster
  // all the same: 7B MLP at two rows 51.7 -> 47.1 us, MLPs of 6144 x 18432 and 8192 x 20480 at one row 85.8 -> 75.7 and 121.7 -> 107.9.)
  bool listed = false, gathered = true;
  for (int p = 0; p < sp.nphase; ++p) {
    listed = listed || sp.ph[p].gather == 0;
    gathered = gathered && sp.ph[p].gather == 2 && (sp.ph[p].use_image == 1 || (sp.ph[p].use_image == 2 && sp.ph[p].N < 6));
  }
  sp.only5 = 1;
  for (int p = 0; p < sp.nphase; ++p)
    if (sp.ph[p].N != 5) sp.only5 = 0;
  sp.form = (int)(listed ? ResidForm::kListed : gathered ? ResidForm::kGathered : ResidForm::kPlaced);
  if (listed)
    for (int p = 0; p < sp.nphase; ++p)
      if (sp.ph[p].gather == 1) sp.ph[p].gather = 0;
  const size_t s_need = 8 * sizeof(uint32_t);
  if (sp.max_share > 1) sp.gpart_slots = (uint32_t)maxR * sp.max_share * sp.part_floats;
  const size_t g_need = (size_t)sp.gpart_slots * sizeof(uint2);
  if (s_need > sync_need) sync_need = s_need;
  if (g_need > gpart_need) gpart_need = g_need;
  return i;
}

// Gathered throughout, lists of 5:8 layers alone have a kernel of their own, with halves and bytes picked by dot products (13B block at one
// row 96.1 -> 87.4 us).  Beside other formats that form costs those more than it brings (6:8 4 to 5 %), and kernels for 4:8 or 6:8 alone
// were slower than the one for all three (235 against 231 us for four 7B layers at 4:8, 191 against 188 at 6:8).
static auto kernel_of(ResidForm form, bool only5) {
  if (form == ResidForm::kPlaced) return stack_kernel<ResidForm::kPlaced, false>;
  if (form == ResidForm::kListed) return stack_kernel<ResidForm::kListed, false>;
  return only5 ? stack_kernel<ResidForm::kGathered, true> : stack_kernel<ResidForm::kGathered, false>;
}

static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace stb

extern "C" int stb_layer_stack_resident_workspace(const stb_step* steps, int count, size_t* bytes) {
  if (!steps || count < 1 || !bytes) return STB_ERR_ARG;
  for (int i = 0; i < count; ++i) {
    const int rc = stb::check_step(steps[i]);
    if (rc != STB_OK) return rc;
  }
  int G = 0;
  int rc = stb::stack_sm_count(&G);
  if (rc != STB_OK) return rc;
  size_t sync_need = 0, gpart_need = 0;
  static thread_local stb::StackParams sp;
  int i = 0;
  while (i < count) {
    i = stb::build_phases(steps, count, i, G, sp, sync_need, gpart_need);
    if (i < 0) return STB_ERR_UNSUPPORTED;
  }
  *bytes = stb::align256(sync_need) + stb::align256(gpart_need);
  return STB_OK;
}

static int stack_resident_impl(const stb_step* steps, int count, void* ws, size_t ws_bytes, int* dev_status, void* stream,
                               bool selftest) {
  if (!steps || count < 1 || !ws) return STB_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(ws) & 255u) return STB_ERR_ARG;
  for (int i = 0; i < count; ++i) {
    const int rc = stb::check_step(steps[i]);
    if (rc != STB_OK) return rc;
  }
  int G = 0;
  int rc = stb::stack_sm_count(&G);
  if (rc != STB_OK) return rc;
  // the whole list must fit the workspace before anything is launched
  size_t sync_need = 0, gpart_need = 0;
  static thread_local stb::StackParams sp;
  {
    int i = 0;
    while (i < count) {
      i = stb::build_phases(steps, count, i, G, sp, sync_need, gpart_need);
      if (i < 0) return STB_ERR_UNSUPPORTED;
    }
  }
  const size_t sync_bytes = stb::align256(sync_need);
  if (ws_bytes < sync_bytes + stb::align256(gpart_need)) return STB_ERR_SIZE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  static bool attr_done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return STB_ERR_CUDA;
  if (!attr_done[dev]) {
    for (auto* kernel : {stb::kernel_of(stb::ResidForm::kGathered, false), stb::kernel_of(stb::ResidForm::kGathered, true),
                         stb::kernel_of(stb::ResidForm::kPlaced, false), stb::kernel_of(stb::ResidForm::kListed, false)})
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stb::kSmemLimit) != cudaSuccess) return STB_ERR_CUDA;
    attr_done[dev] = true;
  }
  int i = 0;
  while (i < count) {
    size_t a = 0, b = 0;
    i = stb::build_phases(steps, count, i, G, sp, a, b);
    if (i < 0) return STB_ERR_UNSUPPORTED;
    sp.sync = static_cast<uint32_t*>(ws);
    sp.gpart = reinterpret_cast<uint2*>(static_cast<uint8_t*>(ws) + sync_bytes);
    sp.dev_status = dev_status;
    sp.wait_limit = selftest ? stb::kSSelftestLimit : stb::kSWaitLimit;
    sp.copies_off = selftest ? 1 : 0;
    const uint32_t smem = sp.x_off + sp.x_bytes;
    if (smem > stb::kSmemLimit) return STB_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)G, 1, 1);
    cfg.blockDim = dim3((unsigned)stb::kSAllThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    // programmatic: the launch is prepared while the kernel before it drains, and its CTAs start as that one's leave (each
    // waits in its first instructions until all of it is complete)
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = 2;
    auto* kernel = stb::kernel_of((stb::ResidForm)sp.form, sp.only5 != 0);
    if (cudaLaunchKernelEx(&cfg, kernel, sp) != cudaSuccess) return STB_ERR_CUDA;
  }
  return STB_OK;
}

extern "C" int stb_layer_stack_resident(const stb_step* steps, int count, void* ws, size_t ws_bytes, int* dev_status,
                                        void* stream) {
  return stack_resident_impl(steps, count, ws, ws_bytes, dev_status, stream, false);
}

extern "C" int stb_layer_stack_resident_wait_selftest(const stb_step* steps, int count, void* ws, size_t ws_bytes,
                                                      int* dev_status, void* stream) {
  if (!dev_status) return STB_ERR_ARG;
  return stack_resident_impl(steps, count, ws, ws_bytes, dev_status, stream, true);
}

extern "C" int stb_layer_stack_resident_host(const stb_step* steps, int count, void* ws, size_t ws_bytes, const void* in_host,
                                             size_t in_bytes, void* out_host, size_t out_bytes, int* dev_status, void* stream) {
  if (!steps || count < 1 || !in_host || !out_host || !steps[0].in || !steps[count - 1].out) return STB_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemcpyAsync(const_cast<void*>(steps[0].in), in_host, in_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return STB_ERR_CUDA;
  const int rc = stb_layer_stack_resident(steps, count, ws, ws_bytes, dev_status, stream);
  if (rc != STB_OK) return rc;
  if (cudaMemcpyAsync(out_host, steps[count - 1].out, out_bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return STB_ERR_CUDA;
  return STB_OK;
}

extern "C" int stb_layer_stack_checksum(const stb_step* steps, int count, unsigned long long* sums, int* dev_status, void* stream) {
  if (!steps || count < 1 || !sums) return STB_ERR_ARG;
  for (int i = 0; i < count; ++i) {
    const int rc = stb::check_step(steps[i]);
    if (rc != STB_OK) return rc;
  }
  int G = 0;
  int rc = stb::stack_sm_count(&G);
  if (rc != STB_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  static bool attr_done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return STB_ERR_CUDA;
  if (!attr_done[dev]) {
    if (cudaFuncSetAttribute(stb::checksum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stb::kSmemLimit) != cudaSuccess) return STB_ERR_CUDA;
    attr_done[dev] = true;
  }
  if (cudaMemsetAsync(sums, 0, sizeof(unsigned long long) * (size_t)count, s) != cudaSuccess) return STB_ERR_CUDA;
  static thread_local stb::StackParams sp;
  int i = 0;
  while (i < count) {
    size_t a = 0, b = 0;
    const int first = i;
    i = stb::build_phases(steps, count, i, G, sp, a, b);
    if (i < 0) return STB_ERR_UNSUPPORTED;
    sp.sync = nullptr; sp.gpart = nullptr; sp.dev_status = dev_status;
    sp.wait_limit = stb::kSWaitLimit; sp.copies_off = 0;
    // the same shared-memory footprint as the arithmetic kernel would have for these steps
    const uint32_t smem = sp.x_off + sp.x_bytes;
    stb::checksum_kernel<<<(unsigned)G, stb::kSAllThreads, smem, s>>>(sp, sums, first);
    if (cudaGetLastError() != cudaSuccess) return STB_ERR_CUDA;
  }
  return STB_OK;
}
