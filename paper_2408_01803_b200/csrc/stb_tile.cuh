// One 32 x 128 tile of packed weights times up to 8 NB batch rows in registers (N = 4, 5, 6), and the residual words of the
// salient columns: the inner pieces of the GEMV kernels.  Activations come from shared memory (or, in position order, any
// memory): lane (g, t) reads those of batch rows g + 8 c; lanes beyond the batch are pointed at zeros.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "stb_decode.cuh"
#include "stb_layout.cuh"
#include "stb_ptx.cuh"

namespace stb {

static __device__ const Meta6Pairs g_meta6_pairs = make_meta6_pairs();

// The joint 6:8 metadata table, kept at shared-memory offset 0: two copies of every entry side by side, for even and for odd lanes, so
// that a pair field of a tile (16 times its entry's number) is the address of the entry.
constexpr uint32_t kMeta6Bytes = kMasks6 * kMasks6 * 16;
__device__ __forceinline__ void fill_meta6(uint8_t* smem, int thread, int threads) {
  for (int i = thread; i < (int)(kMasks6 * kMasks6); i += threads) {
    const uint2 e = *reinterpret_cast<const uint2*>(g_meta6_pairs.v[i]);
    reinterpret_cast<uint4*>(smem)[i] = make_uint4(e.x, e.y, e.x, e.y);
  }
}
constexpr uint32_t kImgWordsPerBlock = 96;    // 6:8 operand-order image: words per block and batch row
constexpr uint32_t kXPad = 64;                // bytes between the rows of the plain copy beyond 2 m: the eight lane groups' loads do not conflict
constexpr uint32_t kImgPad = 16;              // the same beyond the rows of the image
constexpr uint32_t kPosCopies = 16;           // copies of a position table, lane-minor: the look-ups of 16 lanes never conflict
constexpr uint32_t kPosBytes = kPosTableEntries * kPosCopies * 8;
constexpr uint32_t kZeroBytes = 384;          // zeros for the lanes beyond the batch: a block of the image

// where column c of block b stands in the staged activations of a batch row, in halves: in operand order (6:8), word
// ((t 2 + sl) 3 + i) 4 + u of a block = operand register u of chunk i of step sl of lane t, or plainly
__device__ __forceinline__ uint32_t image_word(uint32_t b, uint32_t group) {
  return b * kImgWordsPerBlock + (4u * (group & 1u) + ((group >> 2) & 1u)) * 12u + 2u * (group >> 3) + ((group >> 1) & 1u);
}
__device__ __forceinline__ uint32_t staged_index(bool image, uint32_t b, uint32_t c) {
  const uint32_t pr = (c >> 1) & 3u;
  return image ? 2u * (image_word(b, c >> 3) + (pr < 3u ? 4u * pr : 32u)) + (c & 1u) : b * (uint32_t)kBlock + c;
}
// eight activations (group `group` of block b) into the image of a batch row: lanes t = 2 (G & 1) + p read word i + p of
// group G as chunk i: words 0..2 for p = 0, 1..3 for p = 1
__device__ __forceinline__ void image_store(uint32_t* row, uint32_t b, uint32_t group, const uint32_t (&a)[4]) {
  uint32_t* d = row + image_word(b, group);
  d[0] = a[0]; d[4] = a[1]; d[8] = a[2];
  d[24] = a[1]; d[28] = a[2]; d[32] = a[3];
}

// product of two fp16 pairs given and returned as bit patterns
__device__ __forceinline__ uint32_t hmul2_bits(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// 6:8 through the sparse instruction: the weights stay in rank order and the instruction places them (stb_decode.cuh,
// meta6_nibble).  x: the lane's place in the operand-order image (t 96 bytes into the block's 384).
//
// What bounds it: shared memory, about 93 wavefronts a tile, and 96 clocks (its 149 integer instructions take 75).  With 16-byte table
// entries and the fields loaded one by one a tile took 130 wavefronts (82 of the look-ups, 32 of the fields) and as many clocks.
struct Tile6 { LaneTile<6> lt; uint32_t fld[8]; };
__device__ __forceinline__ void load_tile(const uint8_t* tile, int lane, Tile6& d) {
  load_lane_tile<6>(tile, lane, d.lt, true);
  const uint32_t copy = 8u * ((uint32_t)lane & 1u);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    d.fld[2 * k] = pick_half<false>(d.lt.mask[k], copy);
    d.fld[2 * k + 1] = pick_half<true>(d.lt.mask[k], copy);
  }
}
template <int NB>
__device__ __forceinline__ void tile_mul(const Tile6& d, const uint8_t* smem, const uint8_t* const (&x)[NB], float (&acc)[2][NB][4]) {
  FastRows<6> fr;
  fr.init(d.lt, d.lt.A, d.lt.B);
  // Metadata: fld[4 bb + tq] is the address of the table entry of slot 2 h + bb of lane tq of the quad, for the two rows whose
  // metadata this lane supplies.
  uint32_t E[2][3];
#pragma unroll
  for (int bb = 0; bb < 2; ++bb) {
    uint32_t en[4][2];
#pragma unroll
    for (int tq = 0; tq < 4; ++tq) {
      const uint2 v = *reinterpret_cast<const uint2*>(smem + d.fld[4 * bb + tq]);
      en[tq][0] = v.x; en[tq][1] = v.y;
    }
    meta6_pairs_words(en, E[bb]);
  }
  // the activations of the tile's six chunk positions, once for both halves of the rows (one batch group; of more, as they come)
  uint4 bxs[2][3];
  if (NB == 1) {
#pragma unroll
    for (int sl = 0; sl < 2; ++sl)
#pragma unroll
      for (int i = 0; i < 3; ++i) bxs[sl][i] = *reinterpret_cast<const uint4*>(x[0] + sl * 48 + 16 * i);
  }
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    uint32_t XLh[2][2], XHh[2][2];
#pragma unroll
    for (int jj = 0; jj < 2; ++jj)
#pragma unroll
      for (int sp = 0; sp < 2; ++sp) fr.high(2 * mt + jj, sp, XLh[jj][sp], XHh[jj][sp]);
#pragma unroll
    for (int sl = 0; sl < 2; ++sl) {
      uint32_t R[2][2][3];
#pragma unroll
      for (int jj = 0; jj < 2; ++jj)
#pragma unroll
        for (int h = 0; h < 2; ++h) fr.pairs(2 * mt + jj, 2 * h + sl, XLh[jj][h], XHh[jj][h], R[jj][h]);
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int c = 0; c < NB; ++c) {
          const uint4 bx = NB == 1 ? bxs[sl][i] : *reinterpret_cast<const uint4*>(x[c] + sl * 48 + 16 * i);
          if (mt == 0) mma_sp16832<0>(acc[0][c], R[0][0][i], R[1][0][i], R[0][1][i], R[1][1][i], bx.x, bx.y, bx.z, bx.w, E[sl][i]);
          else mma_sp16832<1>(acc[1][c], R[0][0][i], R[1][0][i], R[0][1][i], R[1][1][i], bx.x, bx.y, bx.z, bx.w, E[sl][i]);
        }
    }
  }
}

// Position order (N = 4, 5, 6): byte-permute decode into m16n8k16 operands.  The position selectors are looked up by keep-mask
// index; each of 16 lanes has a copy of the table in its own pair of banks (ptab: the lane's, prow bytes from entry to entry).
template <int N>
struct TileD { LaneTile<N> lt; uint2 P[16]; };
template <int N>
__device__ __forceinline__ void load_tile(const uint8_t* tile, int lane, const uint8_t* ptab, uint32_t prow, TileD<N>& d) {
  load_lane_tile<N>(tile, lane, d.lt);
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    const uint32_t idx = mask_pairs(N) ? keep_index_of(d.lt.mask, u >> 2, u & 3) : (uint32_t)tile[lane * 16 + u];
    d.P[u] = *reinterpret_cast<const uint2*>(ptab + idx * prow);
  }
}
// activations from global memory, coherent (they may have been written by the kernel that reads them)
__device__ __forceinline__ uint4 ldg_v4_coherent(const void* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
// x: the lane's activations of the block (8 t columns in), in shared memory (kStaged) or global
template <int N, bool kStaged, int NB, bool kDot = false>
__device__ __forceinline__ void tile_mul(const TileD<N>& d, const uint8_t* const (&x)[NB], float (&acc)[2][NB][4]) {
  FastRows<N, kDot> fr;
  fr.init(d.lt, d.lt.A, d.lt.B);
  uint32_t XL[4] = {0, 0, 0, 0}, XH[4] = {0, 0, 0, 0};
  if (N == 5) {
#pragma unroll
    for (int j = 0; j < 4; ++j) fr.high(j, 0, XL[j], XH[j]);
  }
  auto load_x = [&](int c, int s) {
    if (kStaged) return *reinterpret_cast<const uint4*>(x[c] + s * 64);
    uint4 v = make_uint4(0, 0, 0, 0);
    if (x[c]) v = ldg_v4_coherent(x[c] + s * 64);
    return v;
  };
  uint4 xf[4];
  if (NB == 1) {
#pragma unroll
    for (int s = 0; s < 4; ++s) xf[s] = load_x(0, s);
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    uint32_t f[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (N == 6 && (s & 1) == 0) fr.high(j, s >> 1, XL[j], XH[j]);
      fr.slot2(j, s, d.P[4 * j + s].x, d.P[4 * j + s].y, XL[j], XH[j], f[j]);
    }
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      const uint4 v = NB == 1 ? xf[s] : load_x(c, s);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        mma16816(acc[mt][c], f[2 * mt][0], f[2 * mt + 1][0], f[2 * mt][1], f[2 * mt + 1][1], v.x, v.y);
        mma16816(acc[mt][c], f[2 * mt][2], f[2 * mt + 1][2], f[2 * mt][3], f[2 * mt + 1][3], v.z, v.w);
      }
    }
  }
}

// Operand registers of the lane's four rows for four salient slots (a residual word `rw` of a block whose a_sal2 are `a2`): the
// two-bit codes pick the high byte of +1, 0 or -1 (one byte permute per row), two more spread them to fp16 pairs, and one
// fp16 multiply per register (not on the busy integer pipe) scales them by the row's a_sal2: exact, the factors are +-1 and 0.
__device__ __forceinline__ void resid_operands(uint32_t rw, uint2 a2, uint32_t (&fa)[4][2]) {
  const uint32_t code_lo = rw & 0x33333333u, code_hi = (rw >> 2) & 0x33333333u;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t codes = (j & 2) ? code_hi : code_lo;
    const uint32_t unit = prmt(0x00BC003Cu, 0u, (j & 1) ? (codes >> 16) : codes);          // high bytes of +1, 0, -1, 0 by code
    const uint32_t s2 = prmt((j & 2) ? a2.y : a2.x, 0u, (j & 1) ? 0x3232u : 0x1010u);     // (a_sal2, a_sal2) of row j
    fa[j][0] = hmul2_bits(prmt(unit, 0u, 0x1404u), s2);
    fa[j][1] = hmul2_bits(prmt(unit, 0u, 0x3424u), s2);
  }
}
constexpr uint32_t kNoTerms = 0x55555555u;     // a residual word without terms

}  // namespace stb
