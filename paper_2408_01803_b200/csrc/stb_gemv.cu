// stb_gemv: decode GEMV  y[t][i] = sum_j W^[i][j] x[t][j],  batch 1..64, fp32 accumulation.
// The memory-bound decoding stage of Appendix C.2: every packed byte is read once.
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "../../include/stb.h"
#include "stb_decode.cuh"
#include "stb_layout.cuh"
#include "stb_ptx.cuh"
#include "stb_tile.cuh"

namespace cg = cooperative_groups;

namespace stb {

__device__ const Meta6Table g_meta6 = make_meta6_table();

// ------------------------------------------------------------------------------------------
// Tensor-core GEMV of small layers, of chains of small layers and of 17 to 64 batch rows, N = 4, 5, 6, batch <= 8 NB (NB = 1, 2, 4, 8).
//
// Grid: one thread-block cluster of `ksplit` CTAs per row tile (32 rows); CTA k of the cluster
// takes the k-th slice of the 128-column blocks and its warps take contiguous runs of that
// slice.  Each warp streams its tiles from HBM into a private ring in shared memory with 1-D
// bulk copies (kChunk tiles per copy, kDepth copies in flight), reads a tile into registers,
// decodes it into fp16 operand registers (stb_decode.cuh) and multiplies on the tensor cores,
// fp32 accumulators in registers for the whole run:
//   N = 4, 5, and N = 6 beyond 8 batch rows: position-order decode, m16n8k16 (A = 16 rows x 16
//     columns of W^, B = the activations of 8 batch rows read through L1);
//   N = 6 up to 8 batch rows: the weights stay in rank order and the 2:4 sparse instruction
//     (m16n8k32) places them: every pair of kept weights is a 2-of-4 selection from a window of
//     four columns, three overlapping windows per group of 8 (stb_decode.cuh, meta6_nibble);
//     the activations are read three halves wide, for up to two batch rows from a copy of the
//     CTA's slice that is laid out in operand order in shared memory once per CTA.
// The residual term of the salient columns goes through the dense instruction with the salient
// slots of 16 / SPB blocks as its K dimension, after the weight stream.  Partial sums: warps
// through shared memory, CTAs of the cluster through distributed shared memory, both in a fixed
// order.
constexpr int kDepth = 2;     // ring slots per warp
constexpr int kChunk = 2;     // tiles per bulk copy (consecutive blocks of a row tile are contiguous)
constexpr long long kWaitLimit = 2000000000ll;     // about a second of SM clocks
constexpr long long kSelftestWaitLimit = 100000ll;  // the wait self-test gives up after about 50 microseconds

struct GemvSmem {
  uint32_t bars, ring, part, ximg, total;           // byte offsets
  uint32_t tile_stride;
};
// N = 6, up to two batch rows: the CTA's slice of the activations is kept in shared memory in the order the lanes
// consume it: per block and batch row 96 words, word ((t * 2 + sl) * 3 + i) * 4 + u = operand register u of chunk i
// of step sl of lane t (two fp16 each).
constexpr uint32_t kImgMaxBytes = 20 * 1024;
__host__ __device__ inline uint32_t gemv_image_bytes(int N, int NB, int batch, int bpp) {
  const uint32_t bytes = (uint32_t)batch * (uint32_t)bpp * kImgWordsPerBlock * 4u;
  return (N == 6 && NB == 1 && batch <= 2 && bytes <= kImgMaxBytes) ? bytes : 0u;
}
__host__ __device__ inline GemvSmem gemv_smem(int N, int warps, int ksplit, int NB, uint32_t image_bytes) {
  GemvSmem s;
  s.bars = kPosTableEntries * 8;                     // the position table comes first
  s.ring = (s.bars + (uint32_t)(warps * kDepth * 8) + 127u) & ~127u;
  s.tile_stride = (kChunk * tile_bytes(N) + 127u) & ~127u;      // one ring slot = one chunk of tiles
  // the ring is reused for the per-warp partial sums (warps x 32 rows x 8 NB floats) after the main loop
  const uint32_t ring_bytes = (uint32_t)(warps * kDepth) * s.tile_stride, red_bytes = (uint32_t)warps * 32u * 8u * (uint32_t)NB * 4u;
  s.part = s.ring + (ring_bytes > red_bytes ? ring_bytes : red_bytes);
  s.ximg = s.part + (uint32_t)ksplit * 32u * 8u * (uint32_t)NB * 4u;
  s.total = s.ximg + image_bytes;
  return s;
}

// Up to kMaxFused layers that read the same activations (q / k / v, gate / up) run as one grid:
// row tiles [tile_start[i], tile_start[i + 1]) of the grid belong to layer i.
constexpr int kMaxFused = 4;
struct GemvLayers {
  const uint8_t* packed[kMaxFused];
  void* y[kMaxFused];
  size_t ldy[kMaxFused];
  int n[kMaxFused];
  int y_f16[kMaxFused];
  int tile_start[kMaxFused + 1];
  int count;
};

// At most 128 threads per CTA, four CTAs per SM for up to 16 batch rows (a bound of five CTAs, 96
// registers, was measured slower: the spills cost more than the extra resident CTA brings).
constexpr int kGemvMaxThreads = 128;
constexpr int kMaxDevices = 64;
constexpr int kMmaPerSm = 4;
template <int N, int NB, bool kChained, bool kDot>
__global__ void __launch_bounds__(kGemvMaxThreads, NB <= 2 ? kMmaPerSm : 1)
gemv_mma_kernel(const __grid_constant__ GemvLayers layers, int m, const __half* __restrict__ x, int batch,
                size_t ldx, int* dev_status, int lg_ksplit, int bpp, long long wait_limit, int copies_off) {
  // A programmatic dependent of whatever ran before it: prepared while that drains.  Only within a chain (stb_layer_stack,
  // whose packed layers nobody writes meanwhile) may anything be read before that is complete.
  if constexpr (!kChained) { grid_dependency_wait(); grid_launch_dependents(); }
  extern __shared__ __align__(128) uint8_t smem[];
  int li = 0, rt_all = (int)(blockIdx.x >> lg_ksplit);
#pragma unroll
  for (int i = 1; i < kMaxFused; ++i)
    if (i < layers.count && rt_all >= layers.tile_start[i]) li = i;
  const uint8_t* __restrict__ packed = layers.packed[li];
  if constexpr (!kChained) packed = after_dependency_wait(packed);
  void* __restrict__ y = layers.y[li];
  const size_t ldy = layers.ldy[li];
  const int n = layers.n[li], y_f16 = layers.y_f16[li];
  const Header* hdr = reinterpret_cast<const Header*>(packed);
  // every CTA of a cluster takes the same branch here (the header is the same for all)
  if (!header_matches(hdr, n, m, N)) {
    if constexpr (kChained) grid_dependency_wait();     // (what follows on the stream waits for this grid alone)
    if (threadIdx.x == 0 && dev_status) *dev_status = STB_ERR_CORRUPT;
    return;
  }
  const int nblk = m / kBlock;
  const int ksplit = 1 << lg_ksplit;
  // A CTA may write into the shared memory of another CTA of its cluster only once that CTA runs: every CTA
  // arrives here, and waits for the others just before its first remote store (behind the whole weight stream).
  if (ksplit > 1) cluster_arrive();
  const int warps = (int)(blockDim.x >> 5);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int kpart = (int)(blockIdx.x & (unsigned)(ksplit - 1)), rt = rt_all - layers.tile_start[li];
  const int b0 = kpart * bpp, b1 = min(nblk, b0 + bpp);
  const int nbp = max(b1 - b0, 0);
  const BlockInfo* binfo = reinterpret_cast<const BlockInfo*>(packed + sizeof(Header));
  constexpr uint32_t tbytes = tile_bytes(N);
  const uint8_t* rtbase = packed + hdr->tiles_offset + (size_t)rt * hdr->rt_stride;
  const uint8_t* resid_rt = packed + hdr->tiles_offset + hdr->rt_stride * (size_t)hdr->ntile +
                            (size_t)rt * resid_rt_bytes(nblk, hdr->nrw);
  const uint32_t image_bytes = gemv_image_bytes(N, NB, batch, bpp);
  const GemvSmem L = gemv_smem(N, warps, ksplit, NB, image_bytes);

  const uint2* ptab = reinterpret_cast<const uint2*>(smem);
  uint8_t* ring = smem + L.ring + (size_t)warp * kDepth * L.tile_stride;
  const uint32_t bar0 = smem_u32(smem + L.bars) + (uint32_t)warp * kDepth * 8u;

  // this warp's run of blocks
  const int per = (nbp + warps - 1) / warps;
  const int wb0 = b0 + warp * per, wb1 = min(b1, wb0 + per);
  const int cnt = max(wb1 - wb0, 0);

  // Start the weight stream before anything else.  The packed layer is never written by a GEMV,
  // so under a programmatic dependent launch this may run while the previous layer still computes.
  if (lane == 0) {
    for (int i = 0; i < kDepth; ++i) mbar_init(bar0 + 8u * i, 1);
    fence_async_smem();
    for (int i = 0; i < kDepth && i * kChunk < cnt; ++i) {
      const uint32_t bytes = (uint32_t)min(kChunk, cnt - i * kChunk) * tbytes;
      mbar_expect_tx(bar0 + 8u * i, bytes);
      // copies_off (the wait self-test): the barrier is armed but nothing will ever complete it
      if (!copies_off) bulk_g2s(smem_u32(ring + (size_t)i * L.tile_stride), rtbase + (size_t)(wb0 + i * kChunk) * tbytes, bytes, bar0 + 8u * i);
    }
  }
  if (N == 6 && NB == 1) {   // metadata by keep-mask index (256 bytes: an index byte of the tile cannot point past it)
    for (int i = threadIdx.x; i < kMeta6Entries; i += blockDim.x) reinterpret_cast<uint32_t*>(smem)[i] = g_meta6.v[i];
  } else {
    for (int i = threadIdx.x; i < kPosTableEntries; i += blockDim.x) reinterpret_cast<uint2*>(smem)[i] = g_pos_table.v[N][i];
  }

  // Everything below reads the activations (the previous layer's output) or writes y: wait for the
  // previous grid of the stream to have completed (no-op without a programmatic launch), then let
  // the next grid start its own weight stream.
  if constexpr (kChained) { grid_dependency_wait(); grid_launch_dependents(); }
  x = after_dependency_wait(x);
  const uint32_t* ximg = reinterpret_cast<const uint32_t*>(smem + L.ximg);
  const uint32_t img_row_words = (uint32_t)bpp * kImgWordsPerBlock;
  if (N == 6 && NB == 1 && image_bytes != 0u) {
    // one item = the 8 activations of one group of one block of one batch row: a 16-byte load, six 4-byte stores
    // (lanes t = 2 (G & 1) + p read word i + p of group G as chunk i: words 0..2 for p = 0, words 1..3 for p = 1)
    uint32_t* img = reinterpret_cast<uint32_t*>(smem + L.ximg);
    const int items = batch * nbp * 16;
    for (int base = 0; base < items; base += 4 * (int)blockDim.x) {
      uint4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int it = base + k * (int)blockDim.x + (int)threadIdx.x;
        v[k] = make_uint4(0, 0, 0, 0);
        if (it < items) {
          const int r = it / (nbp * 16), q = it - r * nbp * 16;
          v[k] = ldg_nc_v4(x + (size_t)r * ldx + (size_t)b0 * kBlock + (size_t)q * 8);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int it = base + k * (int)blockDim.x + (int)threadIdx.x;
        if (it < items) {
          const int r = it / (nbp * 16), q = it - r * nbp * 16, blk = q >> 4, G = q & 15;
          uint32_t* d = img + (uint32_t)r * img_row_words + (uint32_t)blk * kImgWordsPerBlock +
                        (uint32_t)((4 * (G & 1) + ((G >> 2) & 1)) * 12 + 2 * (G >> 3) + ((G >> 1) & 1));
          d[0] = v[k].x; d[4] = v[k].y; d[8] = v[k].z;
          d[24] = v[k].y; d[28] = v[k].z; d[32] = v[k].w;
        }
      }
    }
  }
  __syncthreads();

  float acc[2][NB][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < NB; ++c)
#pragma unroll
      for (int d = 0; d < 4; ++d) acc[a][c][d] = 0.0f;

  bool failed = false;
  const __half* xrow[NB];
#pragma unroll
  for (int c = 0; c < NB; ++c) xrow[c] = g + 8 * c < batch ? x + (size_t)(g + 8 * c) * ldx + t * 8 : nullptr;
  // N = 6: the lane's activation pairs of a chunk start at column 8 (t >> 1) + 2 (t & 1) of a 32-column step
  const __half* xsp[NB];
#pragma unroll
  for (int c = 0; c < NB; ++c) xsp[c] = xrow[c] ? xrow[c] - t * 8 + 8 * (t >> 1) + 2 * (t & 1) : nullptr;

  // Residual term of the salient columns: the residual words of this warp's run of blocks are numbered
  // consecutively (stb_layout.cuh); one tensor-core step takes 16 salient slots = four words, lane t the t-th.
  // A word's table entry names its block and its four salient columns.
  const ResidWord* rwt = reinterpret_cast<const ResidWord*>(packed + hdr->rwtab_offset);
  uint32_t rw0 = 0, rw1 = 0;
  if (cnt > 0) { rw0 = __ldg(&binfo[wb0].rw_off); rw1 = __ldg(&binfo[wb1 - 1].rw_off) + __ldg(&binfo[wb1 - 1].nrw); }
  struct ResidWords { uint32_t rw, cols, block; uint2 a2; };
  auto fetch = [&](uint32_t step, ResidWords& w) {
    w.rw = 0x55555555u; w.cols = 0u; w.block = (uint32_t)wb0; w.a2 = make_uint2(0u, 0u);
    const uint32_t wi = rw0 + 4u * step + (uint32_t)t;
    if (wi < rw1) {
      const uint2 e = __ldg(reinterpret_cast<const uint2*>(rwt + wi));
      w.block = e.x >> 3; w.cols = e.y;
      // the word's block record in the residual stream: a_sal2 of the lane's four rows, then the block's words
      const uint8_t* rec = resid_rt + resid_block_off((int)w.block, wi - (e.x & 7u));
      w.a2 = __ldg(reinterpret_cast<const uint2*>(rec + resid_a2_off(g, 0)));
      w.rw = __ldg(reinterpret_cast<const uint32_t*>(rec + resid_code_off(e.x & 7u, g)));
    }
  };
  ResidWords rfirst;
  fetch(0u, rfirst);      // in flight during the main loop

  for (int it = 0; it < cnt; ++it) {
    const int ch = it / kChunk, kin = it - ch * kChunk;     // chunk and tile inside the chunk
    const int slot = ch % kDepth;
    const uint32_t bar = bar0 + 8u * slot;
    const int b = wb0 + it;
    // all lanes poll; the verdict is made warp-uniform so that nobody is left at a __syncwarp
    if (kin == 0 && !__all_sync(0xFFFFFFFFu, mbar_wait(bar, (uint32_t)(ch / kDepth) & 1u, wait_limit))) { failed = true; break; }
    const uint8_t* tile = ring + (size_t)slot * L.tile_stride + (size_t)kin * tbytes;
    // release of the ring slot: once the whole chunk is in registers or consumed, refill it
    auto refill = [&]() {
      if (kin == kChunk - 1 || it == cnt - 1) {
        __syncwarp();
        const int nxt = (ch + kDepth) * kChunk;      // first tile of the chunk that reuses this slot
        if (lane == 0 && nxt < cnt) {
          const uint32_t bytes = (uint32_t)min(kChunk, cnt - nxt) * tbytes;
          fence_async_smem();
          mbar_expect_tx(bar, bytes);
          bulk_g2s(smem_u32(ring + (size_t)slot * L.tile_stride), rtbase + (size_t)(wb0 + nxt) * tbytes, bytes, bar);
        }
      }
    };
    if constexpr (N == 6 && NB == 1) {
      // Rank order through the sparse instruction.  This lane's metadata: rows g + 16 (t >> 1) and + 8, the chunks
      // of operand registers 2 h, 2 h + 1 (h = t & 1) of the quad's four lanes, i.e. their slots 2 h and 2 h + 1.
      LaneTile<N> lt;
      load_lane_tile<N>(tile, lane, lt, true);
      refill();
      FastRows<N> fr;
      fr.init(lt, lt.A, lt.B);
      uint32_t E[2][3];
#pragma unroll
      for (int bb = 0; bb < 2; ++bb) {
        uint32_t en[2][4];
#pragma unroll
        for (int tq = 0; tq < 4; ++tq) {
          // the pair field of the two rows whose metadata this lane supplies
          const uint32_t f = (lt.mask[2 * bb + (tq >> 1)] >> (16 * (tq & 1))) & 0xFFFFu;
          en[0][tq] = reinterpret_cast<const uint32_t*>(smem)[pair_field_index(f, 0)];
          en[1][tq] = reinterpret_cast<const uint32_t*>(smem)[pair_field_index(f, 1)];
        }
        meta6_words(en, E[bb]);
      }
      if (image_bytes != 0u) {
        // activations from the CTA's image in shared memory: two rows of the lane at a time (fewer live registers;
        // the 16-byte operand loads are cheap enough to be issued once per row pair)
        const uint32_t* xi0 = ximg + (uint32_t)g * img_row_words + (uint32_t)(b - b0) * kImgWordsPerBlock + (uint32_t)(t * 24);
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
            for (int i = 0; i < 3; ++i) {
              uint4 bx = make_uint4(0, 0, 0, 0);
              if (g < batch) bx = *reinterpret_cast<const uint4*>(xi0 + sl * 12 + 4 * i);
              if (mt == 0) mma_sp16832<0>(acc[0][0], R[0][0][i], R[1][0][i], R[0][1][i], R[1][1][i], bx.x, bx.y, bx.z, bx.w, E[sl][i]);
              else mma_sp16832<1>(acc[1][0], R[0][0][i], R[1][0][i], R[0][1][i], R[1][1][i], bx.x, bx.y, bx.z, bx.w, E[sl][i]);
            }
          }
        }
      } else {
      uint32_t XL6[4][2], XH6[4][2];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int sp = 0; sp < 2; ++sp) fr.high(j, sp, XL6[j][sp], XH6[j][sp]);
#pragma unroll
      for (int sl = 0; sl < 2; ++sl) {
        uint32_t R[4][2][3];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h) fr.pairs(j, 2 * h + sl, XL6[j][h], XH6[j][h], R[j][h]);
        // Activations of chunk i of a step: columns 2 i + 2 (t & 1) + {0, 1} of the group's eight.  Up to two batch
        // rows whose slice is too long for the image: one 4-byte load per register (few lanes are active); more
        // batch rows: the group's 16 bytes through L1, then a select.
        if (batch <= 2) {
#pragma unroll
          for (int i = 0; i < 3; ++i) {
#pragma unroll
            for (int c = 0; c < NB; ++c) {
              uint32_t bx[4] = {0, 0, 0, 0};
              if (xsp[c]) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                  bx[u] = ldg_nc_u32(xsp[c] + (size_t)b * kBlock + 64 * (u >> 1) + 16 * (u & 1) + 32 * sl + 2 * i);
              }
              mma_sp16832<0>(acc[0][c], R[0][0][i], R[1][0][i], R[0][1][i], R[1][1][i], bx[0], bx[1], bx[2], bx[3], E[sl][i]);
              mma_sp16832<1>(acc[1][c], R[2][0][i], R[3][0][i], R[2][1][i], R[3][1][i], bx[0], bx[1], bx[2], bx[3], E[sl][i]);
            }
          }
        } else {
#pragma unroll
          for (int c = 0; c < NB; ++c) {
            uint4 xw[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              xw[u] = make_uint4(0, 0, 0, 0);
              if (xsp[c]) xw[u] = ldg_nc_v4(xsp[c] - 2 * (t & 1) + (size_t)b * kBlock + 64 * (u >> 1) + 16 * (u & 1) + 32 * sl);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              uint32_t bx[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const uint32_t w0 = i == 0 ? xw[u].x : (i == 1 ? xw[u].y : xw[u].z), w1 = i == 0 ? xw[u].y : (i == 1 ? xw[u].z : xw[u].w);
                bx[u] = (t & 1) ? w1 : w0;
              }
              mma_sp16832<0>(acc[0][c], R[0][0][i], R[1][0][i], R[0][1][i], R[1][1][i], bx[0], bx[1], bx[2], bx[3], E[sl][i]);
              mma_sp16832<1>(acc[1][c], R[2][0][i], R[3][0][i], R[2][1][i], R[3][1][i], bx[0], bx[1], bx[2], bx[3], E[sl][i]);
            }
          }
        }
      }
      }
    } else {
    LaneTile<N> lt;
    load_lane_tile<N>(tile, lane, lt);
    refill();
    FastRows<N, kDot> fr;
    fr.init(lt, lt.A, lt.B);
    uint32_t XL[4] = {0, 0, 0, 0}, XH[4] = {0, 0, 0, 0};
    if (N == 5) {
#pragma unroll
      for (int j = 0; j < 4; ++j) fr.high(j, 0, XL[j], XH[j]);
    }
    // all table lookups (and, for up to 16 batch rows, activation loads) of the tile are issued up front
    uint2 P[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) P[u] = ptab[keep_index_of(lt.mask, u >> 2, u & 3)];
    constexpr int XS = NB <= 2 ? 4 : 1;          // activation fragments held at a time: all four steps, or one
    uint4 xf[XS][NB];
    if (NB <= 2) {
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < NB; ++c) {
          xf[s % XS][c] = make_uint4(0, 0, 0, 0);
          if (xrow[c]) xf[s % XS][c] = ldg_nc_v4(xrow[c] + (size_t)b * kBlock + s * 32);
        }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (NB > 2) {
#pragma unroll
        for (int c = 0; c < NB; ++c) {
          xf[0][c] = make_uint4(0, 0, 0, 0);
          if (xrow[c]) xf[0][c] = ldg_nc_v4(xrow[c] + (size_t)b * kBlock + s * 32);
        }
      }
      uint32_t f[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (N == 6 && (s & 1) == 0) fr.high(j, s >> 1, XL[j], XH[j]);
        fr.slot2(j, s, P[4 * j + s].x, P[4 * j + s].y, XL[j], XH[j], f[j]);
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int c = 0; c < NB; ++c) {
          const uint4 xv = xf[s % XS][c];
          mma16816(acc[mt][c], f[2 * mt][0], f[2 * mt + 1][0], f[2 * mt][1], f[2 * mt + 1][1], xv.x, xv.y);
          mma16816(acc[mt][c], f[2 * mt][2], f[2 * mt + 1][2], f[2 * mt][3], f[2 * mt + 1][3], xv.z, xv.w);
        }
    }
    }

  }

  // Residual term of the salient columns, after the main stream (its registers and loads stay out of the main
  // loop): per four residual words one tensor-core step with their 16 salient slots as K.  The lane's word (its
  // codes, the a_sal2 of its rows in the word's block, the salient columns) is fetched one step ahead.
  if (rw1 > rw0 && !failed) {
    const uint32_t nstep = (rw1 - rw0 + 3u) >> 2;
    ResidWords cur = rfirst, nxt;
#pragma unroll 1
    for (uint32_t gi = 0; gi < nstep; ++gi) {
      fetch(gi + 1u, nxt);
      const size_t xoff = (size_t)cur.block * kBlock;
      uint32_t fa[4][2];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t h = (((j & 2) ? cur.a2.y : cur.a2.x) >> (16 * (j & 1))) & 0xFFFFu;
        const uint32_t L2 = prmt(h, 0u, 0x4040u);                 // (lo, 0, lo, 0)
        const uint32_t H2 = prmt(h, h ^ 0x8000u, 0x2521u);        // (hi, 0, hi ^ 0x80, 0)
        const uint32_t sel = resid_selector(cur.rw, j);
        const uint32_t lo4 = prmt(L2, L2, sel), hi4 = prmt(H2, H2, sel);
        fa[j][0] = prmt(lo4, hi4, 0x5140u);
        fa[j][1] = prmt(lo4, hi4, 0x7362u);
      }
      // the four salient columns behind this lane's residual word
      const uint32_t cw = cur.cols;
#pragma unroll
      for (int c = 0; c < NB; ++c) {
        uint2 xr = make_uint2(0, 0);
        if (xrow[c]) {
          const unsigned short* xq = reinterpret_cast<const unsigned short*>(xrow[c] - t * 8 + xoff);
          xr.x = (uint32_t)__ldg(xq + (cw & 0xFFu)) | ((uint32_t)__ldg(xq + ((cw >> 8) & 0xFFu)) << 16);
          xr.y = (uint32_t)__ldg(xq + ((cw >> 16) & 0xFFu)) | ((uint32_t)__ldg(xq + (cw >> 24)) << 16);
        }
        mma16816(acc[0][c], fa[0][0], fa[1][0], fa[0][1], fa[1][1], xr.x, xr.y);
        mma16816(acc[1][c], fa[2][0], fa[3][0], fa[2][1], fa[3][1], xr.x, xr.y);
      }
      cur = nxt;
    }
  }

  if (failed) {
    // give the copies still in flight time to land before the shared memory is given up
    const long long t0 = clock64();
    while (clock64() - t0 < 200000) {}
    if (lane == 0 && dev_status) *dev_status = STB_ERR_TIMEOUT;
  }
  __syncthreads();     // every warp is done with its ring: reuse it for the partial sums

  // red[warp][row 0..31][batch 0..8NB-1]
  constexpr int BW = 8 * NB;
  float* red = reinterpret_cast<float*>(smem + L.ring);
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      float* r0 = red + ((size_t)warp * 32 + (g + 16 * mt)) * BW + 8 * c + 2 * t;
      float* r1 = r0 + 8 * BW;
      r0[0] = acc[mt][c][0]; r0[1] = acc[mt][c][1];
      r1[0] = acc[mt][c][2]; r1[1] = acc[mt][c][3];
    }
  __syncthreads();
  float* part = reinterpret_cast<float*>(smem + L.part);       // [ksplit][32][BW], used on cluster rank 0
  if (ksplit > 1) cluster_wait();
  for (int i = threadIdx.x; i < 32 * BW; i += blockDim.x) {
    float sacc = 0.0f;
    for (int w = 0; w < warps; ++w) sacc += red[(size_t)w * 32 * BW + i];
    if (ksplit == 1) {
      const int row = rt * kTileRows + i / BW, bt = i % BW;
      if (row < n && bt < batch) {
        if (y_f16) static_cast<__half*>(y)[(size_t)bt * ldy + row] = __float2half_rn(sacc);
        else static_cast<float*>(y)[(size_t)bt * ldy + row] = sacc;
      }
    } else {
      float* dst = cg::this_cluster().map_shared_rank(part, 0);
      dst[(size_t)kpart * 32 * BW + i] = sacc;
    }
  }
  if (ksplit == 1) return;
  cg::this_cluster().sync();
  if (kpart == 0) {
    for (int i = threadIdx.x; i < 32 * BW; i += blockDim.x) {
      const int row = rt * kTileRows + i / BW, bt = i % BW;
      if (row < n && bt < batch) {
        float tsum = 0.0f;
        for (int k = 0; k < ksplit; ++k) tsum += part[(size_t)k * 32 * BW + i];
        if (y_f16) static_cast<__half*>(y)[(size_t)bt * ldy + row] = __float2half_rn(tsum);
        else static_cast<float*>(y)[(size_t)bt * ldy + row] = tsum;
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// The GEMV of larger layers, N = 4, 5, 6, up to 16 batch rows (8 NB).
//
// Grid: Q thread-block clusters of `ksplit` CTAs, one CTA of 16 warps per SM.  CTA k of a cluster takes the k-th slice of the
// 128-column blocks of ALL row tiles of the cluster, so that its slice of the activations is staged in shared memory once and
// used for every row tile; its 32 x 128 tiles, in (row tile, block) order, are dealt to the warps as equal contiguous runs.
// gemv_plan takes the split (1, 2, 4, 6 or 8) that is done first.
// Each warp streams its tiles and their residual records from HBM into a private ring (two slots of one or two tiles) with 1-D
// bulk copies, and decodes and multiplies them on the tensor cores, fp32 accumulators in registers (stb_tile.cuh):
//   N = 4, 5        position-order decode, m16n8k16, activations from a plain copy in shared memory
//   N = 6           rank order through the 2:4 sparse instruction, activations from an image in operand order (position order
//                   where the image does not fit)
// The residual term of a chunk of tiles goes through the dense instruction with 16 salient slots as K; the columns behind the
// residual words of the slice are turned into places in the staged activations once per CTA.
// Sums: a warp writes the rows it begins to shared memory and the piece it continues beside it; the CTA adds them in order, the
// cluster adds its CTAs' sums through distributed shared memory, in order.
// What bounds it: the decode with its residual words (about 180 / 190 / 155 clocks per tile and SM at N = 4 / 5 / 6, the integer ALU),
// and a chain of latencies before and after it (header - first tile - staging - sums - cluster: about 10,000 clocks, which is why small
// layers stay with gemv_mma_kernel; launch_mma_b has the rule).
// Against that kernel, three layers in turn, microseconds: 28672 x 8192 4:8 batch 1 56.3 -> 46.5, 5120 x 13824 5:8 batch 8 38.3 -> 22.7,
// 4096 x 11008 6:8 batch 1 17.1 -> 13.1, 11008 x 4096 6:8 batch 16 28.9 -> 18.1, 4096 x 4096 4:8 batch 1 8.9 -> 8.7; 16 rows:
// 5120 x 13824 4:8 34.6 -> 29.0, 5:8 41.4 -> 30.7, 6:8 43.7 -> 28.4; 1500 x 5120 6:8 13 rows 12.8 -> 10.7.
constexpr int kGWarps = 16, kGThreads = kGWarps * 32;
__device__ __forceinline__ int layer_of(const GemvLayers& layers, int rt) {
  int li = 0;
#pragma unroll
  for (int i = 1; i < kMaxFused; ++i)
    if (i < layers.count && rt >= layers.tile_start[i]) li = i;
  return li;
}

// Split and shared memory of a launch (byte offsets; the 6:8 metadata table or the position table comes first).
struct GemvPlan {
  int ksplit, clusters, bs, chunk, image;             // bs: blocks per slice; chunk: tiles per ring slot
  uint32_t zero, bars, masks, head, part, roff, wtab, ring, slot, x, xpitch, total;
};
constexpr uint32_t kGemvSmem = 227 * 1024;
static inline uint32_t gemv_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }
static bool gemv_layout(GemvPlan& p, int N, int batch, int rows, int layers, int image, int chunk) {
  p.image = image; p.chunk = chunk;
  uint32_t o = image ? kMeta6Bytes : kPosBytes;
  p.zero = gemv_up(o, 128) + (image ? kImgPad : kXPad); o = gemv_up(p.zero + kZeroBytes, 16);
  p.bars = o; o += kGWarps * 2 * 8;
  p.masks = o; o += gemv_up((uint32_t)rows * 4u, 16);                         // per row tile: the warps that continue it
  p.head = gemv_up(o, 16); o = p.head + (uint32_t)(kGWarps * 32 * batch) * 4u;                       // sums of the row tile a warp continues
  const unsigned long long part = 128ull * (unsigned long long)rows * batch;   // sums of the CTA's row tiles
  const unsigned long long roff = 4ull * (unsigned long long)layers * (p.bs + 1), wtab = 64ull * (unsigned long long)layers * p.bs;
  p.xpitch = image ? (uint32_t)p.bs * kImgWordsPerBlock * 4u + kImgPad : (uint32_t)p.bs * 256u + kXPad;
  if (part + roff + wtab + (unsigned long long)p.xpitch * batch > kGemvSmem || p.bs * 256 > 65535) return false;
  p.part = gemv_up(o, 16); o = p.part + (uint32_t)part;
  p.roff = o; o += (uint32_t)roff;                                             // residual words before every block of the slice, per layer
  p.wtab = gemv_up(o, 16); o = p.wtab + (uint32_t)wtab;                        // places of the four activations of every residual word
  p.slot = gemv_up((uint32_t)chunk * (tile_bytes(N) + kResidA2Bytes + kMaxResidWords * kResidWordBytes), 128);
  p.ring = gemv_up(o, 128); o = p.ring + kGWarps * 2 * p.slot;
  p.x = o; o += p.xpitch * (uint32_t)batch;
  p.total = o;
  return o <= kGemvSmem;
}

// The tiles of a warp as its copies see them.
struct GemvWalk {
  int left, row, blk;             // tiles left; row tile (of the CTA) and block (of the slice) of the next one
  const uint8_t* tiles;           // of the row tile's slice
  const uint8_t* recs;            // of the row tile, at the slice's first a_sal2
  const uint32_t* roff;           // of the row tile's layer
};

template <int N, int NB, bool kImage>
__global__ void __launch_bounds__(kGThreads, 1)
gemv_stream_kernel(const __grid_constant__ GemvLayers layers, const __grid_constant__ GemvPlan P, int m, const __half* x, int batch, size_t ldx,
                   int* dev_status, long long wait_limit, int copies_off, int chained) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3, tid = threadIdx.x;
  const int nblk = m / kBlock, ksplit = P.ksplit;
  const int kpart = (int)(blockIdx.x % (unsigned)ksplit), cl = (int)(blockIdx.x / (unsigned)ksplit);
  const int b0 = kpart * P.bs, nbp = max(min(nblk - b0, P.bs), 0);              // this CTA's slice of the blocks
  const int R = layers.tile_start[layers.count];
  const int R0 = (int)((long long)R * cl / P.clusters), rows = (int)((long long)R * (cl + 1) / P.clusters) - R0;   // and the cluster's row tiles
  constexpr uint32_t tb = tile_bytes(N);
  // What needs no other memory comes first: the launch is a programmatic dependent of whatever ran before it on the stream.
  // Within a chain (stb_layer_stack, whose packed layers nobody writes meanwhile) the weights may be read before that is done too.
  if (kImage) {
    fill_meta6(smem, tid, kGThreads);
  } else {
    for (int i = tid; i < kPosTableEntries * (int)kPosCopies; i += kGThreads) reinterpret_cast<uint2*>(smem)[i] = g_pos_table.v[N][i / (int)kPosCopies];
  }
  if (tid < (int)kZeroBytes / 4) reinterpret_cast<uint32_t*>(smem + P.zero)[tid] = 0u;
  for (int i = tid; i < rows; i += kGThreads) reinterpret_cast<uint32_t*>(smem + P.masks)[i] = 0u;
  if (!chained) { grid_dependency_wait(); grid_launch_dependents(); }
  // a buffer packed for another shape must not be read as this one (every CTA of the grid comes to the same verdict)
  bool fits = true;
  uint32_t nrw[kMaxFused];
#pragma unroll
  for (int i = 0; i < kMaxFused; ++i)
    if (i < layers.count) {
      const Header* h = reinterpret_cast<const Header*>(layers.packed[i]);
      fits = fits && header_matches(h, layers.n[i], m, N);
      nrw[i] = h->nrw;
    }
  if (!fits) {
    if (chained) grid_dependency_wait();                // (what follows on the stream waits for this grid alone)
    if (tid == 0 && dev_status) *dev_status = STB_ERR_CORRUPT;
    return;
  }
  const uint32_t bar0 = smem_u32(smem + P.bars) + 16u * (uint32_t)warp;
  const uint32_t ring = smem_u32(smem + P.ring) + (uint32_t)warp * 2u * P.slot;
  const uint8_t* ringp = smem + P.ring + (size_t)warp * 2u * P.slot;
  uint32_t* roff_all = reinterpret_cast<uint32_t*>(smem + P.roff);
  // this warp's run of tiles
  const int T = rows * nbp, lo = (int)((long long)T * warp / kGWarps), hi = (int)((long long)T * (warp + 1) / kGWarps);

  GemvWalk w;
  auto enter = [&](int row) {
    const int rt = R0 + row, li = layer_of(layers, rt), rl = rt - layers.tile_start[li];
    const int ntile = layers.tile_start[li + 1] - layers.tile_start[li];
    const uint8_t* base = layers.packed[li] + tiles_offset(nblk);
    uint32_t words = 0;
#pragma unroll
    for (int i = 0; i < kMaxFused; ++i)
      if (i == li) words = nrw[i];
    w.tiles = base + ((size_t)rl * nblk + b0) * tb;
    w.recs = base + (size_t)tb * nblk * ntile + (size_t)rl * resid_rt_bytes(nblk, words) + (size_t)kResidA2Bytes * b0;
    w.roff = roff_all + li * (P.bs + 1);
  };
  auto chunk_of = [&](int left, int blk) { return min(min(P.chunk, left), nbp - blk); };
  w.left = hi - lo; w.row = nbp > 0 ? lo / nbp : 0; w.blk = lo - w.row * nbp;
  // The first chunk's tiles at once and its records as soon as its blocks' word counts are here, which the warp asks for itself
  // (everything later goes by the table below).  A copy may land before its bytes are announced: the barrier's phase cannot
  // end before that, its one arrival.
  if (w.left > 0) {
    enter(w.row);
    const int c = chunk_of(w.left, w.blk);
    if (lane == 0) {
      mbar_init(bar0, 1);
      mbar_init(bar0 + 8u, 1);
      fence_async_smem();
      if (!copies_off) bulk_g2s(ring, w.tiles + (size_t)w.blk * tb, (uint32_t)c * tb, bar0);
      const BlockInfo* bi = reinterpret_cast<const BlockInfo*>(layers.packed[layer_of(layers, R0 + w.row)] + sizeof(Header)) + b0 + w.blk;
      const uint32_t w0 = bi[0].rw_off, nw = bi[0].nrw + (c > 1 ? bi[1].nrw : 0u), rec_b = (uint32_t)c * kResidA2Bytes + nw * kResidWordBytes;
      mbar_expect_tx(bar0, (uint32_t)c * tb + rec_b);
      if (!copies_off) bulk_g2s(ring + (uint32_t)P.chunk * tb, w.recs + (size_t)kResidA2Bytes * w.blk + (size_t)kResidWordBytes * w0, rec_b, bar0);
    }
  }
  for (int i = tid; i < layers.count * (nbp + 1); i += kGThreads) {
    const int li = i / (nbp + 1), k = i - li * (nbp + 1);
    const BlockInfo* bi = reinterpret_cast<const BlockInfo*>(layers.packed[li] + sizeof(Header));
    uint32_t v = 0;
#pragma unroll
    for (int q = 0; q < kMaxFused; ++q)
      if (q == li) v = nrw[q];
    if (b0 + k < nblk) v = bi[b0 + k].rw_off;
    roff_all[li * (P.bs + 1) + k] = v;
  }
  __syncthreads();

  auto advance = [&](int c) {
    w.left -= c; w.blk += c;
    if (w.blk == nbp && w.left > 0) { w.blk = 0; ++w.row; enter(w.row); }
  };
  // next chunk of the walk into ring slot `slot`
  auto issue = [&](uint32_t slot) {
    if (w.left <= 0) return;
    const int c = chunk_of(w.left, w.blk);
    if (lane == 0) {
      const uint32_t w0 = w.roff[w.blk], nw = w.roff[w.blk + c] - w0;
      const uint32_t tile_b = (uint32_t)c * tb, rec_b = (uint32_t)c * kResidA2Bytes + nw * kResidWordBytes, bar = bar0 + 8u * slot, dst = ring + slot * P.slot;
      fence_async_smem();
      mbar_expect_tx(bar, tile_b + rec_b);
      // copies off (the wait self-test): the barrier is armed but nothing will ever complete it
      if (!copies_off) {
        bulk_g2s(dst, w.tiles + (size_t)w.blk * tb, tile_b, bar);
        bulk_g2s(dst + (uint32_t)P.chunk * tb, w.recs + (size_t)kResidA2Bytes * w.blk + (size_t)kResidWordBytes * w0, rec_b, bar);
      }
    }
    advance(c);
  };
  if (w.left > 0) advance(chunk_of(w.left, w.blk));
  issue(1u);
  // where the activations behind the slice's residual words will stand
  uint2* wtab = reinterpret_cast<uint2*>(smem + P.wtab);
  for (int li = 0; li < layers.count; ++li) {
    const uint32_t w0 = roff_all[li * (P.bs + 1)], cnt = roff_all[li * (P.bs + 1) + nbp] - w0;
    const uint2* rwt = reinterpret_cast<const uint2*>(layers.packed[li] + rwtab_offset(nblk)) + w0;
    for (uint32_t i = tid; i < cnt; i += kGThreads) {
      const uint2 e = rwt[i];
      const uint32_t b = (e.x >> 3) - (uint32_t)b0;
      uint32_t at[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) at[k] = staged_index(kImage, b, (e.y >> (8 * k)) & 0xFFu);
      wtab[(size_t)li * kMaxResidWords * P.bs + i] = make_uint2(at[0] | (at[1] << 16), at[2] | (at[3] << 16));
    }
  }

  // Everything below reads the activations (the previous layer's output) or writes y: wait for the
  // previous grid of the stream to have completed, then let the next grid start its own prologue.
  if (chained) { grid_dependency_wait(); grid_launch_dependents(); }
  {
    const int per_row = nbp * 16, items = batch * per_row;
#pragma unroll 1
    for (int first = tid; first < items; first += 4 * kGThreads) {
      uint4 v[4];
      uint32_t at[4];                       // batch row and group, for the stores
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int it = first + k * kGThreads, r = batch == 1 ? 0 : it / per_row, q = it - r * per_row;
        at[k] = ((uint32_t)r << 16) | (uint32_t)q;
        if (it < items) v[k] = ldg_v4_coherent(x + (size_t)r * ldx + (size_t)b0 * kBlock + (size_t)q * 8);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (first + k * kGThreads < items) {
          const uint32_t a[4] = {v[k].x, v[k].y, v[k].z, v[k].w}, q = at[k] & 0xFFFFu;
          uint8_t* row = smem + P.x + (at[k] >> 16) * P.xpitch;
          if (kImage) image_store(reinterpret_cast<uint32_t*>(row), q >> 4, q & 15u, a);
          else *reinterpret_cast<uint4*>(row + 16 * q) = v[k];
        }
    }
  }
  __syncthreads();

  bool failed = false;
  float* part = reinterpret_cast<float*>(smem + P.part);
  {
    const uint8_t* xrow[NB];
    uint32_t live[NB];
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      live[c] = g + 8 * c < batch ? 0xFFFFFFFFu : 0u;
      xrow[c] = live[c] ? smem + P.x + (uint32_t)(g + 8 * c) * P.xpitch : smem + P.zero;
    }
    const uint32_t xstep = kImage ? kImgWordsPerBlock * 4u : 2u * kBlock, xlane = (uint32_t)t * (kImage ? 96u : 16u);
    const uint8_t* ptab = smem + (uint32_t)(lane & (kPosCopies - 1)) * 8u;
    // When a slot is filled again: once its last tile is in registers, in position order after the products (in between, the loads of the
    // activations stay behind it: 28672 x 8192, one row, 49.3 -> 46.3 us at 4:8, 52.5 -> 49.4 at 5:8).
    constexpr bool kBack = !kImage;
    uint32_t slot = 0, parity = 0;
    int left = hi - lo, row = nbp > 0 ? lo / nbp : 0, blk = lo - row * nbp;
    while (left > 0 && !failed) {
      const int first = blk, end = min(nbp, blk + left);
      const int li = layer_of(layers, R0 + row);
      const uint32_t* roff = roff_all + li * (P.bs + 1);
      const uint2* words = wtab + (size_t)li * kMaxResidWords * P.bs;
      const uint32_t wfirst = roff[0];
      float acc[2][NB][4];
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < NB; ++c)
#pragma unroll
          for (int d = 0; d < 4; ++d) acc[a][c][d] = 0.0f;
      while (blk < end) {
        const int cnt = chunk_of(left, blk);
        const uint32_t bar = bar0 + 8u * slot;
        // all lanes poll; the verdict is made warp-uniform
        if (!__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity)) && !__all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, wait_limit))) { failed = true; break; }
        const uint8_t* tile = ringp + slot * P.slot;
        const uint8_t* rec = tile + (uint32_t)P.chunk * tb;
        const uint32_t w0 = roff[blk], na = roff[blk + 1] - w0, nw = roff[blk + cnt] - w0;
        // residual words of the chunk, four (16 salient slots) per tensor-core step, lane t the t-th; before its tiles, whose sum is larger
        // (with them after the tiles 4:8 lost 0.8 % and 5:8 2.2 % of their accuracy against float64)
        auto residual = [&] {
#pragma unroll 1
          for (uint32_t kk = (uint32_t)t; kk < nw + (uint32_t)t; kk += 4u) {
            const uint32_t k = min(kk, nw - 1u);
            const bool second = k >= na;
            uint32_t rw = *reinterpret_cast<const uint32_t*>(rec + k * kResidWordBytes + (second ? 2u * kResidA2Bytes : kResidA2Bytes) + 4 * g), fa[4][2];
            const uint2 a2 = *reinterpret_cast<const uint2*>(rec + (second ? kResidA2Bytes + na * kResidWordBytes : 0u) + 8 * g);
            if (kk >= nw) rw = kNoTerms;
            resid_operands(rw, a2, fa);
            const uint2 at = words[w0 - wfirst + k];
#pragma unroll
            for (int c = 0; c < NB; ++c) {
              const uint16_t* xr = reinterpret_cast<const uint16_t*>(xrow[c]);
              const uint32_t p0 = at.x & live[c], p1 = at.y & live[c];
              const uint32_t q0 = (uint32_t)xr[p0 & 0xFFFFu] | ((uint32_t)xr[p0 >> 16] << 16), q1 = (uint32_t)xr[p1 & 0xFFFFu] | ((uint32_t)xr[p1 >> 16] << 16);
              mma16816(acc[0][c], fa[0][0], fa[1][0], fa[0][1], fa[1][1], q0, q1);
              mma16816(acc[1][c], fa[2][0], fa[3][0], fa[2][1], fa[3][1], q0, q1);
            }
          }
        };
        residual();
#pragma unroll 1
        for (int k = 0; k < cnt; ++k) {
          const uint8_t* xp[NB];
#pragma unroll
          for (int c = 0; c < NB; ++c) xp[c] = xrow[c] + xlane + (live[c] & ((uint32_t)(blk + k) * xstep));
          if constexpr (kImage) {
            Tile6 d;
            load_tile(tile, lane, d);
            if (!kBack && k == cnt - 1) { __syncwarp(); issue(slot); }
            tile_mul<NB>(d, smem, xp, acc);
          } else {
            TileD<N> d;
            load_tile<N>(tile, lane, ptab, kPosCopies * 8u, d);
            if (!kBack && k == cnt - 1) { __syncwarp(); issue(slot); }
            tile_mul<N, true, NB, N == 5>(d, xp, acc);
          }
          tile += tb;
        }
        if (kBack) { __syncwarp(); issue(slot); }
        parity ^= slot;
        slot ^= 1u;
        blk += cnt; left -= cnt;
      }
      if (failed) break;
      // the row tile's sums (or the piece of it): beside the CTA's if another warp began it
      float* dst = first == 0 ? part + (size_t)row * 32 * batch : reinterpret_cast<float*>(smem + P.head) + (size_t)warp * 32 * batch;
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int c = 0; c < NB; ++c)
#pragma unroll
          for (int d = 0; d < 4; ++d) {
            const int r = g + 16 * mt + 8 * (d >> 1), bc = 8 * c + 2 * t + (d & 1);
            if (bc < batch) dst[r * batch + bc] = acc[mt][c][d];
          }
      if (first != 0 && lane == 0) atomicOr(reinterpret_cast<uint32_t*>(smem + P.masks) + row, 1u << warp);
      ++row; blk = 0;
    }
  }
  if (failed) {
    // give the copies still in flight time to land before the shared memory is given up
    const long long t0 = clock64();
    while (clock64() - t0 < 200000) {}
    if (lane == 0 && dev_status) *dev_status = STB_ERR_TIMEOUT;
  }
  __syncthreads();

  // Sums of the CTA: what the row tile's first warp has, then the pieces of the warps after it; four values of one row tile per
  // thread and step (values of a row tile: [row][batch row]).
  const int per4 = 8 * batch, E4 = rows * per4;
  const uint32_t* masks = reinterpret_cast<const uint32_t*>(smem + P.masks);
  const float4* head4 = reinterpret_cast<const float4*>(smem + P.head);
  float4* part4 = reinterpret_cast<float4*>(part);
  auto add = [](float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; };
  auto store = [&](int row, int v4, const float4& s) {
    const int rt = R0 + row, li = layer_of(layers, rt), first = (rt - layers.tile_start[li]) * kTileRows, n = layers.n[li];
    const size_t ldy = layers.ldy[li];
    void* y = layers.y[li];
    const bool f16 = layers.y_f16[li] != 0;
    const float w[4] = {s.x, s.y, s.z, s.w};
    int r = batch == 1 ? 4 * v4 : 4 * v4 / batch, bc = 4 * v4 - r * batch;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (first + r < n) {
        if (f16) static_cast<__half*>(y)[(size_t)bc * ldy + first + r] = __float2half_rn(w[k]);
        else static_cast<float*>(y)[(size_t)bc * ldy + first + r] = w[k];
      }
      if (++bc == batch) { bc = 0; ++r; }
    }
  };
#pragma unroll 1
  for (int e = tid; e < E4; e += kGThreads) {
    const int row = e / per4, v = e - row * per4;
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (nbp > 0) s = part4[e];
#pragma unroll 1
    for (uint32_t mm = masks[row]; mm != 0u; mm &= mm - 1u) add(s, head4[(__ffs(mm) - 1) * per4 + v]);      // in warp order
    if (ksplit == 1) store(row, v, s);
    else part4[e] = s;
  }
  if (ksplit == 1) return;
  // the cluster's CTAs, in order: CTA k finishes the k-th share of the values
  cluster_arrive();
  cluster_wait();
  const int e0 = (int)((long long)E4 * kpart / ksplit), e1 = (int)((long long)E4 * (kpart + 1) / ksplit);
#pragma unroll 1
  for (int e = e0 + tid; e < e1; e += kGThreads) {
    float4 v[8], s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < ksplit) v[k] = *cg::this_cluster().map_shared_rank(part4 + e, k);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < ksplit) add(s, v[k]);
    const int row = e / per4;
    store(row, e - row * per4, s);
  }
  cluster_arrive();        // nobody leaves while its sums are being read
  cluster_wait();
}

// ------------------------------------------------------------------------------------------
// Launch shape: ksplit CTAs per row tile and warps per CTA.  A warp should get a run of several
// tiles (its ring then streams while it decodes) and the grid should have at least two CTAs per
// SM while leaving room on the SM for the next layer's CTAs, which start their own weight
// stream early (programmatic dependent launch).
static void gemv_shape(int n, int m, int& ksplit, int& warps) {
  const int ntile = (n + kTileRows - 1) / kTileRows, nblk = m / kBlock;
  warps = 4;
  int ks = 1;
  while (ks < 8 && ntile * ks < 296 && nblk / (2 * ks * warps) >= 4) ks *= 2;
  ksplit = ks;
}

// kChained: nobody writes the packed layer while the kernel before it on the stream runs.  That is another GEMV of the same
// stb_layer_stack call (`early`: a programmatic dependent of it), or the kernel is launched in stream order.
// kDot: 5:8 picks halves and bytes by dot products (stb_decode.cuh).
template <int N, int NB, bool kChained, bool kDot = N == 5 && NB == 1>
static cudaError_t launch_mma(const GemvLayers& layers, int m, const __half* x, int batch, size_t ldx,
                              int* dev_status, cudaStream_t s, bool early, bool wait_selftest) {
  const int ntile = layers.tile_start[layers.count], nblk = m / kBlock;
  int ksplit, warps;
  gemv_shape(ntile * kTileRows, m, ksplit, warps);
  const int bpp = (nblk + ksplit - 1) / ksplit;
  const GemvSmem L = gemv_smem(N, warps, ksplit, NB, gemv_image_bytes(N, NB, batch, bpp));
  // the shared-memory limit of a kernel is a per-device setting
  static bool attr_done[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices || !attr_done[dev]) {
    e = cudaFuncSetAttribute(gemv_mma_kernel<N, NB, kChained, kDot>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kMaxDevices) attr_done[dev] = true;
  }
  if (L.total > 200 * 1024) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ntile * ksplit), 1, 1);
  cfg.blockDim = dim3((unsigned)(warps * 32), 1, 1);
  cfg.dynamicSmemBytes = L.total;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (ksplit > 1) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = (unsigned)ksplit; at[na].val.clusterDim.y = 1; at[na].val.clusterDim.z = 1;
    ++na;
  }
  if (early) {
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = at; cfg.numAttrs = na;
  int lg = 0;
  while ((1 << lg) < ksplit) ++lg;
  const long long limit = wait_selftest ? kSelftestWaitLimit : kWaitLimit;
  return cudaLaunchKernelEx(&cfg, gemv_mma_kernel<N, NB, kChained, kDot>, layers, m, x, batch, ldx, dev_status, lg, bpp, limit, wait_selftest ? 1 : 0);
}

// Whether a launch is one full wave of CTAs and a small second one with few blocks each: the CTAs of the second have an SM almost to
// themselves, and the longer latency of the dot products outweighs what they spare the full wave (5:8, 22000 x 768, four rows, 9.97 us
// with products, 9.75 with shifts, 19500 x 512 7.94 and 7.77; from 12 blocks or one more CTA per SM on products are level or faster:
// 19500 x 2048 14.2 and 14.6, 25000 x 1408 12.9 and 13.3, 17500 x 768 6.5 and 6.7).
static bool short_second_wave(int ctas, int bpp) {
  int dev = 0, sms = 0;
  if (bpp > 11 || cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
  return ctas > kMmaPerSm * sms && ctas <= (kMmaPerSm + 1) * sms;
}

template <int NB>
static cudaError_t launch_mma_n(int N, const GemvLayers& layers, int m, const __half* x, int batch, size_t ldx,
                                int* dev_status, cudaStream_t s, bool chained, bool selftest) {
  if constexpr (NB == 1) {            // (such a launch has no split)
    if (N == 5 && !chained && short_second_wave(layers.tile_start[layers.count], m / kBlock))
      return launch_mma<5, 1, false, false>(layers, m, x, batch, ldx, dev_status, s, true, selftest);
  }
  // On its own a launch is a programmatic dependent as well, which hides 2 to 4 us of launch but keeps the compiler from reading
  // the weights through the read-only path: with more than eight rows 12% of the time (28672 x 8192 5:8, 16 rows: 99 against
  // 88 us), so that from 16384 tiles on such a launch keeps the stream's order.
  const bool plain = !chained && NB > 1 && (long long)layers.tile_start[layers.count] * (m / kBlock) >= 16384;
  auto* f = N == 4 ? (chained || plain ? launch_mma<4, NB, true> : launch_mma<4, NB, false>)
          : N == 5 ? (chained || plain ? launch_mma<5, NB, true> : launch_mma<5, NB, false>)
                   : (chained || plain ? launch_mma<6, NB, true> : launch_mma<6, NB, false>);
  return f(layers, m, x, batch, ldx, dev_status, s, !plain, selftest);
}

// Clocks that a call of gemv_mma_kernel takes (batch <= 16), from its launch shape: terms fitted to 528 measured calls of all
// three formats, 32 to 32768 tiles, 1 to 16 rows (6% mean error), times the factor for which the choice between the two kernels by
// their costs was best (over those calls 0.9% slower on average than always the faster one).  gemv_stream_kernel has become 3 to 19 %
// faster since, most at 6:8: over 119 calls drawn from the same range the choice is 1.8 % behind the faster kernel (gemv_mma_kernel
// throughout: 18 %; at 6:8 gemv_stream_kernel throughout: 0.2 %).
static double gemv_mma_cost(int N, int row_tiles, int nblk, int batch, int sms) {
  int ksplit, warps;
  gemv_shape(row_tiles * kTileRows, nblk * kBlock, ksplit, warps);
  const int ctas = row_tiles * ksplit, bpp = (nblk + ksplit - 1) / ksplit, per_sm = (ctas + sms - 1) / sms, chain = (bpp + warps - 1) / warps;
  const double clk = (N == 4 ? 100.0 : N == 5 ? 140.0 : 130.0) + (batch > 8 ? 70.0 : 0.0);
  const double cost = 4100.0 + clk * per_sm * bpp + 1000.0 * chain + 250.0 * chain * (per_sm + (double)ctas / sms) + (ksplit > 1 ? 3600.0 : 0.0) +
                      6.0 * batch * bpp + (batch > 8 ? 800.0 : 0.0) + (N == 6 && batch > 2 ? 2100.0 : 0.0);
  return cost * (N == 6 ? 1.1 : 0.95);
}

// Launch of gemv_stream_kernel, batch <= 16: the split of the blocks (1, 2, 4, 6 or 8 slices) that is done first, and the wider ring where
// it fits (clusters of 3, 5 and 7 CTAs measured up to 3 us behind their share of the tiles: an SM of a pair stays idle).  The clocks of a split: the fullest CTA's tiles at their issue rate, its longest warp's tiles at their latency (more
// with a second group of eight rows or single-tile slots), a cluster's sums, the staging, the epilogue (terms fitted to 1900 measured
// calls of the same range, 3% mean error, before the kernel's tiles took 3 to 19 % less).  Returns false where no split fits shared memory.
static bool gemv_plan(int N, int row_tiles, int nblk, int batch, int layers, const int (&most)[9], GemvPlan& best, double& best_cost) {
  bool found = false;
  for (int C = 1; C <= 8; ++C) {
    if (most[C] < 1 || (C > 1 && (C % 2 || nblk < 2 * C))) continue;
    GemvPlan p = {};
    p.ksplit = C;
    p.clusters = row_tiles < most[C] ? row_tiles : most[C];
    p.bs = (nblk + C - 1) / C;
    const int rows = (row_tiles + p.clusters - 1) / p.clusters;
    bool ok = false;
    for (int form = 0; form < 4 && !ok; ++form) {
      const int image = form < 2;
      if (image && N != 6) continue;
      ok = gemv_layout(p, N, batch, rows, layers, image, form % 2 == 0 ? 2 : 1);
    }
    if (!ok) continue;
    const int tiles = rows * p.bs, chain = (tiles + kGWarps - 1) / kGWarps;
    const double clk = N == 5 ? 112.0 : N == 6 && !p.image ? 160.0 : 100.0;
    const double cost = 10000.0 + clk * tiles + ((batch > 8 ? 2400.0 : 1700.0) + (p.chunk == 1 ? 600.0 : 0.0)) * chain +
                        (C > 1 ? 3500.0 - 130.0 * C : 0.0) + 11.0 * batch * p.bs + 23.0 * batch * rows;
    if (!found || cost < best_cost) { best = p; best_cost = cost; found = true; }
  }
  return found;
}

template <int N, int NB, bool kImage>
static cudaError_t launch_stream(const GemvLayers& layers, const GemvPlan& plan, int m, const __half* x, int batch, size_t ldx, int* dev_status, cudaStream_t s,
                                 bool chained, bool wait_selftest, int dev) {
  static bool attr_done[kMaxDevices] = {};          // the shared-memory limit of a kernel is a per-device setting
  if (dev < 0 || dev >= kMaxDevices || !attr_done[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(gemv_stream_kernel<N, NB, kImage>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemvSmem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kMaxDevices) attr_done[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(plan.clusters * plan.ksplit), 1, 1);
  cfg.blockDim = dim3((unsigned)kGThreads, 1, 1);
  cfg.dynamicSmemBytes = plan.total;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (plan.ksplit > 1) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = (unsigned)plan.ksplit; at[na].val.clusterDim.y = 1; at[na].val.clusterDim.z = 1;
    ++na;
  }
  at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[na].val.programmaticStreamSerializationAllowed = 1;
  ++na;
  cfg.attrs = at; cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, gemv_stream_kernel<N, NB, kImage>, layers, plan, m, x, batch, ldx, dev_status,
                            wait_selftest ? kSelftestWaitLimit : kWaitLimit, wait_selftest ? 1 : 0, chained ? 1 : 0);
}

// Clusters of 1 to 8 CTAs (one CTA per SM) that a device holds at once, by their size.  Asked for once per device; several host
// threads may come here at the same time, and all must get the whole answer (the choice of kernel, and with it the order of
// the sums, depends on it).
static cudaError_t gemv_clusters(int dev, int (&most)[9]) {
  static int cached[kMaxDevices][9] = {};
  static std::atomic<bool> filled[kMaxDevices] = {};
  static std::mutex filling;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::unique_lock<std::mutex> lock(filling, std::defer_lock);
  if (!filled[dev].load(std::memory_order_acquire)) lock.lock();
  if (lock.owns_lock() && !filled[dev].load(std::memory_order_relaxed)) {
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(gemv_stream_kernel<4, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemvSmem);
    if (e != cudaSuccess) return e;
    int v[9] = {0, sms};
    for (int C = 2; C <= 8; ++C) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(sms / C * C), 1, 1);
      cfg.blockDim = dim3((unsigned)kGThreads, 1, 1);
      cfg.dynamicSmemBytes = kGemvSmem;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)C; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.attrs = at; cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&v[C], gemv_stream_kernel<4, 1, false>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); v[C] = 0; }
    }
    for (int C = 1; C <= 8; ++C) cached[dev][C] = v[C];
    filled[dev].store(true, std::memory_order_release);
  }
  for (int C = 0; C <= 8; ++C) most[C] = cached[dev][C];
  return cudaSuccess;
}

// Which of the two kernels a launch of up to 16 rows takes.
enum class GemvForm {
  cheapest,     // a launch on its own: the one with the lower cost
  stream,       // gemv_stream_kernel from 1024 tiles on
  mma           // gemv_mma_kernel
};
constexpr long long kStreamTiles = 1024;

// The launches of a chain (stb_layer_stack) mostly take the same kernel: gemv_mma_kernel's CTAs start beside the launch before
// them, those of gemv_stream_kernel, which fill an SM, do not, and each change from one to the other cost about 4 us.  By the mean
// tiles of the chain's launches, measured per decoder layer (QKV, O, gate/up, down; microseconds, gemv_mma_kernel against
// gemv_stream_kernel before its tiles took 3 to 19 % less): mean 832 20.6 / 26.8 (4:8, 2 rows), 25.8 / 33.7 (6:8, 8 rows); 2884 35.5 / 39.6 (4:8), 48.8 / 42.3 (6:8, 8
// rows), 51.0 / 51.4 (6:8, 16 rows); 4266 47.1 / 49.2 (5:8, 8 rows), 59.7 / 53.5 (6:8, 16 rows); 7498 57.4 / 53.8 (4:8, 2 rows),
// 61.8 / 58.1 (5:8, 2 rows), 70.6 / 53.1 (6:8, 4 rows); 12352 84.7 / 66.6 (6:8, 2 rows); 19360 115.4 / 100.7 (5:8, 4 rows).
// `fits`: every launch has a split; `wide`: at least one has double slots (5:8 with a second group of rows needs them: 79.8 / 80.9
// at mean 7498, 16 rows, without, 76.7 / 73.5 at 12 rows with them).
static GemvForm chain_form(int N, int batch, long long mean, bool fits, bool wide) {
  if (!fits || (N == 5 && batch > 8 && !wide)) return GemvForm::mma;
  return mean >= (N != 6 ? 6000 : batch <= 8 ? 2500 : 4000) ? GemvForm::stream : GemvForm::mma;
}

// batch -> number of 8-row batch groups (1, 2, 4 or 8)
static cudaError_t launch_mma_b(int batch, int N, const GemvLayers& layers, int m, const __half* x, size_t ldx,
                                int* dev_status, cudaStream_t s, bool chained, bool selftest, GemvForm form) {
  const int R = layers.tile_start[layers.count], nblk = m / kBlock;
  if (batch <= 16 && form != GemvForm::mma && (form == GemvForm::cheapest || (long long)R * nblk >= kStreamTiles)) {
    int dev = 0, most[9];
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = gemv_clusters(dev, most);
    if (e != cudaSuccess) return e;
    GemvPlan plan;
    double cost = 0.0;
    if (gemv_plan(N, R, nblk, batch, layers.count, most, plan, cost) && (form == GemvForm::stream || cost < gemv_mma_cost(N, R, nblk, batch, most[1]))) {
      if (batch > 8) {
        if (N == 4) return launch_stream<4, 2, false>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
        if (N == 5) return launch_stream<5, 2, false>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
        if (plan.image) return launch_stream<6, 2, true>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
        return launch_stream<6, 2, false>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
      }
      if (N == 4) return launch_stream<4, 1, false>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
      if (N == 5) return launch_stream<5, 1, false>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
      if (plan.image) return launch_stream<6, 1, true>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
      return launch_stream<6, 1, false>(layers, plan, m, x, batch, ldx, dev_status, s, chained, selftest, dev);
    }
  }
  if (batch <= 8) return launch_mma_n<1>(N, layers, m, x, batch, ldx, dev_status, s, chained, selftest);
  if (batch <= 16) return launch_mma_n<2>(N, layers, m, x, batch, ldx, dev_status, s, chained, selftest);
  if (batch <= 32) return launch_mma_n<4>(N, layers, m, x, batch, ldx, dev_status, s, chained, selftest);
  return launch_mma_n<8>(N, layers, m, x, batch, ldx, dev_status, s, chained, selftest);
}

// ------------------------------------------------------------------------------------------
// General kernel: N = 1, 2, 3, 7, 8, batch <= BT.  One CTA per row tile (32 rows), 8 warps split
// the blocks, lane = (g, t); plain position-order decode and fp32 multiply-adds, x read
// through L1.  The four lanes that share a row combine with shuffles, the 8 warps through
// shared memory in a fixed order, so the result is deterministic.
template <int N, int BT>
__global__ void __launch_bounds__(256)
gemv_general_kernel(const uint8_t* __restrict__ packed, int n, int m, const __half* __restrict__ x,
                    int batch, size_t ldx, void* __restrict__ y, int y_f16, size_t ldy, int* dev_status) {
  const Header* hdr = reinterpret_cast<const Header*>(packed);
  if (!header_matches(hdr, n, m, N)) {
    if (threadIdx.x == 0 && dev_status) *dev_status = STB_ERR_CORRUPT;
    return;
  }
  const int nblk = m / kBlock;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int rt = blockIdx.x;
  const BlockInfo* binfo = reinterpret_cast<const BlockInfo*>(packed + sizeof(Header));
  const uint8_t* rtbase = packed + hdr->tiles_offset + (size_t)rt * hdr->rt_stride;
  const uint8_t* resid_rt = packed + hdr->tiles_offset + hdr->rt_stride * (size_t)hdr->ntile +
                            (size_t)rt * resid_rt_bytes(nblk, hdr->nrw);

  float acc[4][BT];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int bt = 0; bt < BT; ++bt) acc[j][bt] = 0.0f;

  for (int b = warp; b < nblk; b += 8) {
    const uint8_t* tile = rtbase + (size_t)b * hdr->tile_bytes;
    LaneTile<N> lt;
    load_lane_tile<N>(tile, lane, lt);
    const uint64_t sal[2] = {binfo[b].salient[0], binfo[b].salient[1]};
    const uint8_t* record = resid_rt + resid_block_off(b, binfo[b].rw_off);
    const int nslot = 4 * (int)binfo[b].nrw;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float alpha[5];
#pragma unroll
      for (int q = 0; q < 4; ++q) alpha[q] = __half2float(__ushort_as_half((unsigned short)scale_bits<N>(lt, j, q)));
      alpha[4] = __half2float(__ushort_as_half((unsigned short)sal2_bits(record, g, j)));
#pragma unroll 1
      for (int s = 0; s < 4; ++s) {
        const int grp = 4 * s + t;
        uint32_t code[8], neg[8];
        plain_slot<N>(lt, 4 * j + s, code, neg);
        const uint32_t salb = (uint32_t)((sal[grp >> 3] >> (8 * (grp & 7))) & 0xFFull);
        int qbase = grp >= 8 ? __popcll(sal[0]) : 0;
        qbase += __popcll(sal[grp >> 3] & ((1ull << (8 * (grp & 7))) - 1ull));
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          float w = 0.0f;
          if (code[c] < 4u) {
            const float s1 = neg[c] ? -1.0f : 1.0f;
            if (code[c] == 3u) {
              const int q = qbase + __popc(salb & ((1u << c) - 1u));
              const uint32_t word = q < nslot ? resid_word(record, (uint32_t)(q >> 2), g) : 0x55555555u;
              const float s2 = resid_code(word, j, q & 3) == 0u ? 1.0f : -1.0f;
              w = __fadd_rn(s1 * alpha[3], s2 * alpha[4]);
            } else {
              w = s1 * (code[c] == 0u ? alpha[0] : (code[c] == 1u ? alpha[1] : alpha[2]));
            }
          }
          v[c] = w;
        }
#pragma unroll
        for (int bt = 0; bt < BT; ++bt) {
          if (bt < batch) {
            const uint4 xv = __ldg(reinterpret_cast<const uint4*>(x + (size_t)bt * ldx + (size_t)b * kBlock + grp * 8));
            const __half2* xh = reinterpret_cast<const __half2*>(&xv);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float2 xf = __half22float2(xh[c]);
              acc[j][bt] = fmaf(v[2 * c], xf.x, acc[j][bt]);
              acc[j][bt] = fmaf(v[2 * c + 1], xf.y, acc[j][bt]);
            }
          }
        }
      }
    }
  }

  // the four lanes t of a row
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int bt = 0; bt < BT; ++bt) {
      float a = acc[j][bt];
      a += __shfl_xor_sync(0xFFFFFFFFu, a, 1);
      a += __shfl_xor_sync(0xFFFFFFFFu, a, 2);
      acc[j][bt] = a;
    }
  __shared__ float red[8][BT][32];
  if (t == 0) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int bt = 0; bt < BT; ++bt) red[warp][bt][g + 8 * j] = acc[j][bt];
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < BT * 32; idx += blockDim.x) {
    const int bt = idx >> 5, l = idx & 31;
    const int row = rt * kTileRows + l;
    if (bt < batch && row < n) {
      float s = 0.0f;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += red[w][bt][l];
      if (y_f16) static_cast<__half*>(y)[(size_t)bt * ldy + row] = __float2half_rn(s);
      else static_cast<float*>(y)[(size_t)bt * ldy + row] = s;
    }
  }
}

template <int N>
static cudaError_t launch_general(const uint8_t* packed, int n, int m, const __half* x, int batch,
                                  size_t ldx, void* y, int y_f16, size_t ldy, int* dev_status, cudaStream_t s) {
  const unsigned grid = (unsigned)((n + kTileRows - 1) / kTileRows);
  if (batch <= 2) gemv_general_kernel<N, 2><<<grid, 256, 0, s>>>(packed, n, m, x, batch, ldx, y, y_f16, ldy, dev_status);
  else if (batch <= 8) gemv_general_kernel<N, 8><<<grid, 256, 0, s>>>(packed, n, m, x, batch, ldx, y, y_f16, ldy, dev_status);
  else gemv_general_kernel<N, 16><<<grid, 256, 0, s>>>(packed, n, m, x, batch, ldx, y, y_f16, ldy, dev_status);
  return cudaGetLastError();
}

}  // namespace stb

static int gemv_impl(const void* packed, int n, int m, int N, const void* x, int batch, size_t ldx,
                     void* y, stb_dtype ydt, size_t ldy, int* dev_status, void* stream, bool chained,
                     bool wait_selftest = false, stb::GemvForm form = stb::GemvForm::cheapest) {
  if (!packed || !x || !y) return STB_ERR_ARG;
  if (n < 1 || m < stb::kBlock || m % stb::kBlock != 0) return STB_ERR_SHAPE;
  if (N < 1 || N > 8) return STB_ERR_NM;
  if (batch < 1 || batch > 64) return STB_ERR_SIZE;
  if (ydt != STB_F32 && ydt != STB_F16) return STB_ERR_UNSUPPORTED;
  const int y_f16 = ydt == STB_F16;
  if (ldx < (size_t)m || ldy < (size_t)n || (ldx % 8) != 0 || (reinterpret_cast<uintptr_t>(x) & 15u)) return STB_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint8_t* p = static_cast<const uint8_t*>(packed);
  const __half* xh = static_cast<const __half*>(x);
  cudaError_t e = cudaSuccess;
  if (N >= 4 && N <= 6) {
    stb::GemvLayers layers = {};
    layers.packed[0] = p; layers.y[0] = y; layers.ldy[0] = ldy; layers.n[0] = n; layers.y_f16[0] = y_f16;
    layers.tile_start[0] = 0; layers.tile_start[1] = (n + stb::kTileRows - 1) / stb::kTileRows; layers.count = 1;
    e = stb::launch_mma_b(batch, N, layers, m, xh, ldx, dev_status, s, chained, wait_selftest, form);
    return e == cudaSuccess ? STB_OK : STB_ERR_CUDA;
  }
  if (wait_selftest) return STB_ERR_UNSUPPORTED;
  // the general kernel takes up to 16 batch rows per launch
  for (int t0 = 0; t0 < batch && e == cudaSuccess; t0 += 16) {
    const int bt = batch - t0 < 16 ? batch - t0 : 16;
    const __half* xc = xh + (size_t)t0 * ldx;
    void* yc = y_f16 ? static_cast<void*>(static_cast<__half*>(y) + (size_t)t0 * ldy)
                     : static_cast<void*>(static_cast<float*>(y) + (size_t)t0 * ldy);
    switch (N) {
      case 1: e = stb::launch_general<1>(p, n, m, xc, bt, ldx, yc, y_f16, ldy, dev_status, s); break;
      case 2: e = stb::launch_general<2>(p, n, m, xc, bt, ldx, yc, y_f16, ldy, dev_status, s); break;
      case 3: e = stb::launch_general<3>(p, n, m, xc, bt, ldx, yc, y_f16, ldy, dev_status, s); break;
      case 7: e = stb::launch_general<7>(p, n, m, xc, bt, ldx, yc, y_f16, ldy, dev_status, s); break;
      case 8: e = stb::launch_general<8>(p, n, m, xc, bt, ldx, yc, y_f16, ldy, dev_status, s); break;
    }
  }
  return e == cudaSuccess ? STB_OK : STB_ERR_CUDA;
}

extern "C" int stb_gemv(const void* packed, int n, int m, int N, const void* x, int batch, size_t ldx,
                        void* y, stb_dtype ydt, size_t ldy, int* dev_status, void* stream) {
  return gemv_impl(packed, n, m, N, x, batch, ldx, y, ydt, ldy, dev_status, stream, false);
}

extern "C" int stb_gemv_wait_selftest(const void* packed, int n, int m, int N, const void* x, int batch, size_t ldx,
                                      void* y, stb_dtype ydt, size_t ldy, int* dev_status, void* stream) {
  if (!dev_status) return STB_ERR_ARG;
  return gemv_impl(packed, n, m, N, x, batch, ldx, y, ydt, ldy, dev_status, stream, false, true);
}

// Steps i..j-1 can share one grid when they read the same activations with the same batch, m and N
// (4, 5 or 6) and none of them writes what another reads: same-input projections of a decoder
// layer (q / k / v, gate / up).
static bool can_fuse(const stb_step& a, const stb_step& b) {
  return a.in == b.in && a.ldin == b.ldin && a.batch == b.batch && a.m == b.m && a.N == b.N && a.N >= 4 && a.N <= 6 &&
         b.out != a.in && b.packed && b.out && b.n >= 1 && (b.odt == STB_F32 || b.odt == STB_F16) && b.ldout >= (size_t)b.n;
}

extern "C" int stb_layer_stack(const stb_step* steps, int count, int* dev_status, void* stream) {
  if (!steps || count < 0) return STB_ERR_ARG;
  for (int k = 0; k < count; ++k)
    if (steps[k].input != STB_IN_PLAIN) return STB_ERR_UNSUPPORTED;      // only the resident kernel forms inputs
  const auto launch_end = [&](int i) {
    int j = i + 1;
    while (j < count && j - i < stb::kMaxFused && can_fuse(steps[i], steps[j])) ++j;
    return j;
  };
  // what chain_form goes by: the tensor-core launches of up to 16 rows
  long long launches = 0, tiles = 0;
  bool fits = true, wide = false;
  int dev = 0, most[9];
  const bool known = count > 1 && cudaGetDevice(&dev) == cudaSuccess && stb::gemv_clusters(dev, most) == cudaSuccess;
  for (int i = 0, j; known && i < count; i = j) {
    j = launch_end(i);
    const stb_step& st = steps[i];
    if (st.N < 4 || st.N > 6 || st.batch < 1 || st.batch > 16 || st.m < stb::kBlock) continue;
    int R = 0;
    for (int k = i; k < j; ++k) R += (steps[k].n + stb::kTileRows - 1) / stb::kTileRows;
    const long long t = (long long)R * (st.m / stb::kBlock);
    ++launches; tiles += t;
    if (t < stb::kStreamTiles) continue;
    stb::GemvPlan plan;
    double cost;
    if (!stb::gemv_plan(st.N, R, st.m / stb::kBlock, st.batch, j - i, most, plan, cost)) fits = false;
    else if (plan.chunk == 2) wide = true;
  }
  const auto form = [&](const stb_step& st) {
    return !known || launches <= 1 ? stb::GemvForm::cheapest : stb::chain_form(st.N, st.batch, tiles / launches, fits, wide);
  };
  int i = 0;
  while (i < count) {
    const stb_step& st = steps[i];
    const int j = launch_end(i);
    // steps after the first start their weight stream while the previous step drains
    const bool chained = i > 0;
    if (j - i == 1) {
      int rc = gemv_impl(st.packed, st.n, st.m, st.N, st.in, st.batch, st.ldin, st.out, st.odt, st.ldout,
                         dev_status, stream, chained, false, form(st));
      if (rc != STB_OK) return rc;
    } else {
      // validate the first step like stb_gemv does; can_fuse has checked what differs in the others
      if (!st.packed || !st.in || !st.out) return STB_ERR_ARG;
      if (st.n < 1 || st.m < stb::kBlock || st.m % stb::kBlock != 0) return STB_ERR_SHAPE;
      if (st.batch < 1 || st.batch > 64) return STB_ERR_SIZE;
      if (st.odt != STB_F32 && st.odt != STB_F16) return STB_ERR_UNSUPPORTED;
      if (st.ldin < (size_t)st.m || st.ldout < (size_t)st.n || (st.ldin % 8) != 0 || (reinterpret_cast<uintptr_t>(st.in) & 15u))
        return STB_ERR_ARG;
      stb::GemvLayers layers = {};
      layers.count = j - i;
      layers.tile_start[0] = 0;
      for (int k = i; k < j; ++k) {
        const stb_step& sk = steps[k];
        layers.packed[k - i] = static_cast<const uint8_t*>(sk.packed);
        layers.y[k - i] = sk.out; layers.ldy[k - i] = sk.ldout; layers.n[k - i] = sk.n; layers.y_f16[k - i] = sk.odt == STB_F16;
        layers.tile_start[k - i + 1] = layers.tile_start[k - i] + (sk.n + stb::kTileRows - 1) / stb::kTileRows;
      }
      cudaStream_t s = static_cast<cudaStream_t>(stream);
      const __half* xh = static_cast<const __half*>(st.in);
      cudaError_t e = stb::launch_mma_b(st.batch, st.N, layers, st.m, xh, st.ldin, dev_status, s, chained, false, form(st));
      if (e != cudaSuccess) return STB_ERR_CUDA;
    }
    i = j;
  }
  return STB_OK;
}

extern "C" int stb_layer_stack_host(const stb_step* steps, int count, const void* in_host, size_t in_bytes,
                                    void* out_host, size_t out_bytes, int* dev_status, void* stream) {
  if (!steps || count < 1 || !in_host || !out_host || !steps[0].in || !steps[count - 1].out) return STB_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemcpyAsync(const_cast<void*>(steps[0].in), in_host, in_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return STB_ERR_CUDA;
  const int rc = stb_layer_stack(steps, count, dev_status, stream);
  if (rc != STB_OK) return rc;
  if (cudaMemcpyAsync(out_host, steps[count - 1].out, out_bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return STB_ERR_CUDA;
  return STB_OK;
}
